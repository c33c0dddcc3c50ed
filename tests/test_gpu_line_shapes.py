"""Which kernel steps a 1-D grid, and in which order its rows are summed: a row shape set by option is the one
``step`` and ``time_kernels`` both use, bit for bit; tuned and cached shapes, which belong to the row kernel, change
nothing where the cooperative kernel steps the grid; ``launch_shapes`` says which of the two it is."""
import numpy as np
import pytest

from fdtd_inputs import spec_1d_slab

pytestmark = pytest.mark.gpu

COOP = 512   # threads of the cooperative kernel, as launch_shapes reports them


def _spec(dtype, nv=64, nz=900):
    sp = spec_1d_slab(nz=nz, slab=(nz // 3, nz // 2), src_k=20, nv=nv, precision="f64" if dtype == "f64" else "f32",
                      f_dtype=dtype, seed=6)
    sp["source"].update(t0=0.5 * sp["source"]["tau"])
    return sp


def _make(sp):
    from paper_2211_05647_gb300 import Solver
    s = Solver.from_spec(sp)
    rng = np.random.default_rng(8)
    nz = sp["grid"]["nz"]
    s.write("ex", rng.standard_normal(nz + 1))
    s.write("hy", rng.standard_normal(nz) / 377.0)
    return s


def _equal(a, b):
    for n in (1, 45):
        a.step(n)
        b.time_kernels(n)
    return all(np.array_equal(a.read(q, device=False), b.read(q, device=False)) for q in ("ex", "hy", "j", "df"))


@pytest.mark.parametrize("dtype,shape,coop", [("f32", (4, 4), True), ("f32", (2, 8), False), ("f32", (1, 16), False),
                                              ("bf16", (4, 2), True), ("bf16", (1, 8), False),
                                              ("f64", (4, 8), False), ("f64", (1, 32), False)])
def test_forced_shape(dtype, shape, coop):
    sp = _spec(dtype)
    a, b = _make(sp), _make(sp)
    for s in (a, b):
        s.set_option("kinetic_shape", shape[0] * 10**6 + shape[1] * 1000)
        got = s.launch_shapes()
        assert (got["kin_vpl"], got["kin_l"], got["block_x"]) == (*shape, COOP if coop else 0)
    assert _equal(a, b)
    a.set_option("kinetic_shape", 0)
    assert a.launch_shapes()["block_x"] == COOP


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_tuned_and_cached_shapes(dtype, tmp_path, monkeypatch):
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("FDTD_PLASMA_TUNE_CACHE", str(cache))
    sp = _spec(dtype)
    t = _make(sp)
    t.set_ports([[300]], np.array([1e10]))      # the graphs step it: the row kernel is tuned and cached
    assert t.launch_shapes()["block_x"] == 0
    assert t.autotune()["kin_vpl"] > 0
    key, rest = cache.read_text().split(maxsplit=1)
    odd = (1, 16) if dtype == "f32" else (1, 8)
    cache.write_text(f"{key} {odd[0]} {odd[1]} 0 0\n")
    a, b = _make(sp), _make(sp)                 # the cooperative kernel steps these
    for s in (a, b):
        assert s.launch_shapes() == {**{k: 0 for k in s.launch_shapes()}, "block_x": COOP, "block_y": 1, "block_z": 1}
    assert _equal(a, b)
    a.set_ports([[300]], np.array([1e10]))      # and now the graphs, with the cached shape
    assert (a.launch_shapes()["kin_vpl"], a.launch_shapes()["kin_l"]) == odd
    c, d = _make(sp), _make(sp)
    c.set_option("kinetic_shape", 2 * 10**6 + (8 if dtype == "f32" else 4) * 1000)
    before = c.read("ex", device=False).copy()
    r = c.autotune()                            # nothing to tune; the option's shape goes back to the default
    assert r["kin_vpl"] == 0 and c.launch_shapes()["block_x"] == COOP
    assert np.array_equal(c.read("ex", device=False), before)
    assert _equal(c, d)


@pytest.mark.parametrize("nz,slab,nv,dtype,coop", [(40000, (1, 40000), 512, "f32", False),
                                                   (400, (100, 200), 1024, "f64", False), (70001, (3, 70), 128, "f64", True),
                                                   (608, (300, 301), 64, "bf16", True), (2000000, (9, 12), 8, "f32", True),
                                                   (5000000, (9, 12), 8, "f32", False)])
def test_what_fits(nz, slab, nv, dtype, coop):
    from paper_2211_05647_gb300 import Solver
    sp = spec_1d_slab(nz=nz, slab=slab, src_k=20, nv=nv, precision="f64" if dtype == "f64" else "f32", f_dtype=dtype)
    s = Solver.from_spec(sp)
    assert s.launch_shapes()["block_x"] == (COOP if coop else 0)
    s.step(3)
    assert s.launch_shapes()["block_x"] == (COOP if coop else 0)
