"""The 1-D cooperative stepping kernel (what ``step`` runs on 1-D grids whose
state fits in the SMs' shared memory) against the separate H, kinetic and E
launches of ``time_kernels``: every field, J and delta f equal bit for bit in
FP32 and BF16, and to a few FP64 roundings in FP64, whose rows take a shape of
their own (J's compensated sum is then formed in another order), at the lines where its ranges can go wrong -- shorter than a range per CTA, one
node more or less than a multiple, plasma on the first and last updated node,
everywhere, in one cell or nowhere, rows of one vector up to the longest a
lane group takes, PEC and Mur ends, the source in the first and last range --
and over call lengths around the source table's 64 steps.  A line too long or
with rows too long for the shared memory keeps the step graphs."""
import numpy as np
import pytest

from fdtd_inputs import critical_density, spec_1d_slab

pytestmark = pytest.mark.gpu

#        nz, slab, source node, nv, Mur ends
LINES = [(3, (1, 3), 1, 8, 1), (4, (2, 3), 3, 4, 0), (9, (0, 0), 4, 8, 1), (607, (1, 607), 606, 31, 1),
         (608, (300, 301), 1, 64, 0), (1201, (200, 900), 100, 64, 1), (5000, (1000, 4500), 1000, 16, 1),
         (70001, (3, 70), 69999, 128, 1)]


def _spec(nz, slab, src, nv, mur, precision, f_dtype):
    sp = spec_1d_slab(nz=nz, slab=slab, src_k=src, nv=nv, precision=precision, f_dtype=f_dtype, seed=4)
    sp["grid"]["mur"] = mur
    sp["source"].update(t0=0.5 * sp["source"]["tau"])
    if slab[1] > slab[0]:   # uneven densities: a row mixed up with its neighbour shows
        d = sp["plasma"]["density"]
        d[slab[0]:slab[1]] = critical_density() * np.linspace(0.1, 0.6, slab[1] - slab[0])
    return sp


def _start(sp):
    from paper_2211_05647_gb300 import Solver
    s = Solver.from_spec(sp)
    rng = np.random.default_rng(2)
    nz = sp["grid"]["nz"]
    s.write("ex", rng.standard_normal(nz + 1))
    s.write("hy", rng.standard_normal(nz) / 377.0)
    return s


def _same(a, b, dtype):
    """FP64: each of up to 140 steps rounds J, hence E, by at most an ulp or two differently, and delta f rows
    decay slower than that: 1e-13 of each quantity's norm."""
    if dtype != "f64":
        return all(np.array_equal(a[q], b[q]) for q in a)
    return all(np.linalg.norm(a[q] - b[q]) <= 1e-13 * np.linalg.norm(b[q]) for q in a)


def _state(s):
    return {n: s.read(n, device=False).copy() for n in ("ex", "hy", "j", "df")}


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("line", LINES)
def test_equals_separate_launches(line, dtype):
    sp = _spec(*line, "f64" if dtype == "f64" else "f32", dtype)
    a, b = _start(sp), _start(sp)
    for n in (1, 2, 63, 66, 7):
        a.step(n)
        b.time_kernels(n)
        ga, gb = _state(a), _state(b)
        assert _same(ga, gb, dtype), n
        assert a.info()[1] == b.info()[1]
    a.reset()   # the step counter starts again; the messages' tags do not
    b.reset()
    a.step(3)
    a.time_kernels(2)   # the device's own step counter follows
    a.step(64)
    b.time_kernels(69)
    assert _same(_state(a), _state(b), dtype)


@pytest.mark.parametrize("sp", [_spec(40000, (1, 40000), 30, 512, 1, "f32", "f32"),
                                _spec(400, (100, 200), 30, 1024, 1, "f64", "f64")], ids=["state", "rows"])
def test_what_does_not_fit_keeps_the_graphs(sp):
    a, b = _start(sp), _start(sp)
    a.step(5)
    b.time_kernels(5)
    ga, gb = _state(a), _state(b)
    assert all(np.array_equal(ga[q], gb[q]) for q in ga)
