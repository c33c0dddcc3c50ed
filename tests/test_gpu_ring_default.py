"""Long FP32 rows whose delta f is just past the size from which the default runs the bulk-copy ring kernel: the
fields, J and delta f of the register kernel of the same row shape, bit for bit."""
import numpy as np
import pytest

from fdtd_inputs import critical_density, spec_2d_cylinder
from tests.adapters import FIELDS

pytestmark = pytest.mark.gpu


#        nodes, delta f (MB), (vectors a lane, lanes), grid: fields that fit L2, or not
@pytest.mark.parametrize("nv,nvp,mb,shape,n", [(16, 16, 256, (8, 8), 640), (32, 16, 256, (8, 16), 640),
                                               (32, 32, 512, (16, 16), 3100)])
def test_default_past_the_ring_threshold(nv, nvp, mb, shape, n, tmp_path, monkeypatch):
    from paper_2211_05647_gb300 import Solver
    monkeypatch.setenv("FDTD_PLASMA_TUNE_CACHE", str(tmp_path / "none.txt"))
    rows = (mb << 20) // (nv * nvp * 4) + 3
    spec = spec_2d_cylinder(n=n, R=2, src=(40, 300), nv=nv, nv_perp=nvp, f_dtype="f32", seed=5)
    d = np.zeros(n * n)
    at = np.arange(n * 60, n * n)
    d[at[at % n > 0][:rows]] = critical_density() * np.linspace(0.05, 0.6, rows)   # (column 0 carries no plasma)
    spec["plasma"]["density"] = d
    spec["source"].update(t0=0.5 * spec["source"]["tau"])
    a, b = Solver.from_spec(spec), Solver.from_spec(spec)
    assert a.plasma_shape()[0] == rows
    b.set_option("kinetic_shape", shape[0] * 10**6 + shape[1] * 1000)
    rng = np.random.default_rng(1)
    v = rng.standard_normal(n * n, dtype=np.float32)
    for s in (a, b):
        s.write("ez", v)
        s.step(5)
    assert np.abs(a.read("j", device=False)).max() > 0
    for q in FIELDS[2] + ["j", "df"]:
        assert bool((a.read(q) == b.read(q)).all()), q
