"""The nonlinear rows on either side of the numbers of rows where the update changes from the staged kernel to the
column walk, against the FP64 oracle, and a sub-domain's rows, which go by the whole grid's number, against the whole
grid's bit for bit."""
import numpy as np
import pytest

from fdtd_inputs import critical_density, spec_2d_cylinder
from tests.adapters import FIELDS, compare, oracle_sim

pytestmark = pytest.mark.gpu


def _spec(rows, nv, nvp, prec, n=120, ny=100):
    """A grid with exactly `rows` plasma cells, in a disc off the centre."""
    spec = spec_2d_cylinder(n=n, ny=ny, cpml=6, R=2, src=(20, 50), nv=nv, nv_perp=nvp, precision=prec, f_dtype=prec,
                            seed=2)
    j, i = np.meshgrid(np.arange(ny), np.arange(n), indexing="ij")
    r2 = ((i - 0.55 * n) ** 2 + (j - 0.5 * ny) ** 2).ravel()
    d = np.zeros(n * ny)
    at = np.argsort(r2, kind="stable")[:rows]
    d[at] = critical_density() * np.linspace(0.5, 0.1, rows)
    spec["plasma"].update(density=d, nonlinear=1)
    spec["source"].update(amp=2e5, t0=0.5 * spec["source"]["tau"])
    return spec


def _edges():
    # two lanes a row: 32 rows a SM; FP64, four lanes: half a row a SM; eight: that, and sixteen rows
    sms = 152
    out = [(32 * sms + k, nv, nvp, prec) for k in (-1, 0) for nv, nvp, prec in ((9, 4, "f64"), (10, 8, "f32"))]
    out += [(r, 9, nvp, "f64") for nvp in (8, 6) for r in (3, sms // 2 - 1, sms // 2)]
    return out + [(r, 8, nvp, "f64") for nvp in (16, 5) for r in (16, 17, sms // 2 - 1, sms // 2)]


@pytest.mark.parametrize("rows,nv,nvp,prec", _edges() + [(40, 64, 16, "f64"), (400, 64, 16, "f64")])
def test_rows_match_oracle(oracle_lib, rows, nv, nvp, prec):
    from paper_2211_05647_gb300 import Solver
    spec = _spec(rows, nv, nvp, prec)
    s, sim = Solver.from_spec(spec), oracle_sim(oracle_lib, spec)
    assert s.plasma_shape()[0] == rows
    s.step(60)
    sim.step(60)
    errs = compare(s, sim, 2)
    assert max(errs.values()) <= (1e-12 if prec == "f64" else 1e-4), errs   # the bounds of every other parity test


@pytest.mark.parametrize("rows,nvp,prec", [(5000, 4, "f64"), (5000, 8, "f32"), (100, 8, "f64"), (90, 16, "f64")])
def test_subdomain_rows_go_by_the_whole_grid(rows, nvp, prec, tmp_path, monkeypatch):
    from paper_2211_05647_gb300 import Solver
    from paper_2211_05647_gb300.decomposed import DecomposedSolver
    monkeypatch.setenv("FDTD_PLASMA_TUNE_CACHE", str(tmp_path / "none.txt"))
    spec = _spec(rows, 16, nvp, prec)
    whole, dec = Solver.from_spec(spec), DecomposedSolver(spec, bounds=[(0, 45), (45, 10), (55, 45)])
    assert all(s.plasma_shape()[0] < rows for s in dec.subs)
    whole.step(60)
    dec.step(60)
    assert np.abs(whole.read("j", device=False)).max() > 0
    for q in FIELDS[2] + ["j", "df"]:
        a, b = dec.read(q), whole.read(q, device=False)
        assert np.array_equal(a, b.reshape(a.shape)), q
