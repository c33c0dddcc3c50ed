"""The nonlinear kinetic update's column walk against the FP64 oracle, at the
velocity grids where its pairing can go wrong: an even and an odd number of
v_par nodes (the odd one has a node that is its own mirror), two and three of
them (no interior pair), fewer pairs than one chunk of loads and one more than
a chunk, columns that fill a vector, leave lanes idle or come one at a time,
more column vectors than a warp has lanes, and the narrow columns that keep
the staged kernel.  The field swings through both signs and is strong enough
for the advection to matter."""
import pytest

from fdtd_inputs import spec_2d_cylinder
from tests.adapters import compare, oracle_sim

pytestmark = pytest.mark.gpu

GRIDS = [(32, 32), (31, 16), (2, 8), (3, 20), (8, 12), (9, 9), (10, 33), (7, 132), (18, 4), (5, 1)]


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("nv,nv_perp", GRIDS)
def test_walk_matches_oracle(oracle_lib, nv, nv_perp, prec):
    from paper_2211_05647_gb300 import Solver
    spec = spec_2d_cylinder(n=40, ny=36, cpml=4, R=7, center=(22, 18), src=(12, 18), wp_w0=0.6, nv=nv,
                            nv_perp=nv_perp, precision=prec, f_dtype=prec, seed=3)
    spec["source"].update(amp=2e5, t0=0.5 * spec["source"]["tau"])
    spec["plasma"]["nonlinear"] = 1
    s, sim = Solver.from_spec(spec), oracle_sim(oracle_lib, spec)
    s.step(90)
    sim.step(90)
    errs = compare(s, sim, 2)
    # the bounds of every other parity test: FP64 1e-12, FP32 1e-4 relative L2
    assert max(errs.values()) <= (1e-12 if prec == "f64" else 1e-4), errs
