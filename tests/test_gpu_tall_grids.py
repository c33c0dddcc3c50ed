"""Long, narrow FP32 grids, whose block counts along y or z come near the 65535 of a launch: every stencil path the
size rules or an option can choose gives the grid-of-cells kernels' fields bit for bit."""
import numpy as np
import pytest

from tests.adapters import FIELDS

pytestmark = pytest.mark.gpu


def _start(dims, cpml):
    from paper_2211_05647_gb300 import Solver
    nx, ny, nz = (*dims, 1)[:3]
    nd = len(dims)
    s = Solver(dict(ndim=nd, nx=nx, ny=ny, nz=nz, dx=1e-3, courant=0.5, cpml_cells=cpml, mur=0, precision="f32"))
    s.set_source(kind="gauss", amp=1.0, tau=1e-11, t0=0.0, i=nx // 2, j=ny // 2, k=nz // 2)
    rng = np.random.default_rng(3)
    for q in FIELDS[nd]:
        s.write(q, rng.standard_normal(nx * ny * nz, dtype=np.float32) / (1.0 if q[0] == "e" else 377.0))
    return s


def _equal(a, b, nd):
    for k in (1, 4, 7):
        a.step(k)
        b.step(k)
    assert all(np.array_equal(a.read(q, device=False), b.read(q, device=False)) for q in FIELDS[nd])


@pytest.mark.parametrize("dims,cpml,rows", [((24, 262144), 0, None), ((24, 262140), 0, None),
                                            ((24, 262144), 4, 4), ((8, 262141), 2, 4), ((8, 65537), 2, 1)])
def test_march_on_tall_grids(dims, cpml, rows):
    """6.3 M cells take the fused march by the size rule; shorter ones by option with the given rows a segment."""
    a, b = _start(dims, cpml), _start(dims, cpml)
    b.set_option("stencil_tz", 0)
    if rows:
        a.set_option("fused_stencils", 1)
        a.set_option("fused_rows", rows)
    assert a.launch_shapes()["fused_rows"] > 0 and b.launch_shapes()["fused_rows"] == 0
    _equal(a, b, 2)


@pytest.mark.parametrize("dims", [(16, 12, 65537), (16, 12, 66000)])
def test_cell_kernels_on_deep_grids(dims):
    """12.6 M cells take the TMA columns by the size rule; turned off, the grid-of-cells kernels cover two planes a
    block, as they do on grids the rule leaves alone (one plane a block would need more than 65535 along z)."""
    a, b = _start(dims, 0), _start(dims, 0)
    b.set_option("stencil_tz", 0)
    assert a.launch_shapes()["stencil_tz"] > 0 and b.launch_shapes()["stencil_tz"] == 0
    assert b.launch_shapes()["block_z"] == 2
    _equal(a, b, 3)


@pytest.mark.parametrize("dims,cpml,fast", [((64, 125000), 8, False), ((64, 125000), 0, True), ((200, 60000), 8, True),
                                            ((196, 60000), 16, False), ((200000, 48), 8, False), ((640, 3, 6668), 0, False),
                                            ((640, 4, 5000), 0, False), ((640, 5, 4000), 0, True),
                                            ((640, 9, 2224), 0, False), ((512, 26, 1000), 8, False),
                                            ((512, 1000, 26), 8, True), ((64, 64, 3000), 8, False),
                                            ((64, 320, 640), 8, True)])
def test_rules_leave_layers_and_thin_grids_alone(dims, cpml, fast):
    a, b = _start(dims, cpml), _start(dims, cpml)
    b.set_option("stencil_tz", 0)
    assert (a.launch_shapes()["fused_rows" if len(dims) == 2 else "stencil_tz"] > 0) == fast
    for s in (a, b):
        s.step(4)
    for q in FIELDS[len(dims)]:
        assert bool((a.read(q) == b.read(q)).all()), q


def _allocated(s):
    return sum(t.numel() for t in s._alloc.live.values())


@pytest.mark.parametrize("n,mb,runs", [(2500, 0, False), (2720, 0, False), (2760, 0, True), (2760, 60, True),
                                       (2760, 70, False), (2996, 70, False), (3004, 70, True)])
def test_march_runs_where_the_fields_have_left_l2(n, mb, runs):
    """Between 6 and 9 M cells the march that the size rule names runs from 7.6 M cells and beside little delta f
    only: the first steps allocate its second field set, or not."""
    rows = mb << 10   # of 256 FP32 nodes
    a, b = _start((n, n), 8), _start((n, n), 8)
    if rows:
        d = np.zeros(n * n)
        at = np.arange(n * 100, n * n)
        d[at[at % n > 0][:rows]] = 1e16
        for s in (a, b):
            s.set_plasma(d, vgrid="cart2d", nv=16, nv_perp=16)
    b.set_option("stencil_tz", 0)
    assert a.launch_shapes()["fused_rows"] > 0
    before = _allocated(a)
    _equal(a, b, 2)
    assert (_allocated(a) - before >= 12 * n * n) == runs
