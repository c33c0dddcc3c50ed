"""The default launch shape of the kinetic rows against the shape whose sums it
forms (forced by option): delta f, J and the fields equal bit for bit, BF16 rows
of 16 to 128 vectors (eight a lane, summed as four), FP32 rows around the ring's
and the block cap's limits, and rows with padding; and the default 2-D and 3-D
stencils of sizes on either side of their rules against one-cell kernels."""
import numpy as np
import pytest

from fdtd_inputs import spec_2d_cylinder, spec_3d_slab
from tests.adapters import FIELDS

pytestmark = pytest.mark.gpu


def _state(s, nd):
    return {n: s.read(n, device=False).copy() for n in FIELDS[nd] + ["j", "df"]}


#       nv, nv_perp, storage -> (vectors a lane, lanes) J is summed in
ROWS = [(16, 8, "bf16", (4, 4)), (16, 16, "bf16", (4, 8)), (31, 16, "bf16", (4, 16)), (32, 31, "bf16", (4, 32)),
        (8, 4, "bf16", (4, 1)), (8, 8, "bf16", (4, 2)), (8, 4, "f32", (2, 4)), (8, 8, "f32", (4, 4)),
        (16, 8, "f32", (4, 8)), (16, 16, "f32", (8, 8)), (31, 16, "f32", (8, 16)), (32, 32, "f32", (16, 16))]


@pytest.mark.parametrize("nv,nvp,dtype,shape", ROWS)
def test_default_rows_sum_as_their_shape(nv, nvp, dtype, shape):
    from paper_2211_05647_gb300 import Solver
    spec = spec_2d_cylinder(n=120, ny=101, cpml=6, R=29, center=(60, 50), src=(30, 50), nv=nv, nv_perp=nvp,
                            f_dtype=dtype, seed=5)
    spec["source"].update(t0=0.5 * spec["source"]["tau"])
    a, b = Solver.from_spec(spec), Solver.from_spec(spec)
    b.set_option("kinetic_shape", shape[0] * 10**6 + shape[1] * 1000)
    for n in (1, 40):
        a.step(n)
        b.step(n)
    ga, gb = _state(a, 2), _state(b, 2)
    assert np.abs(ga["j"]).max() > 0
    assert all(np.array_equal(ga[q], gb[q]) for q in ga)


@pytest.mark.parametrize("dims", [(1500, 1048), (1500, 1049), (2500, 2400), (2500, 2401), (256, 216, 216),
                                  (256, 217, 217)])
def test_default_stencils_equal_one_cell_kernels(dims):
    """2-D: one / four cells a thread at 1.5 M cells, the fused march at 6 M; 3-D: the TMA columns at 12 M."""
    from paper_2211_05647_gb300 import Solver
    nd = len(dims)
    if nd == 2:
        spec = spec_2d_cylinder(n=dims[0], ny=dims[1], R=20, nv=4, nv_perp=4)
    else:
        spec = spec_3d_slab(n=dims[0], ny=dims[1], nz=dims[2], slab=(100, 104), src_k=20, nv=8, f_dtype="f32")
    spec["source"].update(t0=0.3 * spec["source"]["tau"])
    a, b = Solver.from_spec(spec), Solver.from_spec(spec)
    rng = np.random.default_rng(1)
    n = int(np.prod(dims))
    for q in FIELDS[nd]:
        v = rng.standard_normal(n, dtype=np.float32) / (1.0 if q[0] == "e" else 377.0)
        a.write(q, v)
        b.write(q, v)
    b.set_option("stencil_tz", 0)          # grid-of-cells kernels: no march, no TMA
    assert b.launch_shapes()["fused_rows"] == 0 and b.launch_shapes()["stencil_tz"] == 0
    big = n >= (6000000 if nd == 2 else 12000000)
    assert (a.launch_shapes()["fused_rows" if nd == 2 else "stencil_tz"] > 0) == big
    for k in (1, 22):
        a.step(k)
        b.step(k)
    ga, gb = _state(a, nd), _state(b, nd)
    assert all(np.array_equal(ga[q], gb[q]) for q in ga)
