"""The source values of a sequence are tabulated by its first H update: a call of n steps (graphs of 32, 16, ... 1
steps) gives the bits of n calls of one step, for every H kernel that writes the table and every E pass that reads it."""
import pytest

from fdtd_inputs import spec_1d_slab, spec_2d_cylinder, spec_3d_slab

pytestmark = pytest.mark.gpu

CASES = {
    "1d_f32": (lambda: spec_1d_slab(nz=300, slab=(100, 160), nv=8, precision="f32", f_dtype="f32"), {}),
    "2d_odd_f32": (lambda: spec_2d_cylinder(n=61, ny=44, cpml=4, R=8, src=(12, 20), nv=4, nv_perp=4), {}),
    "2d_f64": (lambda: spec_2d_cylinder(n=61, ny=44, cpml=4, R=8, src=(12, 20), nv=4, nv_perp=4, precision="f64",
                                        f_dtype="f64"), {}),
    "2d_tma": (lambda: spec_2d_cylinder(n=64, ny=44, cpml=4, R=8, src=(12, 20), nv=4, nv_perp=4), {"stencil_tz": 8}),
    "2d_march": (lambda: spec_2d_cylinder(n=64, ny=44, cpml=4, R=8, src=(12, 20), nv=4, nv_perp=4),
                 {"fused_rows": 4, "fused_stencils": 1}),
    "2d_tile": (lambda: spec_2d_cylinder(n=64, ny=44, cpml=4, R=8, src=(12, 20), nv=4, nv_perp=4),
                {"fused_rows": 0, "fused_stencils": 1}),
    "3d_odd_f32": (lambda: spec_3d_slab(n=33, cpml=4, slab=(14, 20), src_k=8, nv=4, f_dtype="f32"), {}),
    "3d_tma": (lambda: spec_3d_slab(n=32, cpml=4, slab=(14, 20), src_k=8, nv=4, f_dtype="f32"), {"stencil_tz": 8}),
    "3d_tma_fused": (lambda: spec_3d_slab(n=32, cpml=4, slab=(14, 20), src_k=8, nv=4, f_dtype="f32"),
                     {"stencil_tz": 8, "fused_stencils": 1}),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_sequence_equals_single_steps(case):
    import torch
    from paper_2211_05647_gb300 import Solver
    make, options = CASES[case]
    spec = make()
    a, b = Solver.from_spec(spec), Solver.from_spec(spec)
    ndim = spec["grid"]["ndim"]
    fields = {1: ("ex", "hy"), 2: ("ez", "hx", "hy"), 3: ("ex", "ey", "ez", "hx", "hy", "hz")}[ndim]
    for s in (a, b):
        if ndim == 1:   # a port keeps the 1-D steps in the graphs
            s.set_ports([[5]], [1e9])
        for k, v in options.items():
            s.set_option(k, v)
    n = 0
    for steps in (3, 47, 64, 22):
        a.step(steps)
        for _ in range(steps):
            b.step(1)
        n += steps
        for q in fields:
            x, y = a.read(q).cpu(), b.read(q).cpu()
            assert torch.equal(x, y), (q, n)
        assert a.read(fields[0]).abs().max() > 0
    a.step(3)
    b.time_kernels(3)
    for q in fields:
        assert torch.equal(a.read(q).cpu(), b.read(q).cpu()), q
