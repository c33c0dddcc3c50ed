"""Delta f written on the device between the two halves of a step (where only the row kernel reads it) gives the
bits that the same write before the step gives, for plain and padded rows and for writes by the copy kernel."""
import numpy as np
import pytest

from fdtd_inputs import spec_2d_cylinder

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv,nvp,dtype,prec", [(32, 16, "f32", "f32"), (31, 9, "f32", "f32"), (32, 16, "bf16", "f32"),
                                               (4, 4, "bf16", "f32"), (12, 12, "f64", "f64"), (256, 8, "f32", "f32")])
def test_write_between_halves(nv, nvp, dtype, prec):
    import torch
    from paper_2211_05647_gb300 import Solver
    td = {"f32": torch.float32, "bf16": torch.bfloat16, "f64": torch.float64}[dtype]
    spec = spec_2d_cylinder(n=64, ny=56, cpml=4, R=14, src=(12, 20), nv=nv, nv_perp=nvp, precision=prec, f_dtype=dtype)
    a, b = Solver.from_spec(spec), Solver.from_spec(spec)
    ns, nn = a.plasma_shape()
    gen = torch.Generator().manual_seed(nv + nvp)
    for _ in range(8):
        v = torch.randn(ns * nn, generator=gen, dtype=torch.float64).to(td).cuda()
        a.write("df", v)
        a.step_half(0)
        a.step_half(1)
        b.step_half(0)
        b.write("df", v)
        b.step_half(1)
        for q in ("df", "ez", "j"):
            x, y = a.read(q).cpu(), b.read(q).cpu()
            assert torch.equal(x.view(torch.uint8).flatten(), y.view(torch.uint8).flatten()), q
    assert np.isfinite(a.read("ez").cpu().numpy()).all()
