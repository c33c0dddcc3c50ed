"""Device reads and writes of delta f: the rows of a padded layout packed and
unpacked by the library's kernel equal what the host copies of the same state
give, for every unit the kernel moves (16, 8, 4 and 2 bytes), for rows without
padding, and into device memory that is aligned to an element only."""
import ctypes

import numpy as np
import pytest

from fdtd_inputs import spec_1d_slab, spec_2d_cylinder

pytestmark = pytest.mark.gpu

#        nv, nv_perp, storage: bytes of a row -> widest unit
GRIDS = [(31, 1, "f32"), (31, 1, "bf16"), (31, 1, "f64"), (33, 1, "f64"), (20, 1, "f32"), (62, 1, "bf16"),
         (12, 12, "bf16"), (31, 16, "bf16"), (32, 1, "f32"), (3, 1, "f32"), (1, 2, "bf16")]


def _solver(nv, nvp, dtype):
    from paper_2211_05647_gb300 import Solver
    prec = "f64" if dtype == "f64" else "f32"
    if nvp > 1:
        nv = max(nv, 2)
        spec = spec_2d_cylinder(n=48, ny=40, cpml=4, R=9, src=(12, 20), nv=nv, nv_perp=nvp, precision=prec, f_dtype=dtype)
    else:
        spec = spec_1d_slab(nz=700, slab=(100, 631), nv=nv, precision=prec, f_dtype=dtype)
    return Solver.from_spec(spec)


@pytest.mark.parametrize("nv,nvp,dtype", GRIDS)
def test_device_rows_equal_host_rows(nv, nvp, dtype):
    import torch
    s = _solver(nv, nvp, dtype)
    ns, nn = s.plasma_shape()
    td = {"f32": torch.float32, "bf16": torch.bfloat16, "f64": torch.float64}[dtype]
    vals = torch.randn(ns * nn, generator=torch.Generator().manual_seed(nv), dtype=torch.float64).to(td)
    s.write("df", vals.cuda())                                    # packed -> padded on the device
    host = s.read("df", device=False)
    want = vals.view(ns, nn).float().numpy() if dtype == "bf16" else vals.view(ns, nn).numpy()
    assert np.array_equal(host, want)
    assert torch.equal(s.read("df").cpu(), vals.view(ns, nn))     # padded -> packed on the device
    # a destination that starts one element past an aligned address
    buf = torch.zeros(ns * nn + 1, dtype=td, device="cuda")
    rc = s.lib.fdtd_plasma_read_fields(s.h, 7, ctypes.c_void_p(buf.data_ptr() + buf.element_size()),
                                       s.quantity_bytes("df"), 1)
    assert rc == 0 and torch.equal(buf[1:].cpu(), vals)
    s.write("df", vals)                                           # host write, then a device read of it
    assert torch.equal(s.read("df").cpu().view(-1), vals)
    s.step(2)                                                     # padding nodes are still 0: J stays finite
    assert s.diagnostics()["finite"]


@pytest.mark.parametrize("nz", [4095, 4096, 4097, 50001, 5000000])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_linear_copies(nz, prec):
    """Fields of a line around the sizes where the copy kernel takes over (16 KB) and hands back (16 MB), to and from
    addresses aligned to one element only."""
    import torch
    from paper_2211_05647_gb300 import Solver
    td = torch.float32 if prec == "f32" else torch.float64
    s = Solver(dict(ndim=1, nz=nz, dx=1e-3, courant=0.5, precision=prec))
    v = torch.randn(nz + 2, generator=torch.Generator().manual_seed(nz), dtype=td).cuda()
    for off in (0, 1):
        s.write("ex", v[off:off + nz + 1])
        assert np.array_equal(s.read("ex", device=False), v[off:off + nz + 1].cpu().numpy())
        buf = torch.zeros(nz + 2, dtype=td, device="cuda")
        assert s.lib.fdtd_plasma_read_fields(s.h, 0, ctypes.c_void_p(buf[off:].data_ptr()), s.quantity_bytes("ex"), 1) == 0
        assert torch.equal(buf[off:off + nz + 1], v[off:off + nz + 1]) and float(buf[(1 - off) * (nz + 1)]) == 0.0
