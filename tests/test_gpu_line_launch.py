"""The 1-D cooperative launch where it is refused or held up: while the caller's stream captures."""
import numpy as np
import pytest

from fdtd_inputs import spec_1d_slab

pytestmark = pytest.mark.gpu


def _spec(nz=2000, slab=(900, 1400), nv=64, seed=3):
    sp = spec_1d_slab(nz=nz, slab=slab, src_k=50, nv=nv, precision="f32", seed=seed)
    sp["source"].update(t0=0.5 * sp["source"]["tau"])
    return sp


def _state(s):
    return {q: s.read(q, device=False).copy() for q in ("ex", "hy", "j", "df")}


def _same(a, b):
    a, b = _state(a), _state(b)
    return np.abs(b["j"]).max() > 0 and all(np.array_equal(a[q], b[q]) for q in a)


@pytest.mark.parametrize("before", [0, 5])
def test_step_while_the_stream_captures(before):
    """Refused with an error that leaves the capture and the handle as they were: the first step of a handle as any
    later one, and the handle still takes the cooperative kernel afterwards."""
    import torch
    from paper_2211_05647_gb300 import FdtdError, Solver
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        a, b = Solver.from_spec(_spec(), stream=st), Solver.from_spec(_spec(), stream=st)
        if before:
            a.step(before)
            b.step(before)
        x = torch.zeros(64, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        x += 1
        with pytest.raises(FdtdError):
            a.step(3)
        x += 1
    g.replay()
    torch.cuda.synchronize()
    assert float(x.sum()) == 128.0
    assert a.info()[1] == before and a.launch_shapes()["block_x"] > 0
    with torch.cuda.stream(st):
        for s in (a, b):
            s.step(40)
        assert _same(a, b)
