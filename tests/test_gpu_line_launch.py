"""The 1-D cooperative launch where it is refused or held up: while the caller's stream captures, and on a stream
that may use some of the SMs only; and the bounded wait of its CTAs."""
import ctypes

import numpy as np
import pytest

from fdtd_inputs import spec_1d_slab

pytestmark = pytest.mark.gpu


def _spec(nz=2000, slab=(900, 1400), nv=64, seed=3):
    sp = spec_1d_slab(nz=nz, slab=slab, src_k=50, nv=nv, precision="f32", seed=seed)
    sp["source"].update(t0=0.5 * sp["source"]["tau"])
    return sp


def _make(sp, stream=None):
    """A solver whose plasma is driven from the first step."""
    from paper_2211_05647_gb300 import Solver
    s = Solver.from_spec(sp, stream=stream)
    rng = np.random.default_rng(4)
    nz = sp["grid"]["nz"]
    s.write("ex", rng.standard_normal(nz + 1))
    s.write("hy", rng.standard_normal(nz) / 377.0)
    return s


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
    from paper_2211_05647_gb300 import FdtdError
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        a, b = _make(_spec(), st), _make(_spec(), st)
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


class _GreenStream:
    """A stream of a green context of at least `sms` SMs (driver API; no other process or stream is affected)."""

    def __init__(self, sms):
        import torch
        torch.zeros(1, device="cuda")
        try:
            self.cu = ctypes.CDLL("libcuda.so.1")
            for f in ("cuDeviceGetDevResource", "cuDevSmResourceSplitByCount", "cuDevResourceGenerateDesc",
                      "cuGreenCtxCreate", "cuGreenCtxStreamCreate", "cuStreamDestroy_v2", "cuGreenCtxDestroy"):
                getattr(self.cu, f)
        except (OSError, AttributeError) as e:
            pytest.skip(f"no green contexts here: {e}")
        res = lambda: ctypes.create_string_buffer(144)   # CUdevResource: type, 92 bytes, 48 bytes
        all_sms, part, rest, n = res(), res(), res(), ctypes.c_uint(1)
        desc, self.ctx, self.ptr = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
        self._call("cuDeviceGetDevResource", 0, all_sms, 1)
        self._call("cuDevSmResourceSplitByCount", part, ctypes.byref(n), all_sms, rest, 0, sms)
        self._call("cuDevResourceGenerateDesc", ctypes.byref(desc), part, 1)
        self._call("cuGreenCtxCreate", ctypes.byref(self.ctx), desc, 0, 1)
        self._call("cuGreenCtxStreamCreate", ctypes.byref(self.ptr), self.ctx, 1, 0)
        self.sms = int(np.frombuffer(part.raw[96:100], dtype=np.uint32)[0])
        self.stream = torch.cuda.ExternalStream(self.ptr.value)

    def _call(self, name, *args):
        rc = getattr(self.cu, name)(*args)
        if rc:
            pytest.skip(f"{name}: error {rc}")

    def close(self):
        self.stream.synchronize()
        self._call("cuStreamDestroy_v2", self.ptr)
        self._call("cuGreenCtxDestroy", self.ctx)


@pytest.mark.parametrize("nv,coop", [(64, True), (512, False)])
def test_stream_with_some_of_the_sms(nv, coop):
    """A line whose state fits 16 SMs runs there, one that needs the whole device takes the step graphs; the results
    are those of an ordinary stream."""
    import torch
    sp = _spec(nz=3000, slab=(500, 2900), nv=nv)
    b = _make(sp)
    assert b.launch_shapes()["block_x"] > 0
    g = _GreenStream(16)
    assert 16 <= g.sms < torch.cuda.get_device_properties(0).multi_processor_count
    a = _make(sp, g.stream)
    assert (a.launch_shapes()["block_x"] > 0) == coop
    for n in (1, 70):
        a.step(n)
        b.step(n)
    assert _same(a, b)
    a.close()
    g.close()


def test_wait_gives_up_after_its_limit():
    """A message that never comes is given up on after the limit, not sooner and not never."""
    import time
    from paper_2211_05647_gb300 import FdtdError, Solver, selftest_line_wait
    selftest_line_wait(10)                        # load and warm the module
    t0 = time.perf_counter()
    assert selftest_line_wait(2000) is True
    assert 2e-3 <= time.perf_counter() - t0 < 1.0
    for bad in (0, 10 ** 7):
        with pytest.raises(FdtdError):
            selftest_line_wait(bad)
    s = Solver.from_spec(_spec())
    s.step(20)
    assert s.diagnostics()["finite"]
