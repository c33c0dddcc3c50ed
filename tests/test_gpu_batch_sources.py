"""The batch's tabulated source values: a call longer than one launch's table
equals the same steps in short calls and the runs on the single-run path, bit
for bit, with sources of both kinds, one run without a source, and a batch of so
many runs that a launch holds the fewest steps."""
import numpy as np
import pytest

from fdtd_inputs import batch_runs_1d

pytestmark = pytest.mark.gpu


def _specs(n, nz, steps):
    sp = batch_runs_1d(nruns=n, seed=8, nz_range=nz, nv=16, f_dtype="f32", precision="f32", src_k=20, steps=steps)
    sp[0]["source"]["kind"] = "gauss"
    if n > 1:
        sp[1]["source"] = None
    for s in sp[2:]:
        s["source"].update(t0=0.5 * s["source"]["tau"])
    return sp


def test_long_calls_equal_short_ones():
    from paper_2211_05647_gb300 import Batch, Solver
    sp = _specs(4, (60, 400), 1100)
    a, b = Batch(sp), Batch(sp)
    a.step(1100)
    for _ in range(11):
        b.step(100)
    for r, spec in enumerate(sp):
        s = Solver.from_spec(spec)
        s.step(1100)
        for q in ("ex", "hy"):
            assert np.array_equal(a.read(r, q), b.read(r, q)), (r, q)
            assert np.array_equal(a.read(r, q), s.read(q, device=False)), (r, q)
        s.close()
    assert np.abs(a.read(2, "ex")).max() > 0 and np.abs(a.read(1, "ex")).max() == 0


def test_many_runs():
    """140 000 runs: 32 steps a launch, and more runs than one source launch's grid is high."""
    from paper_2211_05647_gb300 import Batch
    one = _specs(3, (8, 16), 70)
    sp = [one[r % 3] for r in range(140000)]
    a, ref = Batch(sp), Batch(one)
    a.step(70)
    ref.step(70)
    for r in (0, 1, 2, 65533, 65535, 65536, 65537, 131070, 131071, 139999):
        for q in ("ex", "hy", "j"):
            if q != "j" or ref.lib.fdtd_batch_quantity_bytes(ref.h, r % 3, 6):
                assert np.array_equal(a.read(r, q), ref.read(r % 3, q)), (r, q)
