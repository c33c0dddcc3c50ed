"""A run of a batch has the bits it has alone, for rows of every length: the batched kernel's built-in row shape sums
J in the order of the single-run default."""
import numpy as np
import pytest

from fdtd_inputs import batch_runs_1d

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("nv", [3, 8, 12, 20, 32, 64, 100, 128, 200, 256, 300, 512])
def test_batch_equals_single_runs(nv, dtype):
    """BF16: one run a batch, since the stochastic rounding is counted by the batch's row numbers."""
    from paper_2211_05647_gb300 import Batch, Solver
    specs = batch_runs_1d(nruns=3, seed=nv, nz_range=(60, 900), nv=nv, f_dtype=dtype, src_k=20)
    rng = np.random.default_rng(nv)
    for sp in specs:
        sp["source"].update(t0=0.5 * sp["source"]["tau"])
        sp["ex"] = rng.standard_normal(sp["grid"]["nz"] + 1)
    for group in ([specs] if dtype == "f32" else [[sp] for sp in specs]):
        b = Batch(group)
        for r, sp in enumerate(group):
            b.write(r, "ex", sp["ex"])
        b.step(50)
        for r, sp in enumerate(group):
            s = Solver.from_spec(sp)
            s.write("ex", sp["ex"])
            s.step(50)
            assert np.abs(s.read("j", device=False)).max() > 0
            for q in ("ex", "hy", "j", "df"):
                assert np.array_equal(b.read(r, q).ravel(), s.read(q, device=False).ravel()), (r, q)
