"""Batches whose tiles fill the SMs by themselves take the training tile that runs on one CTA: every tile's gradient
and loss equal those of the same rows in batches small enough for the clusters.  The loss is a mean, so a batch of four or
eight times the rows scales every residual's derivative, and each product and sum that follows, by exactly that."""
import math

import pytest

pytestmark = pytest.mark.gpu

NP = 18945
STRIDE = NP + 1      # floats a tile in the workspace: its gradient, then its loss


def _tiles(tr, x, t):
    import torch
    tr.loss_grad(x, t)
    torch.cuda.synchronize()
    off = -tr.ws.data_ptr() % 256
    n = -(-x.shape[0] // 128)
    return tr.ws[off:off + 4 * STRIDE * n].view(torch.float32).view(n, STRIDE).clone()


@pytest.mark.parametrize("rows", [16384, 32768])
def test_tiles_equal_the_clusters(rows):
    import torch
    from paper_2211_05647_gb300 import MlpTrainer
    from paper_2211_05647_gb300 import closure as C
    p = C.init_params(3, "cuda")
    gen = torch.Generator(device="cuda").manual_seed(rows)
    x = torch.randn(rows, 17, generator=gen, device="cuda")
    t = torch.randn(rows, generator=gen, device="cuda")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    part = 4096
    assert 8 * (part // 128) <= 3 * sms < 8 * (rows // 128)
    big = _tiles(MlpTrainer(p, rows), x, t)
    small = MlpTrainer(p, part)
    got = torch.cat([_tiles(small, x[i:i + part].contiguous(), t[i:i + part].contiguous())
                     for i in range(0, rows, part)])
    assert torch.equal(big, got / (rows // part))   # (a power of two: exact)


@pytest.mark.parametrize("rows", [58 * 128, 58 * 128 + 1, 20011])
def test_ragged_large_batches(rows):
    """Gradient and loss against the mean over small batches of the same rows.  A term is rounded to BF16 up to three
    times on either side, at another scale of dy: 2 * 3 * 2^-9 / sqrt(3) of the gradient's norm, the terms' signs
    being random; the FP32 sums' other order is far below that."""
    import torch
    from paper_2211_05647_gb300 import MlpTrainer
    from paper_2211_05647_gb300 import closure as C
    p = C.init_params(4, "cuda")
    gen = torch.Generator(device="cuda").manual_seed(rows)
    x = torch.randn(rows, 17, generator=gen, device="cuda")
    t = torch.randn(rows, generator=gen, device="cuda")
    tr = MlpTrainer(p, rows)
    loss, g = (v.clone() for v in tr.loss_grad(x, t))
    acc, lacc = torch.zeros_like(g, dtype=torch.float64), 0.0
    for i in range(0, rows, 5000):
        n = min(5000, rows - i)
        l, gi = MlpTrainer(p, n).loss_grad(x[i:i + n].contiguous(), t[i:i + n].contiguous())
        acc += gi.double() * (n / rows)
        lacc += float(l) * n / rows
    assert abs(float(loss) - lacc) <= 1e-5 * lacc
    assert float((g.double() - acc).norm() / acc.norm()) <= 7e-3


def test_epoch_of_large_minibatches_equals_its_steps():
    import torch
    from paper_2211_05647_gb300 import MlpTrainer
    from paper_2211_05647_gb300 import closure as C
    from paper_2211_05647_gb300 import fdtd_plasma as F
    lib = F.load_library()
    n, batch = 30000, 10000
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(n, 17, generator=gen, device="cuda")
    t = torch.randn(n, generator=gen, device="cuda")
    pa = C.init_params(3, "cuda")
    pb = pa.clone()
    ta, sep = MlpTrainer(pa, batch, lr=2e-3), MlpTrainer(pb, batch, lr=2e-3)
    ta.epoch(x, t, 9, 0, 0, 6)
    xb, tb = torch.empty(batch, 17, device="cuda"), torch.empty(batch, device="cuda")
    for b in range(n // batch):
        assert lib.fdtd_mlp_gather(x.data_ptr(), t.data_ptr(), n, 9, 0, b * batch, batch, xb.data_ptr(), tb.data_ptr(),
                                   None) == 0
        sep.t = b
        sep.step(xb, tb, lr=2e-3 * 0.5 * (1 + math.cos(math.pi * b / 6)))
    torch.cuda.synchronize()
    assert torch.equal(pa, pb) and torch.equal(ta.m, sep.m)
