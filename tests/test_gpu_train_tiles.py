"""The training kernels at the sizes where a tile of 128 rows or an epoch of
minibatches can go wrong: one row, a row less and more than a CTA's 32 and a
tile's 128, several tiles with a ragged last one, and epochs of one, two and three
minibatches (the rows of the next and the places of the one after are prepared
ahead).  The gradient against FP64, and an
epoch against its separate gather, gradient and Adam calls, bit for bit."""
import math

import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu


def _data(n, seed):
    import torch
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((n, 17)).astype(np.float32)
    t = rng.standard_normal(n).astype(np.float32)
    return x, t, torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()


def _oracle_params(flat):
    o = np.cumsum([0, 17 * 128, 128, 128 * 128, 128, 128, 1])
    w1, b1, w2, b2, w3, b3 = (np.asarray(flat[a:b], dtype=np.float64) for a, b in zip(o[:-1], o[1:]))
    return dict(W1=w1.reshape(17, 128), b1=b1, W2=w2.reshape(128, 128), b2=b2, W3=w3.reshape(128, 1), b3=b3)


@pytest.mark.parametrize("batch", [1, 31, 33, 127, 128, 129, 300])
def test_gradient_of_ragged_batches(batch):
    from paper_2211_05647_gb300 import MlpTrainer
    from paper_2211_05647_gb300 import closure as C
    x, t, xd, td = _data(batch, batch)
    p = C.init_params(7, "cuda")
    loss, grad = MlpTrainer(p, batch).loss_grad(xd, td)
    P = _oracle_params(p.cpu().numpy())
    L, go = M.loss_and_grads(P, x.astype(np.float64), t.astype(np.float64))
    y, _ = M.forward(P, x.astype(np.float64))
    # the forward is within 1e-2 of y's norm, so a residual is off by d; the gradient by d relative to the residual's
    # norm and the 3e-2 of its own BF16 contractions
    d = 1e-2 * np.sqrt(np.mean(np.square(y)))
    assert abs(float(loss.item()) - L) <= 2 * np.sqrt(L) * d + d * d
    g, ref = _oracle_params(grad.cpu().numpy()), go
    num = np.sqrt(sum(np.sum((g[k].ravel() - np.ravel(ref[k])) ** 2) for k in ref))
    den = np.sqrt(sum(np.sum(np.square(ref[k])) for k in ref))
    assert num <= (3e-2 + d / np.sqrt(L)) * den


@pytest.mark.parametrize("n,batch", [(130, 130), (517, 258), (385, 128), (700, 33), (9, 3)])
def test_epoch_equals_its_steps(n, batch):
    import torch
    from paper_2211_05647_gb300 import MlpTrainer
    from paper_2211_05647_gb300 import closure as C
    from paper_2211_05647_gb300 import fdtd_plasma as F
    lib = F.load_library()
    _, _, x, t = _data(n, n)
    pa = C.init_params(3, "cuda")
    pb = pa.clone()
    total = 2 * (n // batch)
    ta, sep = MlpTrainer(pa, batch, lr=2e-3), MlpTrainer(pb, batch, lr=2e-3)
    xb = torch.empty(batch, 17, dtype=torch.float32, device="cuda")
    tb = torch.empty(batch, dtype=torch.float32, device="cuda")
    for ep in range(2):
        ta.epoch(x, t, 9, ep, ep * (n // batch), total)
        for b in range(n // batch):
            assert lib.fdtd_mlp_gather(x.data_ptr(), t.data_ptr(), n, 9, ep, b * batch, batch, xb.data_ptr(),
                                       tb.data_ptr(), None) == 0
            it = ep * (n // batch) + b
            sep.t = it
            sep.step(xb, tb, lr=2e-3 * 0.5 * (1 + math.cos(math.pi * it / total)))
    torch.cuda.synchronize()
    assert torch.equal(pa, pb) and torch.equal(ta.m, sep.m) and torch.equal(ta.v, sep.v)
