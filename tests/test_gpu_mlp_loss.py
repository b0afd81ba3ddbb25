"""The training batch's loss: the same bits in every call, and the mean over the samples.

Tolerance against a 64-bit sum over the library's own FP32 logits: per sample two functions of 2 ulps,
two products and a sum, then 5 + 1 additions and a division in FP32 (the chunks' sum carries its
errors): below 13 x 2^-24 = 8e-7 relative, all terms being positive."""
import numpy as np
import pytest

import paper_1904_11147_gb300 as dgl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 31, 64, 65, 1000, 8192, 20011])
@pytest.mark.parametrize("F", [5, 116])
def test_loss(B, F):
    import torch
    rng = np.random.default_rng(B + F)
    X = torch.from_numpy(rng.standard_normal((B, F)).astype(np.float32)).cuda()
    y = torch.from_numpy((rng.random(B) < 0.3).astype(np.uint8)).cuda()
    net = dgl.MLP(F, seed=3)
    z = torch.empty(B, dtype=torch.float32, device="cuda")
    net.predict(X, z)
    torch.cuda.synchronize()
    z, t = z.cpu().numpy().astype(np.float64), y.cpu().numpy()
    want = (np.where(t == 1, 4.0 * np.logaddexp(0, -z), np.logaddexp(0, z))).mean()
    g0, l0 = net.grad(X, y, pos_weight=4.0)
    assert abs(l0 - want) <= 1e-6 * want
    for _ in range(40):
        g, l = net.grad(X, y, pos_weight=4.0)
        assert l == l0 and np.array_equal(g, g0)
    first = net.train_step(X, y, pos_weight=4.0, lr=1e-3, want_loss=True)
    assert first == l0
