"""The training kernels at the edges of their tiles: 32 and 64 rows a tile,
one CTA up to one per SM, several tiles a CTA, and rows past the batch.

The FP64 gradient of oracle/learned.py is compared per layer with the bar of
test_gpu_learned.py (1e-4 of the layer's largest entry, inputs away from the
ReLU kinks), the loss at 1e-5 relative as there (squares of FP32
residuals, each within about 64 u of its y, added in FP64).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import learned as OL
from paper_1707_01170_gb300 import learned as LS
from paper_1707_01170_gb300 import lrvol as lv
from paper_1707_01170_gb300.synth.lrgen import Stream

pytestmark = pytest.mark.gpu


def _batch(n, seed):
    """Rows whose hidden pre-activations all stay 2e-5 away from 0 (both sides take the same ReLU branch)."""
    p = LS.init_params(seed).astype(np.float64)
    X = (2 * Stream(seed + 1, 16 * n + 8).take(16 * n).reshape(n, 16) - 0.5).astype(np.float32)
    w, h, near = OL.unpack(p), X.astype(np.float64), np.zeros(n, dtype=bool)
    for k in (1, 2, 3):
        z = h @ w[f"W{k}"] + w[f"b{k}"]
        near |= (np.abs(z) < 2e-5).any(axis=1)
        h = np.maximum(z, 0.0)
    X[near] = X[~near][0]
    t = (3 * Stream(seed + 2, n + 8).take(n)).astype(np.float32)
    return p.astype(np.float32), X, t


@pytest.mark.parametrize("n", [1, 31, 32, 33, 49, 50, 64, 65, 97, 4863, 4865, 9728, 9793, 16385])
def test_gradient_at_tile_edges(n):
    p, X, t = _batch(n, 500 + n)
    scratch = torch.full((int(lv.load().lrvol_mlp_scratch_floats(n)) + 64,), 7.0, device="cuda")
    x = torch.from_numpy(X).cuda()
    loss, g = lv.mlp_grad(x, torch.from_numpy(t).cuda(), torch.from_numpy(p).cuda(), scratch=scratch)
    assert bool((scratch[-64:] == 7.0).all())            # nothing past the stated scratch
    want_loss, want = OL.loss_and_grad(p.astype(np.float64), X, t)
    assert abs(float(loss) - want_loss) <= 1e-5 * want_loss
    got, want = OL.unpack(g.cpu().numpy()), OL.unpack(want)
    for k in want:
        assert np.abs(got[k] - want[k]).max() <= 1e-4 * np.abs(want[k]).max() + 1e-12, (n, k)
    again = lv.mlp_grad(x, torch.from_numpy(t).cuda(), torch.from_numpy(p).cuda())[1]
    assert torch.equal(g, again)                          # a fixed order of sums


@pytest.mark.parametrize("n", [1, 40, 8192])
def test_step_applies_the_gradient(n):
    """The step's moments are those of the gradient call, and features may start at any float."""
    p, X, t = _batch(n, 900 + n)
    buf = torch.zeros(16 * n + 1, device="cuda")
    buf[1:] = torch.from_numpy(X).cuda().reshape(-1)
    x, tgt = buf[1:].reshape(n, 16), torch.from_numpy(t).cuda()
    P = torch.from_numpy(p).cuda()
    _, g = lv.mlp_grad(x, tgt, P)
    m, v = torch.zeros_like(P), torch.zeros_like(P)
    lv.mlp_train_step(x, tgt, P, m, v, 1, 1e-3, lv.mlp_scratch(n))
    assert torch.allclose(m, 0.1 * g, rtol=1e-6, atol=0)
    assert torch.allclose(v, 0.001 * g * g, rtol=1e-6, atol=1e-44)
    assert not torch.equal(P.cpu(), torch.from_numpy(p))
