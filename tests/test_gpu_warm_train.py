"""The training step of the warm-start network against FP64 autograd, at row
counts around its tiles: 32 rows per head CTA, 64 per GEMM tile, 128 per row
group of a weight gradient."""

import math

import numpy as np
import pytest
import torch

F, H, O = 256, 256, 16
# Worst-case growth of FP32 rounding in a contraction of length n is n u
# (u = 6e-8).  The longest chain behind a gradient is four contractions of
# length 256 (6e-5) and one over the N <= 1100 rows (6.6e-5).
TOL = 2e-4


def reference(theta, feats, targets, lens):
    th = theta.double().cpu().requires_grad_(True)
    parts, at = [], 0
    for a, b in ((F, H), (H, H), (H, O)):
        parts += [th[at:at + a * b].reshape(a, b), th[at + a * b:at + a * b + b]]
        at += a * b + b
    x = torch.nn.functional.gelu(feats.double().cpu() @ parts[0] + parts[1])
    x = torch.nn.functional.gelu(x @ parts[2] + parts[3])
    mask = torch.arange(O)[None, :] >= lens.cpu()[:, None]
    o = (x @ parts[4] + parts[5]).masked_fill(mask, -math.inf)
    u = torch.exp(o - o.max(1, keepdim=True).values)
    u = u / u.norm(dim=1, keepdim=True)
    loss = (1 - (u * targets.double().cpu()).sum(1) ** 2).mean()
    loss.backward()
    return float(loss.detach()), th.grad


def rows(N, seed, offset=0):
    """N rows; offset > 0 places the features at an address that is only 4-byte aligned."""
    g = np.random.default_rng(seed)
    buf = torch.zeros(N * F + 4, device="cuda")
    feats = buf[offset:offset + N * F].view(N, F)
    feats.copy_(torch.from_numpy((g.random((N, F)) < 0.35).astype(np.float32)))
    lens = torch.from_numpy(np.where(g.random(N) < 0.7, 16, 2).astype(np.int32)).cuda()
    t = np.exp(g.standard_normal((N, O))) * (np.arange(O)[None, :] < lens.cpu().numpy()[:, None])
    targets = torch.from_numpy((t / np.linalg.norm(t, axis=1, keepdims=True)).astype(np.float32)).cuda()
    return feats, targets, lens


@pytest.mark.gpu
@pytest.mark.parametrize("N,offset", [(1, 0), (31, 0), (33, 0), (64, 1), (127, 0), (129, 0), (256, 3), (700, 0),
                                      (1100, 0)])
def test_gradient_matches_fp64_autograd(N, offset):
    from paper_2402_04834_gb300 import warmstart
    net = warmstart.WarmStart(seed=3)
    feats, targets, lens = rows(N, 100 + N, offset)
    assert feats.data_ptr() % 16 == (4 * offset) % 16
    loss, grad = net.gradient(feats, targets, lens)
    want_loss, want = reference(net.theta, feats, targets, lens)
    assert abs(loss - want_loss) <= TOL * abs(want_loss)
    at = 0
    for n in (F * H, H, H * H, H, H * O, O):
        a, b = grad[at:at + n].double().cpu(), want[at:at + n]
        assert float((a - b).norm()) <= TOL * float(b.norm()), (n, at)
        at += n
    again, grad2 = net.gradient(feats, targets, lens)      # every sum has a fixed order
    assert again == loss and torch.equal(grad, grad2)
    before = net.theta.clone()
    net.train_step(feats, targets, lens, lr=1e-3)
    m, v = 0.1 * grad, 0.001 * grad * grad                  # Adam's first step
    step = 1e-3 * (m / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    assert torch.allclose(net.theta, before - step, rtol=0, atol=1e-6)
