"""Network loss, gradient and forward pass at the edges of their tiles (one
row, either side of a 64-row chunk and of a 128-row tile, several K splits)
against the same network in 64 bits with BF16 rounding at the points where the
device rounds.  The device sums in FP32 (relative 1e-6 a sum) and a sum that
falls on the other side of a BF16 rounding moves one value by 2^-9, which a
gradient entry averages over the batch: 2e-3 of a parameter block's norm."""
import numpy as np
import pytest

import oracle as O
import paper_1503_00707_gb300 as D

pytestmark = pytest.mark.gpu


def _bf(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, np.float32)).bfloat16().double().numpy()


def _silu(z):
    return z / (1 + np.exp(-z))


@pytest.mark.parametrize("n", [1, 31, 63, 64, 65, 127, 128, 129, 1000, 1345, 5000])
def test_rows(n):
    g = np.random.default_rng(n)
    blocks = [(g.standard_normal(r * c) * 1.2 / np.sqrt(c), 0.1 * g.standard_normal(nb)) for (r, c), nb in O.MLP_SHAPES]
    p = np.concatenate([np.concatenate(b) for b in blocks]).astype(np.float32)
    x = g.standard_normal((n, 64)).astype(np.float32)
    t = g.standard_normal((n, 64)).astype(np.float32)
    s = D.Solver(D.F32, D.COLL_NONE, 1.0)
    s.set_weights(p)
    # a larger batch first: the work buffers and their padding are reused
    s.mlp_loss_grad(np.ones((n + 200, 64), np.float32), np.zeros((n + 200, 64), np.float32))
    y, (loss, grad) = s.mlp_forward(x), s.mlp_loss_grad(x, t)
    W, b, off = [], [], 0
    for (r, c), nb in O.MLP_SHAPES:
        W.append(p[off:off + r * c].reshape(r, c))
        b.append(p[off + r * c:off + r * c + nb].astype(np.float64))
        off += r * c + nb
    h, z = [_bf(x)], []
    for k in range(4):
        z.append(h[k] @ _bf(W[k]).T + b[k])
        h.append(_bf(_silu(z[k])))
    assert np.linalg.norm(y - z[3]) < 2e-3 * np.linalg.norm(z[3])
    r = z[3] - t
    assert abs(loss - np.mean(r * r)) < 2e-3 * loss
    d, want = 2 * r / (64 * n), [None] * 4
    for k in range(3, -1, -1):
        want[k] = (_bf(d).T @ h[k], d.sum(0))
        if k:
            sg = 1 / (1 + np.exp(-z[k - 1]))
            d = (_bf(d) @ _bf(W[k])) * sg * (1 + z[k - 1] * (1 - sg))
    off = 0
    for k, ((rr, c), nb) in enumerate(O.MLP_SHAPES):
        for q, w in ((rr * c, want[k][0].ravel()), (nb, want[k][1])):
            assert np.linalg.norm(grad[off:off + q] - w) < 2e-3 * np.linalg.norm(w), (k, q)
            off += q
    s.close()
