"""Weight gradients of large batches: batches of up to 12,000 rows sum over
several K splits, larger ones in one chain of the tensor core's accumulator.

A batch's gradient is the mean of its eighths' gradients, and an eighth's output
gradients are exactly eight times the batch's (the scale is a power of two
apart), so every BF16 rounding falls alike and the two differ by their sums
alone.  The accumulator truncates: 2^-23 of the sum, 2^-24 on average, with each
16 rows, so one chain is off by at most (n / 16) 2^-24 of the gradient (measured:
a third of it); a split sum by that of its 1/21 of the rows, and 21 FP32
additions more; the eighths, at most 7,500 rows, likewise."""
import numpy as np
import pytest

import oracle as O
import paper_1503_00707_gb300 as D
from tests.gpu_util import random_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8 * 1500, 8 * 1501, 30000, 60000])
def test_sums_of_large_batches(n):
    g = np.random.default_rng(n)
    x = (g.standard_normal((n, 64)) * 0.5).astype(np.float32)
    t = (-0.4 * x + 0.3 * np.abs(x[:, ::-1]) + 0.05 * g.standard_normal((n, 64))).astype(np.float32)
    s = D.Solver(D.F32, D.COLL_NONE, 1.0)
    s.set_weights(random_params(9))
    loss, grad = s.mlp_loss_grad(x, t)
    m = n // 8
    parts = [s.mlp_loss_grad(x[k * m:(k + 1) * m], t[k * m:(k + 1) * m]) for k in range(8)]
    s.close()
    assert abs(loss - np.mean([p[0] for p in parts])) < 1e-12 * loss
    want = np.mean([p[1].astype(np.float64) for p in parts], axis=0)

    def off(rows):
        splits = min(21, (rows + 63) // 64) if rows <= 12000 else 1
        return (rows / splits / 16 + (21 if splits > 1 else 0)) * 2.0 ** -24

    tol, at = off(n) + off(m), 0
    for k, ((r, c), nb) in enumerate(O.MLP_SHAPES):
        for q in (r * c, nb):
            a, b = grad[at:at + q].astype(np.float64), want[at:at + q]
            # biases are FP32 sums over 128-row tiles
            lim = tol if q == r * c else (n / 128) * 2.0 ** -24 + 8 * 2.0 ** -24
            assert np.linalg.norm(a - b) < lim * np.linalg.norm(b), (k, q)
            at += q
