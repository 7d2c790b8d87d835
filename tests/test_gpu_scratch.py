"""What the library allocates for a call, seen through the caller's allocator:
a network evaluation holds the forward pass's buffers and its rows, not those
of training, which the first gradient adds; the first hard-sphere step takes
its scratch in one block. Results do not depend on which came first."""
import ctypes as C

import numpy as np
import pytest

import paper_1503_00707_gb300 as D
from tests.gpu_util import random_params

pytestmark = pytest.mark.gpu


class Counter:
    """The library's allocations, through torch's allocator."""

    def __init__(self, solver):
        import torch
        torch.cuda.init()
        self.sizes, self.live = [], {}

        def alloc(n, user):
            p = torch.cuda.caching_allocator_alloc(n)
            self.sizes.append(n)
            self.live[p] = n
            return p

        def free(p, user):
            torch.cuda.caching_allocator_delete(p)
            del self.live[p]

        self.fn = (C.CFUNCTYPE(C.c_void_p, C.c_size_t, C.c_void_p)(alloc), C.CFUNCTYPE(None, C.c_void_p, C.c_void_p)(free))
        assert D.lib().dvm_set_allocator(solver._h, C.cast(self.fn[0], C.c_void_p), C.cast(self.fn[1], C.c_void_p), None) == 0


def test_network_buffers_follow_the_call():
    n = 4096
    g = np.random.default_rng(1)
    x, t = g.standard_normal((n, 64)).astype(np.float32), g.standard_normal((n, 64)).astype(np.float32)
    s = D.Solver(D.F32, D.COLL_NONE, 1.0)
    count = Counter(s)
    s.set_weights(random_params(3))
    held = sum(count.live.values())
    y = s.mlp_forward(x)
    # BF16 input and three BF16 activations, and the rows in and out
    assert sum(count.live.values()) - held == n * (2 * 64 + 3 * 2 * 256 + 2 * 4 * 64)
    loss, grad = s.mlp_loss_grad(x, t)
    assert np.array_equal(s.mlp_forward(x[:100]), y[:100])
    # more rows: each set grows by itself; fewer rows after them
    s.mlp_forward(np.concatenate([x, x]))
    again = s.mlp_loss_grad(x, t)
    assert again[0] == loss and np.array_equal(again[1], grad)
    s.close()
    assert not count.live


@pytest.mark.parametrize("n", [8, 16])
def test_first_hard_sphere_step_allocates_once(n):
    s = D.Solver(D.F32, D.COLL_HS, 0.1)
    count = Counter(s)
    s.build_tree(D.tree_spec(3, 1, 1))
    s.set_velocity_grid((n, n, n), (-4.0,) * 3, (4.0,) * 3)
    s.set_collision_tables(32, 5)
    nc = s.ncells
    s.init_maxwellian(np.ones((nc, 1)), np.ones((nc, 1)), np.zeros((nc, 1, 3)), np.ones((nc, 1)))
    before = len(count.sizes)
    s.step(1, 1e-6)
    assert len(count.sizes) - before == 1
    s.step(2, 1e-6)
    assert len(count.sizes) - before == 1
    s.close()
    assert not count.live
