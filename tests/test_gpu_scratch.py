"""What the library allocates for a call, seen through the caller's allocator:
the first hard-sphere step takes its scratch in one block."""
import ctypes as C

import numpy as np
import pytest

import paper_1503_00707_gb300 as D

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
