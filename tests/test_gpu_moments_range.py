"""Moments of a stored f whose values span many binary orders: one value of 1
among values of `low` and below, so that the sums' second and third levels and
their rests carry most of the values; the same scaled down, where warps without
the large value leave the range that needs no scaling.

A thread's 32 values go into integers exactly but for rests below 2^-50 of the
largest |f|, summed in FP32 in at most 60 additions a value: off by at most
60 2^-24 2^-50 nv of it, 2^-53 at 24^3 and 2^-52 at 32^3, and the density takes
four FP64 roundings of 2^-53 more."""
import numpy as np
import pytest

import paper_1503_00707_gb300 as D
from tests.gpu_util import storage_round

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "bf16"])
@pytest.mark.parametrize("n", [(6, 2, 8), (18, 18, 16), (24, 24, 24), (18, 22, 32), (32, 32, 32)])
@pytest.mark.parametrize("scale", [0, -70, -110])
def test_one_large_value(n, prec, scale):
    s = D.Solver({"f32": D.F32, "bf16": D.BF16}[prec], D.COLL_NONE, 1.0)
    s.build_tree(D.tree_spec(3, 1, 1))
    hi = (3.0, 4.0, 5.0)
    s.set_velocity_grid(n, [-h for h in hi], hi)
    g = np.random.default_rng(11)
    low = 2.0 ** -np.array([12.0, 18.0, 27.0, 30.0, 31.0, 36.0, 45.0, 53.0])
    f = low[:, None] * g.uniform(0.5, 1.0, (s.ncells, s.nv))
    f[3] = 0.93 * 2.0 ** -30
    f[np.arange(8), g.integers(0, s.nv, 8)] = 1.0
    f = storage_round(f * 2.0 ** scale, prec)
    s.set_f(f)
    rho, u, T = s.moments()
    xi, dv = s.velocities().astype(np.longdouble), np.prod([2 * h / k for h, k in zip(hi, n)])
    tol = (4 + max(1.0, 2.0 * s.nv / 13824)) * 2.0 ** -53
    for c in range(8):
        fl = f[c].astype(np.longdouble)
        s0 = fl.sum()
        ur, e2 = (xi * fl[:, None]).sum(0) / s0, (np.square(xi).sum(1) * fl).sum() / s0
        assert abs(rho[c] / (s0 * dv) - 1) < tol, c
        # a value's share of a sum is weighted with j <= n_d - 1 of its axis, the
        # large one's with j >= 1
        rest = 60 * 2.0 ** -74 * s.nv
        assert np.all(np.abs(u[c] - ur) < 4 * tol * (np.abs(xi) * fl[:, None]).sum(0) / s0 + rest * np.array(hi)), c
        assert abs(T[c] - (e2 - np.square(ur).sum()) / 3) < 8 * tol * e2 + rest * np.square(hi).sum(), c
    s.close()
