"""Moments of a stored f (dvm_moments) against extended-precision sums, at
the sizes and values where the fixed-point sums change path: one quad of
positions, a partial warp, two quads a thread, positions beyond the two a
thread holds, cells whose scale falls outside the split's range, zeros and
non-finite values."""
import numpy as np
import pytest

import paper_1503_00707_gb300 as D
from tests.gpu_util import storage_round

pytestmark = pytest.mark.gpu

# a thread adds at most 64 terms in a row in FP64 and the tree of the CTA is
# shorter: 64 roundings of 2^-53 bound every sum's error against sum |w f|
TOL = 64 * 2.0 ** -53


@pytest.mark.parametrize("prec", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("n", [(2, 2, 8), (6, 2, 8), (10, 14, 8), (24, 24, 24), (18, 22, 32), (32, 32, 32), (64, 20, 40)])
def test_moments(n, prec):
    s = D.Solver({"f32": D.F32, "bf16": D.BF16, "f64": D.F64}[prec], D.COLL_NONE, 1.0)
    s.build_tree(D.tree_spec(3, 1, 1))
    hi = (3.0, 4.0, 5.0)
    s.set_velocity_grid(n, [-h for h in hi], hi)
    g = np.random.default_rng(5)
    f = np.exp(3.0 * g.standard_normal((s.ncells, s.nv)))
    f[1] *= np.where(g.uniform(size=s.nv) < 0.2, -0.1, 1.0)
    f[2] *= 1e-30
    f[3] *= 1e33
    f[4] = 0.0
    f[5, s.nv // 3] = np.inf
    f[6, s.nv - 1] = np.nan
    f[7] = 1e-6
    f[7, 5] = 1e6
    f = storage_round(f, prec)
    s.set_f(f)
    rho, u, T = s.moments()
    xi, dv = s.velocities().astype(np.longdouble), np.prod([2 * h / k for h, k in zip(hi, n)])
    for c in (0, 1, 2, 3, 7):
        fl = f[c].astype(np.longdouble)
        s0, sa = fl.sum(), np.abs(fl).sum()
        if not np.isfinite(s0):  # the scaled cell overflows FP32 on the largest grid
            assert not np.isfinite(rho[c]) and not np.isfinite(T[c])
            continue
        ur, e2 = (xi * fl[:, None]).sum(0) / s0, (np.square(xi).sum(1) * fl).sum() / s0
        assert abs(rho[c] / (s0 * dv) - 1) < TOL * sa / s0
        scale = (np.abs(xi) * np.abs(fl)[:, None]).sum(0) / s0
        assert np.all(np.abs(u[c] - ur) < 2 * TOL * scale), c
        assert abs(T[c] - (e2 - np.square(ur).sum()) / 3) < 4 * TOL * (np.square(xi).sum(1) * np.abs(fl)).sum() / s0, c
    assert rho[4] == 0.0 and np.isnan(T[4])
    assert not np.isfinite(rho[5]) and not np.isfinite(T[5])
    assert np.isnan(rho[6]) and np.isnan(T[6])
    s.close()
