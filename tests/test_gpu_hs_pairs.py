"""The hard-sphere update on pairs of cells against the oracle where it
changes shape: one cell, an odd number of cells, batches at the limit of the
fixed scratch, nodes on one lane and on a whole warp, and grids too large for
pair tiles, which run one cell at a time."""
import numpy as np
import pytest

import oracle as O
import paper_1503_00707_gb300 as D
import workloads as W
from tests.gpu_util import oracle_for, rel_linf, storage_round

pytestmark = pytest.mark.gpu


def _problem(n, hi, M):
    c = dict(W.CONFIGS["c4_hs_bimodal"])
    # the node spacing is the same on every axis
    nz = (n + 7) // 8 * 8
    ax = (hi, hi, hi * nz / n)
    c.update(base_level=1, max_level=1, pred=0, n=(n, n, nz), lo=tuple(-h for h in ax), hi=ax)
    s, o = D.solver_from_config(c, D.F32, D.COLL_HS), oracle_for(c)
    g = np.random.default_rng(3)
    u = np.zeros((8, 2, 3))
    u[:, 0, 0], u[:, 1, 0] = 0.2 * hi, -0.2 * hi
    u += 0.05 * g.standard_normal(u.shape)
    o.init_maxwellian(np.tile([0.45, 0.55], (8, 1)), np.ones((8, 2)), u, 0.03 * hi * hi * (1 + 0.1 * g.uniform(size=(8, 2))))
    s.set_collision_tables(M, 77)
    o.hs_tables(M, 77)
    return c, s, o


# hs_collide_noalloc takes any number of cells: rows repeat the oracle's eight
@pytest.mark.parametrize("n, hi, M, rows", [(8, 4.0, 128, 1), (8, 4.0, 32, 7), (8, 4.0, 1024, 8), (16, 6.0, 512, 5),
                                            (24, 8.0, 128, 3), (28, 8.0, 64, 9), (8, 4.0, 64, "limit")])
def test_collide_rows(n, hi, M, rows):
    import torch
    c, s, o = _problem(n, hi, M)
    if rows == "limit":
        rows = D.HS_NOALLOC_SCRATCH_BYTES // (8 * s.nv + 40)
    f = storage_round(o.get_f(), "f32")
    o.set_f(f)
    dt = 2e-6
    o.hs_collide(dt, c["kn"])
    want = o.get_f()
    assert rel_linf(want, f) > 1e-5
    which = np.arange(rows) % 8
    buf = torch.from_numpy(f.astype(np.float32)[which]).cuda()
    torch.cuda.synchronize()
    s.hs_collide_noalloc(buf.data_ptr(), rows, dt)
    got = buf.cpu().numpy()
    # as the hard-sphere step's parity bar: FP32 sums of up to 1024 trials
    for k in range(min(rows, 8)):
        assert rel_linf(got[k], want[k]) < 1e-5, k
    assert np.array_equal(got, got[which]) or np.max(np.abs(got - got[which])) < 1e-6 * np.max(np.abs(got))
    s.close()
