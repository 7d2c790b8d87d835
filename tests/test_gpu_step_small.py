"""The step kernel on grids of one to five compute warps per CTA, where the
launch changes form (three or four warps: three CTAs an SM, the sources behind
coarse-fine faces added after the transport loop), against the oracle: transport,
BGK and entropic BGK on a tree with walls, inflow, outflow and hanging faces. FP32 within
1e-5 and BF16 within 1e-2, as the other step tests hold them."""
import numpy as np
import pytest

import oracle as O
import paper_1503_00707_gb300 as D
import workloads as W
from tests.gpu_util import field_errors, pair, rel_linf, same_start

pytestmark = pytest.mark.gpu


# compute warps: 1, 2, 3, 3, 4, 4, 5
@pytest.mark.parametrize("n", [(8, 8, 16), (8, 8, 24), (12, 12, 16), (8, 16, 24), (10, 22, 16), (14, 18, 16), (18, 20, 16)])
@pytest.mark.parametrize("prec, coll", [("f32", "BGK"), ("bf16", "BGK"), ("f32", "BGK_ENTROPIC"), ("f32", "NONE")])
def test_step(n, prec, coll):
    hi = tuple(0.5 * k for k in n)
    c = dict(W.CONFIGS["c2_sphere_m3"], base_level=2, max_level=4, n=n, lo=tuple(-h for h in hi), hi=hi,
             fs_u=(0.5, 0.0, 0.0))
    s, o = pair(c, prec, getattr(D, "COLL_" + coll))
    same_start(s, o, o.get_f(), prec)
    dt = o.dt_cfl(c["cfl"])
    s.step(2, dt)
    o.step(2, dt, getattr(O, "COLL_" + coll), c["kn"])
    bar = 1e-5 if prec == "f32" else 1e-2
    assert rel_linf(s.get_f(), o.get_f()) < bar
    err = field_errors(s.moments(), o.moments())
    assert max(err.values()) < bar, err
    s.close()
