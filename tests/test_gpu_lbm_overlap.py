"""The steps of one lattice Boltzmann call follow each other with overlapped
launches; a call of one step launches plainly. Both are the same operations
on the same values, so f is equal bit for bit."""
import numpy as np
import pytest

import paper_1503_00707_gb300 as D
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1503_00707_gb300 import _build
    _build.build()


@pytest.mark.parametrize("precision", [D.F32, D.F64])
@pytest.mark.parametrize("name,levels", [
    ("l1_2d_disk_d2q9", None), ("l1_2d_disk_d2q9", (3, 5)),                # at most one CTA per SM: overlapped
    ("l2_sphere_d3q19_small", (3, 4)), ("l2_sphere_d3q27_small", (3, 4)),
    ("l2_sphere_d3q19_small", None), ("l2_sphere_d3q27_small", None)])     # larger grids: plain launches
def test_one_call_equals_single_steps(name, levels, precision):
    c = W.CONFIGS[name]
    if levels:
        c = dict(c, base_level=levels[0], max_level=levels[1])
    out = []
    for calls in ([33], [1] * 33):
        s = D.lbm_solver_from_config(c, precision)
        s.lbm_init(*W.lbm_initial_state(c, s.centres()[0]))
        dt = s.lbm_dt_cfl(0.4)
        for n in calls:
            s.lbm_step(n, dt, tau=2 * dt)
        out.append(s.lbm_get_f())
    assert np.array_equal(out[0], out[1])
