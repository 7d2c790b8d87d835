"""Which lattice Boltzmann steps overlap their launches depends on the number of
cells alone (at most 2,048 an SM in FP32, 128 in FP64), whatever size the CTAs
are cut to. On either side of the line, and where the CTA size changes, a block of
steps equals the same steps one call each, bit for bit."""
import numpy as np
import pytest

import paper_1503_00707_gb300 as D
import workloads as W

pytestmark = pytest.mark.gpu


# 152 SMs: the lines lie at 311,296 (FP32) and 19,456 cells (FP64); CTAs have 32
# threads up to 9,727 cells, then 64, 128 and 256 from 38,912
@pytest.mark.parametrize("name, levels, precision", [
    ("l1_2d_disk_d2q9", (6, 6), D.F64), ("l1_2d_disk_d2q9", (7, 7), D.F64), ("l1_2d_disk_d2q9", (8, 8), D.F64),
    ("l1_2d_disk_d2q9", (7, 7), D.F32), ("l1_2d_disk_d2q9", (9, 9), D.F32), ("l1_2d_disk_d2q9", (10, 10), D.F32),
    ("l2_sphere_d3q19_small", (5, 5), D.F32), ("l2_sphere_d3q19_small", (6, 6), D.F32),
    ("l2_sphere_d3q27_small", (5, 6), D.F64)])
def test_block_equals_single_steps(name, levels, precision):
    c = dict(W.CONFIGS[name], base_level=levels[0], max_level=levels[1])
    out = []
    for calls in ([7], [1] * 7):
        s = D.lbm_solver_from_config(c, precision)
        s.lbm_init(*W.lbm_initial_state(c, s.centres()[0]))
        dt = s.lbm_dt_cfl(0.4)
        for n in calls:
            s.lbm_step(n, dt, tau=2 * dt)
        out.append(s.lbm_get_f())
        s.close()
    assert np.array_equal(out[0], out[1])
