"""QQ^T just below and just above the sizes where its one-launch form gives way to the sweeps (by the
points on the elements' upper faces): plain and masked in FP64, after the folded FP64 operator, and
after the FP32 operator, against the oracle."""
import numpy as np
import pytest

import oracle as o
from tests.gpu_common import Case, rel_err

pytestmark = pytest.mark.gpu


def _face_points(nel, p):
    return nel[0] * nel[1] * nel[2] * (3 * (p + 1) ** 2 - 3 * (p + 1) + 1)


@pytest.mark.parametrize("line,nel,p", [
    (375000, (21, 21, 22), 3), (375000, (22, 22, 21), 3), (375000, (13, 13, 13), 7), (375000, (13, 13, 14), 7),
    (700000, (33, 33, 33), 2), (700000, (34, 33, 33), 2), (700000, (20, 19, 20), 5), (700000, (20, 20, 20), 5),
    (1400000, (33, 34, 33), 3), (1400000, (34, 34, 33), 3), (1900000, (64, 64, 66), 1), (1900000, (65, 65, 65), 1)])
def test_both_sides_of_the_line(line, nel, p):
    assert 0.95 < _face_points(nel, p) / line < 1.07
    c = Case(nel, p, seed=2, bc=("N", "D", "D", "N", "N", "D"))
    try:
        se = c.se
        u = np.random.default_rng(5).uniform(-1, 1, c.lv.gid.shape)
        ref = o.qqt(c.lv, u)
        for mask in (0, 1):
            g = c.to_gpu(u)
            se.se_gs(c.m, g, mask)
            assert rel_err(c.to_np(g), c.lv.mask * ref if mask else ref) <= 1e-14
        uc, y = c.random_continuous(3), c.empty()
        ref = o.ax(c.lv, uc)
        se.se_ax(c.m, c.to_gpu(uc), y, se.SE_AX_ASSEMBLE | se.SE_AX_MASK)
        assert rel_err(c.to_np(y), ref) <= 1e-12
        se.se_ax(c.m, c.to_gpu(uc), y, se.SE_AX_ASSEMBLE | se.SE_AX_MASK | se.SE_AX_FP32)
        assert rel_err(c.to_np(y), ref) <= 2e-5
    finally:
        c.close()
