"""FP32 kernels' elements per block: the sizes that the rules choose (by order, and for the local solves
by the level's elements) give bitwise the results of other sizes, since every element is computed by one
block or warp whatever shares it; ragged last blocks included."""
import pytest

from tests.gpu_common import Case

pytestmark = pytest.mark.gpu


# (19, 17, 16) elements at p = 2: above the local solves' line between the two default sizes
@pytest.mark.parametrize("nel,p", [((3, 3, 3), 1), ((5, 3, 3), 3), ((5, 3, 1), 5), ((3, 3, 3), 7), ((3, 1, 3), 9),
                                   ((3, 3, 3), 6), ((3, 3, 3), 10), ((19, 17, 16), 2)])
def test_fp32_results_independent_of_tile(nel, p):
    c = Case(nel, p, seed=4)
    se, torch = c.se, c.torch
    try:
        P = se.se_pmg_setup(c.m, se.pmg_desc((p, 1), se.SE_SMOOTH_ASM, 1, precision=se.SE_FP32)) if p > 1 else None
        u = c.to_gpu(c.random_continuous(5))
        flags = se.SE_AX_ASSEMBLE | se.SE_AX_FP32
        y0, y1, z0, z1 = c.empty(), c.empty(), c.empty(), c.empty()
        se.se_ax(c.m, u, y0, flags)
        if P is not None:
            se.se_pmg_smooth(P, 0, u, z0)
        for ax_ne, fdm_ne in [(1, 1), (2, 4), (4, 8)]:
            se.se_tune_set(p, se.SE_FP32, ax_ne, fdm_ne)
            se.se_ax(c.m, u, y1, flags)
            assert torch.equal(y0, y1)
            if P is not None:
                se.se_pmg_smooth(P, 0, u, z1)
                assert torch.equal(z0, z1)
        se.se_tune_set(p, se.SE_FP32, 0, 0)
        if P is not None:
            se.se_pmg_destroy(P)
    finally:
        c.close()
