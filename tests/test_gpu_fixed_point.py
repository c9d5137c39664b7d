"""The FP64 kernels in block floating point: every order on meshes whose blocks end inside a row of
elements, values at the ends of the exponent range, elements without a common scale (infinities,
NaN: computed in FP64) and elements of zeros, against the oracle.

Tolerance 1e-12 of the largest entry, as the FP64 operator's tests."""
import numpy as np
import pytest

import oracle as o
from tests.gpu_common import Case, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", range(1, 11))
def test_operator_blocks_ending_inside_rows(p):
    c = Case((5, 3, 3), p, seed=60 + p, bc=("D", "N", "N", "D", "D", "D"))
    try:
        se = c.se
        u, y, r = c.random_continuous(3, masked=False), c.empty(), c.empty()
        se.se_ax(c.m, c.to_gpu(u), y, se.SE_AX_ASSEMBLE | se.SE_AX_MASK)
        assert rel_err(c.to_np(y), o.ax(c.lv, u)) <= 1e-12
        um, b = c.lv.mask * u, c.random_continuous(4)
        se.se_residual(c.m, c.to_gpu(b), c.to_gpu(um), r)
        assert rel_err(c.to_np(r), b - o.ax(c.lv, um)) <= 1e-12
    finally:
        c.close()


@pytest.mark.parametrize("p", [2, 5, 7])
@pytest.mark.parametrize("k", [-1010, -960, -900, 900, 990, 1005])
def test_operator_at_the_ends_of_the_range(p, k):
    """A u for u scaled by 2^k (exact): the same result scaled, on both sides of the range of the
    common scale."""
    c = Case((3, 2, 2), p, seed=5)
    try:
        u, y = c.random_continuous(9), c.empty()
        c.se.se_ax(c.m, c.to_gpu(np.ldexp(u, k)), y)
        assert rel_err(np.ldexp(c.to_np(y), -k), o.ax(c.lv, u)) <= 1e-12
    finally:
        c.close()


@pytest.mark.parametrize("p", [1, 4, 7, 10])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e308, 1e-310])
def test_operator_with_one_unscalable_value(p, value):
    """One value of one element: the local operator is not finite exactly where the plain FP64 one is
    not, and unchanged elsewhere; elements of zeros give zeros."""
    c = Case((4, 3, 2), p, seed=6)
    try:
        u = np.random.default_rng(2).uniform(-1, 1, c.lv.gid.shape)
        u[5] = 0.0
        u[9, p // 2, p, 0] = value
        if value == 1e-310:
            u[9] = 0.0
            u[9, p // 2, p, 0] = value
        y = c.empty()
        c.se.se_ax(c.m, c.to_gpu(u), y, 0)
        with np.errstate(all="ignore"):
            ref = o.ax_local(c.lv, u)
        got = c.to_np(y)
        ok = np.isfinite(ref)
        assert np.array_equal(np.isfinite(got), ok)
        for e in range(c.lv.E):
            scale = np.max(np.abs(ref[e][ok[e]]), initial=0.0)
            assert np.max(np.abs(got[e] - ref[e])[ok[e]], initial=0.0) <= 1e-12 * scale + 5e-324, e
    finally:
        c.close()
