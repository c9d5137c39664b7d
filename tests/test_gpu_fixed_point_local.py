"""What the FP64 kernels in block floating point owe a value to: its own lines only.  A large value leaves
the points that no line through it reaches as accurate as plain FP64 does, and a value without a scale
(infinity, NaN, a magnitude at an end of the range) changes no bit of the elements it does not
belong to, however many elements share a block.

Tolerance 1e-12 of the unaffected values' own largest, as the FP64 operator's tests have for whole fields."""
import numpy as np
import pytest

import oracle as o
from tests.gpu_common import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", range(1, 11))
@pytest.mark.parametrize("spike", [1e4, 1e8, 1e12])
def test_operator_away_from_a_large_value(p, spike):
    """One large value at an element's corner: it reaches the three lines through the corner, and through
    the metric terms there the element's three lower faces; A_L u elsewhere is that of u without it."""
    c = Case((3, 2, 2), p, seed=21)
    try:
        u = np.random.default_rng(p).uniform(-1, 1, c.lv.gid.shape)
        u[4, 0, 0, 0] = 0.0
        ref = o.ax_local(c.lv, u)
        u[4, 0, 0, 0] = spike
        y = c.empty()
        c.se.se_ax(c.m, c.to_gpu(u), y, 0)
        got = c.to_np(y)
        # the corner's own value is 0 in the reference: its lines do not touch what is compared
        far, want = got[4, 1:, 1:, 1:], ref[4, 1:, 1:, 1:]
        assert np.max(np.abs(far - want)) <= 1e-12 * np.max(np.abs(want))
        for e in (3, 5):
            assert np.max(np.abs(got[e] - ref[e])) <= 1e-12 * np.max(np.abs(ref[e]))
    finally:
        c.close()


@pytest.mark.parametrize("p", range(1, 11))
@pytest.mark.parametrize("value", [np.inf, np.nan, 1e-300, 5e-324])
def test_operator_elements_do_not_share_a_fallback(p, value):
    """The other elements' bits with and without an element that has no scale, for every block size."""
    c = Case((4, 3, 2), p, seed=22)
    se, torch = c.se, c.torch
    try:
        u = np.random.default_rng(p).uniform(-1, 1, c.lv.gid.shape)
        v = u.copy()
        v[13] *= 0.0 if abs(value) < 1.0 else 1.0
        v[13, 0, p, 0] = value
        y, z, w = c.empty(), c.empty(), c.empty()
        se.se_ax(c.m, c.to_gpu(u), y, 0)
        se.se_ax(c.m, c.to_gpu(v), z, 0)
        others = np.arange(c.lv.E) != 13
        assert np.array_equal(c.to_np(y)[others], c.to_np(z)[others])
        if abs(value) < 1.0:  # an element of one tiny value: plain FP64's result, not zero
            with np.errstate(under="ignore"):
                ref = o.ax_local(c.lv, v)[13]
            assert np.max(np.abs(c.to_np(z)[13] - ref)) <= 1e-12 * np.max(np.abs(ref)) + 2e-323 * 27
        for ne in (1, 2, 3, 5):
            if ne * (p + 1) ** 2 > 512:
                continue
            se.se_tune_set(p, se.SE_FP64, ne, 0)
            se.se_ax(c.m, c.to_gpu(v), w, 0)
            assert np.array_equal(c.to_np(z).view(np.int64)[others], c.to_np(w).view(np.int64)[others])
            assert np.array_equal(c.to_np(z)[13], c.to_np(w)[13], equal_nan=True)
    finally:
        se.se_tune_set(p, se.SE_FP64, 0, 0)
        c.close()
