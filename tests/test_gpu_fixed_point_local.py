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


def _transfer(c, pf, pc):
    se = c.se
    P = se.se_pmg_setup(c.m, se.pmg_desc((pf, pc, 1) if pc > 1 else (pf, 1), se.SE_SMOOTH_JACOBI, 1))
    return P, o.make_level(c.V, c.nel, pc, c.lv.bc, c.amp)


PAIRS = [(2, 1), (3, 1), (3, 2), (4, 2), (5, 3), (6, 4), (7, 5), (8, 4), (9, 5), (10, 4), (10, 9), (10, 1)]


@pytest.mark.parametrize("pf,pc", PAIRS)
def test_prolongation_is_continuous_to_the_last_bit(pf, pc):
    """Every copy of an interface point depends on the interface's values alone, by the same operations."""
    c = Case((4, 3, 3), pf, seed=23, bc=("D", "N", "N", "D", "N", "N"))
    try:
        P, lc = _transfer(c, pf, pc)
        ef = c.empty()
        c.se.se_pmg_prolong(P, 0, c.to_gpu(c.random_continuous(8, lv=lc) * np.exp(3.0)), ef)
        got = c.to_np(ef)
        one = np.zeros(c.lv.n_global)
        one[c.lv.gid] = got
        assert np.array_equal(one[c.lv.gid].view(np.int64), got.view(np.int64))
        c.se.se_pmg_destroy(P)
    finally:
        c.close()


@pytest.mark.parametrize("pf,pc", PAIRS)
@pytest.mark.parametrize("spike", [1e4, 1e12])
def test_transfers_away_from_a_large_value(pf, pc, spike):
    """A large value at an element's corner: J's unit rows keep it from the faces opposite to it in the
    prolongation, and from everything but its own node in the restriction; likewise a large value in
    the element's middle where both orders have that point."""
    c = Case((3, 2, 2), pf, seed=24, bc=("N",) * 6)
    try:
        P, lc = _transfer(c, pf, pc)
        rng = np.random.default_rng(pf)
        ec = rng.uniform(-1, 1, lc.gid.shape)
        ec[4, 0, 0, 0] = 0.0
        ref = o.prolong(c.lv, lc, ec)[4]
        ec[4, 0, 0, 0] = spike
        ef, rc = c.empty(), c.empty(lc.gid.size)
        c.se.se_pmg_prolong(P, 0, c.to_gpu(ec), ef)
        got = c.to_np(ef)[4]
        far = np.zeros(got.shape, bool)
        far[-1], far[:, -1], far[:, :, -1] = True, True, True
        assert np.max(np.abs(got - ref)[far]) <= 1e-13 * np.max(np.abs(ref[far]))
        places = [(0, 0, 0)] + ([(pf // 2,) * 3] if pf % 2 == 0 and pc % 2 == 0 else [])
        for at in places:
            rf = rng.uniform(-1, 1, c.lv.gid.shape)
            rf[(4,) + at] = 0.0
            ref_r = o.restrict(c.lv, lc, rf)
            rf[(4,) + at] = spike
            c.se.se_pmg_restrict(P, 0, c.to_gpu(rf), rc)
            got_r = rc.cpu().numpy().reshape(lc.gid.shape)
            node = lc.gid[(4,) + tuple(pc // 2 if q else 0 for q in at)]
            others = lc.gid != node
            assert np.max(np.abs(got_r - ref_r)[others]) <= 1e-13 * np.max(np.abs(ref_r[others]))
        c.se.se_pmg_destroy(P)
    finally:
        c.close()


@pytest.mark.parametrize("pf,pc", PAIRS)
@pytest.mark.parametrize("value", [np.inf, np.nan, 1e-300, 1e-310])
def test_transfers_elements_do_not_share_a_fallback(pf, pc, value):
    c = Case((6, 2, 2), pf, seed=25, bc=("N",) * 6)
    try:
        P, lc = _transfer(c, pf, pc)
        rng = np.random.default_rng(pc)
        ec, rf = rng.uniform(-1, 1, lc.gid.shape), rng.uniform(-1, 1, c.lv.gid.shape)
        out = []
        for put in (False, True):
            if put:
                for a in (ec, rf):
                    a[8] *= 0.0 if abs(value) < 1.0 else 1.0
                    a[8, 0, 1, 0] = value
            ef, rc = c.empty(), c.empty(lc.gid.size)
            c.se.se_pmg_prolong(P, 0, c.to_gpu(ec), ef)
            c.se.se_pmg_restrict(P, 0, c.to_gpu(rf), rc)
            out.append((c.to_np(ef), rc.cpu().numpy().reshape(lc.gid.shape)))
        others = np.arange(c.lv.E) != 8
        assert np.array_equal(out[0][0][others], out[1][0][others])
        # the restriction adds the element's results to its neighbours' copies
        apart = ~np.isin(lc.gid, lc.gid[8])
        assert np.array_equal(out[0][1][apart], out[1][1][apart])
        if abs(value) < 1.0:
            with np.errstate(under="ignore"):
                ref = o.prolong(c.lv, lc, ec)[8]
            assert np.max(np.abs(out[1][0][8] - ref)) <= 1e-13 * np.max(np.abs(ref)) + 2e-323 * 8
        c.se.se_pmg_destroy(P)
    finally:
        c.close()


@pytest.mark.parametrize("pf,pc", [(2, 1), (5, 3), (8, 4), (10, 9)])
@pytest.mark.parametrize("k", [-953, -952, -940, 996])
def test_transfers_of_cancelling_lines_at_the_ends_of_the_range(pf, pc, k):
    """Odd fields, whose contractions cancel, scaled to the ends of the range of the lines' scale."""
    c = Case((3, 2, 2), pf, seed=26, bc=("N",) * 6)
    try:
        P, lc = _transfer(c, pf, pc)
        def odd(lv, seed):
            v = np.random.default_rng(seed).uniform(0.5, 1, lv.gid.shape)
            v = v - v[:, :, :, ::-1] + 1e-9 * (v[:, :, ::-1] - v)
            return v / np.max(np.abs(v))
        ec, rf = odd(lc, 1), odd(c.lv, 2)
        ef, rc = c.empty(), c.empty(lc.gid.size)
        c.se.se_pmg_prolong(P, 0, c.to_gpu(np.ldexp(ec, k)), ef)
        c.se.se_pmg_restrict(P, 0, c.to_gpu(np.ldexp(rf, k)), rc)
        re, rr = o.prolong(c.lv, lc, ec), o.restrict(c.lv, lc, rf)
        assert np.max(np.abs(np.ldexp(c.to_np(ef), -k) - re)) <= 1e-13 * np.max(np.abs(re))
        assert np.max(np.abs(np.ldexp(rc.cpu().numpy().reshape(rr.shape), -k) - rr)) <= 1e-13 * np.max(np.abs(rr))
        c.se.se_pmg_destroy(P)
    finally:
        c.close()


@pytest.mark.parametrize("kind", ["ras", "asm"])
@pytest.mark.parametrize("p", range(2, 11))
@pytest.mark.parametrize("value", [np.inf, np.nan, 1e-300, 1e-315])
def test_schwarz_elements_do_not_share_a_fallback(p, kind, value):
    """Elements far from a window without a scale keep their bits, whatever the number of elements per
    block; the windows without one do not depend on it either."""
    c = Case((8, 2, 2), p, seed=27)
    se = c.se
    try:
        sched = (p, 1) if p < 4 else (p, p // 2, 1)
        P = se.se_pmg_setup(c.m, se.pmg_desc(sched, se.SE_SMOOTH_RAS if kind == "ras" else se.SE_SMOOTH_ASM, 1))
        r = c.random_continuous(p)
        g = np.zeros(c.lv.n_global)
        g[c.lv.gid] = r
        if abs(value) < 1.0:  # alone in its window and in those beside it
            g[np.unique(c.lv.gid[[e for e in range(c.lv.E) if e % 8 <= 2]])] = 0.0
        g[c.lv.gid[1, p // 2, p // 2, p // 2]] = value
        bad = g[c.lv.gid]
        s, t, w = c.empty(), c.empty(), c.empty()
        se.se_pmg_smooth(P, 0, c.to_gpu(r), s)
        se.se_pmg_smooth(P, 0, c.to_gpu(bad), t)
        far = np.array([e % 8 >= (5 if abs(value) < 1.0 else 4) for e in range(c.lv.E)])
        assert np.array_equal(c.to_np(s)[far], c.to_np(t)[far])
        for ne in (1, 2, 3, 4):
            se.se_tune_set(p, se.SE_FP64, 0, ne)
            se.se_pmg_smooth(P, 0, c.to_gpu(bad), w)
            assert np.array_equal(c.to_np(t), c.to_np(w), equal_nan=True)
        se.se_pmg_destroy(P)
    finally:
        se.se_tune_set(p, se.SE_FP64, 0, 0)
        c.close()
