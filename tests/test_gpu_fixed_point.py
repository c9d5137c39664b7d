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
            assert np.max(np.abs(got[e][ok[e]] - ref[e][ok[e]]), initial=0.0) <= 1e-12 * scale + 5e-324, e
    finally:
        c.close()


def _smoother(c, p, kind):
    sched = (p, 1) if p < 4 else (p, p // 2, 1)
    c.lv.extra["fdm"] = o.fdm_setup(c.lv, c.V, c.amp)
    se = c.se
    return se.se_pmg_setup(c.m, se.pmg_desc(sched, se.SE_SMOOTH_RAS if kind == "ras" else se.SE_SMOOTH_ASM, 1))


@pytest.mark.parametrize("kind", ["ras", "asm"])
@pytest.mark.parametrize("p", range(2, 11))
def test_schwarz_blocks_and_range(p, kind):
    """Element counts that leave a part of the last block empty; the residual scaled by powers of two
    on both sides of the range of the common scale."""
    c = Case((3, 3, 2) if p > 6 else (4, 3, 3), p, seed=80 + p, bc=("D", "D", "N", "D", "D", "N"))
    try:
        P = _smoother(c, p, kind)
        r, s = c.random_continuous(5), c.empty()
        ref = (o.ras if kind == "ras" else o.asm)(c.lv, r)
        for k in (0, -985, -955, -800, 800, 990):
            c.se.se_pmg_smooth(P, 0, c.to_gpu(np.ldexp(r, k)), s)
            assert rel_err(np.ldexp(c.to_np(s), -k), ref) <= 1e-10, k
        c.se.se_pmg_destroy(P)
    finally:
        c.close()


@pytest.mark.parametrize("kind", ["ras", "asm"])
@pytest.mark.parametrize("p,value", [(3, np.inf), (7, np.nan), (8, -np.inf)])
def test_schwarz_with_one_unscalable_value(p, kind, value):
    """The smoother is not finite exactly where the plain FP64 one is not; zeros stay zeros."""
    c = Case((5, 3, 2), p, seed=7)
    try:
        P = _smoother(c, p, kind)
        g = np.random.default_rng(3).uniform(-1, 1, c.lv.n_global)
        g[c.lv.gid[0]] = 0.0
        g[c.lv.gid[14, p // 2, p // 2, p // 2]] = value
        r, s = o.from_global(c.lv, g), c.empty()
        r = np.where(c.lv.mask > 0, r, 0.0)
        with np.errstate(all="ignore"):
            ref = (o.ras if kind == "ras" else o.asm)(c.lv, r)
        ref = np.where(c.lv.mask > 0, ref, 0.0)
        c.se.se_pmg_smooth(P, 0, c.to_gpu(r), s)
        got = c.to_np(s)
        ok = np.isfinite(ref)
        assert not ok.all() and ok.any()
        assert np.array_equal(np.isfinite(got)[c.lv.mask > 0], ok[c.lv.mask > 0])
        scale = np.max(np.abs(ref[ok]))
        both = ok & (c.lv.mask > 0)
        assert np.max(np.abs(got[both] - ref[both])) <= 1e-10 * scale
        c.se.se_pmg_smooth(P, 0, c.to_gpu(np.zeros_like(r)), s)
        assert not c.to_np(s).any()
        c.se.se_pmg_destroy(P)
    finally:
        c.close()


@pytest.mark.parametrize("pf,pc", [(2, 1), (4, 2), (7, 5), (8, 7), (9, 4), (10, 9), (10, 1)])
def test_transfers_range_and_unscalable_values(pf, pc):
    """Both transfers, scaled by powers of two on both sides of the range of the common scale, and with
    one value that has no scale: not finite exactly where plain FP64 is not."""
    c = Case((5, 3, 2), pf, seed=8)
    try:
        se = c.se
        lc = o.make_level(c.V, c.nel, pc, c.lv.bc, c.amp)
        P = se.se_pmg_setup(c.m, se.pmg_desc((pf, pc, 1) if pc > 1 else (pf, 1), se.SE_SMOOTH_JACOBI, 1))
        rf, ec = c.random_continuous(6), c.random_continuous(7, lv=lc)
        rc, ef = c.empty(lc.gid.size), c.empty()
        ref_r, ref_e = o.restrict(c.lv, lc, rf), o.prolong(c.lv, lc, ec)
        for k in (0, -1005, -955, 900, 1005):
            se.se_pmg_restrict(P, 0, c.to_gpu(np.ldexp(rf, k)), rc)
            se.se_pmg_prolong(P, 0, c.to_gpu(np.ldexp(ec, k)), ef)
            assert rel_err(np.ldexp(rc.cpu().numpy().reshape(ref_r.shape), -k), ref_r) <= 1e-13, k
            assert rel_err(np.ldexp(c.to_np(ef), -k), ref_e) <= 1e-13, k
        for value in (np.inf, np.nan):
            bad = ec.copy()
            bad[7, 0, pc, 0] = value
            se.se_pmg_prolong(P, 0, c.to_gpu(bad), ef)
            with np.errstate(all="ignore"):
                ref = o.prolong(c.lv, lc, bad)
            ok = np.isfinite(ref)
            got = c.to_np(ef)
            # every value of the element depends on it (0 inf is NaN in plain FP64 too)
            assert np.array_equal(np.isfinite(got), ok) and not ok[7].any() and ok[8].all()
            assert np.max(np.abs(got[ok] - ref[ok])) <= 1e-13 * np.max(np.abs(ref[ok]))
        se.se_pmg_destroy(P)
    finally:
        c.close()


@pytest.mark.parametrize("nel,p", [((1, 1, 1), 3), ((1, 4, 3), 2), ((5, 1, 2), 7), ((7, 6, 1), 4), ((9, 5, 4), 1),
                                   ((30, 29, 31), 2), ((11, 12, 11), 7), ((16, 15, 14), 7)])
@pytest.mark.parametrize("bc", [("D",) * 6, ("N", "D", "D", "N", "N", "N")])
def test_qqt_one_launch_and_sweeps(nel, p, bc):
    """QQ^T with and without the mask on lattices one element wide in each direction, and on both sides
    of the size where the one-launch form gives way to the sweeps; FP32 within one rounding per sum."""
    c = Case(nel, p, seed=1, bc=bc)
    try:
        u = np.random.default_rng(4).uniform(-1, 1, c.lv.gid.shape)
        for mask in (0, 1):
            g = c.to_gpu(u)
            c.se.se_gs(c.m, g, mask)
            ref = o.qqt(c.lv, u)
            if mask:
                ref = c.lv.mask * ref
            assert rel_err(c.to_np(g), ref) <= 1e-14
        y = c.empty()
        c.se.se_ax(c.m, c.to_gpu(u), y, c.se.SE_AX_ASSEMBLE | c.se.SE_AX_MASK | c.se.SE_AX_FP32)
        assert rel_err(c.to_np(y), o.ax(c.lv, u)) <= 2e-5
    finally:
        c.close()
