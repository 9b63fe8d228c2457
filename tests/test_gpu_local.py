"""Group expansions of the list form (mixed precision) on dense states, against
the oracle and against the pair-by-pair list form; the sizes where the finish
kernel changes its targets per CTA, the FP64 point-vortex shortcut and the
chunked vorticity kernel, against the oracle or the full evaluation.

Tolerances: mixed right-hand sides as everywhere (the FP32 jet's rounding,
5e-6 up to order 6, growing with the order); FP64 1e-12 against the oracle.
Dropping terms below 2^-54 of a jet entry changes an FP64 sum by less than its
rounding, so the shortcut is held to 1e-12 of the full jet too.
"""
import numpy as np
import pytest

import mmvm_inputs
from oracle.diagnostics import vorticity
from oracle.rhs import lam_at, rhs_regrouped
from tests.parity_util import (abs_scale_rows, rhs_error_cond, rhs_error_rows, vel_error,
                               vel_error_cond, vel_error_rows)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mm():
    import paper_1010_2475_gb300 as mm

    mm.load_library()
    return mm


def _dense(n, order, seed):
    """Two patches with ~30 particles per squared core unit: most groups of 32
    are narrower than the expansions' limit."""
    wl = mmvm_inputs.two_patches(n=n, order=order, sigma=0.5, seed=seed)
    if order >= 2:
        rng = np.random.default_rng(seed + 1)
        wl.moments[:, 3:] = rng.normal(size=wl.moments[:, 3:].shape) * 1e-2 \
            * wl.moments[:, :1] * wl.lam0 ** 2
    return wl


# ragged last group, one particle in the last group, one group exactly, coincident centres
@pytest.mark.parametrize("order,n", [(0, 1505), (1, 1504), (2, 1537), (3, 1501), (4, 1999),
                                     (5, 1505), (6, 2017), (6, 32), (7, 1505), (8, 1601)])
def test_group_expansions(mm, order, n, monkeypatch):
    wl = _dense(n, order, 300 + order)
    wl.x[7] = wl.x[8]  # a separation of zero
    nd, nl = mm.pair_variant_counts(order)
    res, work = {}, {}
    for v in (nd, nd + nl - 1):
        monkeypatch.setenv("MMVM_PAIR_VARIANT", str(v))
        for local in ("0", "1"):
            monkeypatch.setenv("MMVM_LOCAL", local)
            monkeypatch.setenv("MMVM_FAR_TREE", "1")
            with mm.Context(order, wl.lam0, wl.nu, mm.MMVM_MIXED_FP32) as ctx:
                ctx.set_state(wl.x, wl.moments, 0.0)
                res[v, local] = ctx.rhs()
                work[v, local] = mm.mmvm_pair_work(ctx.handle)
            near, far_pp, n_m2p, m2p_pairs = work[v, local]
            assert near + far_pp + m2p_pairs == n * n
    rows = np.array(sorted({0, 7, 8, n - 1, *np.random.default_rng(2).choice(n, min(n, 12),
                                                                             replace=False)}))
    ox, oM = rhs_regrouped(wl.x, wl.moments, 0.0, order, wl.lam0, wl.nu, rows=rows)
    sx, sM = abs_scale_rows(wl.x, wl.moments, 0.0, order, wl.lam0, wl.nu, rows)
    tol = 5e-6 * max(1.0, order / 6.0)
    for key, (gx, gM) in res.items():
        assert vel_error_cond(gx[rows], ox, sx) <= tol, key
        if order >= 1:
            assert rhs_error_cond(gM[rows], oM, sM, order, wl.lam0) <= tol, key
    if n > 1000:  # the expansions were really used: other roundings
        assert any(not np.array_equal(res[nd, "0"][i], res[nd, "1"][i]) for i in range(2))


@pytest.mark.parametrize("order,shape,per", [(2, "even", 1), (2, "even", 16), (4, "even", 3),
                                             (6, "uneven", 1), (6, "uneven", 16), (3, "tiny", 16),
                                             (8, "uneven", 4)])
def test_near_shares(mm, order, shape, per, monkeypatch):
    """Near pairs in equal shares: groups cut anywhere, a share of many groups,
    one group in as many shares as it may fall into, more CTAs than shares."""
    n = {"even": 1203, "uneven": 1501, "tiny": 33}[shape]
    wl = mmvm_inputs.random_disk(n=n, order=order, radius=6.0, sigma=0.5, seed=80 + order)
    if shape == "uneven":  # long lists in one corner, short ones elsewhere
        wl.x[:500] = wl.x[:500] * 0.3
        wl.x[500:] = wl.x[500:] * 12.0
    nd, nl = mm.pair_variant_counts(order)
    rows = np.array(sorted({0, n - 1, *range(1, n, max(1, n // 12))}))
    ox, oM = rhs_regrouped(wl.x, wl.moments, 0.0, order, wl.lam0, wl.nu, rows=rows)
    sx, sM = abs_scale_rows(wl.x, wl.moments, 0.0, order, wl.lam0, wl.nu, rows)
    tol = 5e-6 * max(1.0, order / 6.0)
    monkeypatch.setenv("MMVM_LIST_SEGMENTS", str(per))
    for v in range(nd, nd + nl):
        monkeypatch.setenv("MMVM_PAIR_VARIANT", str(v))
        with mm.Context(order, wl.lam0, wl.nu, mm.MMVM_MIXED_FP32) as ctx:
            ctx.set_state(wl.x, wl.moments, 0.0)
            gx, gM = ctx.rhs()
            near, far_pp, n_m2p, m2p_pairs = mm.mmvm_pair_work(ctx.handle)
        assert near + far_pp + m2p_pairs == n * n
        assert vel_error_cond(gx[rows], ox, sx) <= tol
        assert rhs_error_cond(gM[rows], oM, sM, order, wl.lam0) <= tol


# groups of radius 0.6 to 1.2 core sizes, where the remainder of the Gaussian
# part's Taylor series sets the least separation
@pytest.mark.parametrize("order,kind,n", [(4, "patches", 20000), (5, "patches", 20000),
                                          (6, "disk", 16000), (6, "patches", 20000),
                                          (7, "disk", 16000), (8, "disk", 30011)])
def test_expansions_of_moderate_groups(mm, order, kind, n, monkeypatch):
    """No particle's velocity further off than the far field's bound (2e-6 of
    the largest velocity) against the FP64 form."""
    if kind == "patches":
        wl = mmvm_inputs.two_patches(n=n, order=order, sigma=0.1, seed=600 + order)
    else:
        wl = mmvm_inputs.random_disk(n=n, order=order, radius=10.0, sigma=0.5, seed=n)
    wl.moments[:, 3:] = np.random.default_rng(order).normal(size=wl.moments[:, 3:].shape) \
        * 1e-3 * wl.moments[:, :1] * wl.lam0 ** 2
    monkeypatch.setenv("MMVM_PAIR_VARIANT", str(mm.pair_variant_counts(order)[0]))
    monkeypatch.setenv("MMVM_FAR_TREE", "1")
    monkeypatch.setenv("MMVM_LOCAL", "1")
    with mm.Context(order, wl.lam0, wl.nu, mm.MMVM_MIXED_FP32) as ctx:
        ctx.set_state(wl.x, wl.moments, 0.0)
        gx = ctx.rhs()[0]
    monkeypatch.delenv("MMVM_PAIR_VARIANT")
    with mm.Context(order, wl.lam0, wl.nu, mm.MMVM_FP64) as ctx:
        ctx.set_state(wl.x, wl.moments, 0.0)
        rx = ctx.rhs()[0]
    assert vel_error(gx, rx) <= 2e-6


@pytest.mark.parametrize("groups", [1, 2, 3, 64, 65, 127, 128, 129, 130, 258])
def test_tree_levels(mm, groups, monkeypatch):
    """The levels built by one CTA (at most 64 nodes) and those below it, full
    and ragged; every group range against the same groups without a tree."""
    n, order = 32 * groups - 5, 3
    wl = mmvm_inputs.two_patches(n=n, order=order, sigma=0.1, seed=groups)
    wl.moments[:, 3:] = np.random.default_rng(groups).normal(size=wl.moments[:, 3:].shape) \
        * 1e-2 * wl.moments[:, :1] * wl.lam0 ** 2
    nd, nl = mm.pair_variant_counts(order)
    monkeypatch.setenv("MMVM_PAIR_VARIANT", str(nd + nl - 1))
    rows = np.array(sorted({0, n // 2, n - 1, *range(max(0, n - 40), n, 8)}))
    ox, oM = rhs_regrouped(wl.x, wl.moments, 0.0, order, wl.lam0, wl.nu, rows=rows)
    sx, sM = abs_scale_rows(wl.x, wl.moments, 0.0, order, wl.lam0, wl.nu, rows)
    for tree, local in (("1", "1"), ("1", "0"), ("0", "1")):
        monkeypatch.setenv("MMVM_FAR_TREE", tree)
        monkeypatch.setenv("MMVM_LOCAL", local)
        with mm.Context(order, wl.lam0, wl.nu, mm.MMVM_MIXED_FP32) as ctx:
            ctx.set_state(wl.x, wl.moments, 0.0)
            gx, gM = ctx.rhs()
            near, far_pp, n_m2p, m2p_pairs = mm.mmvm_pair_work(ctx.handle)
        assert near + far_pp + m2p_pairs == n * n
        assert vel_error_cond(gx[rows], ox, sx) <= 5e-6
        assert rhs_error_cond(gM[rows], oM, sM, order, wl.lam0) <= 5e-6


@pytest.mark.parametrize("n", [1, 2, 2431, 2433, 4865, 9729, 19457])
def test_finish_shapes(mm, n):
    """One and many targets per finish CTA, full and ragged."""
    wl = mmvm_inputs.random_disk(n=n, order=3, radius=4.0, seed=n) if n > 1 else \
        mmvm_inputs.single_quadrupole(order=3)
    with mm.Context(3, wl.lam0, wl.nu, mm.MMVM_FP64) as ctx:
        ctx.set_state(wl.x, wl.moments, 0.3)
        gx, gM = ctx.rhs()
    rows = np.array(sorted({0, n - 1, n // 2, *range(max(0, n - 3), n)}))
    ox, oM = rhs_regrouped(wl.x, wl.moments, 0.3, 3, wl.lam0, wl.nu, rows=rows)
    lam = lam_at(0.3, wl.lam0, wl.nu)
    if n > 1:
        assert vel_error_rows(gx[rows], ox) <= 1e-12
    assert rhs_error_rows(gM[rows], oM, 3, lam) <= 1e-12


# the group-sorted moment table at 1, 2, 4 and 8 targets per CTA, ragged tails
@pytest.mark.parametrize("order,n", [(0, 1826), (1, 3655), (2, 1), (5, 911), (6, 3651), (6, 913),
                                     (7, 1825), (7, 3650), (8, 2), (8, 1827)])
def test_finish_groups(mm, order, n):
    wl = mmvm_inputs.random_disk(n=n, order=order, radius=4.0, seed=n) if n > 1 else \
        mmvm_inputs.single_quadrupole(order=order)
    with mm.Context(order, wl.lam0, wl.nu, mm.MMVM_FP64) as ctx:
        ctx.set_state(wl.x, wl.moments, 0.3)
        gx, gM = ctx.rhs()
    rows = np.array(sorted({0, n - 1, n // 2, *range(max(0, n - 3), n)}))
    ox, oM = rhs_regrouped(wl.x, wl.moments, 0.3, order, wl.lam0, wl.nu, rows=rows)
    sx, sM = abs_scale_rows(wl.x, wl.moments, 0.3, order, wl.lam0, wl.nu, rows)
    if n > 1:
        assert vel_error_cond(gx[rows], ox, sx) <= 1e-12
    if order >= 1 and n > 1:
        assert rhs_error_cond(gM[rows], oM, sM, order, lam_at(0.3, wl.lam0, wl.nu)) <= 1e-12
    elif order >= 1:
        assert rhs_error_rows(gM[rows], oM, order, lam_at(0.3, wl.lam0, wl.nu)) <= 1e-12


@pytest.mark.parametrize("order", range(9))
def test_fp64_shortcut_matches_full_jet(mm, order):
    wl = mmvm_inputs.two_patches(n=513, order=order, sigma=0.1, seed=40 + order)
    if order >= 2:
        rng = np.random.default_rng(order)
        wl.moments[:, 3:] = rng.normal(size=wl.moments[:, 3:].shape) * 1e-2 \
            * wl.moments[:, :1] * wl.lam0 ** 2
    res = []
    for flags in (0, mm.MMVM_FLAG_NO_FAR_FIELD):
        with mm.Context(order, wl.lam0, wl.nu, mm.MMVM_FP64, flags=flags) as ctx:
            ctx.set_state(wl.x, wl.moments, 0.0)
            res.append(ctx.rhs())
    assert vel_error_rows(res[0][0], res[1][0]) <= 1e-12
    if order >= 2:  # first moments are conserved: at order 1 the rate is 0 up to rounding
        assert rhs_error_rows(res[0][1], res[1][1], order, wl.lam0) <= 1e-12


@pytest.mark.parametrize("order,n,npts", [(0, 2049, 5), (4, 1100, 517), (8, 700, 129), (9, 1, 130)])
def test_vorticity_chunks(mm, order, n, npts):
    wl = mmvm_inputs.random_disk(n=n, order=order, radius=9.0, sigma=0.5, amp=0.05, seed=order)
    pts = np.random.default_rng(order).uniform(-12.0, 12.0, size=(npts, 2))
    with mm.Context(order, wl.lam0, wl.nu, mm.MMVM_FP64) as ctx:
        ctx.set_state(wl.x, wl.moments, 0.0)
        g = ctx.vorticity(pts)
    o = vorticity(wl.x, wl.moments, wl.lam0, order, pts)
    assert np.abs(g - o).max() <= 1e-12 * np.abs(o).max()
