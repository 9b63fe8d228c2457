"""States at the limits of the approximations, in the mixed and the FP64 form:
far from the origin, groups on a line, a strong vortex at the facing end of a
group, domains many core sizes wide, tiny circulations.

References are the FP64 form (fewer than 256 particles, or the full-jet flag:
no approximation) or the oracle.  Tolerances, unless stated at a test: mixed
velocities 2e-6 and moment rates 5e-6 (growing with the order beyond 6) as
everywhere, each particle against the scale of its own pair terms; FP64 1e-12.
"""
import math

import numpy as np
import pytest

import mmvm_inputs
from oracle.rhs import rhs_regrouped
from tests.parity_util import (abs_scale_rows, rhs_error, rhs_error_cond, rhs_error_rows,
                               vel_error, vel_error_cond, vel_error_rows, weights)

pytestmark = pytest.mark.gpu

X_FAR = (20.0, 32.0, 40.0, 50.0, 58.0, 66.0, 74.0, 80.0, 88.0)  # near/far threshold by order
LAM = math.sqrt(0.5)  # core units are the units of length


@pytest.fixture(scope="module")
def mm():
    import paper_1010_2475_gb300 as mm

    mm.load_library()
    return mm


def _rhs(mm, order, lam, x, m, precision, flags=0):
    with mm.Context(order, lam, 1e-3, precision, flags=flags) as ctx:
        ctx.set_state(x, m, 0.0)
        return ctx.rhs()


def _moments(gamma, order, lam, rng, amp=0.1):
    """Circulations gamma, moments of order >= 2 `amp` of them in the weighted norm."""
    m = np.zeros((len(gamma), mmvm_inputs.n_moments(order)))
    m[:, 0] = gamma
    if order >= 2:
        m[:, 3:] = amp * rng.normal(size=m[:, 3:].shape) * gamma[:, None] \
            / np.sqrt(weights(order, lam)[3:])
    return m


def _tol(order):
    return 5e-6 * max(1.0, order / 6.0)


@pytest.mark.parametrize("order", [0, 2, 4, 6, 8])
@pytest.mark.parametrize("state", ["disk", "patches", "clusters"])
def test_fp64_shortcut_far_from_the_origin(mm, order, state):
    """The test for the point-vortex form works on differences of positions:
    at 2e8 units one FP32 step of a coordinate is 16 units, wider than the far
    threshold.  `clusters`: the targets of one warp lie in several clusters 1e8
    units apart, each around a value half way between two FP32 numbers."""
    rng = np.random.default_rng(order)
    n = 504
    if state == "disk":
        x = 8.0 * rng.uniform(-1.0, 1.0, size=(n, 2)) + [2e8 + 8.0, -2e8]
    elif state == "patches":
        x = mmvm_inputs.two_patches(n=n, order=order, sigma=0.1, seed=order).x * 7.0 + [-4e8, 3e6]
    else:
        x = 4.0 * rng.uniform(-1.0, 1.0, size=(n, 2))
        c = (2.0 ** 27 * (1 + np.arange(24))).astype(np.float32)
        x[:, 0] += np.repeat(c.astype(np.float64) + 0.5 * np.spacing(c), 21)
    m = _moments(rng.normal(size=n), order, LAM, rng)
    gx, gM = _rhs(mm, order, LAM, x, m, mm.MMVM_FP64)
    rx, rM = _rhs(mm, order, LAM, x, m, mm.MMVM_FP64, mm.MMVM_FLAG_NO_FAR_FIELD)
    assert vel_error_rows(gx, rx) <= 1e-12
    if order >= 2:
        assert rhs_error_rows(gM, rM, order, LAM) <= 1e-12


@pytest.mark.parametrize("order", range(9))
def test_strong_vortex_at_the_facing_end(mm, order, monkeypatch):
    """Two groups on a line, a strong vortex at the end of one that faces the
    other, at radii and separations through the whole range of the near
    expansions: where a group expansion converges worst, whoever of the pair
    kernels and the expansions takes the pair."""
    widest = (2.0, 2.0, 2.0, 1.8, 1.8, 1.6, 1.7, 1.1, 0.85)[order]
    rng = np.random.default_rng(order)
    monkeypatch.setenv("MMVM_LOCAL", "1")
    monkeypatch.setenv("MMVM_FAR_TREE", "0")
    variant = str(mm.pair_variant_counts(order)[0])
    rows = np.arange(32, 64)
    expanded = 0
    for r in widest * np.array([0.4, 0.55, 0.7, 0.85, 0.999]):
        sep = max(8.0, (2.0 * r + 0.2) ** 2) * 1.001
        while sep < 90.0:
            s = math.sqrt(sep)
            x = rng.uniform(-0.6, 0.6, size=(64, 2)) * [r, 0.2 * r]
            for k in (0, 32):
                x[k], x[k + 1] = [r, 0.0], [-r, 0.0]
                x[k + 2], x[k + 3] = [0.0, 0.15 * r], [0.0, -0.15 * r]
            x[32:, 0] += s
            g = 1e-6 * (1.0 + rng.random(64))
            g[0] = 1.0
            m = _moments(g, order, LAM, rng)
            monkeypatch.delenv("MMVM_PAIR_VARIANT", raising=False)
            rx, rM = _rhs(mm, order, LAM, x, m, mm.MMVM_FP64)
            monkeypatch.setenv("MMVM_PAIR_VARIANT", variant)
            with mm.Context(order, LAM, 1e-3, mm.MMVM_MIXED_FP32) as ctx:
                ctx.set_state(x, m, 0.0)
                gx, gM = ctx.rhs()
                expanded += mm.mmvm_pair_expanded(ctx.handle)
            assert vel_error_rows(gx[rows], rx[rows]) <= 2e-6, (r, sep)
            if order >= 1:
                sM = abs_scale_rows(x, m, 0.0, order, LAM, 1e-3, rows[:8], procs=1)[1]
                assert rhs_error_cond(gM[rows[:8]], rM[rows[:8]], sM, order, LAM) \
                    <= _tol(order), (r, sep)
            sep *= 1.12
    assert expanded > 0


# groups as wide as the expansions' limits: n sets the radius
@pytest.mark.parametrize("order,n", [(0, 4001), (1, 5003), (2, 5003), (2, 12001), (3, 6007),
                                     (4, 9001), (5, 9001), (6, 9001), (6, 16001), (7, 16001),
                                     (8, 30011)])
def test_rates_of_moderate_groups(mm, order, n, monkeypatch):
    """Velocities within 2e-6 of the largest and moment rates within the mixed
    tolerance of the largest against the FP64 form; one vortex of 50 is 100
    times as strong as the others.  The pairs really went through the expansions."""
    rng = np.random.default_rng(n + order)
    wl = mmvm_inputs.random_disk(n=n, order=order, radius=10.0, sigma=0.5, seed=n + order)
    g = np.where(rng.random(n) < 0.02, 100.0, 1.0) * rng.normal(size=n)
    m = _moments(g, order, wl.lam0, rng, 0.01)
    rx, rM = _rhs(mm, order, wl.lam0, wl.x, m, mm.MMVM_FP64)
    monkeypatch.setenv("MMVM_PAIR_VARIANT", str(mm.pair_variant_counts(order)[0]))
    monkeypatch.setenv("MMVM_FAR_TREE", "1")
    for local in ("0", "1"):
        monkeypatch.setenv("MMVM_LOCAL", local)
        with mm.Context(order, wl.lam0, 1e-3, mm.MMVM_MIXED_FP32) as ctx:
            ctx.set_state(wl.x, m, 0.0)
            gx, gM = ctx.rhs()
            expanded = mm.mmvm_pair_expanded(ctx.handle)
        assert (expanded > 0) == (local == "1")
        assert vel_error(gx, rx) <= 2e-6
        if order >= 2:  # first moments are conserved: at order 1 the rate is 0 up to rounding
            assert rhs_error(gM, rM, order, wl.lam0) <= _tol(order)


@pytest.mark.parametrize("order", range(9))
@pytest.mark.parametrize("frac", [0.7, 0.85, 0.99, 1.05])
def test_far_field_of_line_groups(mm, order, frac, monkeypatch):
    """A target group on a line (half length up to the widest that may take a
    local field) and one strong vortex just beyond the far threshold beside it: the
    group's box has no width, so the source is as close to its centre as the
    threshold.  Velocities to 5e-7: a truncation at FP32 rounding (1e-7) and
    the rounding of a far field."""
    r = (2.0, 2.3, 2.5, 2.8, 3.0, 3.2, 3.4, 3.4, 3.2)[order] * frac
    D = math.sqrt(X_FAR[order]) * 1.002
    rng = np.random.default_rng(10 * order + int(10 * frac))
    x = np.zeros((64, 2))
    x[:32, 1] = np.linspace(-r, r, 32)
    x[32:] = rng.uniform(0.0, 0.02, size=(32, 2)) + [D, -0.01]
    g = 1e-6 * (1.0 + rng.random(64))
    g[32] = 1.0
    m = _moments(g, order, LAM, rng)
    monkeypatch.setenv("MMVM_PAIR_VARIANT", str(mm.pair_variant_counts(order)[0]))
    monkeypatch.setenv("MMVM_LOCAL", "1")
    rows = np.arange(32)
    rx, rM = _rhs(mm, order, LAM, x, m, mm.MMVM_FP64)
    sM = abs_scale_rows(x, m, 0.0, order, LAM, 1e-3, rows, procs=1)[1] if order else None
    for tree in ("0", "1"):
        monkeypatch.setenv("MMVM_FAR_TREE", tree)
        gx, gM = _rhs(mm, order, LAM, x, m, mm.MMVM_MIXED_FP32)
        assert vel_error_rows(gx[rows], rx[rows]) <= 5e-7
        if order >= 1:
            assert rhs_error_cond(gM[rows], rM[rows], sM, order, LAM) <= _tol(order)


@pytest.mark.parametrize("order", range(9))
def test_far_nodes_of_local_fields(mm, order, monkeypatch):
    """One strong vortex at the edge of its group that faces a compact target
    group, at every distance from the far threshold on: the widest source
    groups that are taken through their expansions.  Velocities to 5e-7 as above."""
    rng = np.random.default_rng(order)
    monkeypatch.setenv("MMVM_LOCAL", "1")
    monkeypatch.setenv("MMVM_FAR_TREE", "0")
    rows = np.arange(32)
    for ratio in (0.1, 0.14, 0.17, 0.195, 0.21):  # radius / distance of the source group
        for gap in (1.01, 1.5):
            D = math.sqrt(X_FAR[order]) * gap
            r = ratio / (1.0 - ratio) * (D + 0.2)
            x = rng.uniform(-0.1, 0.1, size=(64, 2))
            x[32:] = rng.uniform(-0.6, 0.6, size=(32, 2)) * r + [D + 0.1 + r, 0.0]
            x[32], x[33] = [D + 0.1, 0.0], [D + 0.1 + 2.0 * r, 0.0]
            x[34], x[35] = [D + 0.1 + r, 0.6 * r], [D + 0.1 + r, -0.6 * r]
            g = 1e-6 * (1.0 + rng.random(64))
            g[32] = 1.0
            m = _moments(g, order, LAM, rng)
            monkeypatch.delenv("MMVM_PAIR_VARIANT", raising=False)
            rx, rM = _rhs(mm, order, LAM, x, m, mm.MMVM_FP64)
            monkeypatch.setenv("MMVM_PAIR_VARIANT", str(mm.pair_variant_counts(order)[0]))
            gx, gM = _rhs(mm, order, LAM, x, m, mm.MMVM_MIXED_FP32)
            assert vel_error_rows(gx[rows], rx[rows]) <= 5e-7, (ratio, gap)
            if order >= 1:
                sM = abs_scale_rows(x, m, 0.0, order, LAM, 1e-3, rows, procs=1)[1]
                assert rhs_error_cond(gM[rows], rM[rows], sM, order, LAM) <= _tol(order)


@pytest.mark.parametrize("order", range(9))
@pytest.mark.parametrize("sparse", [False, True])
def test_domains_many_core_sizes_wide(mm, order, sparse, monkeypatch):
    """Source groups and tree nodes whose expansions would leave the FP32 range:
    64 clusters of 32, each 2e3 units wide, over 2e5 units, with (and without) tight
    groups of targets among them."""
    rng = np.random.default_rng(order)
    n = 2048
    c = 2e5 * rng.uniform(-1.0, 1.0, size=(64, 2))
    w = np.where(np.arange(64) % 4 == 0, 2e3 if sparse else 0.5, 2e3)
    x = np.repeat(c, 32, axis=0) + np.repeat(w, 32)[:, None] * rng.uniform(-0.5, 0.5, size=(n, 2))
    m = _moments(rng.normal(size=n), order, LAM, rng)
    rows = np.arange(0, n, 97)
    ox, oM = rhs_regrouped(x, m, 0.0, order, LAM, 1e-3, rows=rows)
    sx, sM = abs_scale_rows(x, m, 0.0, order, LAM, 1e-3, rows, procs=1)
    nd, nl = mm.pair_variant_counts(order)
    for v, tree, local in ((0, "0", "0"), (nd, "0", "0"), (nd, "1", "0"), (nd, "0", "1"),
                           (nd + nl - 1, "1", "1")):
        monkeypatch.setenv("MMVM_PAIR_VARIANT", str(v))
        monkeypatch.setenv("MMVM_FAR_TREE", tree)
        monkeypatch.setenv("MMVM_LOCAL", local)
        gx, gM = _rhs(mm, order, LAM, x, m, mm.MMVM_MIXED_FP32)
        assert np.isfinite(gx).all() and np.isfinite(gM).all(), (v, tree, local)
        assert vel_error_cond(gx[rows], ox, sx) <= 2e-6, (v, tree, local)
        if order >= 1:
            assert rhs_error_cond(gM[rows], oM, sM, order, LAM) <= _tol(order), (v, tree, local)


@pytest.mark.parametrize("order", [0, 2, 6])
def test_clusters_beyond_the_range_of_squared_distances(mm, order, monkeypatch):
    """Two clusters 1e20 units apart do not see each other."""
    rng = np.random.default_rng(order)
    n = 192
    x = rng.uniform(-1.0, 1.0, size=(n, 2))
    m = _moments(rng.normal(size=n), order, LAM, rng)
    nd, nl = mm.pair_variant_counts(order)
    for v, tree, local in ((0, "0", "0"), (nd, "0", "0"), (nd, "1", "0"), (nd, "0", "1"),
                           (nd, "1", "1")):
        monkeypatch.setenv("MMVM_PAIR_VARIANT", str(v))
        monkeypatch.setenv("MMVM_FAR_TREE", tree)
        monkeypatch.setenv("MMVM_LOCAL", local)
        far = x.copy()
        far[96:] += [1e20, 0.0]
        gx, gM = _rhs(mm, order, LAM, far, m, mm.MMVM_MIXED_FP32)
        ox, oM = rhs_regrouped(x[:96], m[:96], 0.0, order, LAM, 1e-3)
        sx, sM = abs_scale_rows(x[:96], m[:96], 0.0, order, LAM, 1e-3, np.arange(96), procs=1)
        assert vel_error_cond(gx[:96], ox, sx) <= 2e-6, (v, tree, local)
        if order >= 1:
            assert rhs_error_cond(gM[:96], oM, sM, order, LAM) <= _tol(order), (v, tree, local)


@pytest.mark.parametrize("first", ["sparse", "dense"])
def test_expansions_follow_the_state(mm, first):
    """Whether compact groups take expansions depends on the state, not on
    the state that the first context of the size class held."""
    order, n = (5, 9001) if first == "sparse" else (3, 9001)
    rng = np.random.default_rng(order)
    out = {}
    for state in (first, {"sparse": "dense", "dense": "sparse"}[first]):
        x = rng.uniform(-1.0, 1.0, size=(n, 2)) * (2000.0 if state == "sparse" else 10.0)
        m = _moments(rng.normal(size=n), order, LAM, rng)
        with mm.Context(order, LAM, 1e-3, mm.MMVM_MIXED_FP32) as ctx:
            ctx.set_state(x, m, 0.0)
            ctx.rhs()
            out[state] = mm.mmvm_pair_expanded(ctx.handle)
    assert out["dense"] > 0 and out["sparse"] == 0


@pytest.mark.parametrize("n", [2, 300])
@pytest.mark.parametrize("order", [0, 2])
def test_circulation_without_a_reciprocal(mm, order, n):
    """A circulation below 2^-1024 has no finite reciprocal; its velocity is that
    of any other particle there."""
    rng = np.random.default_rng(n)
    x = rng.uniform(-1.0, 1.0, size=(n, 2))
    m = _moments(rng.normal(size=n), order, LAM, rng, 0.0)
    m[0] = 0.0
    m[0, 0] = 4e-309
    gx, gM = _rhs(mm, order, LAM, x, m, mm.MMVM_FP64)
    m[0, 0] = 1e-200
    rx, rM = _rhs(mm, order, LAM, x, m, mm.MMVM_FP64)
    assert np.isfinite(gx).all() and np.isfinite(gM).all()
    assert vel_error_rows(gx, rx) <= 1e-12  # 4e-309 keeps 49 bits; products with it round at 5e-324
