"""Skill moments on the GPU: the epilogues of few and of many targets per library
variable, and the paired-FP32 sums against the plain comparator's FP64 ones
(needs a GB300)."""

from __future__ import annotations

import numpy as np
import pytest

from paper_1905_00565_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# Both sides sum the same FP32 predictions, the comparator in FP64.  A paired sum
# carries 48 bits over 256 terms and its shift by the first prediction costs at
# most (range / std)^2 <= 1e3 here: 256 * 2^-48 * 1e3 = 1e-9 in the worst case of
# all roundings one way, 16 * 2^-48 * 1e3 = 6e-11 for independent ones.
MOMENT_TOL = 1e-10


@pytest.fixture(scope="module")
def ccm():
    from paper_1905_00565_gb300 import ccm as c
    return c


def run(ccm, ctx, p, flags=0, plain=False):
    plan = ccm.plan_problem(ctx, p, flags)
    try:
        rho = np.zeros(ccm.rho_shape(p))
        (ccm.ccm_run_plain if plain else ccm.ccm_run)(plan, p.series, rho)
    finally:
        ccm.ccm_plan_destroy(plan)
    return rho


def many_series(n, V, seed):
    rng = np.random.default_rng(seed)
    base = I.logistic_pair(n).astype(np.float64)
    mix = rng.random((V, 2))
    out = mix @ base + 0.05 * rng.standard_normal((V, n))
    out[0] = base[0]
    return np.ascontiguousarray(out.astype(np.float32))


@pytest.mark.parametrize("targets,n", [(11, 1000), (12, 1000), (31, 513), (32, 770), (33, 1287),
                                       (70, 300)])
def test_many_targets_equal_one_by_one(ccm, targets, n):
    """A library variable with many targets gives every target the bits of a plan
    of that pair alone, from brute force and from tables."""
    s = many_series(n, targets + 1, targets)
    kw = dict(E=np.array([1, 3, 10], np.int32), tau=np.array([2], np.int32),
              L=np.array([40, 260], np.int64), r=5, seed=11)
    pairs = np.array([[0, i] for i in range(1, targets + 1)], np.int32)
    ctx = ccm.ccm_context_create(0)
    try:
        for flags in (0, ccm.CCM_NO_TABLE):
            both = run(ccm, ctx, I.Problem(series=s, pairs=pairs, **kw), flags)
            for t in (0, targets // 2, targets - 1):
                one = run(ccm, ctx, I.Problem(series=s, pairs=pairs[t:t + 1], **kw), flags)
                np.testing.assert_array_equal(both[t], one[0])
    finally:
        ccm.ccm_context_destroy(ctx)


def test_repeated_pairs(ccm):
    s = many_series(700, 9, 3)
    pairs = np.array([[0, 1 + i % 8] for i in range(20)] + [[2, 0], [2, 0]], np.int32)
    p = I.Problem(series=s, pairs=pairs, E=np.array([2], np.int32), tau=np.array([1], np.int32),
                  L=np.array([50, 300], np.int64), r=3, seed=5)
    ctx = ccm.ccm_context_create(0)
    try:
        rho = run(ccm, ctx, p)
    finally:
        ccm.ccm_context_destroy(ctx)
    np.testing.assert_array_equal(rho[:8], rho[8:16])
    np.testing.assert_array_equal(rho[:4], rho[16:20])
    np.testing.assert_array_equal(rho[20], rho[21])
    assert np.all(np.isfinite(rho))


@pytest.mark.parametrize("targets", [1, 14])
def test_scaled_shifted_and_sparse_targets(ccm, targets):
    """Targets of extreme scale, far from zero, constant, and mostly zero: the same
    skill as the plain comparator's, and a value exactly where it has one."""
    n = 1100
    s = many_series(n, targets + 1, 7)
    rows = [s[0]]
    rng = np.random.default_rng(2)
    made = [s[1] * np.float32(1e30), s[1] * np.float32(1e-30), s[1] + np.float32(300),
            s[1] * np.float32(1e-41), np.full(n, 0.1, np.float32),
            np.where(rng.random(n) < 0.002, s[1], 0).astype(np.float32)]
    ctx = ccm.ccm_context_create(0)
    try:
        for odd in made:
            series = np.ascontiguousarray(np.stack(rows + [odd] + list(s[2:])))
            p = I.Problem(series=series,
                          pairs=np.array([[0, i] for i in range(1, targets + 1)], np.int32),
                          E=np.array([2, 4], np.int32), tau=np.array([1], np.int32),
                          L=np.array([20, 120, 700], np.int64), r=4, seed=9)
            got, want = run(ccm, ctx, p), run(ccm, ctx, p, plain=True)
            assert np.array_equal(np.isnan(got[1:]), np.isnan(want[1:]))
            nan = np.isnan(got[0]) != np.isnan(want[0])
            if not np.any(np.diff(odd)):          # constant: no skill
                assert np.all(np.isnan(got[0]))
            else:
                assert not np.any(nan)
            fine = np.isfinite(got) & np.isfinite(want)
            np.testing.assert_allclose(got[fine], want[fine], rtol=0, atol=MOMENT_TOL)
    finally:
        ccm.ccm_context_destroy(ctx)


# A tile's sums in FP64 (both sides) and rho's merge differ by orders of summation
# of at most 2560 terms: 2560 * 2^-53 * (range / std)^2 <= 1e-10 as above.
@pytest.mark.parametrize("spike", [1e18, 1e22, 1e25, 1e30, 1e37, -3e38])
@pytest.mark.parametrize("targets", [1, 14])
def test_targets_with_one_huge_value(ccm, targets, spike):
    """One target sample far above the others (a spike, a fill value): libraries that
    miss it predict values whose squares are far below FP32's range beside it."""
    n = 900
    s = many_series(n, targets + 1, 7)
    s[1, 450] = spike
    if targets > 1:
        s[2, 1] = spike                   # at E = 3 no manifold point holds it
    p = I.Problem(series=s, pairs=np.array([[0, i] for i in range(1, targets + 1)], np.int32),
                  E=np.array([1, 3], np.int32), tau=np.array([1], np.int32),
                  L=np.array([20, 120, 600], np.int64), r=6, seed=9)
    ctx = ccm.ccm_context_create(0)
    try:
        for flags in (0, ccm.CCM_NO_TABLE):
            got, want = run(ccm, ctx, p, flags), run(ccm, ctx, p, plain=True)
            assert np.all(np.isfinite(want))
            np.testing.assert_allclose(got, want, rtol=0, atol=MOMENT_TOL)
            one = run(ccm, ctx, I.Problem(series=s, pairs=p.pairs[:1], E=p.E, tau=p.tau, L=p.L,
                                          r=p.r, seed=p.seed), flags)
            np.testing.assert_array_equal(got[:1], one)
    finally:
        ccm.ccm_context_destroy(ctx)


@pytest.mark.parametrize("targets", [1, 3, 14])
def test_targets_of_two_scales(ccm, targets):
    """Values near 1e-12 and a fill value of 9.97e36 at every 97th sample; and two
    values 1e-40 apart, whose differences alone carry the skill."""
    n = 1100
    s = many_series(n, targets + 1, 3)
    rng = np.random.default_rng(4)
    fill = (s[1] * np.float32(1e-12)).astype(np.float32)
    fill[::97] = 9.97e36
    two = np.where(rng.random(n) < 0.5, np.float32(0), np.float32(1e-40))
    two[7] = 1.0
    deep = (s[1] * np.float32(1e-20)).astype(np.float32)   # scaled, these are subnormal
    deep[::211] = 1e37
    ctx = ccm.ccm_context_create(0)
    try:
        for odd in (fill, two, deep):
            series = s.copy()
            series[1] = odd
            p = I.Problem(series=series,
                          pairs=np.array([[0, i] for i in range(1, targets + 1)], np.int32),
                          E=np.array([2, 4], np.int32), tau=np.array([1], np.int32),
                          L=np.array([20, 120, 700], np.int64), r=4, seed=9)
            got, want = run(ccm, ctx, p), run(ccm, ctx, p, plain=True)
            np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
            fine = np.isfinite(want)
            np.testing.assert_allclose(got[fine], want[fine], rtol=0, atol=MOMENT_TOL)
    finally:
        ccm.ccm_context_destroy(ctx)


def test_grouped_realizations_with_a_huge_value(ccm):
    """14 targets whose realizations read their table in groups (240 of them, 12 query
    tiles): the tiles summed again in FP64 have brute force's bits and the comparator's
    sums."""
    n, targets = 3000, 14
    s = many_series(n, targets + 1, 5)
    s[1, 1700] = 1e30
    s[14, 5] = -3e37
    p = I.Problem(series=s, pairs=np.array([[0, i] for i in range(1, targets + 1)], np.int32),
                  E=np.array([3], np.int32), tau=np.array([1], np.int32),
                  L=np.array([600, 2500], np.int64), r=120, seed=9)
    ctx = ccm.ccm_context_create(0)
    try:
        got = run(ccm, ctx, p)
        np.testing.assert_array_equal(got, run(ccm, ctx, p, ccm.CCM_NO_TABLE))
        few = I.Problem(series=s, pairs=p.pairs, E=p.E, tau=p.tau, L=p.L, r=6, seed=p.seed)
        want = run(ccm, ctx, few, plain=True)
        assert np.all(np.isfinite(want))
        np.testing.assert_allclose(got[..., :6], want, rtol=0, atol=MOMENT_TOL)
    finally:
        ccm.ccm_context_destroy(ctx)
