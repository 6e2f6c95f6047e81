"""Sizes at which a size rule changes its path: the query order's sorts, a plan whose
tables do not fit the context's budget, and the scratch of the no-allocation cell
(needs a GB300)."""

from __future__ import annotations

import numpy as np
import pytest

from paper_1905_00565_gb300 import inputs as I
from tests.ccm_check import check_units, run_detailed

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ccm():
    from paper_1905_00565_gb300 import ccm as c
    return c


# The order's bitonic network ends at 512 points, its radix sort at 16384 (runs are
# merged beyond); 96 query tiles (24576 points) is where rho takes a whole warp.
@pytest.mark.parametrize("n_m", [511, 512, 513, 16384, 16385, 24576, 24577, 33000])
def test_orders_and_tile_counts(ccm, n_m):
    E, tau = 2, 3
    p = I.Problem(series=I.logistic_pair(n_m + (E - 1) * tau), pairs=I.BOTH_DIRECTIONS.copy(),
                  E=np.array([E], np.int32), tau=np.array([tau], np.int32),
                  L=np.array([60, 480], np.int64), r=2, seed=11)
    ctx = ccm.ccm_context_create(0)
    try:
        check_units(p, *run_detailed(ccm, ctx, p), which={0, 3, 6})
    finally:
        ccm.ccm_context_destroy(ctx)


def test_tables_give_way_to_the_budget(ccm):
    """A plan's tables shrink, then go, as the budget does; rho stays the same and the
    smallest budget that holds the plan without tables still runs it."""
    p = I.Problem(series=I.logistic_pair(3000), pairs=I.BOTH_DIRECTIONS.copy(),
                  E=np.array([2, 5], np.int32), tau=np.array([1], np.int32),
                  L=np.array([80, 400, 2500], np.int64), r=60, seed=3)

    def footprint(flags, budget):
        ctx = ccm.ccm_context_create(0, budget)
        try:
            plan = ccm.plan_problem(ctx, p, flags)
            try:
                info = ccm.ccm_plan_get_info(plan)
                rho = np.zeros(ccm.rho_shape(p))
                ccm.ccm_run(plan, p.series, rho)
            finally:
                ccm.ccm_plan_destroy(plan)
        finally:
            ccm.ccm_context_destroy(ctx)
        return info["device_bytes"], info["table_bytes"], rho

    full, tables, want = footprint(0, 0)
    bare, none, _ = footprint(ccm.CCM_NO_TABLE, 0)
    assert tables > 0 and none == 0
    seen = set()
    for budget in (full, full - 1, bare + tables // 2, bare + tables // 50, bare):
        size, tab, rho = footprint(0, budget)
        assert size <= budget
        seen.add(tab)
        np.testing.assert_array_equal(rho, want)
    assert 0 in seen
    with pytest.raises(ccm.CCMError) as ei:
        footprint(0, bare - 1)
    assert ei.value.status == ccm.CCM_ETOOLARGE


def test_noalloc_admits_up_to_16_mib(ccm):
    """One query tile and the shortest libraries, where the descriptors weigh most."""
    torch = pytest.importorskip("torch")
    n, L, seed = 256, 3, 7

    def counts(r):
        parts = (112 * r, 12 * r, 4 * r * L, 48 * r, 4 * r, 4, 4, 4 * n, 48, 48 * r, 2112, 56)
        return sum((b + 255) // 256 * 256 for b in parts)

    r = max(q for q in range(70000, 72000) if counts(q) <= 16 << 20)
    p = I.Problem(series=I.logistic_pair(n), pairs=np.array([[0, 1]], np.int32),
                  E=np.array([1], np.int32), tau=np.array([1], np.int32),
                  L=np.array([L], np.int64), r=r, seed=seed)
    ctx = ccm.ccm_context_create(0)
    try:
        plan = ccm.plan_problem(ctx, p, ccm.CCM_NO_TABLE)
        want = np.zeros(ccm.rho_shape(p))
        ccm.ccm_run(plan, p.series, want)
        ccm.ccm_plan_destroy(plan)
    finally:
        ccm.ccm_context_destroy(ctx)
    s = torch.from_numpy(p.series).cuda()
    rho = torch.full((r,), float("nan"), dtype=torch.float64, device="cuda")
    ccm.ccm_run_noalloc(s, 0, 1, 1, 1, L, r, seed, rho)
    np.testing.assert_array_equal(rho.cpu().numpy(), want.reshape(-1))
    more = torch.zeros(r + 1, dtype=torch.float64, device="cuda")
    with pytest.raises(ccm.CCMError) as ei:
        ccm.ccm_run_noalloc(s, 0, 1, 1, 1, L, r + 1, seed, more)
    assert ei.value.status == ccm.CCM_ETOOLARGE


def test_table_beside_a_manifold_too_long_for_one(ccm):
    """A variable with two targets whose E = 10 manifold reads a table while its E = 1
    manifold is longer than any table's (its membership bits alone would fill an
    SM's shared memory)."""
    n, tau = 1_400_000, 155_000                      # N_m = 1400000 and 5000
    rng = np.random.default_rng(5)
    p = I.Problem(series=rng.random((3, n), dtype=np.float32),
                  pairs=np.array([[0, 1], [0, 2]], np.int32), E=np.array([1, 10], np.int32),
                  tau=np.array([tau], np.int32), L=np.array([400], np.int64), r=110, seed=3)
    rho = {}
    ctx = ccm.ccm_context_create(0)
    try:
        for flags in (0, ccm.CCM_NO_TABLE):
            plan = ccm.plan_problem(ctx, p, flags)
            try:
                assert (ccm.ccm_plan_get_info(plan)["table_bytes"] > 0) == (flags == 0)
                rho[flags] = np.zeros(ccm.rho_shape(p))
                ccm.ccm_run(plan, p.series, rho[flags])
            finally:
                ccm.ccm_plan_destroy(plan)
    finally:
        ccm.ccm_context_destroy(ctx)
    assert np.all(np.isfinite(rho[0]))
    np.testing.assert_array_equal(rho[0], rho[ccm.CCM_NO_TABLE])


def test_many_targets_give_way_to_the_budget(ccm):
    """Variables of many targets read a time-major copy of the series; a plan or job that
    does not fit with it runs without, to the same bits."""
    n, V = 20011, 40
    rng = np.random.default_rng(6)
    p = I.Problem(series=rng.random((V, n), dtype=np.float32),
                  pairs=np.array([[0, i] for i in range(1, 15)] + [[1, 0]], np.int32),
                  E=np.array([2], np.int32), tau=np.array([1], np.int32),
                  L=np.array([30], np.int64), r=2, seed=3)
    copy = n * 64 * 4

    def run(budget, flags=ccm.CCM_NO_TABLE):
        ctx = ccm.ccm_context_create(0, budget)
        try:
            plan = ccm.plan_problem(ctx, p, flags)
            try:
                rho = np.zeros(ccm.rho_shape(p))
                ccm.ccm_run(plan, p.series, rho)
                return ccm.ccm_plan_get_info(plan)["device_bytes"], rho
            finally:
                ccm.ccm_plan_destroy(plan)
        finally:
            ccm.ccm_context_destroy(ctx)

    full, want = run(0)
    for budget in (full, full - 1, full - copy):
        size, rho = run(budget)
        assert size <= budget
        np.testing.assert_array_equal(rho, want)
    with pytest.raises(ccm.CCMError) as ei:
        run(full - copy - (1 << 20))
    assert ei.value.status == ccm.CCM_ETOOLARGE
    ctx = ccm.ccm_context_create(0, full - copy)
    try:
        ticket = ccm.ccm_submit(ctx, p.series, p.pairs, p.E, p.tau, p.L, p.r, p.seed)
        rho = np.zeros_like(want)
        for _ in range(600):
            if ccm.ccm_poll(ctx, ticket, rho, 100) == ccm.CCM_OK:
                break
        else:
            pytest.fail("job did not finish")
        np.testing.assert_array_equal(rho, want)
    finally:
        ccm.ccm_context_destroy(ctx)


@pytest.mark.parametrize("n_m", [4096, 4097, 24576])
def test_rho_of_few_and_of_many_targets(ccm, n_m):
    """Up to 1024 targets of more than 16 query tiles take a warp each, more of them four
    lanes each: the same bits, also with tiles summed in FP64 (a spike)."""
    rng = np.random.default_rng(8)
    s = rng.random((3, n_m), dtype=np.float32)
    s[2, n_m // 3] = 1e30
    ctx = ccm.ccm_context_create(0)
    try:
        rho = {}
        for r in (4, 520):
            p = I.Problem(series=s, pairs=np.array([[0, 1], [0, 2]], np.int32),
                          E=np.array([1], np.int32), tau=np.array([1], np.int32),
                          L=np.array([12], np.int64), r=r, seed=3)
            plan = ccm.plan_problem(ctx, p, ccm.CCM_NO_TABLE)
            rho[r] = np.zeros(ccm.rho_shape(p))
            ccm.ccm_run(plan, p.series, rho[r])
            ccm.ccm_plan_destroy(plan)
    finally:
        ccm.ccm_context_destroy(ctx)
    assert np.all(np.isfinite(rho[4]))
    np.testing.assert_array_equal(rho[4], rho[520][..., :4])


@pytest.mark.parametrize("n_m,E,L", [(16385, 1, 3), (16385, 2, 4), (16640, 1, 17), (17001, 2, 2600),
                                     (20000, 1, 2561), (16411, 1, 5003), (16411, 3, 100)])
def test_cells_in_time_order(ccm, n_m, E, L):
    """Above 16384 points a cell's manifold keeps time order and nothing is pruned (a
    search of its own for E <= 2).  The same predictions as ccm_run's in other tiles:
    within the rounding of the sums (256 * 2^-48 * (range / std)^2 of 1e2)."""
    torch = pytest.importorskip("torch")
    n, r = n_m + 2 * (E - 1), 3
    p = I.Problem(series=I.logistic_pair(n), pairs=np.array([[1, 0]], np.int32),
                  E=np.array([E], np.int32), tau=np.array([2], np.int32),
                  L=np.array([L], np.int64), r=r, seed=7)
    ctx = ccm.ccm_context_create(0)
    try:
        plan = ccm.plan_problem(ctx, p, ccm.CCM_NO_TABLE)
        want = np.zeros(ccm.rho_shape(p))
        ccm.ccm_run(plan, p.series, want)
        ccm.ccm_plan_destroy(plan)
    finally:
        ccm.ccm_context_destroy(ctx)
    s = torch.from_numpy(p.series).cuda()
    rho = torch.full((r,), float("nan"), dtype=torch.float64, device="cuda")
    ccm.ccm_run_noalloc(s, 1, 0, E, 2, L, r, 7, rho)
    np.testing.assert_allclose(rho.cpu().numpy(), want.reshape(-1), rtol=0, atol=1e-10)
