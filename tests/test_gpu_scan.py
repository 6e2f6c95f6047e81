"""The grouped table scan and the window sampler at their edges, against brute
force bit for bit and the oracle (needs a GB300)."""

from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1905_00565_gb300 import inputs as I
from tests.ccm_check import check_units, run_detailed

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ccm():
    from paper_1905_00565_gb300 import ccm as c
    return c


def rho_only(ccm, ctx, p, flags):
    plan = ccm.plan_problem(ctx, p, flags)
    try:
        assert (ccm.ccm_plan_get_info(plan)["table_bytes"] > 0) == (flags == 0)
        rho = np.zeros(ccm.rho_shape(p))
        ccm.ccm_run(plan, p.series, rho)
    finally:
        ccm.ccm_plan_destroy(plan)
    return rho


# r: one lane, groups that end inside a cell, exactly at it, and that span cells;
# n: ragged tiles, membership words in shared memory and (20000, 70000) in L2,
# 16- and 32-bit positions; unsorted L
@pytest.mark.parametrize("n,E,L,r,theiler", [
    (700, [1, 10], [400, 690, 300], 33, 0), (2049, [3], [2000, 300, 1024], 31, 0),
    (3000, [2, 9], [2900, 700], 64, 4), (5000, [4], [300, 4999 - 3], 21, 0),
    (20000, [1, 5], [900, 15000], 40, 0), (70000, [3], [20000, 69000], 11, 2)])
def test_scan_equals_brute_force(ccm, n, E, L, r, theiler):
    s = I.add_noise(I.logistic_pair(n), 0.001, 3) if n % 2 else I.logistic_pair(n)
    p = I.Problem(series=s, pairs=I.BOTH_DIRECTIONS.copy(), E=np.array(E, np.int32),
                  tau=np.array([1], np.int32), L=np.array(L, np.int64), r=r, seed=21,
                  theiler=theiler)
    ctx = ccm.ccm_context_create(0)
    try:
        np.testing.assert_array_equal(rho_only(ccm, ctx, p, 0),
                                      rho_only(ccm, ctx, p, ccm.CCM_NO_TABLE))
    finally:
        ccm.ccm_context_destroy(ctx)


@pytest.mark.parametrize("kind", ["clusters", "ints", "few", "line", "zeros"])
def test_rows_of_unusual_distances(ccm, kind):
    """Table rows whose threshold is hard to find: tight clusters 60 octaves of
    squared distance below the manifold's extent, many exact ties (also at
    distance 0), and a one-dimensional manifold."""
    rng = np.random.default_rng(5)
    n = 2600
    if kind == "clusters":      # period 4, near-exact copies of four states
        s = np.tile([0.1, 0.5, 0.35, 0.9], (2, n // 4)) + 1e-6 * rng.random((2, n))
        s[:, ::97] += 3e4
    elif kind == "ints":
        s = rng.integers(0, 3, (2, n))
    elif kind == "few":
        s = rng.integers(0, 40, (2, n)) * 0.25
    elif kind == "line":
        s = np.stack([np.arange(n), np.arange(n)[::-1]]) * 0.125 + 0.01 * rng.random((2, n))
    else:
        s = np.where(rng.random((2, n)) < 0.6, 0.0, rng.random((2, n)))
    p = I.Problem(series=np.ascontiguousarray(s.astype(np.float32)),
                  pairs=I.BOTH_DIRECTIONS.copy(), E=np.array([1, 2, 4], np.int32),
                  tau=np.array([1], np.int32), L=np.array([600, 1900, 2590], np.int64), r=9,
                  seed=6)
    ctx = ccm.ccm_context_create(0)
    try:
        np.testing.assert_array_equal(rho_only(ccm, ctx, p, 0),
                                      rho_only(ccm, ctx, p, ccm.CCM_NO_TABLE))
    finally:
        ccm.ccm_context_destroy(ctx)


# Variables with 13 targets: groups of realizations (lane_group's largest at
# E = 1, 9; smaller ones from the launch's size), membership words in shared
# memory and in L2 (20000, 70000), the one-realization walk (2000), 32-bit rows.
# Rows miss for about one (query, realization) in 10 L: thousands of them here.
@pytest.mark.parametrize("n,E,L,r,theiler", [
    (1500, [1, 9], [1480, 500, 900], 40, 0), (3000, [3], [2900, 700], 80, 0),
    (3000, [2, 6], [2900, 900], 33, 5), (20000, [1], [9000], 19, 0), (2000, [4], [1900], 9, 0),
    (70000, [2], [60000], 10, 0)])
def test_many_targets_equal_brute_force(ccm, n, E, L, r, theiler):
    V = 14
    s, _ = I.logistic_network(V, n, 0.05, 7)
    pairs = np.array([[j, i] for j in range(V) for i in range(V) if i != j], np.int32)
    p = I.Problem(series=s, pairs=pairs, E=np.array(E, np.int32), tau=np.array([1], np.int32),
                  L=np.array(L, np.int64), r=r, seed=4, theiler=theiler)
    ctx = ccm.ccm_context_create(0)
    try:
        np.testing.assert_array_equal(rho_only(ccm, ctx, p, 0),
                                      rho_only(ccm, ctx, p, ccm.CCM_NO_TABLE))
    finally:
        ccm.ccm_context_destroy(ctx)


@pytest.mark.parametrize("theiler", [0, 3])
def test_many_targets_checking_outputs(ccm, theiler):
    """Neighbours, predictions, libraries and counters of the grouped walk."""
    V, n = 13, 6000
    s, _ = I.logistic_network(V, n, 0.05, 9)
    pairs = np.array([[2, i] for i in range(V) if i != 2], np.int32)
    p = I.Problem(series=s, pairs=pairs, E=np.array([2], np.int32), tau=np.array([2], np.int32),
                  L=np.array([1500, 5000], np.int64), r=110, seed=5, theiler=theiler)
    ctx = ccm.ccm_context_create(0)
    try:
        got = run_detailed(ccm, ctx, p, 0)
        want = run_detailed(ccm, ctx, p, ccm.CCM_NO_TABLE)
    finally:
        ccm.ccm_context_destroy(ctx)
    for g, w in zip(got, want):
        np.testing.assert_array_equal(g, w)
    check_units(p, *got, which={0, 219, 220 * 11 + 130})


def test_scan_checking_outputs(ccm):
    """Neighbours, predictions and libraries of the general variant."""
    p = I.Problem(series=I.logistic_pair(1500), pairs=I.BOTH_DIRECTIONS.copy(),
                  E=np.array([1, 6], np.int32), tau=np.array([3], np.int32),
                  L=np.array([500, 1400], np.int64), r=18, seed=2, weight_floor=0.01)
    ctx = ccm.ccm_context_create(0)
    try:
        rho, lib, nbr, xh = run_detailed(ccm, ctx, p)
    finally:
        ccm.ccm_context_destroy(ctx)
    check_units(p, rho, lib, nbr, xh, which={0, 17, 18, 35, 70, 143})


@pytest.mark.parametrize("n,L", [(300, [5, 150, 299, 300]), (9, [4, 9]), (4096, [4, 4095, 2048]),
                                 (65536, [100, 65000])])
def test_libraries_at_the_edges(ccm, n, L):
    """The sampler's window at both ends of its range: the smallest and the full
    library, short and long manifolds."""
    rng = np.random.default_rng(n)
    p = I.Problem(series=rng.random((2, n)).astype(np.float32),
                  pairs=np.array([[0, 1]], np.int32), E=np.array([1], np.int32),
                  tau=np.array([1], np.int32), L=np.array(L, np.int64), r=9, seed=77)
    ctx = ccm.ccm_context_create(0)
    try:
        for flags in (0, ccm.CCM_NO_TABLE):
            _, lib, _, _ = run_detailed(ccm, ctx, p, flags)
            at = 0
            for Lv in L:
                for k in range(p.r):
                    want = oracle.library(n, Lv, 0, 1, 1, k, p.seed)
                    np.testing.assert_array_equal(lib[at:at + Lv], want)
                    at += Lv
    finally:
        ccm.ccm_context_destroy(ctx)
