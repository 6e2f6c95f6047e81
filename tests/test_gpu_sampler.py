"""Library sampler where its key window misses or is left out, and on manifolds too
long for its membership bits (needs a GB300): the libraries of the oracle, as lists
and as membership bits."""

from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1905_00565_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ccm():
    from paper_1905_00565_gb300 import ccm as c
    return c


def libraries(ccm, ctx, p, flags=0):
    plan = ccm.plan_problem(ctx, p, flags)
    try:
        info = ccm.ccm_plan_get_info(plan)
        rho = np.zeros(ccm.rho_shape(p))
        lib = np.zeros(info["library_entries"], np.int32)
        ccm.ccm_run_ex(plan, p.series, rho, libraries=lib)
        return rho, lib, info["table_bytes"]
    finally:
        ccm.ccm_plan_destroy(plan)


def check(p, lib):
    at = 0
    for (j, _) in p.pairs:
        for E in p.E:
            n_m = p.n - (int(E) - 1) * int(p.tau[0])
            for L in p.L:
                for k in range(p.r):
                    want = oracle.library(n_m, int(L), int(j), int(E), int(p.tau[0]), k, p.seed)
                    np.testing.assert_array_equal(lib[at:at + L], want, err_msg=f"E={E} L={L} k={k}")
                    at += int(L)


# 4 keys: no window of three standard deviations fits, but where nearly every point
# is a member; 8 sd / 0.9 keys: a window of +-4 sd that some units miss; 0: the default.
@pytest.mark.parametrize("window", [0, 1, 4, 110, 150, 200])
def test_selection_without_its_window(ccm, monkeypatch, window):
    monkeypatch.setenv("CCM_SAMPLER_WINDOW", str(window))
    p = I.Problem(series=I.logistic_pair(1203), pairs=I.BOTH_DIRECTIONS.copy(),
                  E=np.array([2, 4], np.int32), tau=np.array([1], np.int32),
                  L=np.array([6, 60, 500, 1199, 1200], np.int64), r=60, seed=21)
    ctx = ccm.ccm_context_create(0)
    try:
        rho, lib, tables = libraries(ccm, ctx, p)
        assert tables > 0                            # some as bits, some as lists
        check(p, lib)
        brute, lib2, _ = libraries(ccm, ctx, p, ccm.CCM_NO_TABLE)
    finally:
        ccm.ccm_context_destroy(ctx)
    np.testing.assert_array_equal(lib2, lib)
    np.testing.assert_array_equal(brute, rho)


@pytest.mark.parametrize("window", [0, 2])
@pytest.mark.parametrize("n_m", [1 << 20, (1 << 20) + 1, (1 << 20) + 77])
def test_manifolds_around_the_bits_limit(ccm, monkeypatch, n_m, window):
    monkeypatch.setenv("CCM_SAMPLER_WINDOW", str(window))
    rng = np.random.default_rng(1)
    p = I.Problem(series=rng.random((2, n_m + 1), dtype=np.float32),
                  pairs=np.array([[1, 0]], np.int32), E=np.array([2], np.int32),
                  tau=np.array([1], np.int32), L=np.array([40, 700], np.int64), r=2, seed=5)
    ctx = ccm.ccm_context_create(0)
    try:
        rho, lib, _ = libraries(ccm, ctx, p)
    finally:
        ccm.ccm_context_destroy(ctx)
    assert np.all(np.isfinite(rho))
    check(p, lib)
