"""Tables of series with few distinct values (needs a GB300): a row's threshold falls
on a tie, up to an index, and must still give the brute-force neighbours bit for
bit."""

from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1905_00565_gb300 import inputs as I
from tests.ccm_check import run_detailed, split

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ccm():
    from paper_1905_00565_gb300 import ccm as c
    return c


def made(kind, V, n, seed):
    rng = np.random.default_rng(seed)
    x = rng.random((V, n))
    if kind == "periodic":            # 271 values, each at equally spaced indices
        x = np.stack([np.tile(v, n // 271 + 1)[:n] for v in rng.random((V, 271))])
    elif kind == "settled":           # constant from a third on: the tie fills the series
        x[:, n // 3:] = 0.5
    elif kind == "late":              # the tied indices all lie at the end
        x[:, -n // 4:] = 0.25
    elif kind == "levels":            # quantised: ties at every distance
        x = rng.integers(0, 6, (V, n))
    elif kind == "binary":
        x = rng.integers(0, 2, (V, n))
    elif kind == "constant":
        x[:] = 0.3
        x[1:] = rng.random((V - 1, n))
    elif kind == "signed zeros":
        x = rng.choice([-0.0, 0.0, 1e-3, -1e-3], (V, n))
    elif kind == "far":               # a few points far from a dense cluster
        x = 1e-6 * x
        x[:, ::97] += 1e6
    return np.ascontiguousarray(x.astype(np.float32))


@pytest.mark.parametrize("kind", ["periodic", "settled", "late", "levels", "binary", "constant",
                                  "signed zeros", "far"])
@pytest.mark.parametrize("n,E,L", [(1025, 1, [300, 1000]), (2049, 2, [60, 700, 2000]),
                                   (3000, 6, [100, 2900]), (6100, 1, [150, 5000])])
def test_tied_rows_equal_brute_force(ccm, kind, n, E, L):
    s = made(kind, 3, n, 7)
    p = I.Problem(series=s, pairs=np.array([[0, 1], [1, 0], [1, 2]], np.int32),
                  E=np.array([E], np.int32), tau=np.array([1], np.int32),
                  L=np.array(L, np.int64), r=40, seed=11)
    ctx = ccm.ccm_context_create(0)
    try:
        rho, lib, nbr, xh = run_detailed(ccm, ctx, p)
        rb, lb, nb, xb = run_detailed(ccm, ctx, p, ccm.CCM_NO_TABLE)
        plan = ccm.plan_problem(ctx, p)
        try:
            assert ccm.ccm_plan_get_info(plan)["table_bytes"] > 0
            replay = np.zeros_like(rho)
            ccm.ccm_run(plan, p.series, replay)
        finally:
            ccm.ccm_plan_destroy(plan)
    finally:
        ccm.ccm_context_destroy(ctx)
    np.testing.assert_array_equal(nbr, nb)
    np.testing.assert_array_equal(xh, xb)
    np.testing.assert_array_equal(rho, rb)
    np.testing.assert_array_equal(replay, rho)
    # (predictions of values that cancel are no measure against 64 bits; the lists are)
    for (u, j, i, E_u, tau, L_u, k, n_m, l_g, n_g, _) in split(p, lib, nbr, xh):
        if u in (0, len(L) * 40 - 1, len(L) * 120 - 1):
            _, l_o, n_o, _ = oracle.ccm_unit(p.series, j, i, E_u, tau, L_u, k, p.seed, keep=True)
            np.testing.assert_array_equal(l_g, l_o)
            np.testing.assert_array_equal(n_g, n_o)
