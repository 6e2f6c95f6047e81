"""The autotuner's saved choices (needs a GB300): rows of other kernels, or of the
format without a revision, are not taken; its own are."""

from __future__ import annotations

import os
import time

import numpy as np
import pytest

from paper_1905_00565_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_choices_of_other_kernels_are_measured_again(monkeypatch, tmp_path):
    torch = pytest.importorskip("torch")
    from paper_1905_00565_gb300 import ccm
    cache = tmp_path / "autotune.tsv"
    monkeypatch.setenv("CCM_AUTOTUNE_CACHE", str(cache))
    device = torch.cuda.get_device_name(0)
    old = [f"{device}\t2\t0\t8\n", f"{device}\trsomething-else\t2\t0\t8\n"]
    cache.write_text("".join(old))
    # 2.2e11 query-library pairs, most of them read from tables
    p = I.Problem(series=I.logistic_pair(10001), pairs=I.BOTH_DIRECTIONS.copy(),
                  E=np.array([2], np.int32), tau=np.array([1], np.int32),
                  L=np.array([60, 9000], np.int64), r=1220, seed=2)

    def run(flags=0):
        ctx = ccm.ccm_context_create(0)
        try:
            plan = ccm.plan_problem(ctx, p, flags)
            try:
                rho = np.zeros(ccm.rho_shape(p))
                ccm.ccm_run(plan, p.series, rho)
            finally:
                ccm.ccm_plan_destroy(plan)
        finally:
            ccm.ccm_context_destroy(ctx)
        return rho, cache.read_text().splitlines(keepends=True)

    monkeypatch.setenv("CCM_TABLE_CROSSOVER", "20")   # L = 60 stays with brute force
    first, rows = run()
    assert rows[:2] == old and len(rows) == 3         # measured, and saved
    name, revision, E, variant, merge = rows[2].rstrip("\n").split("\t")
    assert (name, E) == (device, "2") and revision.startswith("r")
    second, again = run()
    assert again == rows                              # its own row is taken
    np.testing.assert_array_equal(first, second)
    assert os.path.exists(cache)


def test_nothing_to_measure_runs_nothing(monkeypatch, tmp_path):
    """A plan whose libraries all read tables has no brute-force items to time: its first
    run, like any other with device buffers and a caller's stream, only enqueues (the
    measurement waits for the stream)."""
    torch = pytest.importorskip("torch")
    from paper_1905_00565_gb300 import ccm
    monkeypatch.setenv("CCM_AUTOTUNE_CACHE", str(tmp_path / "none.tsv"))
    p = I.Problem(series=I.logistic_pair(10001), pairs=I.BOTH_DIRECTIONS.copy(),
                  E=np.array([2], np.int32), tau=np.array([1], np.int32),
                  L=np.array([8000, 9000], np.int64), r=600, seed=2)
    flags = ccm.CCM_INPUT_ON_DEVICE | ccm.CCM_OUTPUT_ON_DEVICE
    series = torch.from_numpy(p.series).cuda()
    rho = torch.zeros(ccm.rho_shape(p), dtype=torch.float64, device="cuda")
    stream = torch.cuda.Stream()
    ctx = ccm.ccm_context_create(0)
    try:
        for first in (False, True):              # the first plan loads the kernels
            plan = ccm.plan_problem(ctx, p, flags | (0 if first else ccm.CCM_NO_AUTOTUNE))
            info = ccm.ccm_plan_get_info(plan)
            assert info["pair_count"] >= 2e11 and info["n_work_items"] == 0
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                torch.cuda._sleep(1_000_000_000)  # about half a second
            t0 = time.perf_counter()
            ccm.ccm_run(plan, series, rho, stream)
            enqueued = time.perf_counter() - t0
            busy = not stream.query()
            torch.cuda.synchronize()
            ccm.ccm_plan_destroy(plan)
            assert busy and enqueued < 0.25, enqueued
    finally:
        ccm.ccm_context_destroy(ctx)
    assert bool(torch.isfinite(rho).all())
