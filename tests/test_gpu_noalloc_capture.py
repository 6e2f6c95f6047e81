"""ccm_run_noalloc inside a stream capture (needs a GB300): its launches carry the
programmatic attribute, and the graph must replay them in order, on new series
values in the same buffers and with the capturing stream's own work around them."""

from __future__ import annotations

import numpy as np
import pytest

from paper_1905_00565_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,E,L,r", [(300, 3, 40, 5), (1000, 1, 400, 60), (9000, 6, 1500, 8),
                                     (20000, 2, 100, 20)])
def test_captured_cell_replays(n, E, L, r):
    torch = pytest.importorskip("torch")
    from paper_1905_00565_gb300 import ccm
    first = I.logistic_pair(n)
    other = np.ascontiguousarray(first[::-1] * np.float32(0.7) + np.float32(0.1))
    stream = torch.cuda.Stream()
    series = torch.from_numpy(first).cuda()
    doubled = torch.empty_like(series)
    rho = torch.zeros(r, dtype=torch.float64, device="cuda")
    half = torch.empty_like(rho)
    torch.cuda.synchronize()

    def direct(values):
        out = torch.zeros(r, dtype=torch.float64, device="cuda")
        ccm.ccm_run_noalloc(torch.from_numpy(values).cuda() * 2, 1, 0, E, 1, L, r, 5, out)
        return out.cpu().numpy()

    want = [direct(first), direct(other)]       # also the set-up call before the capture
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        torch.mul(series, 2, out=doubled)       # a kernel of the caller's before ...
        ccm.ccm_run_noalloc(doubled, 1, 0, E, 1, L, r, 5, rho, torch.cuda.current_stream())
        torch.mul(rho, 0.5, out=half)           # ... and behind
    for values, expect in ((first, want[0]), (other, want[1]), (first, want[0])):
        series.copy_(torch.from_numpy(values))
        rho.zero_()
        half.zero_()
        torch.cuda.synchronize()
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(rho.cpu().numpy(), expect)
        np.testing.assert_array_equal(half.cpu().numpy(), expect * 0.5)
