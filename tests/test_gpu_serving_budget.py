"""Requests that just fit the serving budget (GPU): each is accepted, runs and is right, with no room for the copy
with 16-byte rows or for the closed diagonal block beside it."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_round64 import graph

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def exact(n, large):
    """A request's matrix and panels; on the per-round kernels their panel buffer as well."""
    ld = (n + 255) // 256 * 256
    return n * n * 4 + 64 * ld * 4 + 256 + (128 * ld * 4 if large else 0)


@pytest.mark.parametrize("n", [64, 65, 101, 301, 1000])
@pytest.mark.parametrize("large", [False, True])
@pytest.mark.parametrize("spare", [0, 4096, 40000])
def test_request_that_just_fits_runs(lib, n, large, spare):
    _, _, _, W = graph(n, n)
    E = oracle.fw(W.astype(np.int64))
    with lib.Handle(device=0, memory_budget=exact(n, large) + spare, serving_large_n=n if large else 0) as h:
        for _ in range(2):
            t = h.submit(torch.from_numpy(W).cuda())
            assert h.wait(t, 20000) == 0
            out = torch.empty((n, n), dtype=torch.int32, device="cuda")
            h.fetch(t, out)
            torch.cuda.synchronize()
            np.testing.assert_array_equal(out.cpu().numpy().astype(np.int64), E)
            assert h.release(t) == 0


def test_many_requests_on_a_small_budget_all_finish(lib):
    ns = [65, 130, 201, 64, 97, 300, 33, 150]
    graphs = [graph(n, n)[3] for n in ns]
    with lib.Handle(device=0, memory_budget=exact(300, False) + 5000) as h:
        ts = [h.submit(torch.from_numpy(W).cuda()) for W in graphs]
        for t, n, W in zip(ts, ns, graphs):
            assert h.wait(t, 20000) == 0
            out = torch.empty((n, n), dtype=torch.int32, device="cuda")
            h.fetch(t, out)
            torch.cuda.synchronize()
            assert h.release(t) == 0
            np.testing.assert_array_equal(out.cpu().numpy().astype(np.int64), oracle.fw(W.astype(np.int64)))
