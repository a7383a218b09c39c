"""Batches whose graphs all take a single round (n <= 64), which need neither the task plan nor, without copies, the
output pass (GPU)."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_round64 import graph

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ns", [[1], [2, 1, 3], [31, 33, 64], [63, 64], [64, 4, 60], [64, 65]])
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("pad", [0, 3])
def test_one_round_batches_match_oracle(lib, ns, directed, pad):
    Ws = [graph(n, n + 1, directed)[3] if n > 2 else np.array([[0, 7], [7 if not directed else 5, 0]], np.int32)[:n, :n]
          for n in ns]
    with lib.Handle(device=0) as h:
        for in_place in (False, True):
            ins, outs = [], []
            for W in Ws:
                n = W.shape[0]
                buf = torch.full((n, n + pad), 5, dtype=torch.int32, device="cuda")
                buf[:, :n] = torch.from_numpy(W).cuda()
                ins.append(buf)
                outs.append(buf if in_place else torch.full_like(buf, 5))
            h.solve_batch(ins, outs)
            assert h.last_status() == 0
            for W, D in zip(Ws, outs):
                n = W.shape[0]
                np.testing.assert_array_equal(D[:, :n].cpu().numpy().astype(np.int64), oracle.fw(W.astype(np.int64)))
                assert bool((D[:, n:] == 5).all())
        bad = torch.tensor([[0, -1], [4, 0]], dtype=torch.int32, device="cuda")
        h.solve_batch([ins[0], bad], [torch.empty_like(ins[0]), torch.empty_like(bad)])
        assert h.last_status() == 1  # the input check still runs
