"""A call that fails while it holds the handle's lock returns its error (GPU)."""
import json
import threading

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_failed_allocation_in_autotune_returns(lib, tmp_path):
    """Cached shapes for every size up to 2^19, and a matrix of 2^20 that no device holds: the allocation fails and
    the handle stays usable.  In a thread of its own, so that a call that never returns fails the test."""
    cache = tmp_path / "tune.json"
    name = torch.cuda.get_device_properties(0).name
    cache.write_text(json.dumps({"entries": [{"gpu": name, "dtype": 0, "n": 128 << i, "bk": 64, "tma": 3, "ms": 1.0}
                                             for i in range(13)]}))
    h = lib.Handle(device=0)
    seen = []

    def tune():
        try:
            h.autotune("int32", 1 << 20, str(cache))
        except lib.ApspError as e:
            seen.append(e.name)
    t = threading.Thread(target=tune, daemon=True)
    t.start()
    t.join(30)
    assert not t.is_alive()
    assert seen == ["APSP_E_CUDA"]
    W = np.where(np.eye(70) > 0, 0, 9).astype(np.int32)
    D = h.solve_t("int32", torch.from_numpy(W).cuda()).cpu().numpy()
    assert h.last_status() == 0
    np.testing.assert_array_equal(D.astype(np.int64), oracle.fw(W.astype(np.int64)))
    h.close()
