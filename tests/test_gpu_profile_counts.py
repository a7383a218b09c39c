"""The relaxation counts that a profiled solve reports (GPU)."""
import pytest

from tests.test_gpu_round64 import graph, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,directed", [(1000, False), (1000, True), (65, False), (64, False)])
def test_profiled_relaxations_follow_the_mode(lib, n, directed):
    """Two panels of (n - w) w^2 relaxations a round, one in symmetric mode, which the device chooses here."""
    _, _, _, W = graph(n, 5, directed)
    widths = [min(64, n - p) for p in range(0, n, 64)]
    one_panel = float(sum((n - w) * w * w for w in widths))
    with lib.Handle(device=0) as h:
        h.profile(True)
        for _ in range(2):  # a second solve chooses anew
            h.solve_t("int32", to_dev(W, "int32", (n + 3) // 4 * 4))
            p = h.profile_read()
            assert p[2][2] == (2.0 if directed else 1.0) * one_panel
