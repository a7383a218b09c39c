"""Which Phase-3 kernel a solve runs, and its result at the sizes of each route (GPU): the single launch where it is
the default and where it is asked for, one launch per round where a default single launch runs as that."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_parity import dense_on_device, er_edges

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
INF = oracle.INF32


def solve_rows(h, dt, n, directed, count):
    """`count` seeded rows of an in-place solve and the oracle's; the number of kernels launched."""
    s, d, w = er_edges(n, seed=n + directed, deg=4.0, wmax=60, directed=directed)
    if dt == "fp32":
        W = dense_on_device(n, s, d, w, np.int32, INF, directed).to(torch.float32)
        W[W >= INF] = float("inf")
    else:
        W = dense_on_device(n, s, d, w, np.int32 if dt == "int32" else np.int16, INF if dt == "int32" else 0x7FFF,
                            directed)
    rows = np.sort(np.random.default_rng(n).choice(n, size=count, replace=False))
    before = h.launch_count
    h.solve_t(dt, W, W)
    assert h.last_status() == 0
    launches = h.launch_count - before
    got = W[torch.from_numpy(rows).cuda().long()].cpu().numpy()
    del W
    torch.cuda.empty_cache()
    if dt == "u16":
        got = oracle.unpack_u16(got.view(np.uint16))
    elif dt == "fp32":
        got = np.where(np.isinf(got), INF, got.astype(np.float64))  # small whole numbers: exact
    return got.astype(np.int64), oracle.dijkstra(n, s, d, w, rows, directed=directed), launches


# the largest sizes of the single launch's table, and a packed 16-bit one in which its panel tasks fall between tiles
@pytest.mark.parametrize("dt,n,directed", [("int32", 24000, False), ("int32", 24000, True), ("u16", 8200, False),
                                           ("u16", 49000, False)])
def test_single_launch_asked_for_sampled_rows(lib, dt, n, directed):
    with lib.Handle(device=0, phase3_variant=5) as h:
        got, exp, launches = solve_rows(h, dt, n, directed, 128)
    assert launches < 16
    np.testing.assert_array_equal(got, exp)


# both sides of every line of solve_phase3; a single launch of all rounds, or two launches a round
@pytest.mark.parametrize("dt,n,single", [
    ("int32", 6200, False), ("int32", 7679, False), ("int32", 7680, True), ("int32", 8200, True),
    ("int32", 14335, True), ("int32", 14336, False), ("u16", 9215, False), ("u16", 9216, True),
    ("u16", 32767, True), ("u16", 32768, False), ("fp32", 6200, False), ("fp32", 12000, False)])
def test_default_route_by_n_and_dtype(lib, dt, n, single):
    with lib.Handle(device=0) as h:
        got, exp, launches = solve_rows(h, dt, n, False, 64)
    assert launches < 16 if single else launches >= 2 * (n // 64)
    np.testing.assert_array_equal(got, exp)


@pytest.mark.parametrize("n", [8200, 14000])
def test_default_single_launch_directed_rows(lib, n):
    with lib.Handle(device=0) as h:
        got, exp, launches = solve_rows(h, "int32", n, True, 64)
    assert launches < 16
    np.testing.assert_array_equal(got, exp)


def test_single_launch_solves_after_its_waits_timed_out(lib):
    n = 6200
    with lib.Handle(device=0, phase3_variant=5) as h:
        assert h.check_bounded_wait(1 << 10) == 7  # APSP_E_TIMEOUT
        got, exp, launches = solve_rows(h, "int32", n, False, 64)
    assert launches < 16
    np.testing.assert_array_equal(got, exp)
