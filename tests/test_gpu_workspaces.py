"""The copies with 16-byte rows that unaligned matrices and products run on (GPU): calls under stream capture,
on several streams, and in sequences of growing sizes."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_round64 import back, graph, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def capture(fn):
    g = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=side):
        fn()
    return g


# a handle that is warm for the size can be captured: nothing may be allocated then
@pytest.mark.parametrize("dtype", ["int32", "u16", "fp32"])
@pytest.mark.parametrize("symmetric,warm", [(0, "aligned"), (1, "aligned"), (2, "aligned"), (0, "unaligned"),
                                            (1, "unaligned"), (2, "unaligned")])
def test_unaligned_solve_under_capture(lib, dtype, symmetric, warm):
    n = 301
    _, _, _, W = graph(n, n)
    E = oracle.fw(W.astype(np.int64))
    Wa, Wu = to_dev(W, dtype, 304), to_dev(W, dtype, n)
    D = torch.full_like(Wu, 5)
    with lib.Handle(device=0, symmetric=symmetric) as h:
        if warm == "aligned":
            h.solve_t(dtype, Wa, torch.empty_like(Wa))
        else:
            h.solve_t(dtype, Wu, D)
        D.fill_(5)
        g = capture(lambda: h.solve_t(dtype, Wu, D))
        for _ in range(2):
            D.fill_(5)
            g.replay()
            torch.cuda.synchronize()
            assert h.last_status() == 0
            np.testing.assert_array_equal(back(D, n, dtype), E)
        del g


@pytest.mark.parametrize("wider", [False, True])
def test_captured_solve_outlives_the_copy_of_its_size(lib, wider):
    """A larger unaligned solve (more vertices, or wider elements) replaces the handle's copy; a graph captured
    before still replays right."""
    n, m = 301, 900
    _, _, _, W = graph(n, n)
    E = oracle.fw(W.astype(np.int64))
    Wu, Wm = to_dev(W, "u16", n), graph(m, m)[3]
    D = torch.full_like(Wu, 5)
    with lib.Handle(device=0) as h:
        Wa = to_dev(Wm, "int32", m)  # rows of 16 bytes
        h.solve_t("int32", Wa, torch.empty_like(Wa))  # the panel buffer for m vertices, no copy
        h.solve_t("u16", Wu, D)
        g = capture(lambda: h.solve_t("u16", Wu, D))
        Wb = to_dev(W, "int32", n) if wider else to_dev(Wm, "int32", m + 1)
        h.solve_t("int32", Wb, torch.empty_like(Wb))
        D.fill_(5)
        g.replay()
        torch.cuda.synchronize()
        assert h.last_status() == 0
        np.testing.assert_array_equal(back(D, n, "u16"), E)
        del g


def test_unaligned_product_under_capture(lib):
    m, k, n = 400, 300, 401
    rng = np.random.default_rng(3)
    A, B, C = (rng.integers(0, 5000, size=s) for s in ((m, k), (k, n), (m, n)))
    Ad, Bd, Cd = (torch.from_numpy(x.astype(np.int32)).cuda() for x in (A, B, C))
    with lib.Handle(device=0) as h:
        big = [torch.zeros((512, 512), dtype=torch.int32, device="cuda") for _ in range(3)]
        h.minplus(*big)  # warm: the workspace for A transposed
        torch.cuda.synchronize()
        g = capture(lambda: h.minplus(Ad, Bd, Cd))
        g.replay()
        torch.cuda.synchronize()
        assert h.last_status() == 0
        np.testing.assert_array_equal(Cd.cpu().numpy(), oracle.minplus(A, B, C))
        del g


@pytest.mark.parametrize("dtype", ["int32", "u16"])
def test_unaligned_products_on_several_streams(lib, dtype):
    """Products without 16-byte rows on two streams of one handle, between aligned ones: each is its own."""
    rng = np.random.default_rng(8)
    npdt = {"int32": np.int32, "u16": np.int16}[dtype]
    jobs = []
    for m, k, n in ((400, 300, 401), (600, 250, 301), (300, 500, 333), (700, 201, 255), (512, 512, 512)):
        A, B, C = (rng.integers(0, 9000, size=x) for x in ((m, k), (k, n), (m, n)))
        jobs.append((oracle.minplus(A, B, C), [torch.from_numpy(x.astype(npdt)).cuda() for x in (A, B, C)]))
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    with lib.Handle(device=0) as h:
        for rep in range(20):
            outs = []
            for i, (E, (A, B, C)) in enumerate(jobs[:4]):
                with torch.cuda.stream(streams[i % 2]):
                    outs.append((E, h.minplus(A, B, C.clone())))
            with torch.cuda.stream(streams[0]):  # 16-byte rows: the handle's own A^T
                E, (A, B, C) = jobs[4]
                outs.append((E, h.minplus(A, B, C.clone())))
            torch.cuda.synchronize()
            for E, D in outs:
                np.testing.assert_array_equal(D.cpu().numpy().astype(np.int64), E)


def test_growing_unaligned_sizes_reuse_the_copy(lib):
    """Sizes that share the panel buffer (steps of 256 vertices) share the copy too: a reallocation would
    synchronize the device in a call that is asynchronous."""
    buf = torch.empty(2559 * 2559, dtype=torch.int32, device="cuda")
    with lib.Handle(device=0, symmetric=2) as h:
        free = None
        for n in (2305, 2401, 2503, 2559):
            W = buf[:n * n].view(n, n)
            W.fill_(7).fill_diagonal_(0)
            h.solve_t("int32", W, W)
            torch.cuda.synchronize()
            now = torch.cuda.mem_get_info()[0]
            free = now if free is None else free
            assert now == free, n
            assert h.last_status() == 0 and int(W.max()) == 7 and int(W[n - 1, 0]) == 7
