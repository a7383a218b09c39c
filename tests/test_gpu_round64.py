"""64-wide rounds in two launches, cut left-over tiles, aligned copies, the batched kernel's modes and the
whole-matrix passes, at the sizes where each can go wrong, against the oracle (GPU).  int32 and packed 16-bit are
exact; fp32 runs on whole-number weights, whose sums are exact too."""
import numpy as np
import pytest

import gen
import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
INF = oracle.INF32
TD = {"int32": torch.int32, "u16": torch.int16, "fp32": torch.float32}


def graph(n, seed, directed=False, deg=5.0):
    """Edges and the dense int32 matrix of an ER graph plus a path (directed: each edge one way only)."""
    s, d, w = gen.er_graph(n, seed, avg_degree=deg, wmax=90)
    W = np.full((n, n), INF, np.int32)
    np.minimum.at(W, (s, d), w)
    if not directed:
        np.minimum.at(W, (d, s), w)
    np.fill_diagonal(W, 0)
    return s, d, w, W


def to_dev(W, dtype, ld):
    n = W.shape[0]
    inf = {"int32": INF, "u16": 0x7FFF, "fp32": np.inf}[dtype]
    buf = torch.full((n, ld), 3, dtype=TD[dtype], device="cuda")
    buf[:, :n] = torch.from_numpy(np.where(W >= INF, inf, W.astype(np.float64))).cuda().to(TD[dtype])
    return buf


def back(D, n, dtype):
    a = D[:, :n].cpu().numpy().astype(np.float64)
    return np.where(a >= (0x7FFF if dtype == "u16" else INF), INF, a).astype(np.int64)


# the edges of a round, of a tile and of a panel chunk; rows with and without 16-byte alignment
@pytest.mark.parametrize("dtype", ["int32", "u16", "fp32"])
@pytest.mark.parametrize("n", [65, 79, 127, 129, 191, 193, 257, 383, 449, 641])
@pytest.mark.parametrize("directed", [False, True])
def test_rounds_at_edges(lib, dtype, n, directed):
    _, _, _, W = graph(n, n, directed)
    E = oracle.fw(W.astype(np.int64))
    with lib.Handle(device=0) as h:
        for ld in (n, (n + 7) // 8 * 8, (n + 7) // 8 * 8 + 64):
            Wd = to_dev(W, dtype, ld)
            D = h.solve_t(dtype, Wd, torch.full_like(Wd, 5))
            assert h.last_status() == 0
            np.testing.assert_array_equal(back(D, n, dtype), E)
            assert bool((D[:, n:] == 5).all())  # nothing is written past the n columns
            h.solve_t(dtype, Wd, Wd)  # in place
            np.testing.assert_array_equal(back(Wd, n, dtype), E)


# sizes whose last wave of tiles is cut into k-parts (2 and 4), ragged columns among them
@pytest.mark.parametrize("dtype", ["int32", "fp32"])
@pytest.mark.parametrize("n,ld,directed", [(2200, 2200, False), (2299, 2304, False), (2562, 2568, False),
                                           (1790, 1792, True)])
def test_cut_tiles(lib, dtype, n, ld, directed):
    s, d, w, W = graph(n, n, directed, deg=4.0)
    E = oracle.dijkstra(n, s, d, w, np.arange(n), directed=directed)
    with lib.Handle(device=0, phase3_variant=4, block_k=64) as h:
        D = h.solve_t(dtype, to_dev(W, dtype, ld))
        assert h.last_status() == 0
    np.testing.assert_array_equal(back(D, n, dtype), E)


def test_base_not_16_byte_aligned(lib):
    n = 300
    _, _, _, W = graph(n, 3)
    buf = torch.empty(n * n + 1, dtype=torch.int32, device="cuda")
    Wd = buf[1:].view(n, n)  # rows of 1200 bytes from a base that is not 16-byte aligned
    Wd.copy_(torch.from_numpy(W))
    E = oracle.fw(W.astype(np.int64))
    with lib.Handle(device=0) as h:
        D = torch.empty(n * n + 2, dtype=torch.int32, device="cuda")[2:].view(n, n)
        h.solve_t("int32", Wd, D)
        np.testing.assert_array_equal(D.cpu().numpy().astype(np.int64), E)
        h.solve_batch([Wd], [D.zero_()])
        np.testing.assert_array_equal(D.cpu().numpy().astype(np.int64), E)


def test_batch_directed_and_undirected_aligned_and_not(lib):
    """Per-graph symmetry, single-round graphs, copies with 16-byte rows and in-place graphs in one launch."""
    gs = [(n, directed) for n in (1, 33, 64, 65, 127, 130, 260, 515) for directed in (False, True)]
    Ws = [graph(n, 10 + n, directed)[3] if n > 1 else np.zeros((1, 1), np.int32) for n, directed in gs]
    with lib.Handle(device=0) as h:
        ins = [to_dev(W, "int32", W.shape[0] + (4 if i % 3 == 0 else 0)) for i, W in enumerate(Ws)]
        outs = [x if i % 2 else torch.empty_like(x) for i, x in enumerate(ins)]
        h.solve_batch(ins, outs)
        assert h.last_status() == 0
        for W, D in zip(Ws, outs):
            np.testing.assert_array_equal(back(D, W.shape[0], "int32"), oracle.fw(W.astype(np.int64)))


@pytest.mark.parametrize("n", [63, 64, 65, 200, 257])
def test_input_pass_checks_every_block(lib, n):
    """A negative weight, a weight above INF, a non-zero diagonal or one asymmetric entry at the corners and in the
    middle of the matrix are found (the last only changes the mode: the result stays exact)."""
    _, _, _, W = graph(n, n)
    spots = [(0, n - 1), (n - 1, 0), (n // 2, n // 3), (n // 3, n // 2), (n - 1, n - 2)]
    with lib.Handle(device=0) as h:
        for r, c in spots:
            for bad, status in ((-1, 1), (INF + 1, 4)):
                V = W.copy()
                V[r, c] = bad
                h.solve_t("int32", torch.from_numpy(V).cuda())
                assert h.last_status() == status, (r, c, bad)
            V = W.copy()
            V[r, c] = 1  # now directed
            D = h.solve_t("int32", torch.from_numpy(V).cuda())
            assert h.last_status() == 0
            np.testing.assert_array_equal(D.cpu().numpy().astype(np.int64), oracle.fw(V.astype(np.int64)))
        V = W.copy()
        V[n - 1, n - 1] = 2
        h.solve_t("int32", torch.from_numpy(V).cuda())
        assert h.last_status() == 1


@pytest.mark.parametrize("dtype", ["int32", "u16", "fp32"])
@pytest.mark.parametrize("m,k,n", [(257, 260, 301), (301, 203, 333), (128, 1000, 129)])
def test_minplus_unaligned_rows(lib, dtype, m, k, n):
    """Products whose B and C have no 16-byte rows, above the size from which they run on copies."""
    rng = np.random.default_rng(m * n)
    inf = 0x7FFF if dtype == "u16" else INF
    mats = []
    for shape in ((m, k), (k, n), (m, n)):
        x = rng.integers(0, 2000, size=shape)
        x[rng.random(shape) < 0.2] = inf
        mats.append(x)
    E = oracle.minplus(*mats)
    A, B, C = (torch.from_numpy(np.where(x >= inf, np.inf, x) if dtype == "fp32" else x).to(TD[dtype]).cuda()
               for x in mats)
    with lib.Handle(device=0) as h:
        h.minplus(A, B, C)
    got = C.cpu().numpy().astype(np.float64)
    np.testing.assert_array_equal(np.where(got >= inf, inf, got).astype(np.int64), np.minimum(E, inf))
