"""The 16-bit bound on graphs as deep as they have vertices (GPU): unit-weight paths, where the relaxation has to
run a hop for every vertex before its keys are final.  The bound of a path that starts at vertex 0 is 2 (n - 1)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
INF = 1073741823
ORDERS = ("ascending", "descending", "shuffled")


def path_ids(n, order, seed=0):
    """The vertices along the path; vertex 0 at one end."""
    ids = np.arange(n)
    if order == "descending":
        ids[1:] = ids[:0:-1]
    elif order == "shuffled":
        ids[1:] = np.random.default_rng([n, seed]).permutation(ids[1:])
    return ids


def path_edges(ids, order, seed=0):
    """(src, dst) int32 on the GPU, listed along the path, against it or shuffled."""
    e = np.arange(len(ids) - 1)
    if order == "descending":
        e = e[::-1]
    elif order == "shuffled":
        e = np.random.default_rng([len(ids), seed, 1]).permutation(e)
    return tuple(torch.from_numpy(x.astype(np.int32)).cuda() for x in (ids[e], ids[e + 1]))


def path_dense(ids):
    n = len(ids)
    W = torch.full((n, n), INF, dtype=torch.int32, device="cuda")
    i = torch.from_numpy(ids).cuda()
    W[i[:-1], i[1:]] = 1
    W[i[1:], i[:-1]] = 1
    W.fill_diagonal_(0)
    return W


def check_path(h, ids, order, seed=0):
    n = len(ids)
    assert h.int16_bound(path_dense(ids)) == (2 * (n - 1), True), (n, order)
    s, d = path_edges(ids, order, seed)
    w = torch.ones(n - 1, dtype=torch.int16, device="cuda")
    D = h.solve_edges("u16", s, d, w, n)  # raises when the bound refuses the graph
    assert h.last_status() == 0
    row = np.empty(n, np.int64)
    row[ids] = np.arange(n)  # distances from vertex 0
    np.testing.assert_array_equal(D[0].cpu().numpy().astype(np.int64), row)


@pytest.mark.parametrize("order", ORDERS)
def test_bound_of_every_short_path(lib, order):
    with lib.Handle(device=0) as h:
        for n in range(2, 131):
            check_path(h, path_ids(n, order), order)


@pytest.mark.parametrize("order", ORDERS)
@pytest.mark.parametrize("n", [1000, 2030, 16000])
def test_bound_of_long_paths(lib, n, order):
    with lib.Handle(device=0) as h:
        check_path(h, path_ids(n, order), order)


def test_bound_beside_a_batched_launch(lib):
    """The relaxation's blocks then run when the batched kernel leaves room for them, not together."""
    n = 1024
    g = torch.Generator(device="cuda").manual_seed(1)
    Ws = []
    for _ in range(64):
        W = torch.randint(1, 1000, (n, n), generator=g, device="cuda", dtype=torch.int32)
        Ws.append(W.fill_diagonal_(0))
    Ds = [torch.empty_like(W) for W in Ws]
    ids = path_ids(2030, "shuffled", 7)
    W0, (s, d) = path_dense(ids), path_edges(ids, "shuffled", 7)
    w = torch.ones(len(ids) - 1, dtype=torch.int16, device="cuda")
    side = torch.cuda.Stream()
    with lib.Handle(device=0) as hb, lib.Handle(device=0) as h:
        hb.solve_batch(Ws, Ds)
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            for _ in range(6):
                hb.solve_batch(Ws, Ds)
        main = torch.cuda.Stream()
        with torch.cuda.stream(main):
            assert h.int16_bound(W0) == (2 * 2029, True)
            D = h.solve_edges("u16", s, d, w, len(ids))
        torch.cuda.synchronize()
        assert int(D[0].max()) == 2029
