"""The packed 16-bit min-plus product over the whole 16-bit range (GPU): a sum above 0xFFFF wraps in its own element
and leaves the neighbouring one alone, on every route of the product."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def reference(A, B, C):
    C = C.copy()
    for t in range(A.shape[1]):
        np.minimum(C, A[:, t:t + 1] + B[t:t + 1, :], out=C)  # uint16 arithmetic: modulo 2^16
    return C


def dev16(a, pad):
    buf = torch.full((a.shape[0], a.shape[1] + pad), -1, dtype=torch.int16, device="cuda")
    buf[:, :a.shape[1]] = torch.from_numpy(a.view(np.int16)).cuda()
    return buf[:, :a.shape[1]]


# a single element; 16-byte rows (the TMA-fed kernel); rows without, below and above the size from which the product
# runs on copies; more k-steps than one stage holds; both kinds of rows above the size from which the operands are
# looked at first
@pytest.mark.parametrize("m,k,n,pad", [(1, 1, 1, 0), (128, 64, 256, 0), (131, 130, 264, 0), (130, 70, 251, 0),
                                       (257, 260, 300, 1), (400, 300, 401, 0), (1024, 1000, 1032, 0),
                                       (1001, 1001, 1003, 0)])
@pytest.mark.parametrize("wide", ["many", "few", "A", "B", "none"])
def test_u16_product_wraps_in_its_own_element(lib, m, k, n, pad, wide):
    rng = np.random.default_rng([m, k, n, len(wide)])

    def draw(shape, share):
        a = rng.integers(0, 4000, size=shape).astype(np.uint16)
        a[rng.random(shape) < 0.1] = 0x7FFF
        big = rng.random(shape) < share
        a[big] = rng.integers(0x8000, 0x10000, size=int(big.sum())).astype(np.uint16)
        return a
    # with few large values most results stay ordinary sums, whose neighbours wrap
    A = draw((m, k), {"many": 0.5, "few": 0.02, "A": 0.02}.get(wide, 0.0))
    B = draw((k, n), {"many": 0.5, "few": 0.02, "B": 0.02}.get(wide, 0.0))
    C = rng.integers(0, 0x8000, size=(m, n)).astype(np.uint16)
    Cd = dev16(C, pad)
    with lib.Handle(device=0) as h:
        h.minplus(dev16(A, pad), dev16(B, pad), Cd)
        assert h.last_status() == 0
    np.testing.assert_array_equal(Cd.cpu().numpy().view(np.uint16), reference(A, B, C))


def test_one_wide_element_at_the_edges_is_seen(lib):
    """A single element above 0x7FFF in the last row or column of A or B decides for the loop that allows it."""
    m, k, n = 1001, 1001, 1003
    rng = np.random.default_rng(9)
    for which, r, c in (("A", 0, 0), ("A", m - 1, k - 1), ("B", 0, n - 1), ("B", k - 1, 0)):
        A = rng.integers(0, 4000, size=(m, k)).astype(np.uint16)
        B = rng.integers(0, 4000, size=(k, n)).astype(np.uint16)
        if which == "A":  # every sum of that row and k-step wraps: next to nothing is shorter
            A[r, c] = 0xFFFF
            B[c, :] = np.where(np.arange(n) % 2 == 0, 2, 4000)
        else:
            B[r, c] = 0xFFFF
            A[:, r] = 2
        C = np.full((m, n), 0x7FFF, np.uint16)
        Cd = dev16(C, 0)
        with lib.Handle(device=0) as h:
            h.minplus(dev16(A, 0), dev16(B, 0), Cd)
        np.testing.assert_array_equal(Cd.cpu().numpy().view(np.uint16), reference(A, B, C), err_msg=f"{which} {r} {c}")
