"""What FP64 digit products must prove before they are taken.  Only the last
block of K and the last block of C's rows hold anything, so C's lower left block
is one leaf product.  Its terms cancel in pairs, exactly and in order, and one
pair of 2^-33 stays: FP64 has 2^-66 there, digit products have not (they drop
it).  The magnitude digits add up to `total` units over the first 128 of K; where
the integer operand sums of the depth (2^14 2^(depth - 7) sqrt(2) units for rows
without slack), the dropped products and the running sum may be off by more
than that proves, the product is redone in FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def last_block(K, a, b, full):
    """One row of A's last block and one column of B's: K - 2 terms that cancel
    in pairs (digits a and b over the first 128, then 64 where `full`), then the
    small pair, and a one on each side that sets the scale."""
    x, y = np.zeros(K), np.zeros(K)
    k = np.arange(K)
    sign = 1.0 - 2.0 * (k % 2)
    head = (k < 128) & (k < K - 4)
    x[head], y[head] = sign[head] * a / 64, b / 64
    if full:
        tail = (k >= 128) & (k < K - 4)
        x[tail], y[tail] = sign[tail], 1.0
    x[K - 4], y[K - 3] = 1.0, 1.0  # (beside zeros)
    x[K - 2] = y[K - 2] = 2.0 ** -33
    return x, y


# (192, 1): 64 terms are left of a leaf side of 128, 60 of them 2 x 2 units
@pytest.mark.parametrize("n,d,L,a,b,total", [(192, 1, 128, 2, 2, 240), (1024, 2, 256, 2, 3, 768), (2048, 3, 256, 3, 4, 1536),
                                             (128, 0, 128, 2, 2, 496)])
def test_unproven_products_are_redone(stark_lib, n, d, L, a, b, total):
    S = stark_lib
    at = n - L if n % L == 0 else n // L * L  # first row and K position of the last block
    K = n - at
    x, y = last_block(K, a, b, L > 128)
    assert int(np.sum(np.abs(x[:128]) * np.abs(y[:128]) * 4096)) == total
    A, B = np.zeros((n, n)), np.zeros((n, n))
    A[at:, at:] = x
    B[at:, :L] = y[:, None]
    if n % L:  # the rows that padding leaves the leaf's other products
        A[at - L + K:at, at:] = x
    with S.Plan(n, d, S.DType.F64) as p:
        assert p.leaf == L and p.tile == (128, 128)
        C = p.mul(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()).cpu().numpy()
        p.check()
    assert np.all(C[at:, :min(L, n)] == 2.0 ** -66)
