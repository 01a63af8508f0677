"""FP64 sides that leave the last block of K a few inputs only (n mod leaf side
in 1..15).  Products of that block alone are held to the same proof as all
others: with the scale running along those few terms, C's lower left quadrant,
which has no other products, is accurate term by term, as in FP64."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -53


@pytest.mark.parametrize("n,L", [(129, 128), (137, 128), (143, 128)])
def test_few_terms_in_the_last_block(stark_lib, n, L):
    S = stark_lib
    k = n - L
    rng = np.random.default_rng(n)
    A, B = rng.uniform(-1, 1, (n, n)), np.zeros((n, n))
    B[L:, :L] = rng.uniform(0.5, 1, (k, L))
    # the scale of A falls along K as that of B rises
    s = 2.0 ** -np.linspace(0, 60, k) if k > 1 else np.ones(1)
    A[L:, L:] = rng.uniform(0.5, 1, (k, k)) * s
    B[L:, :L] *= s[::-1, None]
    with S.Plan(n, 1, S.DType.F64) as p:
        assert p.leaf == L
        C = p.mul(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()).cpu().numpy()
        p.check()
    want = oracle.gemm_classical(A, B)
    low = slice(L, n), slice(0, L)
    assert np.all(np.abs(C - want)[low] <= 2 * (k + 2) * U * (np.abs(A) @ np.abs(B))[low])


@pytest.mark.parametrize("n,d", [(129, 1), (143, 1), (193, 1), (389, 2), (777, 2), (897, 3), (963, 2), (1351, 3), (1793, 4)])
def test_sides_with_few_inputs_in_the_last_block(stark_lib, n, d):
    # ordinary inputs are proven there: repeatable bit for bit, which the
    # additions of a redone product are not
    S = stark_lib
    rng = np.random.default_rng(n)
    A, B = rng.uniform(-1, 1, (n, n)), rng.uniform(-1, 1, (n, n))
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    with S.Plan(n, d, S.DType.F64) as p:
        assert p.tile == (128, 128)
        C = p.mul(dA, dB)
        for _ in range(3):
            assert torch.equal(p.mul(dA, dB), C)
        p.check()
        part = sum(p.mul_leaves(dA, dB, lo, hi) for lo, hi in ((0, 2), (2, p.leaves)))
    want = oracle.gemm_classical(A, B)
    # an error of 1e-11 is far above rounding (n u sqrt(n) 2^d) and far below one lost digit product
    assert np.abs(C.cpu().numpy() - want).max() <= 1e-11
    assert np.abs(part.cpu().numpy() - want).max() <= 1e-11
