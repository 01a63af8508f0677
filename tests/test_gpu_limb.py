"""The I64 and F64 leaves as digit products on the tensor cores (leaf sides of
at least 128): exact integers, FP64 within the classical bound, and the
products whose accuracy the digits cannot prove redone on the CUDA cores.

Sizes sit at the edges of the tiling: one tile, a size just above it, leaf
sides of 64 mod 128 (half a tile outside the plane, a last superchunk of 64 of
K), padded and ragged sides, depths 0 to 4."""
import numpy as np
import pytest

import oracle
from paper_1811_07325_gb300 import synth

torch = pytest.importorskip("torch")
U = 2.0 ** -53
SIZES = [(128, 0), (129, 0), (300, 0), (512, 0), (191, 1), (256, 1), (513, 2), (400, 1), (700, 2), (777, 2), (1024, 3),
         (1100, 3), (2100, 4)]


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def strassen_bound(n, d, L, A, B):
    """Higham, Accuracy and Stability, Thm 23.2, for ours and the oracle's rounding."""
    return 2 * ((12 ** d * (L * L + 5 * L) - 5 * n) + n) * U * np.abs(A).max() * np.abs(B).max()


# ------------------------------------------------------------------ CPU: the arithmetic
def digits(q):
    """Eight balanced base-256 digits of an integer mod 2^64, least significant first."""
    t = (q + 0x8080808080808080) % 2 ** 64
    return [((t >> (8 * i)) & 255) - 128 for i in range(8)]


def test_digits_recover_products_mod_2_64():
    rng = np.random.default_rng(5)
    edge = [0, 1, -1, 127, 128, -128, -129, 2 ** 63 - 1, -2 ** 63, 0x7F7F7F7F7F7F7F7F, 0x8080808080808080]
    vals = edge + [int(x) for x in rng.integers(-2 ** 63, 2 ** 63 - 1, 40)]
    for x in vals:
        dx = digits(x)
        assert all(-128 <= v <= 127 for v in dx)
        for y in vals:
            dy = digits(y)
            low = sum(dx[i] * dy[j] << (8 * (i + j)) for i in range(8) for j in range(8) if i + j <= 7)
            assert (low - x * y) % 2 ** 64 == 0


def test_fixed_point_products_are_within_the_stated_error():
    # |x| <= 2^e as round(x 2^(62 - e)), the digit products of weight >= 256^7:
    # a K-term sum is off by at most K (2 * 2^-63 (1 + 2^-63) + 7 * 2^14 (256^6 + ...) 2^-124) R C < K 2^-59 R C
    from fractions import Fraction
    rng = np.random.default_rng(6)
    for K in (1, 7, 64):
        for spread in (0, 20, 60):
            x = rng.uniform(-1, 1, K) * 2.0 ** -rng.integers(0, spread + 1, K)
            y = rng.uniform(-1, 1, K) * 2.0 ** -rng.integers(0, spread + 1, K)
            e, f = (int(np.ceil(np.log2(np.abs(v).max()))) for v in (x, y))
            total = 0
            for a, b in zip(x, y):
                da = digits(round(Fraction(a) * Fraction(2) ** (62 - e)))[::-1]
                db = digits(round(Fraction(b) * Fraction(2) ** (62 - f)))[::-1]
                total += sum(da[i] * db[j] * 256 ** (14 - i - j) for i in range(8) for j in range(8) if i + j <= 7)
            want = sum(Fraction(a) * Fraction(b) for a, b in zip(x, y))
            got = Fraction(total) * Fraction(2) ** (e + f - 124)
            assert abs(got - want) <= K * Fraction(2) ** (-59 + e + f)


# ------------------------------------------------------------------ GPU
@pytest.mark.gpu
@pytest.mark.parametrize("n,d", SIZES)
def test_int64_any_entries_exact(stark_lib, n, d):
    S = stark_lib
    A = synth.integers(n, 31 + n, 0, -2 ** 63, 2 ** 63 - 1)
    B = synth.integers(n, 31 + n, 1, -2 ** 63, 2 ** 63 - 1)
    A[0, :] = -2 ** 63  # every digit at the end of its range
    B[:, 0] = -(0x8080808080808080 - 2 ** 63)
    with S.Plan(n, d, S.DType.I64) as p:
        assert p.tile == (128, 128)
        C = p.mul(dev(A), dev(B))
        p.check()
    assert np.array_equal(C.cpu().numpy(), oracle.gemm_classical(A, B))


@pytest.mark.gpu
@pytest.mark.parametrize("n,d", SIZES)
def test_f64_within_classical_bound_and_repeatable(stark_lib, n, d):
    S = stark_lib
    A, B = synth.uniform(n, 32 + n, 0), synth.normal(n, 32 + n, 1).astype(np.float64)
    want = oracle.gemm_classical(A, B)
    with S.Plan(n, d, S.DType.F64) as p:
        assert p.tile == (128, 128)
        dA, dB = dev(A), dev(B)
        C = p.mul(dA, dB).cpu().numpy()
        again = p.mul(dA, dB).cpu().numpy()
        p.check()
        L = p.leaf
    assert np.array_equal(C, again)
    if d == 0:
        assert np.all(np.abs(C - want) <= 2 * (n + 2) * U * (np.abs(A) @ np.abs(B)))
    else:
        assert np.abs(C - want).max() <= strassen_bound(n, d, L, A, B)


@pytest.mark.gpu
def test_f64_unproven_products_are_redone(stark_lib):
    S = stark_lib
    n = 256
    R = synth.normal(n, 33, 0).astype(np.float64)
    s = np.logspace(-12, 12, n)
    cases = [(np.eye(n), R),                      # one term per element
             (R * s, R / s[:, None]),             # the scale runs along K
             (R * 1e-250, R * 1e200),             # exponents outside the digits' range
             (np.tril(R), np.triu(R))]            # few terms near the corners
    with S.Plan(n, 0, S.DType.F64) as p:
        for A, B in cases:
            C = p.mul(dev(A), dev(B)).cpu().numpy()
            p.check()
            assert np.all(np.abs(C - oracle.gemm_classical(A, B)) <= 2 * (n + 2) * U * (np.abs(A) @ np.abs(B)))
        A, B = R.copy(), R.copy()
        A[3, 5], B[7, 2], B[9, 4] = np.inf, np.nan, -np.inf
        C = p.mul(dev(A), dev(B)).cpu().numpy()
        with np.errstate(invalid="ignore"):
            want = A @ B
        assert np.array_equal(np.isnan(C), np.isnan(want))
        assert np.array_equal(C[np.isinf(want)], want[np.isinf(want)])
        # and a clean product on the same plan afterwards
        C = p.mul(dev(R), dev(R)).cpu().numpy()
        assert np.all(np.abs(C - oracle.gemm_classical(R, R)) <= 2 * (n + 2) * U * (np.abs(R) @ np.abs(R)))
        # zero rows and columns need no proof
        Z = R.copy()
        Z[100:] = 0
        assert np.array_equal(p.mul(dev(Z), dev(Z.T)).cpu().numpy()[100:], np.zeros((n - 100, n)))


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [2.0 ** -1, 2.0 ** -30])
@pytest.mark.parametrize("d", [1, 2])
def test_f64_row_blocks_of_different_scale(stark_lib, d, scale):
    # rows of the lower half (columns of B's left half) scaled: by one half the
    # quadrants share an exponent and the operand sums are integer sums, by
    # 2^-30 they do not; C21 has products of the scaled blocks only, and is
    # accurate at its own scale
    S = stark_lib
    n = 512
    A, B = synth.uniform(n, 35, 0), synth.normal(n, 35, 1).astype(np.float64)
    A[n // 2:] *= scale
    B[:, : n // 2] *= scale
    want = oracle.gemm_classical(A, B)
    with S.Plan(n, d, S.DType.F64) as p:
        C = p.mul(dev(A), dev(B)).cpu().numpy()
        p.check()
        L = p.leaf
    assert np.abs(C - want).max() <= strassen_bound(n, d, L, A, B)
    h = slice(n // 2, n), slice(0, n // 2)
    assert np.abs(C - want)[h].max() <= strassen_bound(n, d, L, A[h[0]], B[:, h[1]])


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,n,d,peel", [("I64", 600, 1, False), ("F64", 600, 1, False), ("I64", 650, 2, True),
                                            ("F64", 650, 2, True)])
def test_limb_leaf_ranges_traversal_and_capture(stark_lib, dtype, n, d, peel):
    # partial products (added into C) sum to the product; the depth-first
    # traversal (CUDA cores) agrees; a captured product replays
    S = stark_lib
    if dtype == "I64":
        A, B = synth.integers(n, 34, 0, -2 ** 62, 2 ** 62), synth.integers(n, 34, 1, -2 ** 62, 2 ** 62)
    else:
        A, B = synth.uniform(n, 34, 0), synth.uniform(n, 34, 1)
    want = oracle.gemm_classical(A, B)
    dA, dB = dev(A), dev(B)
    with S.Plan(n, d, S.DType[dtype], peel=peel) as p:
        tol = 0 if dtype == "I64" else strassen_bound(n, d, p.leaf, A, B) * 4

        def same(C):
            C = C.cpu().numpy()
            assert np.array_equal(C, want) if dtype == "I64" else np.abs(C - want).max() <= tol

        total = torch.zeros_like(dA)
        for lo, hi in ((0, 3), (3, 4), (4, p.leaves)):
            total += p.mul_leaves(dA, dB, lo, hi)
        same(total)
        C = p.mul(dA, dB)
        same(C)
        g = torch.cuda.CUDAGraph()
        C.zero_()
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            p.mul(dA, dB, C)
        g.replay()
        torch.cuda.synchronize()
        same(C)
        p.set_traversal(1)
        same(p.mul(dA, dB))
        p.set_traversal(0)
        same(p.mul(dA, dB))
        p.check()
