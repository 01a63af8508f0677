"""FP64 products from digit products are no less accurate than FP64 itself, by
measured error and not by a bound: the RMS error against the exact product
stays within the oracle's, which adds and multiplies in FP64 in the same
recursion (a product that is redone on the CUDA cores has that error, up to
the order of its additions: 10 %).

An entry is A1 + A2 2^-22, of about 26 bits and 22 bits, so the exact product
comes from four int64 ones, rounded to a whole number (the errors are tens to
hundreds).  Besides plain data: rows and columns with one element far above the
rest, which set the scale of the digits, in all rows or in every third one
(neighbouring rows then have unlike units)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ONE = 2.0 ** 26


def entries(kind, n, seed):
    """(A1, A2), (B1, B2): two n x n matrices with entries of about ONE."""
    rng = np.random.default_rng(seed)

    def matrix(top):
        if kind == "uniform":
            return rng.uniform(-1, 1, (n, n))
        if kind == "normal":
            return rng.standard_normal((n, n))
        x = rng.uniform(0.9, 1.1, (n, n)) * rng.choice([-1, 1], (n, n))
        rows = np.arange(0, n, 3 if kind == "mixed" else 1)
        x[rows, rng.integers(0, n, rows.size)] = rng.uniform(top / 2 + 1, top - 1, rows.size)
        return x

    def parts(x):
        high = np.rint(x * ONE).astype(np.int64)
        return high, rng.integers(-(1 << 21), 1 << 21, (n, n))

    return parts(matrix(32)), parts(np.ascontiguousarray(matrix(16).T))


def exact_product(A, B):
    low = (oracle.gemm_classical(A[0], B[1]) + oracle.gemm_classical(A[1], B[0])) * 2.0 ** -22
    return oracle.gemm_classical(A[0], B[0]) + np.rint(low + oracle.gemm_classical(A[1], B[1]) * 2.0 ** -44).astype(np.int64)


def rms(C, exact):
    return np.sqrt(np.mean((np.rint(C).astype(np.int64) - exact).astype(np.float64) ** 2))


@pytest.mark.parametrize("kind", ["uniform", "normal", "outliers", "mixed"])
@pytest.mark.parametrize("n,d", [(1024, 0), (1024, 1), (1024, 2), (1024, 3), (1088, 0)])
def test_f64_error_is_no_larger_than_in_fp64(stark_lib, kind, n, d):
    S = stark_lib
    A, B = entries(kind, n, 61)
    exact = exact_product(A, B)
    Af, Bf = (x[0] + x[1] * 2.0 ** -22 for x in (A, B))
    want = rms(oracle.strassen(Af, Bf, d), exact)
    with S.Plan(n, d, S.DType.F64) as p:
        C = p.mul(torch.from_numpy(Af).cuda(), torch.from_numpy(Bf).cuda())
        p.check()
    got = rms(C.cpu().numpy(), exact)
    print(f"{kind} n={n} d={d}: {got / want:.3f}")
    assert got <= 1.1 * want, (got, want)
