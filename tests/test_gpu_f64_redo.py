"""FP64 products that are redone on the CUDA cores give up their digit products
early: the flag goes up in the first tiles, in a middle one, in the last, or in
the bounds (NaN), with several tiles for every SM and with fewer tiles than SMs;
whole, ragged and peeled sides, whole products and leaf ranges.  The result is
FP64's, and a clean product on the same plan follows.  A redone product takes
little more than the same leaves on the CUDA cores (a depth-first plan's)."""
import numpy as np
import pytest

import oracle
from paper_1811_07325_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -53


def bound(n, d, L, A, B):
    """Higham, Accuracy and Stability, Thm 23.2, for ours and the oracle's rounding."""
    return 2 * ((12 ** d * (L * L + 5 * L) - 5 * n) + n) * U * np.abs(A).max() * np.abs(B).max()


@pytest.mark.parametrize("n,d,peel", [(1024, 1, False), (1024, 2, False), (1100, 3, False), (300, 1, False), (1001, 2, False),
                                      (1030, 2, True), (2100, 4, False), (700, 0, False)])
@pytest.mark.parametrize("where", ["all", "first", "middle", "last", "nan"])
def test_redone_products(stark_lib, n, d, peel, where):
    S = stark_lib
    R, T = synth.uniform(n, 71, 0), synth.uniform(n, 71, 1)
    A = R.copy()
    if where == "all":
        A = np.tril(R)
    elif where == "nan":
        A[n // 2, 3] = np.nan
    else:  # one row that has one large element and is small beside it
        row = {"first": 0, "middle": n // 2, "last": n - 1}[where]
        A[row] *= 1e-9
        A[row, n // 3] = 1.0
    dA, dB, dR = (torch.from_numpy(x).cuda() for x in (A, T, R))
    want, clean = oracle.gemm_classical(A, T), oracle.gemm_classical(R, T)
    with S.Plan(n, d, S.DType.F64, peel=peel) as p:
        tol = bound(n, d, p.leaf, R, T)
        for C in (p.mul(dA, dB), p.mul_leaves(dA, dB, 0, p.leaves // 2) + p.mul_leaves(dA, dB, p.leaves // 2, p.leaves)):
            C = C.cpu().numpy()
            p.check()
            if where == "nan":
                # the recursion spreads a NaN over its row and column classes, and at depth 0 to its row alone
                assert np.isnan(C[n // 2]).all() and (d > 0 or np.isnan(C).sum() == n)
            else:
                assert np.abs(C - want).max() <= tol
        assert np.abs(p.mul(dR, dB).cpu().numpy() - clean).max() <= tol
        p.check()


def test_redone_products_take_the_cuda_cores_time(stark_lib):
    S = stark_lib
    n, d = 2048, 1
    A, B = torch.eye(n, dtype=torch.float64, device="cuda"), torch.rand((n, n), dtype=torch.float64, device="cuda")
    C = torch.empty_like(A)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def best(p):
        times = []
        for _ in range(6):
            e0.record()
            p.mul(A, B, C)
            e1.record()
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        return min(times)

    with S.Plan(n, d, S.DType.F64) as p:
        redone = best(p)
        assert (C - B).abs().max().item() <= 16 * U  # (sums of up to four entries below one, and their differences)
        p.set_traversal(1)
        direct = best(p)
        p.check()
    # bounds and the digits' divide on top: 0.1 of 13 ms (the leaves' digit products are another 0.45)
    assert redone <= 1.03 * direct, (redone, direct)
