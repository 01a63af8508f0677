"""Device memory of F64 and I64 plans off the digit-product path: depth-first
and sharded plans hold their subtrees' operands at 8 bytes an element and
nothing else (no product planes, no side arrays), and get all of it back with
the whole breadth-first product.  The tables' share is taken from a plan of
the same depth whose leaves (side 64) never have digit planes."""
import numpy as np
import pytest

import oracle
from paper_1811_07325_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def tables(S, dt, d):
    with S.Plan(64 << d, d, dt) as p:
        assert p.leaf == 64
        return p.workspace_bytes - 2 * p.leaves * 64 * 64 * 8


@pytest.mark.parametrize("dtype,bound", [("F64", 0), ("I64", 0), ("I64", 8)])
def test_workspace_off_the_breadth_first_product(stark_lib, dtype, bound):
    S = stark_lib
    dt = S.DType[dtype]
    n, d = 512, 2
    fixed = tables(S, dt, d)
    lim = bound or 1 << 20
    A, B = synth.integers(n, 51, 0, -lim, lim), synth.integers(n, 51, 1, -lim, lim)
    want = oracle.gemm_classical(A, B)
    if dtype == "F64":  # (integers below 2^53, with rounding errors below one half)
        A, B = A.astype(np.float64), B.astype(np.float64)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    with S.Plan(n, d, dt) as p:
        if bound:
            p.set_input_bound(bound)
        whole = p.workspace_bytes
        L, P = p.leaf, p.leaves

        def right():
            assert np.array_equal(np.rint(p.mul(dA, dB).cpu().numpy()), want)
            p.check()

        right()
        p.set_traversal(1)
        assert p.workspace_bytes == fixed + 2 * (P // 7) * L * L * 8
        if bound:  # declared again on a depth-first plan
            p.set_input_bound(0)
            p.set_input_bound(bound)
            assert p.workspace_bytes == fixed + 2 * (P // 7) * L * L * 8
        right()
        p.set_traversal(0)
        assert p.workspace_bytes == whole
        right()
        total = torch.zeros_like(dA)
        for lo, hi, planes in ((0, 20, 21), (20, P, 35)):  # (whole subtrees of 7 leaves)
            p.set_shard(lo, hi)
            assert p.workspace_bytes == fixed + 2 * planes * L * L * 8
            total += p.mul_leaves(dA, dB, lo, hi)
            p.check()
        assert np.array_equal(np.rint(total.cpu().numpy()), want)
        p.set_shard(1, P)  # (every subtree, but not the whole product)
        assert p.workspace_bytes == fixed + 2 * P * L * L * 8
        p.set_shard(0, P)
        assert p.workspace_bytes == whole
        right()
