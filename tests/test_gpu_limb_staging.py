"""Host products of an F64 or I64 plan on a nearly full device: the staging sets
come before the digit planes.  With room for fewer than six matrices left, the
plan falls back to 8 bytes an operand element, whose products are right."""
import numpy as np
import pytest

import oracle
from paper_1811_07325_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,bound", [("F64", 0), ("I64", 0), ("I64", 8)])
def test_staging_comes_before_digit_planes(stark_lib, dtype, bound):
    S = stark_lib
    n, d = 4096, 2
    lim = bound or 1 << 20
    A, B = synth.integers(n, 52, 0, -lim, lim), synth.integers(n, 52, 1, -lim, lim)
    want = oracle.gemm_classical(A, B)
    if dtype == "F64":  # (integers below 2^53, with rounding errors below one half)
        A, B = A.astype(np.float64), B.astype(np.float64)
    with S.Plan(n, d, S.DType[dtype]) as p:
        if bound:
            p.set_input_bound(bound)
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        fill = torch.empty(free - (300 << 20), dtype=torch.uint8, device="cuda")  # two matrices of 128 MiB stay
        try:
            C = p.mul_host(A, B)
            again = p.mul_host(A, B)
        finally:
            del fill
            torch.cuda.empty_cache()
        assert np.array_equal(np.rint(C), want) and np.array_equal(np.rint(again), want)
        p.set_traversal(1)
        p.set_traversal(0)
        elems = p.leaves * p.leaf ** 2  # operands, a bounded plan's products, and tables
        assert p.workspace_bytes < elems * (16 + (4 if bound else 0)) + (1 << 20)
        assert np.array_equal(np.rint(p.mul_host(A, B)), want)
