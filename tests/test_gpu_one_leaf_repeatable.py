"""A one-leaf product (depth 0) with the default combine is repeatable bit for
bit: every element of C has one contribution, or two of them (K slices) added
to zero.  Sizes at which the tiles leave most SMs idle, whole and ragged, and
a C through the staging copy; sixty runs of each, which the arrival order of
more slices does not survive."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["F32_SPLIT_BF16", "F32_SPLIT_TF32", "F32_SPLIT_FP16"])
@pytest.mark.parametrize("n", [130, 256, 512, 513, 1001])
def test_one_leaf_products_are_repeatable(stark_lib, dtype, n):
    S = stark_lib
    gen = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn((n, n), generator=gen, device="cuda")
    B = torch.randn((n, n), generator=gen, device="cuda")
    with S.Plan(n, 0, S.DType[dtype]) as p:
        first = p.mul(A, B).clone()
        for _ in range(60):
            assert torch.equal(p.mul(A, B), first)
        p.check()


@pytest.mark.parametrize("dtype", ["F32_SPLIT_BF16", "F32_SPLIT_TF32", "F32_SPLIT_FP16"])
@pytest.mark.parametrize("lo,hi", [(0, 1), (1, 3), (4, 7)])
def test_leaf_ranges_with_few_contributions_are_repeatable(stark_lib, dtype, lo, hi):
    # one leaf, two leaves (M2 and M3 meet in C22), three (M5 and M7 meet in C11): at most two additions to zero
    S = stark_lib
    n = 512
    gen = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn((n, n), generator=gen, device="cuda")
    B = torch.randn((n, n), generator=gen, device="cuda")
    with S.Plan(n, 1, S.DType[dtype]) as p:
        first = p.mul_leaves(A, B, lo, hi).clone()
        for _ in range(60):
            assert torch.equal(p.mul_leaves(A, B, lo, hi), first)
        p.check()
