"""Small split-fp32 products: both operands divided (and C cleared) in one
launch, a tile's K range cut into slices while the tiles leave the SMs idle,
a single leaf stored straight into C, and the copy out of a staging C.  The
sizes take 8, 4, 2 and 1 slices, whole and ragged sides, and a C that tensor
maps cannot address; every element against the oracle's bound."""
import numpy as np
import pytest

import bounds
import oracle
from paper_1811_07325_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def check(S, dtype, n, d, L, C, A, B):
    A64, B64 = A.astype(np.float64), B.astype(np.float64)
    bound = bounds.componentwise_c(dtype, L, d, 0) * bounds.majorant(oracle, A64, B64, d, L)
    if dtype in bounds.FLOOR:
        bound = bound + bounds.FLOOR[dtype] * bounds.floor_majorant(oracle, A64, B64, d, L)
    assert np.all(np.abs(C.cpu().numpy().astype(np.float64) - oracle.gemm_classical(A64, B64)) <= bound)


# 128-wide tiles: 256/0 and 130/0 (L = 256) in 4 slices or more, 512/0 in 8, 512/1 in 4, 1024/0 in 2, 300/0 (L = 384)
# in 2, 1100/0 (L = 1152) in 1, 900/1 (28 tiles of 256) in 1 or, with 3xTF32, pairs in 2; 1280/0 (25 tiles) in 1 or
# pairs in 2; 1536/0 (36 tiles) stored by 144 CTAs; 1792/0 (49) and 2048/0 by pairs
@pytest.mark.parametrize("dtype", ["F32_SPLIT_BF16", "F32_SPLIT_TF32", "F32_SPLIT_FP16"])
@pytest.mark.parametrize("n,d", [(256, 0), (512, 0), (512, 1), (1024, 0), (1100, 0), (300, 0), (900, 1), (2048, 0),
                                 (130, 0), (257, 0), (1001, 0), (2047, 0), (1280, 0), (1536, 0), (1792, 0)])
def test_small_products(stark_lib, dtype, n, d):
    S = stark_lib
    A, B = synth.normal(n, 41 + n, 0), synth.normal(n, 41 + n, 1)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    with S.Plan(n, d, S.DType[dtype]) as p:
        C = torch.full((n, n), float("nan"), device="cuda")
        check(S, dtype, n, p.depth, p.leaf, p.mul(dA, dB, C), A, B)
        # a C (and inputs) that start off a 16-byte boundary
        raw = torch.full((n * n + 1,), float("nan"), device="cuda")
        view = raw[1:].view(n, n)
        ua = torch.empty(n * n + 1, device="cuda")[1:].view(n, n).copy_(dA)
        check(S, dtype, n, p.depth, p.leaf, p.mul(ua, dB, view), A, B)
        assert torch.isnan(raw[0])
        # the leaves one by one add up to the product, and a captured product replays
        total = sum(p.mul_leaves(dA, dB, l, l + 1) for l in range(p.leaves))
        assert (total - C).abs().max() <= 1e-5 * C.abs().max()
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            p.mul(dA, dB, C)
        C.fill_(float("nan"))
        for _ in range(2):
            g.replay()
        torch.cuda.synchronize()
        check(S, dtype, n, p.depth, p.leaf, C, A, B)
        p.check()


@pytest.mark.parametrize("dtype", ["F32_SPLIT_BF16", "F32_SPLIT_TF32"])
def test_single_leaf_members_of_batches_and_the_server(stark_lib, dtype):
    S = stark_lib
    sizes = [256, 130, 512, 301, 640]
    ins = [(synth.normal(n, 42 + n, 0), synth.normal(n, 42 + n, 1)) for n in sizes]
    dev = [tuple(torch.from_numpy(x).cuda() for x in p) for p in ins]
    Cs = [torch.full((n, n), float("nan"), device="cuda") for n in sizes]
    with S.Batch(sizes, 0, S.DType[dtype]) as b:
        for _ in range(2):  # recorded, then replayed
            b.mul([a for a, _ in dev], [x for _, x in dev], Cs)
            b.check()
    for n, C, (A, B) in zip(sizes, Cs, ins):
        check(S, dtype, n, 0, (n + 127) // 128 * 128, C, A, B)
        C.fill_(float("nan"))
    torch.cuda.synchronize()
    with S.Server(8 << 30, 2) as srv:
        ids = [srv.submit(a, x, C, S.DType[dtype]) for (a, x), C in zip(dev, Cs)]
        srv.drain()
        assert all(srv.poll(i) == (True, S.Status.OK) for i in ids)
    torch.cuda.synchronize()
    for n, C, (A, B) in zip(sizes, Cs, ins):  # (the server chooses the depth: the bound of depth 1 covers it)
        check(S, dtype, n, 1, (n + 255) // 256 * 128, C, A, B)
