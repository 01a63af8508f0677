"""The depth that the autotuner takes (depth -1) costs no accuracy: at sizes
where two depths differ by a microsecond or two and by up to a factor of two in
error (3xFP16, 3xTF32: the deeper is the more accurate; small 3xBF16: the
shallower), batch members, requests and plans have the error of the more
accurate depth, measured against FP64 and not against the bound.  The members
at explicit depths have the same kernels and inputs, so their errors are equal
up to the order of additions; 10 % stands for that."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,sizes,depth", [("F32_SPLIT_FP16", [448, 576, 640, 704, 768], 1),
                                               ("F32_SPLIT_TF32", [384, 448, 704, 768, 1024], 1),
                                               ("F32_SPLIT_BF16", [256, 512, 1024], 0)])
def test_automatic_depth_has_the_error_of_the_accurate_one(stark_lib, dtype, sizes, depth):
    S = stark_lib
    dt = S.DType[dtype]
    gen = torch.Generator(device="cuda").manual_seed(7)
    As = [torch.randn((n, n), generator=gen, device="cuda") for n in sizes]
    Bs = [torch.randn((n, n), generator=gen, device="cuda") for n in sizes]
    want = [a.double() @ b.double() for a, b in zip(As, Bs)]

    def errors(Cs):
        return [((c.double() - w).norm() / w.norm()).item() for c, w in zip(Cs, want)]

    def batch(d):
        Cs = [torch.empty_like(a) for a in As]
        with S.Batch(sizes, d, dt) as b:
            b.mul(As, Bs, Cs)
            b.check()
        return errors(Cs)

    limit = [1.1 * e for e in batch(depth)]
    member = batch(-1)
    Cs = [torch.empty_like(a) for a in As]
    torch.cuda.synchronize()
    with S.Server(8 << 30, 2) as srv:
        ids = [srv.submit(a, b, c, dt) for a, b, c in zip(As, Bs, Cs)]
        srv.drain()
        assert all(srv.poll(i) == (True, S.Status.OK) for i in ids)
    torch.cuda.synchronize()
    request = errors(Cs)
    for i, n in enumerate(sizes):
        with S.Plan(n, -1, dt) as p:
            Cs[i] = p.mul(As[i], Bs[i])
            p.check()
    plan = errors(Cs)
    for got in (member, request, plan):
        assert all(e <= m for e, m in zip(got, limit)), (got, limit)
