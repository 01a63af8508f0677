"""The work that the library's speed is measured on.

Each case is one call (or one graph replay, or one burst of requests) through
the public entry points of ``paper_1811_07325_gb300.stark``: ``Plan.mul`` for
a single product, ``Batch.mul`` for many, ``Server.submit``/``drain`` for
requests.  Sizes are those of the repository's benchmark and tests (n = 1024
in FP64 at depth 3; n = 4096 in FP64 and int64; n = 16384 in fp32 with split
leaves; 64 products of sizes 512 to 4096; a stream of requests of sizes 256
and up), with the smallest and ragged sizes of the same ranges beside them.
"""
import math
import random

import torch

from paper_1811_07325_gb300 import stark

DTYPES = {
    "bf16": stark.DType.F32_SPLIT_BF16,
    "tf32": stark.DType.F32_SPLIT_TF32,
    "fp16": stark.DType.F32_SPLIT_FP16,
    "f64": stark.DType.F64,
    "i64": stark.DType.I64,
}
SPLIT = ("bf16", "tf32", "fp16")

# Member sizes of a batch, as in the benchmark's batched workload.
BATCH_SIZES = (512, 768, 1024, 1536, 2048, 3072, 4096)
SERVE_LOW, SERVE_HIGH = 256, 4096


def _mul(dtype, n, depth, combine=0, promotion=0, bound=0):
    return {"kind": "mul", "dtype": dtype, "n": n, "depth": depth, "combine": combine, "promotion": promotion,
            "bound": bound}


def listed():
    return [
        # one small product, depth chosen by the library: what a caller with
        # many little matrices waits for (launches and latency)
        {"name": "bf16_n256", **_mul("bf16", 256, -1)},
        # a ragged size that no tile divides and whose rows TMA cannot address
        {"name": "bf16_n1001", **_mul("bf16", 1001, -1)},
        # the middle of the served and batched sizes, as a single product
        {"name": "bf16_n2048", **_mul("bf16", 2048, -1)},
        # 3xTF32 leaves at the size of the depth sweep
        {"name": "tf32_n4096_d2", **_mul("tf32", 4096, 2)},
        # the FP32-accurate configuration: 3xFP16 with promoted accumulation
        {"name": "fp16_n8192_d2_promoted", **_mul("fp16", 8192, 2, combine=2, promotion=256)},
        # the headline: n = 16384, depth 2, 3xBF16, reproducible combine
        {"name": "bf16_n16384_d2", **_mul("bf16", 16384, 2, combine=2)},
        # plain Strassen in FP64 at the paper's smallest size, 128 x 128 leaves
        {"name": "f64_n1024_d3", **_mul("f64", 1024, 3)},
        # plain Strassen in FP64 at GPU scale
        {"name": "f64_n4096_d2", **_mul("f64", 4096, 2)},
        # exact integers with no declared bound (entries of any size)
        {"name": "i64_n4096_d2", **_mul("i64", 4096, 2)},
        # exact integers in [-16, 16], the bound declared to the plan
        {"name": "i64_n4096_d1_bound16", **_mul("i64", 4096, 1, bound=16)},
        # the batched form: 64 products of mixed sizes in one call
        {"name": "batch64_bf16", "kind": "batch", "dtype": "bf16", "count": 64, "sizes_seed": 1},
        # the served form: a burst of requests of mixed sizes, submitted and drained
        {"name": "serve32_bf16", "kind": "serve", "dtype": "bf16", "count": 32, "sizes_seed": 2},
    ]


def _log_uniform(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["split", "split", "split", "f64", "i64", "bound", "batch", "serve"])
    if kind == "split":
        dtype = rng.choice(SPLIT)
        n = _log_uniform(rng, 128, 12288)
        if rng.random() < 0.5:  # half of the sizes are whole multiples of 64
            n = max(128, n // 64 * 64)
        depth = rng.choice([-1, -1, 0, 1, 2, 3]) if n >= 1024 else rng.choice([-1, 0, 1])
        combine = rng.choice([0, 2])
        # promotion needs leaf sides that are multiples of 256
        promotion = 256 if depth >= 0 and (n + (128 << depth) - 1) // (128 << depth) % 2 == 0 \
            and rng.random() < 0.5 else 0
        return _mul(dtype, n, depth, combine=combine, promotion=promotion)
    if kind == "f64":
        n = _log_uniform(rng, 192, 4096)
        depths = [-1, 0, 1] if n < 512 else [-1, 0, 1, 2, 3] if n <= 3072 else [-1, 2, 3]
        return _mul("f64", n, rng.choice(depths))
    if kind == "i64":
        n = _log_uniform(rng, 192, 4096)
        return _mul("i64", n, rng.choice([-1, 0, 1, 2, 3]) if n >= 512 else rng.choice([-1, 0, 1]))
    if kind == "bound":
        # leaf sides that are multiples of 128 and within the exactness bound
        depth = rng.choice([1, 2])
        leaf = 128 * rng.randint(2, 16 if depth == 1 else 8)
        return _mul("i64", (leaf << depth) - rng.choice([0, 0, 1, 30]), depth, bound=16)
    if kind == "batch":
        return {"kind": "batch", "dtype": rng.choice(SPLIT), "count": rng.randint(4, 64),
                "sizes_seed": rng.randint(1, 1 << 20)}
    return {"kind": "serve", "dtype": rng.choice(["bf16", "fp16"]), "count": rng.randint(4, 32),
            "sizes_seed": rng.randint(1, 1 << 20)}


def _sizes(case):
    if case["kind"] == "mul":
        return [case["n"]]
    rng = random.Random(case["sizes_seed"])
    if case["kind"] == "batch":
        return [rng.choice(BATCH_SIZES) for _ in range(case["count"])]
    return [_log_uniform(rng, SERVE_LOW, SERVE_HIGH) for _ in range(case["count"])]


def _inputs(case, seed):
    """[(A, B)] of the case, from the seed alone."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def one(n):
        if case["dtype"] == "i64":
            if case["bound"]:
                b = case["bound"]
                return torch.randint(-b, b + 1, (n, n), generator=gen, device="cuda", dtype=torch.int64)
            return torch.randint(-(1 << 62), 1 << 62, (n, n), generator=gen, device="cuda", dtype=torch.int64)
        if case["dtype"] == "f64":  # uniform [-1, 1)
            return torch.rand((n, n), generator=gen, device="cuda", dtype=torch.float64) * 2 - 1
        if case["kind"] == "batch":
            return torch.rand((n, n), generator=gen, device="cuda", dtype=torch.float32) * 2 - 1
        return torch.randn((n, n), generator=gen, device="cuda", dtype=torch.float32)

    return [(one(n), one(n)) for n in _sizes(case)]


def prepare(case, seed):
    pairs = _inputs(case, seed)
    As, Bs = [p[0] for p in pairs], [p[1] for p in pairs]
    Cs = [torch.empty_like(a) for a in As]
    dt = DTYPES[case["dtype"]]
    state = {"kind": case["kind"], "dt": dt, "As": As, "Bs": Bs, "Cs": Cs}
    if case["kind"] == "mul":
        plan = stark.Plan(case["n"], case["depth"], dt)
        if case["bound"]:
            plan.set_input_bound(case["bound"])
        if case["combine"]:
            plan.set_combine(case["combine"])
        if case["promotion"]:
            plan.set_promotion(case["promotion"])
        state["plan"] = plan
    elif case["kind"] == "batch":
        state["batch"] = stark.Batch([a.shape[0] for a in As], -1, dt)
    else:
        state["server"] = stark.Server(32 << 30, 4)
        torch.cuda.synchronize()  # the server works on streams of its own
    return state


def run(state):
    As, Bs, Cs = state["As"], state["Bs"], state["Cs"]
    if state["kind"] == "mul":
        return state["plan"].mul(As[0], Bs[0], Cs[0])
    if state["kind"] == "batch":
        state["batch"].mul(As, Bs, Cs)
        return Cs
    server = state["server"]
    ids = [server.submit(a, b, c, state["dt"]) for a, b, c in zip(As, Bs, Cs)]
    server.drain()
    for rid in ids:
        server.poll(rid)
    return Cs


def work(case):
    esz = 8 if case["dtype"] in ("f64", "i64") else 4
    sizes = _sizes(case)
    nbytes = sum(3 * n * n * esz for n in sizes)
    # leaf arithmetic of the method: 7/8 of the classical products per level,
    # three half-precision products for each one of the split dtypes
    levels = max(case.get("depth", 0), 0)
    terms = 3 if case["dtype"] in SPLIT else 1
    flops = sum(2.0 * n ** 3 for n in sizes) * (7.0 / 8.0) ** levels * terms
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    if case["dtype"] == "i64":
        return None  # whole numbers: compared as they are
    out = [a.double() @ b.double() for a, b in _inputs(case, seed)]
    return out[0] if case["kind"] == "mul" else out
