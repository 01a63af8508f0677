// divide_pair.cu -- the split-fp32 divide of both operands at depth <= 2 in
// one launch (two at depth 2), which also clears C (or its staging copy) where the combine adds
// into it: grid z is A, B, clear.  For small products the phases before the
// leaf kernel are launches, not bytes: cleared and divided by a memset and two
// kernels, n = 256 spent 16 of its 27 us there.  The leaf kernel that follows
// may start its prologue while this one runs (programmatic dependent launch).
#include "divide_impl.cuh"

namespace stark {
namespace {

// SIDES 0: A (and the clear after it), 1: B (the same), 2: both.  Depth 2 runs
// A and B in turn: its code is unrolled over 49 planes, and blocks of both sides
// on one SM fetched it past each other (3xTF32 at n = 1536 34.8 us in turn, 46.4
// together; 3xFP16 at n = 1694 29.3 and 38.4).  Depths 0 and 1 are faster
// together (3xTF32 at n = 1536, depth 1: 23.0 in turn, 17.9).
template <int OUT, int D, int SIDES>
__global__ void __launch_bounds__(256, 2)
    divide_pair_kernel(DivideArgs a, DivideArgs b, int vec_a, int vec_b, float* zero, int64_t zero_count) {
  grid_launch_dependents();
  // (the clear goes last, its lines are still in L2 when the leaf kernel adds:
  // first, 3xTF32 at n = 4096, depth 2 took 542 instead of 531 us)
  if (SIDES != 1 && blockIdx.z == 0) {
    divide_body<float, OUT, D, 0, 4, 0>(a, vec_a);
  } else if (SIDES != 0 && blockIdx.z == (SIDES == 1 ? 0 : 1)) {
    divide_body<float, OUT, D, 1, 4, 0>(b, vec_b);
  } else {
    const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x, step = (int64_t)gridDim.x * 256;
    for (int64_t i = t; i < zero_count / 4; i += step)
      reinterpret_cast<float4*>(zero)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t < zero_count % 4) zero[zero_count / 4 * 4 + t] = 0.f;
  }
}

template <int OUT, int D>
cudaError_t launch(const DivideArgs& a, const DivideArgs& b, void* zero, int64_t zero_bytes, cudaStream_t st) {
  if (a.L % 4 != 0 || a.ld < a.n) return cudaErrorInvalidValue;
  auto vec = [](const DivideArgs& x) { return x.ld % 4 == 0 && (reinterpret_cast<uintptr_t>(x.X) & 15) == 0 ? 1 : 0; };
  const int64_t blocks = (a.L * (a.L / 4) + 255) / 256;
  if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
  const auto go = [&](auto kernel, int parts, void* clear) {
    kernel<<<dim3((unsigned)blocks, 1, clear ? parts + 1 : parts), 256, 0, st>>>(
        a, b, vec(a), vec(b), static_cast<float*>(clear), zero_bytes / 4);
    count_launch();
    return cudaGetLastError();
  };
  if constexpr (D < 2) {
    return go(divide_pair_kernel<OUT, D, 2>, 2, zero);
  } else {
    const cudaError_t e = go(divide_pair_kernel<OUT, D, 0>, 1, nullptr);
    return e == cudaSuccess ? go(divide_pair_kernel<OUT, D, 1>, 1, zero) : e;
  }
}

template <int OUT>
cudaError_t by_depth(const DivideArgs& a, const DivideArgs& b, int depth, void* zero, int64_t bytes, cudaStream_t st) {
  switch (depth) {
    case 0: return launch<OUT, 0>(a, b, zero, bytes, st);
    case 1: return launch<OUT, 1>(a, b, zero, bytes, st);
    case 2: return launch<OUT, 2>(a, b, zero, bytes, st);
    default: return cudaErrorInvalidValue;
  }
}

__global__ void __launch_bounds__(256) unstage_kernel(const float* __restrict__ src, int64_t ld, float* __restrict__ C,
                                                     int64_t n) {
  for (int64_t r = blockIdx.y; r < n; r += gridDim.y)
    for (int64_t c = (int64_t)blockIdx.x * 1024 + threadIdx.x; c < n && c < (int64_t)(blockIdx.x + 1) * 1024; c += 256)
      C[r * n + c] = __ldcs(src + r * ld + c);
}

}  // namespace

cudaError_t launch_divide_pair(const DivideArgs& a, const DivideArgs& b, int depth, OutMode out, void* zero,
                               int64_t zero_bytes, cudaStream_t st) {
  if (out == kOutSplitBf16) return by_depth<kOutSplitBf16>(a, b, depth, zero, zero_bytes, st);
  if (out == kOutSplitTf32) return by_depth<kOutSplitTf32>(a, b, depth, zero, zero_bytes, st);
  if (out == kOutSplitFp16) return by_depth<kOutSplitFp16>(a, b, depth, zero, zero_bytes, st);
  return cudaErrorInvalidValue;
}

// (A pitched device copy took 9.6 us at n = 1001.)
cudaError_t launch_unstage(const float* src, int64_t ld, float* C, int64_t n, int num_sms, cudaStream_t st) {
  const int64_t cols = (n + 1023) / 1024, rows = n < 16 * num_sms ? n : 16 * num_sms;
  unstage_kernel<<<dim3((unsigned)cols, (unsigned)rows), 256, 0, st>>>(src, ld, C, n);
  count_launch();
  return cudaGetLastError();
}

}  // namespace stark
