// divide_limb.cu -- the divide phase (Alg. 3) of the I64 and F64 limb leaves:
// every leaf operand sum, formed as in divide.cu, is written as eight fp16
// digit planes (leaf_limb.cu).  Both operands go in one launch (grid z), at
// every depth; the prefixes of depths 3 and 4 are the grid's y dimension.
#include "divide_impl.cuh"

namespace stark {
namespace {

template <typename Tin, int D>
__global__ void __launch_bounds__(256, 2) divide_limb_kernel(DivideArgs a, DivideArgs b, int vec_a, int vec_b) {
  if (blockIdx.z == 0)
    divide_body<Tin, kOutLimbs, D, 0, 2, 0>(a, vec_a);
  else
    divide_body<Tin, kOutLimbs, D, 1, 2, 0>(b, vec_b);
}

template <typename Tin, int D>
cudaError_t launch(const DivideArgs& a, const DivideArgs& b, cudaStream_t st) {
  if (a.L % 2 != 0 || a.ld < a.n) return cudaErrorInvalidValue;
  auto vec = [](const DivideArgs& x) { return x.ld % 2 == 0 && (reinterpret_cast<uintptr_t>(x.X) & 15) == 0 ? 1 : 0; };
  const int64_t blocks = (a.L * (a.L / 2) + 255) / 256;
  if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
  constexpr int F = D < 2 ? 0 : D - 2;
  divide_limb_kernel<Tin, D><<<dim3((unsigned)blocks, (unsigned)pow7c(F), 2), 256, 0, st>>>(a, b, vec(a), vec(b));
  count_launch();
  return cudaGetLastError();
}

template <typename Tin>
cudaError_t by_depth(const DivideArgs& a, const DivideArgs& b, int depth, cudaStream_t st) {
  switch (depth) {
    case 0: return launch<Tin, 0>(a, b, st);
    case 1: return launch<Tin, 1>(a, b, st);
    case 2: return launch<Tin, 2>(a, b, st);
    case 3: return launch<Tin, 3>(a, b, st);
    case 4: return launch<Tin, 4>(a, b, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_divide_limbs(const DivideArgs& a, const DivideArgs& b, int depth, InType in, cudaStream_t st) {
  if (in == kInI64) return by_depth<int64_t>(a, b, depth, st);
  if (in == kInF64) return by_depth<double>(a, b, depth, st);
  return cudaErrorInvalidValue;
}

}  // namespace stark
