// divide_limb.cu -- the divide phase (Alg. 3) of the I64 and F64 limb leaves:
// every leaf operand sum, formed as in divide.cu, is written as eight fp16
// digit planes (leaf_limb.cu).  Both operands go in one launch (grid z), at
// every depth; the prefixes of depths 3 and 4 are the grid's y dimension.
#include "divide_impl.cuh"

namespace stark {
namespace {

// (One level in registers and seven times the blocks for small leaves was
// slower: int64, n = 1024, depth 3, 126 instead of 57 us.)
// F64 sums are integer sums where this thread's row (columns) have a common
// exponent (limb_bounds.cu): fp64 additions, two a clock and SM, and a
// conversion per leaf instead of one per input made the pass with its bounds 581
// instead of 512 us at n = 4096, depth 2.
template <typename Tin, int D, int SIDE>
__device__ __forceinline__ void limb_body(const DivideArgs& a, int vec) {
  if constexpr (std::is_same_v<Tin, double> && D <= kLimbFixedDepth) {
    const int64_t pos = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, per_row = a.L / 2;
    if (pos >= a.L * per_row) return;
    const int64_t i = pos / per_row, j = pos % per_row * 2;
    const bool fixed = a.common[SIDE == 0 ? i : j] != kLimbZeroRow && a.common[SIDE == 0 ? i : j + 1] != kLimbZeroRow;
    if (fixed) {
      divide_body<FixedF64, kOutLimbs, D, SIDE, 2, 0>(a, vec);
      return;
    }
  }
  divide_body<Tin, kOutLimbs, D, SIDE, 2, 0>(a, vec);
}

template <typename Tin, int D>
__global__ void __launch_bounds__(256, 2) divide_limb_kernel(DivideArgs a, DivideArgs b, int vec_a, int vec_b) {
  if (blockIdx.z == 0)
    limb_body<Tin, D, 0>(a, vec_a);
  else
    limb_body<Tin, D, 1>(b, vec_b);
}

// The plain fp64 operands of a product that is redone (a.gate set): both
// divides and, on the last z, C cleared, in one launch that usually does
// nothing.
template <int D>
__global__ void __launch_bounds__(256, 2) redo_divide_kernel(DivideArgs a, DivideArgs b, int vec_a, int vec_b,
                                                            unsigned long long* C) {
  if (*(volatile const int*)a.gate == 0) return;
  if (blockIdx.z == 0) {
    divide_body<double, kOutPlain, D, 0, 2, 0>(a, vec_a);
  } else if (blockIdx.z == 1) {
    divide_body<double, kOutPlain, D, 1, 2, 0>(b, vec_b);
  } else if (blockIdx.y == 0) {
    for (int64_t r = blockIdx.x; r < a.n; r += gridDim.x)
      for (int64_t c = threadIdx.x; c < a.n; c += 256) C[r * a.ld + c] = 0ull;
  }
}

int vec2_ok(const DivideArgs& x) { return x.ld % 2 == 0 && (reinterpret_cast<uintptr_t>(x.X) & 15) == 0 ? 1 : 0; }

template <typename Tin, int D>
cudaError_t launch(const DivideArgs& a, const DivideArgs& b, cudaStream_t st) {
  if (a.L % 2 != 0 || a.ld < a.n) return cudaErrorInvalidValue;
  const int64_t blocks = (a.L * (a.L / 2) + 255) / 256;
  if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
  constexpr int F = D < 2 ? 0 : D - 2;
  divide_limb_kernel<Tin, D><<<dim3((unsigned)blocks, (unsigned)pow7c(F), 2), 256, 0, st>>>(a, b, vec2_ok(a), vec2_ok(b));
  count_launch();
  return cudaGetLastError();
}

template <int D>
cudaError_t launch_redo(const DivideArgs& a, const DivideArgs& b, void* C, cudaStream_t st) {
  const int64_t blocks = (a.L * (a.L / 2) + 255) / 256;
  if (blocks > 0x7FFFFFFF || !a.gate) return cudaErrorInvalidValue;
  constexpr int F = D < 2 ? 0 : D - 2;
  redo_divide_kernel<D><<<dim3((unsigned)blocks, (unsigned)pow7c(F), 3), 256, 0, st>>>(
      a, b, vec2_ok(a), vec2_ok(b), static_cast<unsigned long long*>(C));
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

cudaError_t launch_redo_divide(const DivideArgs& a, const DivideArgs& b, int depth, void* C, cudaStream_t st) {
  switch (depth) {
    case 0: return launch_redo<0>(a, b, C, st);
    case 1: return launch_redo<1>(a, b, C, st);
    case 2: return launch_redo<2>(a, b, C, st);
    case 3: return launch_redo<3>(a, b, C, st);
    case 4: return launch_redo<4>(a, b, C, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace stark
