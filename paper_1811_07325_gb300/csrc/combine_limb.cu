// combine_limb.cu -- the combine of Alg. 5 for the F64 and I64 limb leaves as
// an ordered pass over stored leaf products.
//
// A leaf product adds into up to 2^d quadrants of C.  As 64-bit reductions in
// the leaf epilogue these came in bursts (all SMs end a tile together) at
// 225 G/s for fp64, 33 us of every 150 us tile at n = 4096, depth 2, and
// cleared C first; stored products cost 8 bytes per element instead, and this
// pass reads them once and writes every element of C once.  A level takes its
// additions as Alg. 1 writes them (C11 = M1 + M4 - M5 + M7, ...): 8 per four
// elements, 5.5 per element of C at depth 2 against 9 by the expanded sums,
// which matters because the SM adds two fp64 numbers a clock.
//
// One launch folds one or two levels; depths 3 and 4 take two launches, the
// first into planes of the products two levels up.
//
// The bounded integer leaves (fp32 products holding integers of at most 2^24,
// leaf_tc.cu) take the same pass with their own input type: as 64-bit
// reductions of 256 bytes a row piece from the epilogue, one per target, they
// kept the copy engine busy for 230 of the 350 us at n = 4096, depth 1.
#include <type_traits>

#include "stark_internal.h"

namespace stark {
namespace {

template <typename T, int W>
struct Cols {
  T v[W];
};
template <typename T, int W>
__device__ __forceinline__ Cols<T, W> operator+(const Cols<T, W>& a, const Cols<T, W>& b) {
  Cols<T, W> r;
#pragma unroll
  for (int e = 0; e < W; ++e) r.v[e] = a.v[e] + b.v[e];
  return r;
}
template <typename T, int W>
__device__ __forceinline__ Cols<T, W> operator-(const Cols<T, W>& a, const Cols<T, W>& b) {
  Cols<T, W> r;
#pragma unroll
  for (int e = 0; e < W; ++e) r.v[e] = a.v[e] - b.v[e];
  return r;
}

// Quadrants of a product from its seven sub-products.
template <typename V>
__device__ __forceinline__ void fold(const V (&m)[7], V (&c)[4]) {
  c[0] = ((m[0] + m[3]) - m[4]) + m[6];
  c[1] = m[2] + m[4];
  c[2] = m[1] + m[3];
  c[3] = ((m[0] - m[1]) + m[2]) + m[5];
}

// A thread owns W columns of one position (r, c) of the L x L leaf grid of one
// product (blockIdx.y) D levels up: 7^D vectors in, 4^D out.
template <typename T, typename TM, int D, int W>
__global__ void __launch_bounds__(256, W == 1 ? 4 : 2)
    combine_limb_kernel(const TM* __restrict__ M, int64_t L, T* __restrict__ out, int64_t out_plane, int64_t ld, int64_t n,
                        const int* __restrict__ skip) {
  using V = Cols<T, W>;
  if (skip && *skip != 0) return;
  const int64_t pos = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (pos >= L * (L / W)) return;
  const int64_t r = pos / (L / W), c = pos % (L / W) * W;
  constexpr int P = D == 0 ? 1 : D == 1 ? 7 : 49;
  const TM* src = M + (int64_t)blockIdx.y * P * L * L + r * L + c;
  out += (int64_t)blockIdx.y * out_plane;
  auto load = [&](int leaf) {
    V x;
    if constexpr (sizeof(TM) == 4) {  // integers held in fp32
      static_assert(W == 2, "8-byte loads");
      const float2 f = __ldcs(reinterpret_cast<const float2*>(src + (int64_t)leaf * L * L));
      x.v[0] = (T)(long long)__float2int_rn(f.x);
      x.v[1] = (T)(long long)__float2int_rn(f.y);
    } else if constexpr (W == 2) {
      const int4 raw = __ldcs(reinterpret_cast<const int4*>(src + (int64_t)leaf * L * L));
      x = *reinterpret_cast<const V*>(&raw);
    } else {
      x.v[0] = __ldcs(src + (int64_t)leaf * L * L);
    }
    return x;
  };
  const bool vec = W == 2 && (ld & 1) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  auto store = [&](int64_t row, int64_t col, const V& v) {
    if (row >= n || col >= n) return;
    T* dst = out + row * ld + col;
    if (vec && col + W <= n) {
      *reinterpret_cast<int4*>(dst) = *reinterpret_cast<const int4*>(&v);
    } else {
#pragma unroll
      for (int e = 0; e < W; ++e)
        if (col + e < n) dst[e] = v.v[e];
    }
  };
  if constexpr (D == 0) {
    store(r, c, load(0));
  } else if constexpr (D == 1) {
    V m[7], q[4];
#pragma unroll
    for (int i = 0; i < 7; ++i) m[i] = load(i);
    fold(m, q);
#pragma unroll
    for (int k = 0; k < 4; ++k) store(r + (k >> 1) * L, c + (k & 1) * L, q[k]);
  } else {
    // the outer level's sums grow product by product, in Alg. 1's order
    V s[16];
#pragma unroll
    for (int i = 0; i < 7; ++i) {
      V m[7], q[4];
#pragma unroll
      for (int k = 0; k < 7; ++k) m[k] = load(i * 7 + k);
      fold(m, q);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        // M1: 11 22; M2: 21 -22; M3: 12 22; M4: 11 21; M5: -11 12; M6: 22; M7: 11
        if (i == 0) s[k] = s[12 + k] = q[k];
        if (i == 1) s[8 + k] = q[k], s[12 + k] = s[12 + k] - q[k];
        if (i == 2) s[4 + k] = q[k], s[12 + k] = s[12 + k] + q[k];
        if (i == 3) s[k] = s[k] + q[k], s[8 + k] = s[8 + k] + q[k];
        if (i == 4) s[k] = s[k] - q[k], s[4 + k] = s[4 + k] + q[k];
        if (i == 5) s[12 + k] = s[12 + k] + q[k];
        if (i == 6) s[k] = s[k] + q[k];
      }
    }
#pragma unroll
    for (int o = 0; o < 4; ++o)
#pragma unroll
      for (int k = 0; k < 4; ++k)
        store(r + (2 * (o >> 1) + (k >> 1)) * L, c + (2 * (o & 1) + (k & 1)) * L, s[4 * o + k]);
  }
}

template <typename T, int D, typename TM>
cudaError_t fold_levels(const TM* M, int64_t L, int64_t products, T* out, int64_t out_plane, int64_t ld, int64_t n,
                        const int* skip, cudaStream_t st) {
  constexpr int W = std::is_same_v<TM, double> && D == 2 ? 1 : 2;
  const int64_t blocks = (L * (L / W) + 255) / 256;
  if (L % 2 != 0 || blocks > 0x7FFFFFFF || products > 65535) return cudaErrorInvalidValue;
  combine_limb_kernel<T, TM, D, W><<<dim3((unsigned)blocks, (unsigned)products), 256, 0, st>>>(M, L, out, out_plane, ld, n, skip);
  count_launch();
  return cudaGetLastError();
}

template <typename T, typename TM>
cudaError_t by_depth(const void* Mv, int depth, int64_t L, int64_t n, void* Cv, int64_t ldc, void* tmp, const int* skip,
                     cudaStream_t st) {
  const TM* M = static_cast<const TM*>(Mv);
  T* C = static_cast<T*>(Cv);
  T* mid = static_cast<T*>(tmp);
  const int64_t side = 4 * L;
  cudaError_t e;
  switch (depth) {
    case 0: return fold_levels<T, 0>(M, L, 1, C, 0, ldc, n, skip, st);
    case 1: return fold_levels<T, 1>(M, L, 1, C, 0, ldc, n, skip, st);
    case 2: return fold_levels<T, 2>(M, L, 1, C, 0, ldc, n, skip, st);
    case 3:
      e = fold_levels<T, 2>(M, L, 7, mid, side * side, side, side, skip, st);
      return e != cudaSuccess ? e : fold_levels<T, 1>(static_cast<const T*>(mid), side, 1, C, 0, ldc, n, skip, st);
    case 4:
      e = fold_levels<T, 2>(M, L, 49, mid, side * side, side, side, skip, st);
      return e != cudaSuccess ? e : fold_levels<T, 2>(static_cast<const T*>(mid), side, 1, C, 0, ldc, n, skip, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_combine_limb(const void* M, int depth, int64_t L, int64_t n, void* C, int64_t ldc, void* tmp,
                                InType t, const int* skip, cudaStream_t st) {
  switch (t) {
    case kInF64: return by_depth<double, double>(M, depth, L, n, C, ldc, tmp, skip, st);
    case kInI64: return by_depth<unsigned long long, unsigned long long>(M, depth, L, n, C, ldc, tmp, skip, st);
    default: return by_depth<unsigned long long, float>(M, depth, L, n, C, ldc, tmp, skip, st);
  }
}

}  // namespace stark
