// limb_bounds.cu -- what the F64 limb leaves need before their divide: for
// every leaf operand row of A and column of B an exponent e with |x| <= 2^e
// for all its elements, and the flag that sends a product to the CUDA cores.
//
// The bound comes from the inputs, not from the operand sums: one read of A
// and B gives the largest magnitude of every row (column) within every
// quadrant column (row) block of the deepest level, and a leaf's bound is the
// sum of its quadrants' maxima in the order of the divide's own additions, so
// by monotonicity of rounding no rounded operand sum exceeds it.  The read is
// bound by HBM; reducing the operand sums themselves would read them 7/4
// times per level instead of once.
#include "divide_impl.cuh"

namespace stark {
namespace {

// Magnitude bits: integer order is magnitude order, NaN above infinity.
__device__ __forceinline__ unsigned long long mag_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// Upper bound s 2^(2 (b - 1023)) of a sum of squares, in fp32 beside the biased
// exponent b of an early element (the FP64 pipe does two operations a clock):
// every element is rounded up to 21 significant bits from its high word, every
// addition rounds up.  Elements below 2^-60 of the base count as that.
struct SquareSum {
  float s = 0.f;
  int b = 0;
  uint32_t limit = 1;  // high words from here on move the base

  __device__ __forceinline__ void rebase(int to) {
    const int e = 2 * (b - to) > -126 ? 2 * (b - to) : -126;
    s = __fmul_ru(s, __uint_as_float((uint32_t)(127 + e) << 23));
    b = to;
  }
  // before add(): `hi`, the largest high word of the elements to come
  __device__ __forceinline__ void prepare(uint32_t hi) {
    if (hi >= limit) {
      rebase((int)(hi >> 20));
      limit = (uint32_t)(b + 32) << 20;
    }
  }
  __device__ __forceinline__ void add(unsigned long long mag) {
    const int t = max((int)(uint32_t)(mag >> 32) + 1 - (b << 20), -(60 << 20));
    const float f = __uint_as_float((uint32_t)(t + (127 << 20)) << 3);
    s = __fmaf_ru(f, f, s);
  }
  __device__ __forceinline__ void merge(float s2, int b2) {
    const int top = b > b2 ? b : b2;
    rebase(top);
    SquareSum o;
    o.s = s2;
    o.b = b2;
    o.rebase(top);
    s = __fadd_ru(s, o.s);
  }
  __device__ __forceinline__ double root() const {
    return (double)__fsqrt_ru(s) * __hiloint2double((b > 1 ? b : 1) << 20, 0);
  }
};

// blockIdx.z == 0: a warp takes one row of A in one column block; 1: a block
// takes 32 columns of B in one row block.  Rows and columns beyond n are zero.
__global__ void __launch_bounds__(256) limb_max_kernel(LimbBoundsArgs a) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int blocks = 1 << a.depth;
  const int64_t L = a.L;
  if (blockIdx.x == 0 && blockIdx.z == 0 && threadIdx.x == 0) *a.flag = 0;
  if (blockIdx.z == 0) {
    for (int64_t u = (int64_t)blockIdx.x * 8 + warp; u < a.npad * blocks; u += (int64_t)gridDim.x * 8) {
      const int64_t row = u / blocks, q = u % blocks;
      unsigned long long m = 0;
      SquareSum sq;
      if (row < a.n) {
        const int64_t c0 = q * L > a.koff ? q * L - a.koff : 0;
        const int64_t c1 = (q + 1) * L - a.koff < a.n ? (q + 1) * L - a.koff : a.n;
        const double* p = a.A + row * a.ld;
        int64_t c = c0 + lane;
        for (; c + 96 < c1; c += 128) {
          const unsigned long long x0 = mag_bits(p[c]), x1 = mag_bits(p[c + 32]), x2 = mag_bits(p[c + 64]),
                                   x3 = mag_bits(p[c + 96]);
          const unsigned long long g = max(max(x0, x1), max(x2, x3));
          m = max(m, g);
          sq.prepare((uint32_t)(g >> 32));
          sq.add(x0);
          sq.add(x1);
          sq.add(x2);
          sq.add(x3);
        }
        for (; c < c1; c += 32) {
          const unsigned long long x = mag_bits(p[c]);
          m = max(m, x);
          sq.prepare((uint32_t)(x >> 32));
          sq.add(x);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        sq.merge(__shfl_xor_sync(0xffffffffu, sq.s, o), __shfl_xor_sync(0xffffffffu, sq.b, o));
      }
      if (lane == 0) {
        a.max_a[q * a.npad + row] = __longlong_as_double((long long)m);
        a.norm_a[q * a.npad + row] = sq.root();
      }
    }
  } else {
    __shared__ unsigned long long part[8][32];
    __shared__ float part_s[8][32];
    __shared__ int part_b[8][32];
    const int64_t groups = a.npad / 32;
    for (int64_t u = blockIdx.x; u < groups * blocks; u += gridDim.x) {
      const int64_t col = u % groups * 32 + lane, q = u / groups;
      const int64_t r0 = q * L > a.koff ? q * L - a.koff : 0;
      const int64_t r1 = (q + 1) * L - a.koff < a.n ? (q + 1) * L - a.koff : a.n;
      unsigned long long m = 0;
      SquareSum sq;
      if (col < a.n) {
        const double* p = a.B + col;
        int64_t r = r0 + warp;
        for (; r + 56 < r1; r += 64) {
          unsigned long long x[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) x[e] = mag_bits(p[(r + 8 * e) * a.ld]);
          unsigned long long g = x[0];
#pragma unroll
          for (int e = 1; e < 8; ++e) g = max(g, x[e]);
          m = max(m, g);
          sq.prepare((uint32_t)(g >> 32));
#pragma unroll
          for (int e = 0; e < 8; ++e) sq.add(x[e]);
        }
        for (; r < r1; r += 8) {
          const unsigned long long x = mag_bits(p[r * a.ld]);
          m = max(m, x);
          sq.prepare((uint32_t)(x >> 32));
          sq.add(x);
        }
      }
      part[warp][lane] = m;
      part_s[warp][lane] = sq.s;
      part_b[warp][lane] = sq.b;
      __syncthreads();
      if (warp == 0) {
#pragma unroll
        for (int w = 1; w < 8; ++w) {
          m = max(m, part[w][lane]);
          sq.merge(part_s[w][lane], part_b[w][lane]);
        }
        a.max_b[q * a.npad + col] = __longlong_as_double((long long)m);
        a.norm_b[q * a.npad + col] = sq.root();
      }
      __syncthreads();
    }
  }
}

// One thread per (leaf, row of A) and (leaf, column of B).  Per depth, so that
// the terms sit in registers and their loads are in flight together (33 us at
// n = 1024, depth 3, with a loop over a local array).
// Grid y 2 and 3: the common exponents.  A row position i of the L x L leaf
// grid sees 4^D input quadrants; where their largest magnitudes (zeros aside)
// lie within a factor of four, all are turned to integers by one exponent
// ec = e(largest) + D, the operand sums are integer sums, and a leaf's digits
// are the sum shifted by ec - e(leaf): off by at most 2^(D + 2) of the 2^-62 R
// units per term, still 2^-57 R at depth 3, where an fp64 sum is rounded to
// 2^-53 (not at depth 4, where the check would allow twice as much for it).
template <int D>
__global__ void __launch_bounds__(256) limb_exp_kernel(LimbBoundsArgs a, int64_t leaves) {
  const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
  const int side = blockIdx.y & 1;
  if (blockIdx.y >= 2) {
    if (t >= a.L) return;
    const double* mq = side == 0 ? a.max_a : a.max_b;
    unsigned long long mx = 0, mn = ~0ull;
    for (int q = 0; q < (1 << D); ++q)  // blocks along K, then along the rows of A (columns of B)
#pragma unroll
      for (int r = 0; r < (1 << D); ++r) {
        const unsigned long long b = mag_bits(mq[q * a.npad + r * a.L + t]);
        mx = max(mx, b);
        if (b != 0) mn = min(mn, b);
      }
    const int ex = (int)(mx >> 52);
    int32_t ec = mx == 0 ? 0 : ex - 1023 + ((mx & 0xFFFFFFFFFFFFFull) ? 1 : 0) + D;
    // (magnitude bits: two exponents apart is a factor of four)
    if (D > kLimbFixedDepth || (mx != 0 && (ex == 2047 || ex < 8 || mn + (2ull << 52) < mx))) ec = kLimbZeroRow;
    (side == 0 ? a.common_a : a.common_b)[t] = ec;
    return;
  }
  if (t >= leaves * a.L) return;
  const int leaf = (int)(t / a.L);
  const int64_t i = t % a.L;  // row (side 0) or column (side 1) of the leaf
  const double* mx = side == 0 ? a.max_a : a.max_b;
  TermPair tp[D > 0 ? D : 1];
  int x = leaf;
#pragma unroll
  for (int k = D - 1; k >= 0; --k) {
    tp[k] = side == 0 ? terms_of<0>(x % 7) : terms_of<1>(x % 7);
    x /= 7;
  }
  // the divide adds level by level, the last level outermost: term u (bit k:
  // second term of level k + 1), folded pairwise from the top level down
  const double* nm = side == 0 ? a.norm_a : a.norm_b;
  double v[1 << D], w2[1 << D];
#pragma unroll
  for (int u = 0; u < (1 << D); ++u) {
    int64_t row = 0, col = 0;
    bool present = true;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const int q = (u >> k) & 1 ? tp[k].qb : tp[k].qa;
      present = present && q >= 0;
      row += (int64_t)((q >> 1) & 1) * (a.npad >> (k + 1));
      col += (int64_t)(q & 1) * (a.npad >> (k + 1));
    }
    v[u] = w2[u] = 0.0;
    if (present) {
      const int64_t at = side == 0 ? col / a.L * a.npad + row + i : row / a.L * a.npad + col + i;
      v[u] = mx[at];
      w2[u] = nm[at];
    }
  }
  // S_1 sums pairs that differ in bit 0 (the top level), S_2 in bit 1, ...
#pragma unroll
  for (int w = (1 << D) / 2; w > 0; w /= 2)
#pragma unroll
    for (int u = 0; u < w; ++u) {
      v[u] = v[2 * u] + v[2 * u + 1];
      w2[u] = w2[2 * u] + w2[2 * u + 1];
    }
  const unsigned long long b = mag_bits(v[0]);
  int32_t e = kLimbZeroRow, h = a.log_l + 2;
  if (b != 0) {
    const int ex = (int)(b >> 52);
    e = ex - 1023 + ((b & 0xFFFFFFFFFFFFFull) ? 1 : 0);  // smallest e with bound <= 2^e (normal numbers)
    if (ex == 2047 || e < -400 || e > 400) {
      *(volatile int*)a.flag = 1;
      e = 0;  // (any value: the product is redone)
    }
    // N <= 2^(half / 2), from the norm's high word plus one (the sums above
    // round to nearest); N >= R / 2, as every block's norm is at least its maximum
    const uint32_t nh = (uint32_t)((unsigned long long)__double_as_longlong(w2[0]) >> 32) + 1u;
    const int half = 2 * ((int)(nh >> 20) - 1023) + ((nh & 0xFFFFFu) <= 0x6A09Du ? 1 : 2);  // (0x1.6A09Ep0 <= sqrt(2))
    h = min(max(a.log_l + 2 * e - half, 0), a.log_l + 2);
  }
  (side == 0 ? a.expA : a.expB)[t] = e;
  (side == 0 ? a.slackA : a.slackB)[t] = h;
}

template <int D>
void launch_exp(const LimbBoundsArgs& a, int64_t leaves, cudaStream_t st) {
  limb_exp_kernel<D><<<dim3((unsigned)((leaves * a.L + 255) / 256), 4), 256, 0, st>>>(a, leaves);
}

}  // namespace

cudaError_t launch_limb_bounds(const LimbBoundsArgs& a, cudaStream_t st) {
  int64_t leaves = 1;
  for (int k = 0; k < a.depth; ++k) leaves *= 7;
  const int64_t units = a.npad << a.depth;  // rows of A; a block of 8 warps or 32 columns of B per 8 of them
  const int64_t blocks = (units + 31) / 32;
  limb_max_kernel<<<dim3((unsigned)(blocks < 2432 ? blocks : 2432), 1, 2), 256, 0, st>>>(a);
  count_launch();
  switch (a.depth) {
    case 0: launch_exp<0>(a, leaves, st); break;
    case 1: launch_exp<1>(a, leaves, st); break;
    case 2: launch_exp<2>(a, leaves, st); break;
    case 3: launch_exp<3>(a, leaves, st); break;
    case 4: launch_exp<4>(a, leaves, st); break;
    default: return cudaErrorInvalidValue;
  }
  count_launch();
  return cudaGetLastError();
}

}  // namespace stark
