// leaf_limb.cu -- exact int64 and FP64 leaf products (Alg. 4) on the tensor
// cores, from operands split into eight signed base-256 digits ("limbs").
//
// The CUDA cores multiply 64-bit integers at 6.85 TOP/s and FP64 at
// 1.25 TFLOP/s; the tensor cores run fp16 products three orders of magnitude
// faster.  A digit in [-128, 127] is exact in fp16, a product of two at most
// 2^14, and a sum of up to 1024 such products exact in the fp32 accumulator,
// so a digit GEMM over K <= 128 with at most eight products per k (or K <= 256
// with four) is exact
// integer arithmetic.  With x = sum_i x_i 256^i and y likewise,
//   I64  x y mod 2^64 = sum_{s <= 7} 256^s D_s,      D_s = sum_{i+j=s} x_i y_j
// (the divide writes plane i = digit i, least significant first), and
//   F64  x y ~= sum_{s <= 7} 256^(14-s) D_s, planes most significant first:
// an operand row (column of B) is scaled by a power of two to integers of at
// most 2^62 and the digit products below 256^7 are dropped.  36 digit
// products replace one 64-bit product: at most 52 T(FL)OP/s at the measured
// fp16 rate of 1869 TFLOP/s.
//
// One CTA per SM takes 128 x 128 tiles of the leaves in turn:
//   warp 0      TMA producer: quads (four digit planes of 128 rows or columns
//               x 32 of K, 32 KB, one or two copies) into six shared-memory slots
//   warp 1      TMEM allocation, MMA issuer
//   warps 4..11 epilogue: two warps per TMEM lane quarter, 64 columns each
//               (two warpgroups with 208 registers a thread, the first one
//               keeps 88; 128 x 88 + 256 x 208 are the 384 x 168 of the launch).
//               Each phase's diagonals are drained from TMEM, converted to
//               int32 (exact) and added into a 64-bit running sum held in
//               registers; after the last superchunk the sums (F64: rescaled
//               and rounded once) are stored, for a whole product, or added into
//               the leaf's C targets by atomics, for a range of its leaves.
//
// Order of the products.  TMEM holds four 128 x 128 accumulators, so K runs in
// superchunks of 256 with three phases: twice, for each 128 of K, diagonals
// 7, 6, 5, 4 on accumulators 0, 1, 2, 3 over all digits (26 products a block;
// quads A0-3, B0-3, B4-7, A4-7 of each K block), then for all 256 diagonals
// 3, 2, 1, 0 on accumulators 3, 2, 1, 0 over the low four digits (10 products,
// at most four per diagonal, so exact over twice the K).  A block of 32 of K costs 72 MMAs for
// 192 KB of operands.  Each phase ends its accumulators one after another in
// the order in which the other phase starts on them, so that the epilogue
// drains one while the tensor cores fill the others.  All of this order is
// fixed at compile time: with the tiles taken one by one from a table of
// steps, the issuing thread needed 760 cycles a step on its own and the
// kernel ran at 30 % of the fp16 rate (6.5 ms for 49 leaves of side 1024).
//
// F64 accuracy.  R and C are the powers of two that bound a row of the left
// operand and a column of the right one, k the terms that are not padding and u
// 2^-53.  A k-term FP64 dot product is bound to k u sum |a||b|; against the exact
// product of its operands the digits' is off by at most
//   drop     k 7.03 2^-62 R C: the digit products below 256^7, 7 of up to 2^14 at
//            256^6, 6 at 256^5, ...;
//   operand  for operand elements off by eps R (eps C), eps (R sum |b| +
//            C sum |a|), where sum |b| <= sqrt(k) times b's 2-norm.  An fp64 sum
//            is rounded to a digit unit, eps = 2^-63; an integer sum (depths 1 to
//            3, limb_bounds.cu) is off by up to eps = 2^(depth - 60);
//   sum      half a unit of the running sum for every diagonal that is rounded
//            to it, two or three in 128 of K.  The sum keeps 64 bits, so its unit
//            follows from the most that the product can be: by Cauchy and Schwarz
//            at most the product of the 2-norms of its row and column, which
//            limb_bounds.cu has as R C 2^l (2^l >= L) less the slacks of both.
//            With the slack of its own row and the least of its warp's 64
//            columns, the unit is 2^(l - 62) R C less that: at most 2^-60 of
//            those bounds' product unless a column stands out among the 64.
//            (With the unit of rows without slack, rows of 1024 elements of about
//            one with a single one of up to 32 were off by 5 times as much as
//            in FP64.)
// and by one rounding of the result, u sum |a||b|, of FP64's k.  So the digits
// keep FP64's bound unless nearly every |a||b| is far below R C (badly scaled
// or sparse rows), and the kernel proves for each element that it is not: over
// the first 128 of K the digit products of magnitudes, sum |a_0||b_0|, must reach
// LimbNeed, else it raises `flag` and the product is redone on the CUDA cores
// (as for infinities, NaN and exponents outside +-400, flagged by the bounds
// kernel).  A magnitude digit is 64 at the bound and may be rounded up from one
// half, so T units are at least T / 4 / 64^2 R C of sum |a||b|, and the three
// errors ask for 225, 2^14 eps / u (...) and 16 a rounded diagonal (plan.cu; 1 %
// is for the digit's half and a bit, k / (k - 1) for the result's rounding).
// These are bounds.  The errors themselves are an order of magnitude below
// FP64's on data without structure (tests/test_gpu_f64_accuracy.py).  The worst
// kind met is entries whose bits end at the top bit of a digit, 31 to 33 bits
// below R: that digit is -128 or 0, and the dropped products add up, 2^-64 R C a
// term.  At 512 units that was 1.07 times FP64's error; kLimbLeast is 640.
// Padding leaves every leaf at least 64 terms to prove it by (limb_k_offset in
// plan.cu).
//
// Splitting operands so that slices multiply without rounding, and summing the
// slices' products, is Ozaki's scheme (Ozaki, Ogita, Oishi and Rump 2012).
#include <cstring>

#include "leaf_common.cuh"

namespace stark {
namespace {

constexpr int kThreadsL = 384;
constexpr int kDigits = 8;
constexpr int kQuadBytes = 32768;                  // four digit planes: 128 rows x 64 bytes (A), or two 64-column
                                                   // chunks of 32 rows x 128 bytes each (B)
constexpr int kQuads = 6;
constexpr int kEpiStride = 72;                     // bytes per staged row of 8 results: 64, and 8 so that the
                                                   // rows start in different banks
constexpr int kEpiBytes = 8 * (32 * kEpiStride + 256);  // and the exponents of each warp's 64 columns
constexpr int kBarBytes = 8 * (2 * kQuads + 8) + 16;
constexpr int kSmemLimb = kQuads * kQuadBytes + kEpiBytes + 1024 + kBarBytes;
static_assert(kSmemLimb <= 232448, "shared memory per CTA");
// acc + v 2^32, on the high word alone.
__device__ __forceinline__ long long add_high(long long acc, uint32_t v) {
  const uint32_t hi = (uint32_t)((unsigned long long)acc >> 32) + v;
  return (long long)(((unsigned long long)hi << 32) | (uint32_t)acc);
}

// acc + v mul.  (The sums are kept mod 2^64: only the last one has to fit.)
__device__ __forceinline__ long long add_wide(long long acc, int v, int mul) {
  return (long long)((unsigned long long)acc + (unsigned long long)((long long)v * mul));
}

// v * 2^e rounded to nearest (ties away), from integer operations (the FP64
// pipe does two operations a clock); |result| stays in the normal range.
__device__ __forceinline__ unsigned long long scaled_double_bits(long long v, int e) {
  const long long sign = v >> 63;
  unsigned long long u = (unsigned long long)((v ^ sign) - sign);
  const int lz = __clzll((long long)u);
  u <<= lz & 63;  // bit 63 set
  // 53 bits and the rounding; a carry to 2^53 goes into the exponent
  const unsigned long long m = (u >> 11) + ((u >> 10) & 1ull);
  const unsigned long long bits = ((unsigned long long)(unsigned)(e + 1085 - lz) << 52) + m;
  return v == 0 ? 0ull : bits | ((unsigned long long)sign & 0x8000000000000000ull);
}

template <bool F64>
__global__ void __launch_bounds__(kThreadsL, 1)
    leaf_limb_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const __grid_constant__ CUtensorMap tmSA, const __grid_constant__ CUtensorMap tmSB,
                     const LeafLimbArgs p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  unsigned char* smem = smem_raw + ((1024 - (raw_addr & 1023)) & 1023);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t epi_base = sbase + kQuads * kQuadBytes;
  const uint32_t bar_base = epi_base + kEpiBytes;
  auto full_bar = [&](int s) { return bar_base + 8 * s; };
  auto empty_bar = [&](int s) { return bar_base + 8 * (kQuads + s); };
  auto accf_bar = [&](int a) { return bar_base + 8 * (2 * kQuads + a); };
  auto acce_bar = [&](int a) { return bar_base + 8 * (2 * kQuads + 4 + a); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kQuads * kQuadBytes + kEpiBytes + 8 * (2 * kQuads + 8));
  // F64: set by the producer, ahead of the barrier of a tile's first quad, once
  // the product's flag is up: the product is redone, and no role goes on
  volatile int* stop = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x / 32;
  const int lane = threadIdx.x % 32;
  const int tiles = (p.L + 127) / 128;  // per side: a leaf side of 64 mod 128 ends in a tile half outside the plane
  const int per_leaf = tiles * tiles;
  const int num_items = (p.leaf_end - p.leaf_begin) * per_leaf;
  const int kblocks = p.L / 32;         // even
  const int chunks = (kblocks + 3) / 4;  // 128 of K each, the last one possibly 64

  if (threadIdx.x == 0) {
    *stop = 0;
    for (int s = 0; s < kQuads; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 4; ++a) {
      mbar_init(accf_bar(a), 1);
      mbar_init(acce_bar(a), 8);
    }
    fence_mbar_init();
    prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
    if (warp == 0 && lane == 0) {
      // ---------------------------------------------------------- producer

      const uint64_t pol_a = policy_evict_normal();
      const uint64_t pol_b = policy_evict_last();  // a leaf's B panels are re-read by its rows of tiles
      int slot = 0;
      uint32_t phase = 0;  // parity of the ring's turns
      uint32_t armed = 0, armed_phase = 0;
      bool ok = true;
      // the next free slot (0: none in time)
      auto next = [&]() -> uint32_t {
        if (!mbar_wait_bounded(empty_bar(slot), phase ^ 1, p.err, kDevTimeoutEmpty, p.timeout_ns)) return 0;
        mbar_arrive_expect_tx(full_bar(slot), kQuadBytes);
        return sbase + (uint32_t)slot * kQuadBytes;
      };
      auto done = [&]() {
        armed |= 1u << slot;
        armed_phase = (armed_phase & ~(1u << slot)) | (phase << slot);
        if (++slot == kQuads) {
          slot = 0;
          phase ^= 1;
        }
        return true;
      };
      auto load_a = [&](int k, int m0, int plane) -> bool {
        const uint32_t st = next();
        if (!st) return false;
        tma_load_3d(st, &tmA, k, m0, plane, full_bar(slot), pol_a);
        return done();
      };
      auto load_b = [&](int k, int n0, int plane) -> bool {
        const uint32_t st = next();
        if (!st) return false;
        tma_load_3d(st, &tmB, n0, k, plane, full_bar(slot), pol_b);
        tma_load_3d(st + kQuadBytes / 2, &tmB, n0 + 64, k, plane, full_bar(slot), pol_b);
        return done();
      };
      for (int item = blockIdx.x; ok && item < num_items; item += gridDim.x) {
        const int leaf = p.leaf_begin + item / per_leaf;  // workspace plane
        const int tile = item % per_leaf;
        const int m0 = tile / tiles * 128, n0 = tile % tiles * 128;
        if (F64 && *(volatile const int*)p.flag != 0) {
          if (!mbar_wait_bounded(empty_bar(slot), phase ^ 1, p.err, kDevTimeoutEmpty, p.timeout_ns)) {
            ok = false;
          } else {
            *stop = 1;
            mbar_arrive(full_bar(slot));
          }
          break;
        }
        if (F64) {
          // magnitudes: the four K blocks of 32 take the place of the digits
          uint32_t st = next();
          if ((ok = st != 0)) {
            for (int q = 0; q < 4; ++q) tma_load_3d(st + q * 8192, &tmSA, q * 32, m0, leaf, full_bar(slot), pol_a);
            done();
            st = next();
            if ((ok = st != 0)) {
              for (int q = 0; q < 4; ++q)
                for (int c = 0; c < 2; ++c)
                  tma_load_3d(st + c * (kQuadBytes / 2) + q * 4096, &tmSB, n0 + c * 64, q * 32, leaf, full_bar(slot),
                              pol_b);
              done();
            }
          }
        }
        const int plane = leaf * kDigits;
        for (int k0 = 0; ok && k0 < p.L; k0 += 256) {
          const int k1 = k0 + 256 < p.L ? k0 + 256 : p.L;
          for (int k = k0; ok && k < k1; k += 32)
            ok = load_a(k, m0, plane) && load_b(k, n0, plane) && load_b(k, n0, plane + 4) && load_a(k, m0, plane + 4);
          for (int k = k0; ok && k < k1; k += 32) ok = load_a(k, m0, plane) && load_b(k, n0, plane);
        }
      }
      if (!ok) {
        // copies already issued land before the CTA can exit
        for (int t = 0; t < kQuads; ++t)
          if (armed & (1u << t)) mbar_wait_bounded(full_bar(t), (armed_phase >> t) & 1, nullptr, 0, 200000000ull);
      }
    }
    if (warp == 1 && lane == 0) {
      // ---------------------------------------------------------- MMA issuer

      constexpr uint32_t IDESC = idesc_as_fp16(make_idesc<128, 128, false, true>());
      int slot = 0;
      uint32_t phase = 0;      // parity of the ring's turns
      uint32_t acc_phase = 0;  // bit a: parity of accumulator a's uses so far
      bool ok = true, issued = false;
      // descriptors: the high words are constant, the low words count 16 bytes
      constexpr uint32_t kHiA = (512u >> 4) | (1u << 14) | (4u << 29);   // 64-byte swizzle, 8-row groups of 512 bytes
      constexpr uint32_t kHiB = (1024u >> 4) | (1u << 14) | (2u << 29);  // 128-byte swizzle, 8 K rows of 1024 bytes
      auto lo_a = [&](int sl) { return ((sbase + (uint32_t)sl * kQuadBytes) >> 4) | (1u << 16); };
      auto lo_b = [&](int sl) { return ((sbase + (uint32_t)sl * kQuadBytes) >> 4) | ((kQuadBytes / 2 >> 4) << 16); };
      // the next quad in load order: its slot (-1: not in time)
      auto take = [&]() -> int {
        if (!mbar_wait_bounded(full_bar(slot), phase, p.err, kDevTimeoutFull, p.timeout_ns)) return -1;
        const int sl = slot;
        if (++slot == kQuads) {
          slot = 0;
          phase ^= 1;
        }
        return sl;
      };
      auto wait_free = [&](int a) -> bool {
        if (!mbar_wait_bounded(acce_bar(a), ((acc_phase >> a) & 1) ^ 1, p.err, kDevTimeoutAccEmpty, p.timeout_ns))
          return false;
        acc_phase ^= 1u << a;
        return true;
      };
      // digit i of quad a times digit j of quad b (both 0..3 within the quad)
      auto mul = [&](uint32_t a, uint32_t b, int i, int j, int acc, bool first) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const uint64_t da = ((uint64_t)kHiA << 32) | (a + (uint32_t)(i * 512 + k * 2));
          const uint64_t db = ((uint64_t)kHiB << 32) | (b + (uint32_t)(j * 256 + k * 128));
          mma_f16(tmem_base + (uint32_t)acc * 128u, da, db, IDESC, first && k == 0 ? 0u : 1u);
        }
      };
      // diagonals 7..4 of a K block: by diagonal (the first block after a low
      // phase; it starts the accumulators in the order that phase frees them),
      // or by quad (the others; quads are freed early and the last block of a
      // phase ends 4, 5, 6, 7)
      auto high_first = [&]() -> bool {
        int sa[2], sb[2];
        if ((sa[0] = take()) < 0 || (sb[0] = take()) < 0 || (sb[1] = take()) < 0 || (sa[1] = take()) < 0) return false;
        tc_fence_after();
        const uint32_t a[2] = {lo_a(sa[0]), lo_a(sa[1])}, b[2] = {lo_b(sb[0]), lo_b(sb[1])};
#pragma unroll
        for (int s = 7; s >= 5; --s) {
          if (!wait_free(7 - s)) return false;
          tc_fence_after();
#pragma unroll
          for (int i = 0; i <= s; ++i) mul(a[i >> 2], b[(s - i) >> 2], i & 3, (s - i) & 3, 7 - s, i == 0);
        }
        if (!wait_free(3)) return false;
        tc_fence_after();
        mul(a[1], b[0], 0, 0, 3, true);  // (4, 0)
        mma_commit(empty_bar(sa[1]));
        mul(a[0], b[1], 0, 0, 3, false);  // (0, 4)
        mma_commit(empty_bar(sb[1]));
#pragma unroll
        for (int i = 1; i <= 3; ++i) mul(a[0], b[0], i, 4 - i, 3, false);
        mma_commit(empty_bar(sa[0]));
        mma_commit(empty_bar(sb[0]));
        return true;
      };
      auto high_next = [&](bool first, bool last) -> bool {
        int sa[2], sb[2];
        if ((sa[0] = take()) < 0 || (sb[0] = take()) < 0) return false;
        tc_fence_after();
        const uint32_t a0 = lo_a(sa[0]), b0 = lo_b(sb[0]);
#pragma unroll
        for (int s = 4; s <= 6; ++s)
#pragma unroll
          for (int i = s - 3; i <= 3; ++i) {
            if (i == s - 3 && first) {
              if (!wait_free(7 - s)) return false;
              tc_fence_after();
            }
            mul(a0, b0, i, s - i, 7 - s, i == s - 3 && first);
          }
        if ((sb[1] = take()) < 0) return false;
        tc_fence_after();
        const uint32_t b1 = lo_b(sb[1]);
#pragma unroll
        for (int s = 4; s <= 7; ++s)
#pragma unroll
          for (int i = 0; i <= s - 4; ++i) {
            if (s == 7 && i == 0 && first) {
              if (!wait_free(0)) return false;
              tc_fence_after();
            }
            mul(a0, b1, i, s - 4 - i, 7 - s, s == 7 && i == 0 && first);
          }
        mma_commit(empty_bar(sa[0]));
        mma_commit(empty_bar(sb[1]));
        if ((sa[1] = take()) < 0) return false;
        tc_fence_after();
        const uint32_t a1 = lo_a(sa[1]);
#pragma unroll
        for (int s = 4; s <= 7; ++s) {
#pragma unroll
          for (int i = 0; i <= s - 4; ++i) mul(a1, b0, i, s - 4 - i, 7 - s, false);
          if (last) mma_commit(accf_bar(7 - s));
        }
        mma_commit(empty_bar(sb[0]));
        mma_commit(empty_bar(sa[1]));
        return true;
      };
      // diagonals 3..0 of a K block on accumulators 3..0
      auto low = [&](bool first, bool last) -> bool {
        int sa, sb;
        if ((sa = take()) < 0 || (sb = take()) < 0) return false;
        tc_fence_after();
        const uint32_t a = lo_a(sa), b = lo_b(sb);
        if (first) {
#pragma unroll
          for (int s = 3; s >= 0; --s) {
            if (!wait_free(s)) return false;
            tc_fence_after();
#pragma unroll
            for (int i = 0; i <= s; ++i) mul(a, b, i, s - i, s, i == 0);
          }
        } else {
#pragma unroll
          for (int s = 0; s <= 3; ++s) {
#pragma unroll
            for (int i = 0; i <= s; ++i) mul(a, b, i, s - i, s, false);
            if (last) mma_commit(accf_bar(s));
          }
        }
        mma_commit(empty_bar(sa));
        mma_commit(empty_bar(sb));
        return true;
      };
      // the magnitude products; `go_on` false: the product is redone
      auto check = [&](bool& go_on) -> bool {
        int sa, sb;
        if ((sa = take()) < 0) return false;
        if (*stop) {
          go_on = false;
          if (!wait_free(3)) return false;
          mbar_arrive(accf_bar(3));  // (in place of the MMAs' commit)
          return true;
        }
        if ((sb = take()) < 0 || !wait_free(3)) return false;
        tc_fence_after();
        const uint32_t a = lo_a(sa), b = lo_b(sb);
#pragma unroll
        for (int q = 0; q < 4; ++q) mul(a, b, q, q, 3, q == 0);
        mma_commit(accf_bar(3));
        mma_commit(empty_bar(sa));
        mma_commit(empty_bar(sb));
        return true;
      };
      for (int item = blockIdx.x; ok && item < num_items; item += gridDim.x) {
        if (F64) {
          bool go_on = true;
          ok = check(go_on);
          if (!go_on) break;
        }
        for (int b0 = 0; ok && b0 < kblocks; b0 += 8) {
          const int b1 = b0 + 8 < kblocks ? b0 + 8 : kblocks;
          issued = true;
          ok = high_first();
          for (int b = b0 + 1; ok && b < b1; ++b) ok = high_next((b & 3) == 0, (b & 3) == 3 || b == b1 - 1);
          for (int b = b0; ok && b < b1; ++b) ok = low(b == b0, b == b1 - 1);
        }
      }
      if (!ok && issued) {
        // MMAs in flight finish before TMEM is released: a commit to a
        // barrier nobody waits on any more, and its arrival awaited briefly
        mma_commit(accf_bar(0));
        spin_ns(2000000ull);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
    const int quarter = warp & 3;
    const int half = (warp - 4) >> 2;
    const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * 64);
    const uint32_t ebuf = epi_base + (uint32_t)(warp - 4) * (32 * kEpiStride + 256);
    const uint32_t fbuf = ebuf + 32 * kEpiStride;
    uint32_t acc_phase = 0;
    int shift = p.shift;  // F64: 2^shift of 256^7 is the unit of this thread's sums
    bool ok = true;
    long long sum[64];
    auto wait_acc = [&](int a) -> bool {
      if (!mbar_wait_bounded(accf_bar(a), (acc_phase >> a) & 1, p.err, kDevTimeoutAccFull, p.timeout_ns)) return false;
      acc_phase ^= 1u << a;
      if (F64) __syncwarp();  // (rows of unlike shift part in drain's branch)
      tc_fence_after();
      return true;
    };
    auto free_acc = [&](int a) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce_bar(a));
    };
    // diagonal s, held in accumulator a
    auto drain = [&](int a, int s) -> bool {
      if (!wait_acc(a)) return false;
      // I64: 256^s.  F64: 256^(7-s) in units of 2^shift (contributions below
      // the unit are rounded)
      const int sh = F64 ? 8 * (7 - s) - shift : 8 * s;
      const uint32_t col = lane_base + (uint32_t)(a * 128);
      uint32_t r0[32], r1[32];
      tmem_ld_32x32b_x32(col, r0);
      tmem_ld_32x32b_x32(col + 32, r1);
      tmem_ld_wait();
      free_acc(a);  // the additions need only registers
      if (sh >= 32) {
        const uint32_t mul = 1u << (sh - 32);
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          sum[e] = add_high(sum[e], (uint32_t)__float2int_rn(__uint_as_float(r0[e])) * mul);
          sum[32 + e] = add_high(sum[32 + e], (uint32_t)__float2int_rn(__uint_as_float(r1[e])) * mul);
        }
      } else {
        // v 2^sh = (v scale) mul, rounded where sh < 0 (|v| <= 2^24)
        const int ms = sh < 0 ? 0 : sh == 31 ? 30 : sh;
        const float scale = F64 ? (sh < 0 ? __int_as_float((127 + sh) << 23) : sh == 31 ? 2.f : 1.f) : 1.f;
        const int mul = 1 << ms;
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          sum[e] = add_wide(sum[e], __float2int_rn(__uint_as_float(r0[e]) * scale), mul);
          sum[32 + e] = add_wide(sum[32 + e], __float2int_rn(__uint_as_float(r1[e]) * scale), mul);
        }
      }
      return true;
    };
    for (int item = blockIdx.x; ok && item < num_items; item += gridDim.x) {
      const int leaf = p.leaf_begin + item / per_leaf;
      const int tile = item % per_leaf;
      const int row0 = tile / tiles * 128 + quarter * 32, row = row0 + lane;  // in the leaf plane
      const int col0 = tile % tiles * 128 + half * 64;
      auto fexp = [&](int c) {  // exponent of column col0 + c
        int f;
        asm volatile("ld.shared.s32 %0, [%1];" : "=r"(f) : "r"(fbuf + 4u * (uint32_t)c));
        return f;
      };
      if (F64) {
        const int32_t* fb = p.expB + (int64_t)leaf * p.L;
        const int ea = row < p.L ? p.expA[(int64_t)leaf * p.L + row] : kLimbZeroRow;
        const int none = p.shift - 4;  // the most slack there is
        int slack = none;              // the least of this warp's columns
        __syncwarp();  // (the previous tile's exponents have been read)
#pragma unroll
        for (int h = 0; h < 64; h += 32) {
          const bool in = col0 + h + lane < p.L;
          const int f = in ? fb[col0 + h + lane] : kLimbZeroRow;
          asm volatile("st.shared.s32 [%0], %1;" ::"r"(fbuf + 4u * (uint32_t)(h + lane)), "r"(f) : "memory");
          if (in) slack = min(slack, p.slackB[(int64_t)leaf * p.L + col0 + h + lane]);
        }
        __syncwarp();
        slack = __reduce_min_sync(0xffffffffu, slack);
        const int slack_a = row < p.L ? p.slackA[(int64_t)leaf * p.L + row] : none;
        shift = p.shift - (slack + slack_a) / 2;
        // the magnitude check of every element that can be non-zero
        const LimbNeed q = p.need[leaf];
        const float need = fmaxf(kLimbLeast, q.drop + q.operand * (exp2f(-0.5f * slack_a) + exp2f(-0.5f * slack)) +
                                                 q.sum * exp2f((float)(shift - p.shift)));
        if (!wait_acc(3) || *stop) break;
        bool bad = false;
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
          uint32_t r[16];
          tmem_ld_32x32b_x16(lane_base + 3u * 128u + (uint32_t)(j * 16), r);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            if (!(__uint_as_float(r[e]) >= need) && ea != kLimbZeroRow && fexp(j * 16 + e) != kLimbZeroRow) bad = true;
          }
        }
        free_acc(3);
        if (bad) *(volatile int*)p.flag = 1;
      }
#pragma unroll
      for (int e = 0; e < 64; ++e) sum[e] = 0;
#pragma unroll 1
      for (int c = 0; ok && c < chunks; ++c) {
        // in the order in which the issuer finishes them: 4..7, then 0..3
#pragma unroll 1
        for (int x = 0; ok && x < 4; ++x) ok = drain(3 - x, x + 4);
        if ((c & 1) || c == chunks - 1) {
#pragma unroll 1
          for (int x = 0; ok && x < 4; ++x) ok = drain(x, x);
        }
      }
      if (!ok) break;
      // combine: the row segment goes into every C target of the leaf
      const int ea = F64 && row < p.L ? p.expA[(int64_t)leaf * p.L + row] : 0;
      const int nt = p.ccount[leaf];
      const CTarget* tg = p.ctab + (int64_t)leaf * p.maxT;
      unsigned long long* C = static_cast<unsigned long long*>(p.C);
      // (one copy of this code, the next 8 columns' sums moving down: unrolled
      // over the 64 columns it was 40 KB that every tile fetched anew)
#pragma unroll 1
      for (int j = 0; j < 8; ++j) {
        unsigned long long v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          // (a zero row or column has a zero sum, whatever its exponent says)
          v[e] = F64 ? scaled_double_bits(sum[e], ea + fexp(j * 8 + e) + shift - 68)
                     : (unsigned long long)sum[e];
        }
#pragma unroll
        for (int e = 0; e < 56; ++e) sum[e] = sum[e + 8];
        // turned in shared memory so that a warp writes four row pieces of 64
        // bytes at a time (per-row bulk reductions of 64 bytes from the staged
        // rows took 20 us a tile: the copy engine's rate of small operations)
        __syncwarp();
#pragma unroll
        for (int e = 0; e < 8; ++e)
          asm volatile("st.shared.u64 [%0], %1;" ::"r"(ebuf + (uint32_t)(lane * kEpiStride + e * 8)), "l"(v[e]) : "memory");
        __syncwarp();
        unsigned long long w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          asm volatile("ld.shared.u64 %0, [%1];" : "=l"(w[i]) : "r"(ebuf + (uint32_t)((4 * i + lane / 8) * kEpiStride + (lane % 8) * 8)));
        const int wr = row0 + lane / 8, wc = col0 + j * 8 + lane % 8;  // of w[0]; w[i] is 4 i rows below
        if (p.store) {
          const bool in_c = p.store == p.C;
          const int64_t lim = in_c ? p.n : p.L, ld = in_c ? p.ldc : p.L;
          if (wc < lim) {
            unsigned long long* dst = static_cast<unsigned long long*>(p.store) +
                                      (in_c ? 0 : (int64_t)leaf * p.L * p.L) + (int64_t)wr * ld + wc;
#pragma unroll
            for (int i = 0; i < 8; ++i)
              if (wr + 4 * i < lim) dst[4 * i * ld] = w[i];
          }
        } else if (wc < p.L) {
#pragma unroll 1
          for (int t = 0; t < nt; ++t) {
            const CTarget c = tg[t];
            const int64_t gcol = (int64_t)c.col_off + wc;
            if (gcol >= p.n) continue;
            const int64_t rows = min((int64_t)p.L - wr, p.n - c.row_off - wr);  // rows from w[0]'s on that exist
            unsigned long long* dst = C + ((int64_t)c.row_off + wr) * p.ldc + gcol;
#pragma unroll
            for (int i = 0; i < 8; ++i)
              if (4 * i < rows) {
                if (F64)
                  atomicAdd(reinterpret_cast<double*>(dst + 4 * i * p.ldc),
                            __longlong_as_double((long long)(c.sign > 0 ? w[i] : w[i] ^ 0x8000000000000000ull)));
                else
                  atomicAdd(dst + 4 * i * p.ldc, c.sign > 0 ? w[i] : 0ull - w[i]);
              }
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, 512);
}

template <bool F64>
cudaError_t launch(const LeafLimbArgs& a, const CUtensorMap* tmA, const CUtensorMap* tmB, const CUtensorMap* tmSA,
                   const CUtensorMap* tmSB, int num_sms, cudaStream_t st) {
  if (a.L < 128 || a.L % 64 != 0) return cudaErrorInvalidValue;
  const int64_t tiles = (a.L + 127) / 128;
  const int64_t items = (int64_t)(a.leaf_end - a.leaf_begin) * tiles * tiles;
  auto kern = leaf_limb_kernel<F64>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimb);
  if (e != cudaSuccess) return e;
  if (items <= 0) return cudaSuccess;
  if (items > 0x7FFFFFFF - num_sms) return cudaErrorInvalidValue;
  const int grid = (int)(items < num_sms ? items : num_sms);
  kern<<<grid, kThreadsL, kSmemLimb, st>>>(*tmA, *tmB, *tmSA, *tmSB, a);
  count_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_leaf_limb(const LeafLimbArgs& a, const CUtensorMap* tmA, const CUtensorMap* tmB,
                             const CUtensorMap* tmSA, const CUtensorMap* tmSB, bool f64, int num_sms,
                             cudaStream_t st) {
  if (f64) return launch<true>(a, tmA, tmB, tmSA, tmSB, num_sms, st);
  return launch<false>(a, tmA, tmB, tmA, tmB, num_sms, st);
}

}  // namespace stark
