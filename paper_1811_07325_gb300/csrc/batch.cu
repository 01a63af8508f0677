// batch.cu -- many independent products in one grouped, graph-captured pass.
//
// Each member keeps its own plan (operand planes, C-target table, operand
// tensor maps).  One stark_batch_mul enqueues, for every member, the divide of
// A and B with the clearing of C, and a few persistent grouped leaf launches
// whose work items are (member, leaf, tile) triples: the 7^d leaf products of
// their members share the GPU, and each item's epilogue combines into its own
// member's C.  The whole sequence is captured once in a CUDA graph and
// replayed while the pointers are unchanged.
//
// Depth per member: given, or chosen by the autotuner, which times the
// candidate (depth, leaf tile) pairs on the device (one warm-up and three
// rounds of two timed products per candidate on scratch inputs) and caches the winner per
// size class and dtype for the process.  The tile candidates are CTA pairs
// on 256 x 256 tiles (cta_group::2; leaf sides that are multiples of 256)
// and single CTAs on 128 x 128 tiles.  Members whose tile is 256 share up to
// three grouped launches of CTA pairs, the others one of single CTAs.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <tuple>
#include <vector>

#include "plan.h"
#include "stark_internal.h"

namespace stark {
namespace {

std::mutex g_tune_mu;
// (n class, dtype) -> (depth, tile)
std::map<std::pair<int64_t, int>, std::pair<int, int>> g_tuned;

// Relative RMS error of a grouped member's product of N(0, 1) inputs, as
// measured: the split's, doubled by every level, and the tensor cores'
// accumulation, in proportion to the K that one accumulation spans.
double relative_error(const stark_plan_s& p) {
  const double split = (p.dt == STARK_F32_SPLIT_BF16 ? 4.4e-6 : 1e-7) * (double)(1 << p.depth);
  const double sums =
      (p.dt == STARK_F32_SPLIT_TF32 ? 7.0e-9 : p.dt == STARK_F32_SPLIT_FP16 ? 3.6e-9 : 3.4e-9) * (double)p.L;
  return std::sqrt(split * split + sums * sums);
}

// Device time (ms) of one product of side n at `depth` with leaf tiles of
// width `tile` (256: CTA pairs; 128: single CTAs) as a grouped member runs it
// (whole K ranges), the best of three rounds, and its error.
float time_depth(int64_t n, int depth, stark_dtype dt, int tile, void* A, void* B, void* C, cudaStream_t s,
                 double* error) {
  stark_plan_s p;
  p.whole_k = true;
  if (plan_init(&p, n, depth, dt) != STARK_OK) {
    plan_release(&p);
    return -1.f;
  }
  if (tile == 128 && p.bn == 256) {  // single CTAs on 128-wide tiles (operand maps do not depend on it)
    p.bn = 128;
    p.pair_mode = 0;
  } else if (tile != p.bn) {
    plan_release(&p);
    return -1.f;
  }
  *error = relative_error(p);
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  float ms = -1.f;
  if (plan_run(&p, A, B, C, 0, p.P, s) == STARK_OK) {
    bool ok = true;
    for (int round = 0; round < 3 && ok; ++round) {  // the best of three rounds of two
      cudaEventRecord(e0, s);
      for (int r = 0; r < 2 && ok; ++r) ok = plan_run(&p, A, B, C, 0, p.P, s) == STARK_OK;
      cudaEventRecord(e1, s);
      float t = 0;
      if (ok && cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&t, e0, e1) == cudaSuccess && t > 0 &&
          (ms < 0 || t / 2 < ms))
        ms = t / 2;
    }
  }
  cudaStreamSynchronize(s);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  plan_release(&p);
  cudaGetLastError();
  return ms;
}

}  // namespace

// Measured depth choice for n x n products (cached per process): one for a plan,
// a batch's member and a request, by the product's time and error as a member
// (a plan's K slices only lower its error at the same depth).
void autotune(int64_t n_req, stark_dtype dt, int* depth_out, int* tile_out) {
  // size class: n rounded up to 64 (n <= 1024), 128 (n <= 2048), else 256
  const int64_t q = n_req <= 1024 ? 64 : n_req <= 2048 ? 128 : 256;
  const int64_t n = (n_req + q - 1) / q * q;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tuned.find({n, (int)dt});
    if (it != g_tuned.end()) {
      *depth_out = it->second.first;
      *tile_out = it->second.second;
      return;
    }
  }
  int best = choose_depth(n, dt);
  int best_tile = (padded_side(n, best, dt) >> best) % 256 == 0 ? 256 : 128;
  const size_t bytes = (size_t)n * n * element_size(dt);
  void *A = nullptr, *B = nullptr, *C = nullptr;
  cudaStream_t s = nullptr;
  if (n > 0 && cudaMalloc(&A, bytes) == cudaSuccess && cudaMalloc(&B, bytes) == cudaSuccess &&
      cudaMalloc(&C, bytes) == cudaSuccess && cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) == cudaSuccess) {
    cudaMemsetAsync(A, 0x3c, bytes, s);  // bounded, nonzero values
    cudaMemsetAsync(B, 0x3c, bytes, s);
    struct Candidate {
      int depth, tile;
      float ms;
      double error;
    };
    std::vector<Candidate> tried;
    float best_ms = 1e30f;
    for (int d = 0; d <= 3; ++d) {
      if ((padded_side(n, d, dt) >> d) < tile_granularity(dt)) continue;
      if (d > 0 && (n >> d) < 128) break;
      const bool wide = (padded_side(n, d, dt) >> d) % 256 == 0;
      for (int tile : {256, 128}) {
        if (tile == 256 && !wide) continue;
        Candidate c{d, tile, 0.f, 0.0};
        c.ms = time_depth(n, d, dt, tile, A, B, C, s, &c.error);
        if (c.ms > 0) {
          tried.push_back(c);
          best_ms = std::min(best_ms, c.ms);
        }
      }
    }
    // of those within 3 us and 1 % of the fastest the most accurate one (of
    // equals the faster).  The depths differ by up to a factor of two in error
    // and, up to n = 1024, by one to three microseconds in time.  By time alone
    // a one-leaf product, stored without a clear (3xFP16, n = 576: 15.5 us, and
    // 17.0 at depth 1), would take many of these sizes from the depth of half
    // its error.  Over 43 size classes up to n = 12288 and three dtypes the
    // pick was within 3 us of the fastest and, from n = 2304 on, within 1 %.
    const Candidate* pick = nullptr;
    for (const Candidate& c : tried)
      if (c.ms <= 1.01f * best_ms + 3e-3f &&
          (!pick || c.error < 0.99 * pick->error || (c.error < 1.01 * pick->error && c.ms < pick->ms)))
        pick = &c;
    if (pick) {
      best = pick->depth;
      best_tile = pick->tile;
    }
  }
  if (s) cudaStreamDestroy(s);
  cudaFree(A);
  cudaFree(B);
  cudaFree(C);
  cudaGetLastError();
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tuned[{n, (int)dt}] = {best, best_tile};
  *depth_out = best;
  *tile_out = best_tile;
}

int autotune_depth(int64_t n, stark_dtype dt) {
  int d = 0, tile = 128;
  autotune(n, dt, &d, &tile);
  return d;
}

}  // namespace stark

struct stark_batch_s {
  stark_dtype dt = STARK_F32_SPLIT_BF16;
  int bn = 128;     // 256 when any member runs 256-wide tiles
  // the grouped leaf launches: members [first, first + count) of the sorted
  // order, whose items are numbered from 0; the 256-wide ones come first
  struct Launch {
    int first, count, items;
    bool wide;
  };
  std::vector<Launch> launches;
  std::vector<stark_plan_s*> plans;
  std::vector<stark::GroupDesc> host_desc;
  stark::GroupDesc* d_desc = nullptr;
  int64_t total_items = 0;
  int* d_err = nullptr;
  cudaStream_t cap = nullptr;  // private capture stream
  // the members' clears and divides are captured on kForks side streams
  // forked from `cap`, so the graph runs them concurrently (small members'
  // kernels are launch- and latency-bound one after another)
  static constexpr int kForks = 8;
  static constexpr int kMaxLaunches = 4;
  cudaStream_t side[kForks] = {};
  cudaStream_t leaf[kMaxLaunches] = {};  // branches of the leaf launches
  cudaEvent_t fork_ev = nullptr;
  cudaEvent_t join_ev[kForks] = {};
  cudaGraphExec_t exec = nullptr;
  std::vector<int> caller_index;  // caller's index of each (size-sorted) member
  std::vector<int> tiles;         // leaf tile width of each member (caller's order)
  std::vector<const void*> last;  // pointers the graph was captured with
  int64_t replays = 0;
};

using namespace stark;

static void batch_free(stark_batch_s* b) {
  if (b->exec) cudaGraphExecDestroy(b->exec);
  for (auto* p : b->plans) {
    plan_release(p);
    delete p;
  }
  cudaFree(b->d_desc);
  cudaFree(b->d_err);
  if (b->cap) cudaStreamDestroy(b->cap);
  for (int i = 0; i < stark_batch_s::kForks; ++i) {
    if (b->side[i]) cudaStreamDestroy(b->side[i]);
    if (b->join_ev[i]) cudaEventDestroy(b->join_ev[i]);
  }
  for (cudaStream_t l : b->leaf)
    if (l) cudaStreamDestroy(l);
  if (b->fork_ev) cudaEventDestroy(b->fork_ev);
  cudaGetLastError();
  delete b;
}

extern "C" {

stark_status stark_batch_create(int32_t count, const int64_t* n, int depth, stark_dtype dt, stark_batch_t* out) {
  if (!out || !n || count <= 0 || count > 4096 || depth < -1 || depth > kMaxDepth) return STARK_EINVAL;
  *out = nullptr;
  if (!is_split(dt)) return STARK_EUNSUPPORTED;
  for (int i = 0; i < count; ++i)
    if (n[i] <= 0 || n[i] > (int64_t)1 << 20) return STARK_EINVAL;
  if (!device_is_sm100_family()) return STARK_EUNSUPPORTED;
  auto* b = new (std::nothrow) stark_batch_s();
  if (!b) return STARK_ENOMEM;
  b->dt = dt;
  stark_status st = STARK_OK;
  // members in order of decreasing size so the big tiles start first
  std::vector<int> order(count);
  for (int i = 0; i < count; ++i) order[i] = i;
  b->plans.assign(count, nullptr);
  b->tiles.assign(count, 128);
  for (int i = 0; i < count && st == STARK_OK; ++i) {
    int d = depth, tile = 0;
    if (depth < 0) autotune(n[i], dt, &d, &tile);
    auto* p = new (std::nothrow) stark_plan_s();
    if (!p) {
      st = STARK_ENOMEM;
      break;
    }
    b->plans[i] = p;
    st = plan_init(p, n[i], d, dt);
    // the tuned tile, or 256-wide wherever the leaf side allows it
    if (st == STARK_OK) b->tiles[i] = (p->L % 256 == 0 && tile != 128) ? 256 : 128;
  }
  if (st != STARK_OK) {
    batch_free(b);
    return st;
  }
  // members on 256-wide tiles (CTA pairs) first, then the rest on 128-wide
  // tiles; largest products first in each
  const std::vector<int> tiles = b->tiles;
  auto wide = [&](int i) { return tiles[i] == 256; };
  std::sort(order.begin(), order.end(), [&](int x, int y) {
    if (wide(x) != wide(y)) return wide(x);
    return b->plans[x]->n > b->plans[y]->n;
  });
  int split = 0;
  while (split < count && wide(order[split])) ++split;
  b->bn = split > 0 ? 256 : 128;
  // The 256-wide members in up to three launches, so that the divides of the
  // later ones run under the leaf products of the earlier ones (a leaf kernel
  // leaves the SMs threads and registers for them).  The first gets an eighth
  // of the work, the second three eighths: its divides take a quarter to a
  // third of its leaf time.  Not when all the divides together move less than
  // 256 MB, about 40 us.
  int64_t divide_bytes = 0;
  double work = 0;
  auto leaf_work = [&](const stark_plan_s* p) { return (double)p->P * p->L * p->L * p->L; };
  for (int k = 0; k < split; ++k) {
    const stark_plan_s* p = b->plans[order[k]];
    divide_bytes += 2 * p->n * p->n * 4 + operand_bytes(p->n, p->depth, dt);
    work += leaf_work(p);
  }
  std::vector<int> cuts;  // ends of the launches
  if (divide_bytes >= (int64_t)256 << 20) {
    double done = 0;
    for (int k = 0; k + 1 < split && cuts.size() < 2; ++k) {
      done += leaf_work(b->plans[order[k]]);
      if (done >= work * (cuts.empty() ? 0.125 : 0.5)) cuts.push_back(k + 1);
    }
  }
  if (split > 0) cuts.push_back(split);
  if (split < count) cuts.push_back(count);
  b->host_desc.resize(count);
  int first = 0;
  for (int end : cuts) {
    int64_t items = 0;
    for (int k = first; k < end; ++k) {
      stark_plan_s* p = b->plans[order[k]];
      const int bn = k < split ? 256 : 128;
      GroupDesc& g = b->host_desc[k];
      std::memset(&g, 0, sizeof(g));
      g.tmA = p->tmA;
      if (dt == STARK_F32_SPLIT_TF32 && !p->tf32_mn) {
        // K-major tf32 Y; 256-wide members run CTA pairs: each CTA loads 128 Y rows
        if (!make_tmap_planes(&g.tmB, p->Y, true, p->L, 2 * p->P, bn == 256 ? 128 : bn)) st = STARK_EUNSUPPORTED;
      } else {
        g.tmB = p->tmB;
      }
      g.item_base = (int32_t)items;
      g.P = (int32_t)p->P;
      g.L = (int32_t)p->L;
      g.ctab = p->d_ctab;
      g.ccount = p->d_ccount;
      g.maxT = p->maxT;
      g.n = p->n;
      // 256-wide members: 256 x 256 pair tiles (CTA pairs); others 128 x 128
      items += bn == 256 ? p->P * (p->L / 256) * (p->L / 256) : p->P * (p->L / 128) * (p->L / 128);
    }
    if (items > 0x7FFFFFFF) st = STARK_EINVAL;
    b->launches.push_back({first, end - first, (int)items, first < split});
    b->total_items += items;
    first = end;
  }
  // keep the member order used by the descriptors
  std::vector<stark_plan_s*> sorted(count);
  for (int k = 0; k < count; ++k) sorted[k] = b->plans[order[k]];
  b->last.clear();
  if (st == STARK_OK && (cudaMalloc(&b->d_desc, sizeof(GroupDesc) * count) != cudaSuccess ||
                         cudaMalloc(&b->d_err, sizeof(int)) != cudaSuccess ||
                         cudaMemset(b->d_err, 0, sizeof(int)) != cudaSuccess ||
                         cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking) != cudaSuccess ||
                         cudaEventCreateWithFlags(&b->fork_ev, cudaEventDisableTiming) != cudaSuccess))
    st = STARK_ENOMEM;
  for (int i = 0; i < stark_batch_s::kForks && st == STARK_OK; ++i)
    if (cudaStreamCreateWithFlags(&b->side[i], cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->join_ev[i], cudaEventDisableTiming) != cudaSuccess)
      st = STARK_ENOMEM;
  for (size_t i = 0; i < b->launches.size() && st == STARK_OK; ++i)
    if (cudaStreamCreateWithFlags(&b->leaf[i], cudaStreamNonBlocking) != cudaSuccess) st = STARK_ENOMEM;
  if (st != STARK_OK) {
    batch_free(b);
    return st;
  }
  // members are kept in the descriptor order; remember the caller's index
  b->plans = sorted;
  b->caller_index = order;
  *out = b;
  return STARK_OK;
}

stark_status stark_batch_destroy(stark_batch_t b) {
  if (!b) return STARK_OK;
  cudaDeviceSynchronize();
  batch_free(b);
  return STARK_OK;
}

stark_status stark_batch_tile(stark_batch_t b, int32_t index, int32_t* tile_n) {
  if (!b || !tile_n || index < 0 || index >= (int32_t)b->tiles.size()) return STARK_EINVAL;
  *tile_n = b->tiles[index];
  return STARK_OK;
}

stark_status stark_batch_depth(stark_batch_t b, int32_t index, int32_t* depth) {
  if (!b || !depth || index < 0 || index >= (int32_t)b->plans.size()) return STARK_EINVAL;
  for (size_t k = 0; k < b->plans.size(); ++k)
    if (b->caller_index[k] == index) {
      *depth = b->plans[k]->depth;
      return STARK_OK;
    }
  return STARK_EINVAL;
}

stark_status stark_batch_info(stark_batch_t b, int32_t* tile_n, int64_t* work_items, int64_t* workspace_bytes,
                              int64_t* graph_replays) {
  if (!b) return STARK_EINVAL;
  if (tile_n) *tile_n = b->bn;
  if (work_items) *work_items = b->total_items;
  if (workspace_bytes) {
    int64_t w = 0;
    for (auto* p : b->plans) w += p->ws_bytes;
    *workspace_bytes = w;
  }
  if (graph_replays) *graph_replays = b->replays;
  return STARK_OK;
}

stark_status stark_batch_mul(stark_batch_t b, const void* const* A, const void* const* B, void* const* C,
                             void* stream) {
  if (!b || !A || !B || !C) return STARK_EINVAL;
  const int count = (int)b->plans.size();
  std::vector<const void*> ptrs((size_t)count * 3);
  for (int k = 0; k < count; ++k) {
    const int i = b->caller_index[k];
    if (!A[i] || !B[i] || !C[i]) return STARK_EINVAL;
    ptrs[3 * k] = A[i];
    ptrs[3 * k + 1] = B[i];
    ptrs[3 * k + 2] = C[i];
  }
  cudaStream_t s = (cudaStream_t)stream;
  if (ptrs != b->last || !b->exec) {
    // new pointers: refresh the C maps and re-record the graph (the device
    // descriptors may be read by a replay still in flight, so wait first)
    if (cudaDeviceSynchronize() != cudaSuccess) return STARK_ECUDA;
    for (int k = 0; k < count; ++k) {
      GroupDesc& g = b->host_desc[k];
      void* Cuser = const_cast<void*>(ptrs[3 * k + 2]);
      const bool staged = plan_uses_cstage(b->plans[k], Cuser);
      g.C = static_cast<float*>(staged ? b->plans[k]->cstage : Cuser);
      g.ldc = staged ? staged_ld(g.n) : g.n;
      // (one leaf: each element of C is stored once, not added into a cleared C)
      g.use_tma_c = make_tmap_c(&g.tmC, g.C, g.n, g.ldc) ? (b->plans[k]->depth == 0 ? 2 : 1) : 0;
    }
    if (cudaMemcpy(b->d_desc, b->host_desc.data(), sizeof(GroupDesc) * count, cudaMemcpyHostToDevice) !=
        cudaSuccess)
      return STARK_ECUDA;
    if (b->exec) {
      cudaGraphExecDestroy(b->exec);
      b->exec = nullptr;
    }
    cudaGraph_t graph = nullptr;
    if (cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return STARK_ECUDA;
    stark_status st = STARK_OK;
    // fork: members' clears and divides on the side streams in the order of
    // the leaf launches, each of which joins its own members' and runs on a
    // branch of its own (a later launch takes SMs as the tail of an earlier one
    // frees them)
    constexpr int F = stark_batch_s::kForks;
    if (cudaEventRecord(b->fork_ev, b->cap) != cudaSuccess) st = STARK_ECUDA;
    for (int i = 0; i < F && st == STARK_OK; ++i)
      if (cudaStreamWaitEvent(b->side[i], b->fork_ev, 0) != cudaSuccess) st = STARK_ECUDA;
    size_t branches = 0;  // leaf streams that are part of the capture
    for (size_t q = 0; q < b->launches.size() && st == STARK_OK; ++q) {
      const auto& run = b->launches[q];
      for (int k = run.first; k < run.first + run.count && st == STARK_OK; ++k) {
        stark_plan_s* p = b->plans[k];
        const GroupDesc& g = b->host_desc[k];
        st = plan_divide_clear(p, ptrs[3 * k], ptrs[3 * k + 1], g.use_tma_c == 2 ? nullptr : g.C,
                               (size_t)p->n * g.ldc * sizeof(float), b->side[k % F]);
      }
      for (int i = 0; i < F && st == STARK_OK; ++i)
        if (cudaEventRecord(b->join_ev[i], b->side[i]) != cudaSuccess ||
            cudaStreamWaitEvent(b->leaf[q], b->join_ev[i], 0) != cudaSuccess)
          st = STARK_ECUDA;
        else
          branches = q + 1;
      if (st != STARK_OK) break;
      LeafTcArgs a{};
      a.err = b->d_err;
      a.timeout_ns = kDefaultTimeoutNs;
      const bool tf32 = b->dt == STARK_F32_SPLIT_TF32;
      a.b_mn = tf32 && b->plans[0]->tf32_mn;  // every member has the plan default
      a.fp16 = b->dt == STARK_F32_SPLIT_FP16 ? 1 : 0;
      a.groups = b->d_desc + run.first;
      a.ngroups = run.count;
      a.total_items = run.items;
      if ((run.wide ? launch_leaf_tc2_grouped(a, tf32, device_sm_count(), b->leaf[q])
                    : launch_leaf_tc_grouped(a, tf32, 128, device_sm_count(), b->leaf[q])) != cudaSuccess)
        st = STARK_ECUDA;
    }
    // join (also after an error, so the capture can end)
    for (int i = 0; i < F; ++i)
      if (cudaEventRecord(b->join_ev[i], b->side[i]) != cudaSuccess ||
          cudaStreamWaitEvent(b->cap, b->join_ev[i], 0) != cudaSuccess)
        st = STARK_ECUDA;
    for (size_t q = 0; q < branches; ++q)
      if (cudaEventRecord(b->fork_ev, b->leaf[q]) != cudaSuccess ||
          cudaStreamWaitEvent(b->cap, b->fork_ev, 0) != cudaSuccess)
        st = STARK_ECUDA;
    if (st == STARK_OK) {
      // members combined into a staging copy: move the result into C
      for (int k = 0; k < count && st == STARK_OK; ++k)
        if (b->host_desc[k].C != ptrs[3 * k + 2])
          st = plan_copy_cstage(b->plans[k], const_cast<void*>(ptrs[3 * k + 2]), b->cap);
    }
    const cudaError_t ec = cudaStreamEndCapture(b->cap, &graph);
    if (st != STARK_OK || ec != cudaSuccess) {
      if (graph) cudaGraphDestroy(graph);
      cudaGetLastError();
      return st != STARK_OK ? st : STARK_ECUDA;
    }
    const cudaError_t ei = cudaGraphInstantiate(&b->exec, graph, 0);
    cudaGraphDestroy(graph);
    if (ei != cudaSuccess) {
      b->exec = nullptr;
      cudaGetLastError();
      return STARK_ECUDA;
    }
    b->last = ptrs;
  }
  if (cudaGraphLaunch(b->exec, s) != cudaSuccess) {
    cudaGetLastError();
    return STARK_ECUDA;
  }
  ++b->replays;
  return STARK_OK;
}

stark_status stark_batch_check(stark_batch_t b, void* stream) {
  if (!b) return STARK_EINVAL;
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return STARK_ECUDA;
  int e = 0;
  if (cudaMemcpy(&e, b->d_err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return STARK_ECUDA;
  if (e != 0) {
    cudaMemset(b->d_err, 0, sizeof(int));
    return STARK_ETIMEOUT;
  }
  return STARK_OK;
}

}  // extern "C"
