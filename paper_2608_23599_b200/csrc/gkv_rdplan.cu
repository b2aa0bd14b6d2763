// RD allocator on the device (Sec. 3.3): the level plan of every stream from its block masses m_b and
// range proxies e_b, the same plan the host allocator makes from the same numbers, bit for bit.
//
// "b bits suffice for block b iff y_b = m_b e_b <= tau (2^b - 1)"; levels snap up to the ladder
// (y <= tau: centroid, <= 3 tau: 2 bits, <= 15 tau: 4, <= 255 tau: 8, else exact); pinned blocks (attention
// sinks, the recent window) stay exact; no level rises above the block's present one (Sec. 3.2) nor, with
// the age constraint, above that of any younger unpinned block.  tau is the smallest of the
// breakpoints {0} u {y_b / k : k in 1, 3, 15, 255} whose plan fits the bit budget.  The bit count never
// increases with tau, so the breakpoints are sorted and bisected; every test is a parallel pass over
// the blocks (thresholds, a suffix minimum for the age constraint, a sum of block sizes).  All
// arithmetic on y and tau is IEEE binary64 (exact products of two fp32, correctly rounded divisions),
// which is what makes the plan independent of who computes it.
//
// One CTA per stream.  Only the y are sorted: divided by k they are four sorted lists, and the smallest breakpoint of all
// whose plan fits is found by bisecting the longest remaining list and cutting all of them at the value tried.
// Shared memory: the four lists (the first one padded to a power of two for the sort), y by block, and the working
// levels.  Bound by latency (a bulk ingest waits for the plan): about fourteen tests of a few hundred cycles.  With all
// 4 n + 1 breakpoints in one bitonic sort a plan of 256 blocks took 28.9 us, 20.4 now.
#include <cuda_runtime.h>

#include <cstdint>

#include "gkv_internal.h"
#include "gkv_layout.cuh"

namespace gkv {
namespace {

constexpr int kPlanThreads = 1024;
constexpr unsigned kPlanAll = 0xffffffffu;

// (32 bits hold the bits of 4095 blocks of 256 values a token: 1.07e9)
__device__ __forceinline__ uint32_t plan_block_bits(int level, uint32_t nval_tok) {
  if (level == 16) return 16u * kBlock * nval_tok;
  if (level == 1) return 16u * nval_tok;
  return static_cast<uint32_t>(level) * kBlock * nval_tok + (kBlock * nval_tok / kGroup) * 32u;
}

constexpr int kPlanLists = 5;                // y / 1, y / 3, y / 15, y / 255, and 0
struct PlanShared {
  int min[kPlanThreads / 32];
  uint32_t bits[kPlanThreads / 32];
  int lo[kPlanLists], hi[kPlanLists];        // candidates below lo are too small, from hi on they fit
  int pick;                                  // list that is bisected, -1 = done
  double tau;                                // value tried
  // the result (fields of its own: a warp may still be on its way out of the search, reading `pick`, when they are written)
  int found;
  double best;
  int eligible;
};

// Levels of the plan for threshold tau into lv[] (shared) and the plan's bits (returned to every thread).
// Thread t owns the blocks [t * per, min(n, (t + 1) * per)).
__device__ uint32_t plan_for_tau(const RdPlanParams& p, const double* y, const TableEntry* table, int n, int per, double tau,
                                           int8_t* lv, PlanShared& sh) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, n_warps = blockDim.x >> 5;
  const int b0 = min(n, t * per), b1 = min(n, b0 + per);
  const int recent = p.retire_after / kBlock;
  const double t3 = tau * 3.0, t15 = tau * 15.0, t255 = tau * 255.0;
  // thresholds, pins and "never above the present level"; the chunk's minimum over unpinned blocks
  int cmin = 127;
  for (int b = b0; b < b1; ++b) {
    const double yb = y[b];
    int L = yb <= tau ? 1 : (yb <= t3 ? 2 : (yb <= t15 ? 4 : (yb <= t255 ? 8 : 16)));
    const bool pinned = b < p.n_sink_blocks || (n - 1 - b) < recent;
    if (pinned) L = 16;
    if (p.use_prev) {
      const int prev = static_cast<int>(table[b].level);
      if (prev < L) L = prev;
    }
    lv[b] = static_cast<int8_t>(L);
    if (!pinned) cmin = min(cmin, L);
  }
  const uint32_t nval = static_cast<uint32_t>(p.nval_tok);
  uint32_t bits = 0;
  if (p.monotone) {
    // level of a block <- minimum over the unpinned blocks at or after it (younger ones have higher
    // indices): a suffix scan over the threads' chunk minima
    int suf = cmin;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_down_sync(kPlanAll, suf, d);
      if (lane + d < 32) suf = min(suf, o);
    }
    if (lane == 0) sh.min[warp] = suf;
    __syncthreads();
    const int later = (lane < n_warps && lane > warp) ? sh.min[lane] : 127;       // the warps after this one
    int run = __reduce_min_sync(kPlanAll, later);
    const int next = __shfl_down_sync(kPlanAll, suf, 1);                           // the lanes after this one
    if (lane < 31) run = min(run, next);
    for (int b = b1 - 1; b >= b0; --b) {
      const bool pinned = b < p.n_sink_blocks || (n - 1 - b) < recent;
      if (!pinned) {
        run = min(run, static_cast<int>(lv[b]));
        lv[b] = static_cast<int8_t>(run);
      }
      bits += plan_block_bits(lv[b], nval);
    }
  } else {
    for (int b = b0; b < b1; ++b) bits += plan_block_bits(lv[b], nval);
    __syncthreads();                     // the last test's total has been read
  }
  // sum over the CTA (integers: any order)
  bits = __reduce_add_sync(kPlanAll, bits);
  if (lane == 0) sh.bits[warp] = bits;
  __syncthreads();
  return __reduce_add_sync(kPlanAll, lane < n_warps ? sh.bits[lane] : 0u);
  // (sh.min and sh.bits are rewritten behind the next test's first barrier only)
}

__global__ void __launch_bounds__(kPlanThreads) rd_plan_kernel(const RdPlanParams p) {
  extern __shared__ __align__(16) unsigned char plan_sm[];
  __shared__ PlanShared sh;
  const int s = blockIdx.x, t = threadIdx.x, n = p.n, n_thr = blockDim.x;
  double* list0 = reinterpret_cast<double*>(plan_sm);                // [pad] y ascending
  double* rest = list0 + p.pad;                                      // [3][n] divided by 3, 15, 255
  double* y = rest + 3 * n + 1;                                      // [n] by block, behind a fifth list: 0
  int8_t* lv = reinterpret_cast<int8_t*>(y + n);                     // [n]
  const float* mass = p.mass + static_cast<size_t>(s) * p.mass_stride;
  const float* range = p.range + static_cast<size_t>(s) * p.range_stride;
  const TableEntry* table = p.table + static_cast<size_t>(s) * p.table_stride;
  if (t < kPlanLists) {
    sh.lo[t] = 0;
    sh.hi[t] = t < 4 ? n : 1;
  }
  if (t == 0) sh.eligible = 0;
  for (int b = t; b < p.pad; b += n_thr) {
    double yb = __longlong_as_double(0x7ff0000000000000ll);          // +inf padding
    if (b < n) y[b] = yb = static_cast<double>(mass[b]) * static_cast<double>(range[b]);
    list0[b] = yb;
  }
  __syncthreads();
  // bitonic sort, ascending: thread t takes the pairs t, t + n_thr, ... of a stage; pair q of distance j is the elements
  // i = 2 q - (q mod j) and i + j, so a warp's 32 pairs cover the same 64 elements in every stage of distance <= 32
  for (int k = 2; k <= p.pad; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int q = t; q < p.pad / 2; q += n_thr) {
        const int i = 2 * q - (q & (j - 1)), l = i + j;
        const double a = list0[i], b = list0[l];
        const bool up = (i & k) == 0;
        if ((a > b) == up) {
          list0[i] = b;
          list0[l] = a;
        }
      }
      // the next stage's distance decides whether other warps' elements come into play
      const int next = j > 1 ? j >> 1 : k;
      if (next > 32 || j > 32) __syncthreads();
      else __syncwarp();
    }
  }
  __syncthreads();
  for (int b = t; b < n; b += n_thr) {
    const double yb = list0[b];
    rest[b] = yb / 3.0;
    rest[n + b] = yb / 15.0;
    rest[2 * n + b] = yb / 255.0;
  }
  if (t == 0) rest[3 * n] = 0.0;
  auto cand = [&](int list, int i) { return list0[(list == 0 ? 0 : p.pad + (list - 1) * n) + i]; };
  // the smallest candidate whose plan fits (bits never increase with tau)
  const int per = (n + n_thr - 1) / n_thr;
  const unsigned long long budget = p.budget_bits >= p.tail_bits ? p.budget_bits - p.tail_bits : 0ull;
  const bool any_room = p.budget_bits >= p.tail_bits;
  __syncthreads();
  while (true) {                                                     // uniform for the CTA
    if (t < 32) {
      const int len = t < kPlanLists ? sh.hi[t] - sh.lo[t] : 0;
      const int longest = __reduce_max_sync(kPlanAll, len);
      const int pick = __ffs(static_cast<int>(__ballot_sync(kPlanAll, len == longest))) - 1;
      if (t == 0) {
        sh.pick = longest > 0 ? pick : -1;
        if (longest > 0) sh.tau = cand(pick, (sh.lo[pick] + sh.hi[pick]) >> 1);
      }
    }
    __syncthreads();
    if (sh.pick < 0) break;
    const double tau = sh.tau;
    const bool fits = plan_for_tau(p, y, table, n, per, tau, lv, sh) <= budget && any_room;
    // cut every list: at its first candidate >= tau, or behind its last one <= tau
    if (t < kPlanLists) {
      int lo = sh.lo[t], hi = sh.hi[t];
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const double v = cand(t, mid);
        if (fits ? v >= tau : v > tau) hi = mid;
        else lo = mid + 1;
      }
      (fits ? sh.hi[t] : sh.lo[t]) = lo;
    }
    __syncthreads();
  }
  if (t == 0) {
    double best = __longlong_as_double(0x7ff0000000000000ll);
    bool found = false;
    for (int l = 0; l < kPlanLists; ++l)
      if (sh.hi[l] < (l < 4 ? n : 1)) {
        found = true;
        best = fmin(best, cand(l, sh.hi[l]));
      }
    sh.found = found;
    sh.best = found ? best : fmax(list0[n - 1], 0.0);                // no plan fits: the largest candidate's
  }
  __syncthreads();
  const bool miss = !sh.found;
  plan_for_tau(p, y, table, n, per, sh.best, lv, sh);
  __syncthreads();
  int8_t* out = p.levels_out + static_cast<size_t>(s) * p.out_stride;
  int eligible = 0;
  for (int b = t; b < n; b += n_thr) {
    out[b] = lv[b];
    eligible += b >= p.n_sink_blocks && lv[b] != 16;
  }
  if (t == 0 && miss) atomicOr(p.miss_flag, 1u);
  if (p.res_count) {
    eligible = __reduce_add_sync(kPlanAll, eligible);
    if ((t & 31) == 0) atomicAdd(&sh.eligible, eligible);
    __syncthreads();
    if (t == 0) p.res_count[s] = min(min(p.n_res, kBlock * sh.eligible), p.res_cap);
  }
}

}  // namespace

size_t rd_plan_smem_bytes(int n, int* pad_out) {
  int pad = 2;
  while (pad < n) pad <<= 1;
  if (pad_out) *pad_out = pad;
  return static_cast<size_t>(pad + 4 * n + 1) * sizeof(double) + static_cast<size_t>(n) + 16;
}

cudaError_t launch_rd_plan(const RdPlanParams& p, int n_streams, cudaStream_t st) {
  const size_t bytes = rd_plan_smem_bytes(p.n, nullptr);
  if (bytes > 48 * 1024) {
    static std::atomic<uint64_t> done{0};
    const cudaError_t e = raise_smem_limit(rd_plan_kernel, rd_plan_smem_bytes(kRdPlanMaxBlocks, nullptr), done);
    if (e != cudaSuccess) return e;
  }
  // a block per thread, as far as there are threads
  const int threads = p.pad < 32 ? 32 : (p.pad < kPlanThreads ? p.pad : kPlanThreads);
  rd_plan_kernel<<<n_streams, threads, bytes, st>>>(p);
  return cudaGetLastError();
}

}  // namespace gkv
