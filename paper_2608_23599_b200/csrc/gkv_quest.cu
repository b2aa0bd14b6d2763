// Compressed-Quest page scorer and top-k selection (paper Sec. 3.5), also used for the exact
// residual's top fraction (Sec. 3.4).
//
// Score of a page for one query head: acc <- fma(q_d, q_d >= 0 ? max_d : min_d, acc) for
// d = 0..127 in order, fp32.  q_d and the box bounds are bf16, so every product is exact in fp32
// and the fma rounds exactly like "exact product, then add": the order of d is the only thing
// that fixes the bits.  Boxes are stored channel-major ([stream][channel][min|max][page]) so a
// warp's loads run along pages and coalesce.
//
// Selection: k largest scores, ties to the lower index, emitted in ascending index order
// (the threshold on an order-preserving key first, then an ordered compaction).
#include "gkv_internal.h"

namespace gkv {
namespace {

// One CTA scores 2 THREADS consecutive pages of one stream, two neighbouring pages per thread.  The 256 box rows of
// the stream (channel x min|max) are streamed through shared memory in chunks of
// kQRows rows with 16-byte cp.async copies, STAGES - 1 chunks in flight, so that the loads are wide, contiguous
// and deep while every thread still adds its pages' channels strictly in order.  Two shapes: 128 pages and a ring of four
// chunks where there are many pages, 64 pages and all eight chunks in flight where CTAs of that size fit the GPU
// at once and the time is that of one round of loads (selection and read, 32 streams: 512 pages 31.2 -> 27.7 us, 1024 pages
// 33.3 -> 30.5; beyond one wave, at 1536 pages, 37.1 instead of 35.4).
//
// The choice between maximum and minimum depends on the sign of q_d only, so it is made once, when the query is
// staged: acc <- fma(max(q, 0), hi, fma(min(q, 0), lo, acc)), where one of the two products is a zero that leaves
// acc as it is.  Two pages share an instruction (packed fp32 pairs, each half rounded as usual), which leaves 18
// instructions per channel and two pages for four heads; with a select per head and one page per thread it was 40,
// and the kernel was bound by instruction issue.  (Selection and read of 2048 pages x 32 streams: 37.0 -> 32.4 us a
// layer with this and the selection below.)
constexpr int kQRows = 32;                                   // rows per chunk = 16 channels x (min, max)
constexpr int kQChunks = 2 * kD / kQRows;                    // 8
constexpr int kQSmallCtas = 148 * 5;

__device__ __forceinline__ void q_cp_async16(uint32_t dst, const void* src, bool on) {
  const uint32_t n = on ? 16u : 0u;                          // 0 source bytes: the 16 bytes are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ uint64_t q_pair(float x, float y) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};\n" : "=l"(v) : "f"(x), "f"(y));
  return v;
}
// two bf16 numbers as a pair of fp32
__device__ __forceinline__ uint64_t q_pair_bf16(uint32_t u) { return q_pair(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)); }
__device__ __forceinline__ uint64_t q_fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// GROUP = query heads per KV head, a compile-time bound: a run-time bound would leave the unused
// heads' instructions in the loop, predicated off but still issued.
template <int GROUP, int THREADS, int STAGES>
__global__ void __launch_bounds__(THREADS) quest_score_kernel(const uint16_t* __restrict__ boxes, int box_stride,
                                                                int n_pages, const uint16_t* __restrict__ q,
                                                                int n_kv_heads, int reduce,
                                                                float* __restrict__ scores, int score_stride) {
  constexpr int group = GROUP, kQThreads = THREADS, kQStages = STAGES, kQPages = 2 * THREADS;
  constexpr int kQRowBytes = kQPages * 2, kQChunkBytes = kQRows * kQRowBytes, kQPieces = kQRowBytes / 16;      // 16-byte pieces per row
  // launched with programmatic stream serialisation: returns once the previous kernel of the stream
  // has completed (the launch itself overlaps that kernel's tail)
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  extern __shared__ __align__(16) uint8_t qsm[];
  // per channel and head the pairs (q+, q+) and (q-, q-)
  ulonglong2* qs = reinterpret_cast<ulonglong2*>(qsm + kQStages * kQChunkBytes);       // [128][GROUP]
  const int stream = blockIdx.y, tid = threadIdx.x;
  const int page0 = blockIdx.x * kQPages;
  const uint16_t* rows = boxes + static_cast<size_t>(stream) * kD * 2 * box_stride + page0;
  const uint32_t stage0 = static_cast<uint32_t>(__cvta_generic_to_shared(qsm));
  // chunk c -> stage c % kQStages: row r of the chunk is box row c * kQRows + r; a piece
  // of 16 bytes is 8 pages; pieces that start beyond the row's end (box_stride) are zero-filled
  auto issue = [&](int c) {
    const uint32_t dst = stage0 + (c % kQStages) * kQChunkBytes;
#pragma unroll
    for (int i = 0; i < kQRows * kQPieces / kQThreads; ++i) {
      const int piece = tid + i * kQThreads, r = piece / kQPieces, col = piece % kQPieces;
      const bool on = page0 + 8 * col < box_stride;
      q_cp_async16(dst + r * kQRowBytes + col * 16, rows + static_cast<size_t>(c * kQRows + r) * box_stride + (on ? 8 * col : 0), on);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
#pragma unroll
  for (int c = 0; c < kQStages - 1; ++c) issue(c);
  {
    const uint32_t* q2 = reinterpret_cast<const uint32_t*>(q + static_cast<size_t>(stream) * group * kD);      // [batch][n_q_heads], KV heads in order
#pragma unroll
    for (int h = 0; h < GROUP; ++h)
#pragma unroll
      for (int at = tid; at < kD / 2; at += kQThreads) {
        const uint32_t u = q2[h * (kD / 2) + at];
        const float v[2] = {__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float up = fmaxf(v[k], 0.f), dn = fminf(v[k], 0.f);
          qs[(2 * at + k) * GROUP + h] = make_ulonglong2(q_pair(up, up), q_pair(dn, dn));
        }
      }
  }
  uint64_t acc[GROUP];
#pragma unroll
  for (int h = 0; h < GROUP; ++h) acc[h] = 0ull;
#pragma unroll 1
  for (int c = 0; c < kQChunks; ++c) {
    if (c + kQStages - 1 < kQChunks) issue(c + kQStages - 1);
    else asm volatile("cp.async.commit_group;\n" ::: "memory");          // keeps the group count uniform
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kQStages - 1) : "memory");
    __syncthreads();                                   // chunk c (and, the first time, the query) is visible to all
    const uint8_t* st = qsm + (c % kQStages) * kQChunkBytes + tid * 4;
    const ulonglong2* qc = qs + c * (kQRows / 2) * GROUP;
#pragma unroll
    for (int i = 0; i < kQRows / 2; ++i) {
      const uint64_t lo = q_pair_bf16(*reinterpret_cast<const uint32_t*>(st + (2 * i) * kQRowBytes));
      const uint64_t hi = q_pair_bf16(*reinterpret_cast<const uint32_t*>(st + (2 * i + 1) * kQRowBytes));
#pragma unroll
      for (int h = 0; h < GROUP; ++h) {
        const ulonglong2 qv = qc[i * GROUP + h];
        acc[h] = q_fma2(qv.x, hi, q_fma2(qv.y, lo, acc[h]));
      }
    }
    __syncthreads();                                   // the stage may be refilled
  }
  const int p0 = page0 + 2 * tid;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (p0 + k >= n_pages) return;
    float s0 = __uint_as_float(static_cast<uint32_t>(acc[0] >> (32 * k)));
#pragma unroll
    for (int h = 1; h < GROUP; ++h) {
      const float s1 = __uint_as_float(static_cast<uint32_t>(acc[h] >> (32 * k)));
      s0 = (reduce == 0) ? fmaxf(s0, s1) : __fadd_rn(s0, s1);
    }
    scores[static_cast<size_t>(stream) * score_stride + p0 + k] = s0;
  }
}

// Order-preserving key: larger score <-> larger key; -0 and +0 map to the same key.
__device__ __forceinline__ uint32_t score_key(float s) {
  const uint32_t f = __float_as_uint(s + 0.0f);
  return (f & 0x80000000u) ? ~f : (f | 0x80000000u);
}

constexpr int kTopkThreads = 1024;

// Selection with every key in registers: warp w holds the keys of the elements [32 PER w, 32 PER (w + 1)), lane l those at
// l, l + 32, ... of them (its loads are 128 bytes a warp).  The k-th largest
// key is bracketed by counting: lo <= it <= hi, three probes a round, the keys at or above each counted with warp
// reductions and one barrier.  The search ends early when exactly k keys lie at or above lo.  One sum over the
// warps then gives every selected element its place in index order.  (A radix select puts its first digit, sign and
// exponent, of nearly all scores into a few bins whose shared-memory counters are then incremented one by one, and its
// compaction took four barriers per 1024 elements: 29 us for 16,384 scores of 32 streams, 18.7 us this way.)
template <int PER>
__global__ void __launch_bounds__(kTopkThreads) topk_regs_kernel(const float* __restrict__ scores, int score_stride, int n,
                                                                 const int32_t* __restrict__ k_per_stream, int k_uniform,
                                                                 int32_t* __restrict__ idx_out, int idx_stride) {
  constexpr uint32_t kAll = 0xffffffffu;
  __shared__ uint2 s_cnt[2][32];
  __shared__ uint32_t s_scan[32];
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int stream = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_warps = blockDim.x >> 5;
  const float* sc = scores + static_cast<size_t>(stream) * score_stride;
  int32_t* out = idx_out + static_cast<size_t>(stream) * idx_stride;
  const uint32_t k = static_cast<uint32_t>(min(k_per_stream ? k_per_stream[stream] : k_uniform, n));
  if (static_cast<int>(k) <= 0) return;
  uint32_t key[PER];                                 // 0 past the end: below every probe
  uint32_t mn = kAll, mx = 0u;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = warp * (32 * PER) + j * 32 + lane;
    key[j] = i < n ? max(score_key(sc[i]), 1u) : 0u;
    if (i < n) {
      mn = min(mn, key[j]);
      mx = max(mx, key[j]);
    }
  }
  mn = __reduce_min_sync(kAll, mn);
  mx = __reduce_max_sync(kAll, mx);
  if (lane == 0) s_cnt[1][warp] = make_uint2(mn, mx);
  __syncthreads();
  {
    const uint2 v = lane < n_warps ? s_cnt[1][lane] : make_uint2(kAll, 0u);
    mn = __reduce_min_sync(kAll, v.x);
    mx = __reduce_max_sync(kAll, v.y);
  }
  uint32_t lo = mn, hi = mx, n_lo = static_cast<uint32_t>(n);      // n_lo keys are >= lo; fewer than k are > hi
  int round = 0;
  while (lo < hi && n_lo != k) {                     // uniform for the CTA
    const uint32_t range = hi - lo, step = range / 4 + 1;
    const uint32_t p1 = lo + min(step, range), p2 = lo + min(2 * step, range), p3 = lo + static_cast<uint32_t>(min(3ull * step, static_cast<unsigned long long>(range)));
    uint32_t c12 = 0, c3 = 0;                        // counts of a thread <= 32, of the CTA <= 32,768: 16 bits each
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      c12 += (key[j] >= p1 ? 1u : 0u) + (key[j] >= p2 ? 0x10000u : 0u);
      c3 += key[j] >= p3 ? 1u : 0u;
    }
    c12 = __reduce_add_sync(kAll, c12);
    c3 = __reduce_add_sync(kAll, c3);
    if (lane == 0) s_cnt[round & 1][warp] = make_uint2(c12, c3);
    __syncthreads();                                 // (the other buffer is rewritten only behind the next barrier)
    const uint2 v = lane < n_warps ? s_cnt[round & 1][lane] : make_uint2(0u, 0u);
    c12 = __reduce_add_sync(kAll, v.x);
    c3 = __reduce_add_sync(kAll, v.y);
    const uint32_t c1 = c12 & 0xffffu, c2 = c12 >> 16;
    if (c3 >= k) {
      lo = p3;
      n_lo = c3;
    } else if (c2 >= k) {
      lo = p2;
      n_lo = c2;
      hi = p3 - 1;
    } else if (c1 >= k) {
      lo = p1;
      n_lo = c1;
      hi = p2 - 1;
    } else {
      hi = p1 - 1;
    }
    ++round;
  }
  // taken: the keys above `thr`, and of those equal to `eq` the first ones in index order until k are taken
  const bool all = n_lo == k;                        // exactly the keys at or above lo
  const uint32_t thr = all ? lo - 1 : lo, eq = all ? 0u : lo;
  uint32_t mine = 0;                                 // the warp's: above | equal << 16
#pragma unroll
  for (int j = 0; j < PER; ++j) mine += (key[j] > thr ? 1u : 0u) + ((eq != 0u && key[j] == eq) ? 0x10000u : 0u);
  mine = __reduce_add_sync(kAll, mine);
  if (lane == 0) s_scan[warp] = mine;
  __syncthreads();
  const uint32_t ws = lane < n_warps ? s_scan[lane] : 0u;
  const uint32_t total = __reduce_add_sync(kAll, ws);
  const uint32_t before = __reduce_add_sync(kAll, lane < warp ? ws : 0u);
  const uint32_t need = k - (total & 0xffffu);       // equal keys taken
  uint32_t above = before & 0xffffu, equal = before >> 16;
  const uint32_t below = (1u << lane) - 1u;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const bool gt = key[j] > thr, same = eq != 0u && key[j] == eq;
    const uint32_t bg = __ballot_sync(kAll, gt), bs = __ballot_sync(kAll, same);
    const uint32_t at_eq = equal + __popc(bs & below);
    if (gt || (same && at_eq < need)) out[above + __popc(bg & below) + min(at_eq, need)] = warp * (32 * PER) + j * 32 + lane;
    above += __popc(bg);
    equal += __popc(bs);
  }
}

// Longer lists: radix select over the scores in global memory, ordered compaction.
__global__ void __launch_bounds__(kTopkThreads) topk_kernel(const float* __restrict__ scores, int score_stride,
                                                            int n, const int32_t* __restrict__ k_per_stream,
                                                            int k_uniform, int32_t* __restrict__ idx_out,
                                                            int idx_stride) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t s_prefix, s_remaining;
  __shared__ uint32_t warp_sel[32], warp_eq[32];
  __shared__ uint32_t base_sel, base_eq;
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int stream = blockIdx.x, tid = threadIdx.x;
  const float* sc = scores + static_cast<size_t>(stream) * score_stride;
  int32_t* out = idx_out + static_cast<size_t>(stream) * idx_stride;
  int k = k_per_stream ? k_per_stream[stream] : k_uniform;
  if (k > n) k = n;
  if (k <= 0) return;
  if (tid == 0) {
    s_prefix = 0;
    s_remaining = static_cast<uint32_t>(k);
  }
  // radix select, most significant byte first: find the key of the k-th largest score
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    for (int i = tid; i < 256; i += kTopkThreads) hist[i] = 0;
    __syncthreads();
    const uint32_t prefix = s_prefix;
    const uint32_t pmask = pass == 0 ? 0u : (0xffffffffu << (shift + 8));
    for (int i = tid; i < n; i += kTopkThreads) {
      const uint32_t key = score_key(sc[i]);
      if ((key & pmask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
    }
    __syncthreads();
    // The digit of the k-th largest is the t with c[t] >= rem > c[t + 1], c[t] = sum_{j >= t} hist[j].
    // Warp 0: lane l owns bins 255 - 8 l .. 248 - 8 l (from the top), a shuffle scan joins the lanes.
    if (tid < 32) {
      const uint32_t rem = s_remaining;
      uint32_t own[8], tot = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        own[j] = hist[255 - 8 * tid - j];
        tot += own[j];
      }
      uint32_t incl = tot;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t up = __shfl_up_sync(0xffffffffu, incl, d);
        if (tid >= d) incl += up;
      }
      uint32_t above = incl - tot;                  // count in bins above this lane's eight
      if (above < rem && incl >= rem) {             // exactly one lane
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (above < rem && above + own[j] >= rem) {
            s_prefix = prefix | (static_cast<uint32_t>(255 - 8 * tid - j) << shift);
            s_remaining = rem - above;
            above = rem;                            // done: no later bin matches
          } else {
            above += own[j];
          }
        }
      }
    }
    __syncthreads();
  }
  const uint32_t thr = s_prefix;          // key of the k-th largest
  const uint32_t need_eq = s_remaining;   // how many elements equal to thr are taken (lowest indices)
  if (tid == 0) {
    base_sel = 0;
    base_eq = 0;
  }
  __syncthreads();
  // ordered compaction in index order
  const int lane = tid & 31, wid = tid >> 5;
#pragma unroll 1
  for (int i0 = 0; i0 < n; i0 += kTopkThreads) {
    const int i = i0 + tid;
    uint32_t key = 0;
    bool gt = false, eq = false;
    if (i < n) {
      key = score_key(sc[i]);
      gt = key > thr;
      eq = key == thr;
    }
    // rank of this element among the equal ones (exclusive, in index order)
    const uint32_t eq_ballot = __ballot_sync(0xffffffffu, eq);
    const uint32_t eq_before_w = __popc(eq_ballot & ((1u << lane) - 1u));
    if (lane == 0) warp_eq[wid] = __popc(eq_ballot);
    __syncthreads();
    uint32_t eq_before = base_eq + eq_before_w;
    for (int w2 = 0; w2 < wid; ++w2) eq_before += warp_eq[w2];
    const bool take = gt || (eq && eq_before < need_eq);
    const uint32_t sel_ballot = __ballot_sync(0xffffffffu, take);
    const uint32_t sel_before_w = __popc(sel_ballot & ((1u << lane) - 1u));
    if (lane == 0) warp_sel[wid] = __popc(sel_ballot);
    __syncthreads();
    uint32_t pos = base_sel + sel_before_w;
    for (int w2 = 0; w2 < wid; ++w2) pos += warp_sel[w2];
    if (take && pos < static_cast<uint32_t>(k)) out[pos] = i;
    __syncthreads();
    if (tid == 0) {
      uint32_t te = 0, ts = 0;
      for (int w2 = 0; w2 < 32; ++w2) {
        te += warp_eq[w2];
        ts += warp_sel[w2];
      }
      base_eq += te;
      base_sel += ts;
    }
    __syncthreads();
  }
}

}  // namespace

namespace {
template <int GROUP, int THREADS, int STAGES>
cudaError_t launch_quest_shape(const uint16_t* boxes, int box_stride, int n_pages, const uint16_t* q, int n_streams, int n_kv_heads,
                               int reduce, float* scores, int score_stride, cudaStream_t st) {
  const size_t smem = static_cast<size_t>(STAGES) * kQRows * THREADS * 4 + static_cast<size_t>(GROUP) * kD * 16;
  static std::atomic<uint64_t> done{0};
  const cudaError_t e = raise_smem_limit(quest_score_kernel<GROUP, THREADS, STAGES>, smem, done);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((n_pages + 2 * THREADS - 1) / (2 * THREADS), n_streams);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, quest_score_kernel<GROUP, THREADS, STAGES>, boxes, box_stride, n_pages, q, n_kv_heads, reduce, scores, score_stride);
}
template <int GROUP>
cudaError_t launch_quest_group(const uint16_t* boxes, int box_stride, int n_pages, const uint16_t* q, int n_streams, int n_kv_heads,
                               int reduce, float* scores, int score_stride, cudaStream_t st) {
  // CTAs of 64 pages that an SM holds at once: five (shared memory, four query heads)
  if (static_cast<long long>((n_pages + 63) / 64) * n_streams <= kQSmallCtas)
    return launch_quest_shape<GROUP, 32, kQChunks>(boxes, box_stride, n_pages, q, n_streams, n_kv_heads, reduce, scores, score_stride, st);
  return launch_quest_shape<GROUP, 64, 4>(boxes, box_stride, n_pages, q, n_streams, n_kv_heads, reduce, scores, score_stride, st);
}
}  // namespace

cudaError_t launch_quest_scores(const uint16_t* boxes, int box_stride, int n_pages, const uint16_t* q,
                                int n_streams, int n_kv_heads, int group, int reduce, float* scores,
                                int score_stride, cudaStream_t st) {
  if (n_pages <= 0) return cudaSuccess;
#define GKV_QUEST_CASE(G) \
  case G: return launch_quest_group<G>(boxes, box_stride, n_pages, q, n_streams, n_kv_heads, reduce, scores, score_stride, st);
  switch (group) {
    GKV_QUEST_CASE(1)
    GKV_QUEST_CASE(2)
    GKV_QUEST_CASE(3)
    GKV_QUEST_CASE(4)
    GKV_QUEST_CASE(5)
    GKV_QUEST_CASE(6)
    GKV_QUEST_CASE(7)
    GKV_QUEST_CASE(8)
    default: return cudaErrorInvalidValue;
  }
#undef GKV_QUEST_CASE
}

cudaError_t launch_topk(const float* scores, int score_stride, int n, const int32_t* k_per_stream, int k_uniform,
                        int32_t* idx_out, int idx_stride, int n_streams, cudaStream_t st) {
  if (n <= 0 || n_streams <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_streams);
  cfg.blockDim = dim3(kTopkThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
#define GKV_TOPK_CASE(PER)                                                                                                  \
  if (n <= PER * kTopkThreads) {                                                                                           \
    cfg.blockDim = dim3(static_cast<unsigned>((n + 32 * PER - 1) / (32 * PER) * 32));                                      \
    return cudaLaunchKernelEx(&cfg, topk_regs_kernel<PER>, scores, score_stride, n, k_per_stream, k_uniform, idx_out, idx_stride); \
  }
  GKV_TOPK_CASE(4)
  GKV_TOPK_CASE(16)
  GKV_TOPK_CASE(32)
#undef GKV_TOPK_CASE
  return cudaLaunchKernelEx(&cfg, topk_kernel, scores, score_stride, n, k_per_stream, k_uniform, idx_out, idx_stride);
}

}  // namespace gkv
