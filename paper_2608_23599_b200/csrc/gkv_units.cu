// Work lists of the decode kernel, made on the device from the block table (one CTA per stream).
//
// A stream's items (closed blocks, the tail, groups of 16 exact residual rows) become units: an item, a run of up to 16
// neighbouring centroid blocks that does not cross a multiple of 16, or, in small workloads, a part of a block.  The
// units are put in order of falling cost and dealt to the stream's warps in rounds: the costliest unit of a round goes to
// the warp that has least so far, the next one to the next warp, up to the first warp that already has more than the least
// laden one will have with its unit.  So every warp ends up with about the same cost whatever the order of levels along
// the context, and with about the same share of every level.  (Dealing forth and back without a look at
// what a warp has balances the cost as well, but leaves the 8-bit blocks to the warps that have an exact one: 64 streams
// of 32,757 tokens took 73.6 us a call instead of 72.3.  One unit to every warp in every round leaves a warp with an exact
// block 12 % more than the others where the rest is cheap: 64 streams with exact residual rows 32.7 us a call.  Classes in a
// fixed order, exact blocks first and centroid runs last, 256 exact tokens, centroids and 10 % exact rows: 32.2 us a call for 64
// streams of 32,747 tokens, 21.6 for 32, 21.1 for 64 of 16,384; by falling cost 31.75, 19.8 and 20.3.)
//
// The first round hands the costliest units (of whole blocks the exact ones, then 8-bit ones) to the first warps, and a CTA is a window of
// consecutive warps: the warps are walked with a golden-ratio stride, so that every window holds the same mixture of
// levels.  Warps of one SM share its issue slots, and a CTA whose warps all run the issue-heavy levels would finish
// last.  Within its list a warp takes the units alternately from both ends (a byte-heavy unit after an issue-heavy one: its
// two-stage pipeline always has a long compute to hide a long copy behind) and starts at a place of its own, which
// keeps both kinds of step in every SM at all times.  Every place follows from an item's rank, so the lists, and with
// them the order of every sum, do not depend on timing.
//
// Bound by latency: a few barriers per 512 items and a sort of the warps per round.  The host's dealing (a sort and a
// heap per stream) took 780 us for 32 streams of 256 blocks whose plans differ; the host's part is now the streams' cost
// and warp counts, 35 us with the launches.
#include "gkv_internal.h"

namespace gkv {
namespace {

constexpr int kUnitThreads = 512, kUnitWarps = kUnitThreads / 32;
constexpr unsigned kUnitAll = 0xffffffffu;
constexpr int kUnitHandBits = 12;           // a warp's number in a sort key
static_assert(148 * kDecodeCtasPerSm * kDecodeWarps + 1 < (1 << kUnitHandBits), "a stream's warps fit a sort key");

__global__ void __launch_bounds__(kUnitThreads) units_kernel(const __grid_constant__ UnitsParams p) {
  __shared__ int s_base[kUnitClasses], s_start[kUnitClasses + 1], s_at[kUnitWarps][kUnitClasses];
  extern __shared__ __align__(16) uint32_t s_key[];            // [pad] load / 16 << 12 | warp; later where a list begins
  const int s = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const StreamPlan plan = p.plans[s];
  const TableEntry* table = p.table + static_cast<size_t>(s) * p.table_stride;
  const int n_items = p.n_closed + 1 + (plan.n_res + 15) / 16;
  const int nw = plan.n_warps;

  // the place of an item's class in the order of falling cost (-1: the item is part of an earlier unit, or past the end), its
  // unit word without the tile mask, its parts
  const int at2 = p.place[kClass2Bits], at4 = p.place[kClass4Bits];
  auto classify = [&](int it, uint32_t& word, int& parts) -> int {
    const int level = it < p.n_closed ? static_cast<int>(table[it].level) : 0;
    const bool cent = it < p.n_closed && level != 16 && level != 8 && level != 4 && level != 2;
    const uint32_t group = (__ballot_sync(kUnitAll, cent) >> (lane & 16)) & 0xffffu;      // items of the aligned group of 16
    const int pos = lane & 15;
    word = static_cast<uint32_t>(it) | (1u << 24);
    parts = 1;
    if (it >= n_items) return -1;
    if (cent) {
      if (pos > 0 && ((group >> (pos - 1)) & 1u)) return -1;
      const int run = __ffs(static_cast<int>(~(group >> pos))) - 1;
      word = static_cast<uint32_t>(it) | (static_cast<uint32_t>(run) << 24);
      return p.place[22 - run];
    }
    if (it > p.n_closed) return p.place[5];
    if (it == p.n_closed) {
      parts = p.split_all ? 4 : 1;
      return p.place[4];
    }
    if (level == 16) {
      parts = p.split ? 4 : 1;
      return p.place[0];
    }
    parts = p.split_all ? 2 : 1;
    return level == 8 ? p.place[1] : (level == 2 ? at2 : at4);
  };
  auto clear = [&]() {
    for (int i = tid; i < kUnitWarps * kUnitClasses; i += kUnitThreads) s_at[i / kUnitClasses][i % kUnitClasses] = 0;
  };

  // pass 1: units of every class, then where the classes begin in the order of falling cost
  if (tid < kUnitClasses) s_base[tid] = 0;
  __syncthreads();
  for (int c0 = 0; c0 < n_items; c0 += kUnitThreads) {
    uint32_t word;
    int parts;
    const int cls = classify(c0 + tid, word, parts);
    const uint32_t peers = __match_any_sync(kUnitAll, cls);
    if (cls >= 0 && lane == __ffs(static_cast<int>(peers)) - 1) atomicAdd(&s_base[cls], __popc(peers) * parts);
  }
  __syncthreads();
  if (warp == 0) {
    const int n = lane < kUnitClasses ? s_base[lane] : 0;
    int incl = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int up = __shfl_up_sync(kUnitAll, incl, d);
      if (lane >= d) incl += up;
    }
    if (lane < kUnitClasses) s_base[lane] = s_start[lane] = incl - n;
    if (lane == kUnitClasses) s_start[lane] = incl;
  }
  clear();
  const int pad = p.pad;                               // a power of two, at least the warps of any stream
  uint32_t* s_mix = s_key + pad;                       // [pad] a warp's 2-bit units, and its 4-bit ones << 16
  uint32_t* s_cnt = s_mix + pad;                       // [pad] units of a warp
  uint32_t* hand_of = s_cnt + pad;                     // [n_units] a rank's place in its list << 12 | the warp that it goes to
  for (int i = tid; i < pad; i += kUnitThreads) {
    s_key[i] = i < nw ? static_cast<uint32_t>(i) : 0xffffffffu;
    s_mix[i] = 0u;
    s_cnt[i] = 0u;
  }
  __syncthreads();

  // The deal: per round the warps in order of what they have, those left out that have more than the least laden one
  // will have with its unit.  A thread's ranks only grow, so its class does, too.
  const int n_units = plan.n_units;
  int cls_at = 0, cls_base = 0, base = 0;
  auto deal = [&](int rank, uint32_t key) -> uint32_t {
    if (rank >= n_units) return key;
    const uint32_t hand = key & ((1u << kUnitHandBits) - 1u);
    hand_of[rank] = (s_cnt[hand]++ << kUnitHandBits) | hand;                         // (one unit per warp and round)
    while (cls_at < kUnitClasses - 1 && rank >= s_start[cls_at + 1]) ++cls_at;
    if (cls_at == at2 || cls_at == at4) s_mix[hand] += cls_at == at2 ? 1u : 0x10000u;
    return key + (static_cast<uint32_t>(p.cost[cls_at]) / 16 << kUnitHandBits);
  };
  // keys below this take part in the round that begins with rank `base`; least is the smallest key
  auto limit = [&](uint32_t least) -> uint32_t {
    while (cls_base < kUnitClasses - 1 && base >= s_start[cls_base + 1]) ++cls_base;
    return ((least >> kUnitHandBits) + static_cast<uint32_t>(p.cost[cls_base]) / 16) << kUnitHandBits;
  };
  if (p.dealt && nw <= 64) {
    // one warp, two keys a lane (places lane and lane + 32), sorted with shuffles
    if (warp == 0) {
      uint32_t k0 = lane < nw ? static_cast<uint32_t>(lane) : 0xffffffffu, k1 = lane + 32 < nw ? static_cast<uint32_t>(lane + 32) : 0xffffffffu;
      while (base < n_units) {
        if (base > 0) {
#pragma unroll
          for (int k = 2; k <= 64; k <<= 1) {
#pragma unroll
            for (int j = k >> 1; j > 0; j >>= 1) {
              if (j == 32) {
                const uint32_t lo = min(k0, k1);
                k1 = max(k0, k1);
                k0 = lo;
              } else {
                const uint32_t o0 = __shfl_xor_sync(kUnitAll, k0, j), o1 = __shfl_xor_sync(kUnitAll, k1, j);
                const bool first = (lane & j) == 0, up0 = (lane & k) == 0, up1 = ((lane + 32) & k) == 0;
                k0 = first == up0 ? min(k0, o0) : max(k0, o0);
                k1 = first == up1 ? min(k1, o1) : max(k1, o1);
              }
            }
          }
        }
        const uint32_t lim = limit(__shfl_sync(kUnitAll, k0, 0));
        const bool in0 = k0 < lim || lane == 0, in1 = k1 < lim;      // the least laden warp always: every round ends with fewer units left
        if (in0) k0 = deal(base + lane, k0);
        if (in1) k1 = deal(base + lane + 32, k1);
        base += __popc(__ballot_sync(kUnitAll, in0)) + __popc(__ballot_sync(kUnitAll, in1));
        __syncwarp();
      }
    }
  } else if (p.dealt) {
    int small = 128;
    while (small < nw) small <<= 1;
    while (base < n_units) {
      if (base > 0) {
        for (int k = 2; k <= small; k <<= 1) {
          for (int j = k >> 1; j > 0; j >>= 1) {
            for (int q = tid; q < small / 2; q += kUnitThreads) {
              const int i = 2 * q - (q & (j - 1)), l = i + j;
              const uint32_t x = s_key[i], y = s_key[l];
              if ((x > y) == ((i & k) == 0)) {
                s_key[i] = y;
                s_key[l] = x;
              }
            }
            __syncthreads();
          }
        }
      }
      const uint32_t lim = limit(s_key[0]);
      int m = 1, end = nw;                             // how many keys, in order, are below the limit (the first one is)
      while (m < end) {
        const int mid = (m + end) >> 1;
        if (s_key[mid] < lim) m = mid + 1;
        else end = mid;
      }
      __syncthreads();
      for (int i = tid; i < m; i += kUnitThreads) s_key[i] = deal(base + i, s_key[i]);
      base += m;
      __syncthreads();
    }
  } else {
    const int full = n_units / nw;
    for (int i = tid; i < nw; i += kUnitThreads) s_cnt[i] = static_cast<uint32_t>(full + (i < n_units - full * nw));
  }
  __syncthreads();
  // where the warps' lists begin (the keys are done with)
  if (warp == 0) {
    uint32_t at = static_cast<uint32_t>(plan.unit_base);
    for (int i0 = 0; i0 < nw; i0 += 32) {
      const uint32_t n = i0 + lane < nw ? s_cnt[i0 + lane] : 0u;
      uint32_t incl = n;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t up = __shfl_up_sync(kUnitAll, incl, d);
        if (lane >= d) incl += up;
      }
      if (i0 + lane < nw) s_key[i0 + lane] = at + incl - n;
      at += __shfl_sync(kUnitAll, incl, 31);
    }
  }
  __syncthreads();

  // pass 2: every unit's rank, and from it its warp and its place in the warp's list
  for (int c0 = 0; c0 < n_items; c0 += kUnitThreads) {
    uint32_t word;
    int parts;
    const int cls = classify(c0 + tid, word, parts);
    const uint32_t peers = __match_any_sync(kUnitAll, cls);
    if (cls >= 0 && lane == __ffs(static_cast<int>(peers)) - 1) s_at[warp][cls] = __popc(peers) * parts;
    __syncthreads();
    if (tid < kUnitClasses) {
      int at = s_base[tid];
#pragma unroll
      for (int w = 0; w < kUnitWarps; ++w) {
        const int n = s_at[w][tid];
        s_at[w][tid] = at;
        at += n;
      }
      s_base[tid] = at;
    }
    __syncthreads();
    if (cls >= 0) {
      int rank = s_at[warp][cls] + __popc(peers & ((1u << lane) - 1u)) * parts;
      for (int t = 0; t < parts; ++t, ++rank) {
        if (rank >= n_units) break;               // (never: the host counts units by the same rule)
        const uint32_t mask = parts == 4 ? (1u << t) : (parts == 2 ? (t ? 12u : 3u) : 15u);
        const uint32_t to = p.dealt ? hand_of[rank] : 0u;
        const int r = p.dealt ? static_cast<int>(to >> kUnitHandBits) : rank / nw;
        const int d = p.dealt ? static_cast<int>(to & ((1u << kUnitHandBits) - 1u)) : rank - r * nw;
        const int k = static_cast<int>(static_cast<long long>(d) * plan.stride_inv % nw);
        const int m = static_cast<int>(s_cnt[d]);
        // the unit's number in its list from the narrowest level on (2-bit blocks are dealt before 4-bit ones)
        const int z = m - 1 - (cls == at2 ? r + static_cast<int>(s_mix[d] >> 16) : (cls == at4 ? r - static_cast<int>(s_mix[d] & 0xffffu) : r));
        const int place = z < (m + 1) / 2 ? 2 * z : 2 * (m - 1 - z) + 1;
        p.units[s_key[d] + (place + m - (k * 5) % m) % m] = word | (mask << 20);
      }
    }
    __syncthreads();
    clear();
    __syncthreads();
  }

  // the warps' descriptors: the head groups of a stream get the same lists and neighbouring warps, so that the second
  // reader of a block finds it in L2; one partial row per (CTA, head group)
  auto describe = [&](int k, int hg, int partial) {
    const int d = static_cast<int>(static_cast<long long>(k) * plan.stride % nw);
    const int begin = static_cast<int>(s_key[d]);
    return WarpDesc{hg, begin, begin + static_cast<int>(s_cnt[d]), partial};
  };
  if (p.cluster > 0) {
    // CTAs of the head group's own, its warps dealt round by round to them
    const int room = p.cluster * kDecodeWarps;
    for (int i = tid; i < room * p.head_groups; i += kUnitThreads) {
      const int g = i / room, at = i - g * room, k = (at % kDecodeWarps) * p.cluster + at / kDecodeWarps;
      p.warps[plan.warp_base + i] = k < nw ? describe(k, s * p.head_groups + g, 0) : WarpDesc{-1, 0, 0, 0};
    }
    return;
  }
  for (int i = tid; i < nw * p.head_groups; i += kUnitThreads) {
    const int g = i / nw, k = i - g * nw, hg = s * p.head_groups + g, w0 = plan.warp_base + g * nw, w = w0 + k;
    p.warps[w] = describe(k, hg, p.parts[hg].begin + w / kDecodeWarps - w0 / kDecodeWarps);
  }
  if (s == static_cast<int>(gridDim.x) - 1)
    for (int w = plan.warp_base + nw * p.head_groups + tid; w < p.n_warps; w += kUnitThreads) p.warps[w] = WarpDesc{-1, 0, 0, 0};
}

}  // namespace

cudaError_t launch_units(UnitsParams p, int n_streams, int max_units, cudaStream_t st) {
  // the ranks' warps in shared memory; a context of more than kUnitsDealt units per stream (2.8 million tokens) is dealt
  // round by round without a look at what a warp has
  constexpr int kUnitsDealt = 45056;
  constexpr size_t kMost = (static_cast<size_t>(3) << kUnitHandBits) * sizeof(uint32_t) + kUnitsDealt * sizeof(uint32_t);      // 224 KB
  p.dealt = max_units <= kUnitsDealt;
  const size_t bytes = (static_cast<size_t>(p.pad) * 3 + (p.dealt ? static_cast<size_t>(max_units) : 0)) * sizeof(uint32_t);
  if (bytes > 40 * 1024) {
    static std::atomic<uint64_t> done{0};
    const cudaError_t e = raise_smem_limit(units_kernel, kMost, done);
    if (e != cudaSuccess) return e;
  }
  units_kernel<<<n_streams, kUnitThreads, bytes, st>>>(p);
  return cudaGetLastError();
}

}  // namespace gkv
