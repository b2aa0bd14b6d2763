// What the CTAs of a cluster send one another at the end of a read: every CTA has a row of accumulators and of pairs
// (running maximum, sum), and finishes a share of the channels over all rows.  A value goes straight to the CTA that finishes its channel,
// whose mbarrier counts the bytes.  Sizes, places and the wait for the bytes are here without the instructions, so that they can be run on a
// host as well.
#pragma once
#include "gkv_internal.h"

namespace gkv {

constexpr int kExchangeChannels = kHeadsPerWarp * kD;                    // accumulators of a row
constexpr int kExchangeFloats = kExchangeChannels + kMaxCluster;         // [CTA][share]: shares are rounded up
constexpr int kExchangePairs = kMaxCluster * kHeadsPerWarp;              // [CTA][head]
constexpr int kExchangeBytes = 8 + kExchangeFloats * 4 + kExchangePairs * 8;      // behind the mbarrier

// channels that a CTA finishes (the last one may have fewer)
__host__ __device__ constexpr int exchange_share(int cluster) { return (kExchangeChannels + cluster - 1) / cluster; }
// where the owner of a channel, channel / share, keeps the value that CTA `from` sends
__host__ __device__ constexpr int exchange_slot(int share, int from, int channel) { return from * share + channel % share; }
// bytes that reach CTA `rank`: from every CTA, itself included, its channels and the pairs of all heads
__host__ __device__ constexpr int exchange_bytes_expected(int cluster, int rank) {
  const int share = exchange_share(cluster), rest = kExchangeChannels - rank * share;
  return cluster * ((share < rest ? share : rest) * 4 + kHeadsPerWarp * 8);
}

// A thread's wait for the bytes of all CTAs.  A CTA must not leave while another may still send to it: its shared memory is gone
// then.  When the polls run out (a peer is waiting for a copy that does not come, for as many polls of its own) it reports that and stays until every
// other thread of the cluster has come here too or has left, which none does before it has sent: all waits in front are bounded, so this one ends.
// What was sent then is on its way, and the bytes are polled for once more.  False: some never came.
// (Out of line behind the first poll, which sleeps on the mbarrier and as a rule suffices: inline the unused code made a call over 1000 tokens 6.45 -> 6.49 us.)
template <class Io>
__host__ __device__ __attribute__((noinline)) bool await_late_exchange(Io io, int polls) {
  for (int i = 0; i < polls; ++i)
    if (io.poll()) return true;
  io.report();
  io.meet();
  for (int i = 0; i < polls; ++i)
    if (io.poll()) return true;
  return false;
}
template <class Io>
__host__ __device__ inline bool await_exchange(const Io& io, int polls) {
  return io.poll() || await_late_exchange(io, polls);
}

}  // namespace gkv
