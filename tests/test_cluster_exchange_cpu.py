"""The exchange between the CTAs of a cluster at the end of a read, run on host threads from the kernel's own header: the bytes that
each CTA is told to wait for are the bytes that are sent to it, every value has a place of its own, and no CTA leaves while another may still
send to it, also when a wait runs out because one of them is late or its bytes are lost."""
import os
import shutil
import subprocess

import pytest

from paper_2608_23599_b200 import build as _build

HARNESS = r"""
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <set>
#include <thread>
#include <vector>
#include "gkv_exchange.h"
using namespace gkv;

static int geometry() {
  for (int n = 2; n <= kMaxCluster; ++n) {
    const int share = exchange_share(n);
    std::vector<int> bytes(n, 0);
    std::vector<std::set<int>> used(n);
    for (int from = 0; from < n; ++from) {
      for (int c = 0; c < kExchangeChannels; ++c) {
        const int owner = c / share, at = exchange_slot(share, from, c);
        if (owner >= n || at < 0 || at >= kExchangeFloats || !used[owner].insert(at).second) return 1;
        bytes[owner] += 4;
      }
      for (int to = 0; to < n; ++to) bytes[to] += kHeadsPerWarp * 8;
    }
    for (int r = 0; r < n; ++r) {
      if (bytes[r] != exchange_bytes_expected(n, r) || share > kDecodeWarps * 32) return 2;
      // the thread that finishes channel r * share + t reads slot c * share + t of every CTA c
      for (int c = 0; c < n; ++c)
        for (int t = 0; t < share && r * share + t < kExchangeChannels; ++t)
          if (exchange_slot(share, c, r * share + t) != c * share + t) return 3;
    }
  }
  return 8 + kExchangeFloats * 4 + kMaxCluster * kHeadsPerWarp * 8 <= kExchangeBytes ? 0 : 4;
}

struct Cta {
  std::atomic<bool> here{true};
  std::atomic<int> due{0};       // bytes still to come
};
struct Cluster {
  std::vector<Cta> cta;
  std::mutex mu;
  std::condition_variable cv;
  int threads, arrived = 0, gone = 0;
  std::atomic<int> to_the_gone{0}, reports{0}, incomplete{0};
  Cluster(int n, int per) : cta(n), threads(n * per) {}
};
struct HostIo {
  Cluster& k;
  int rank;
  bool poll() const {
    std::this_thread::sleep_for(std::chrono::milliseconds(1));
    return k.cta[rank].due == 0;
  }
  void report() const { ++k.reports; }
  void meet() const {           // returns when every thread that has not left has come here
    std::unique_lock<std::mutex> lock(k.mu);
    ++k.arrived;
    k.cv.notify_all();
    k.cv.wait(lock, [&] { return k.arrived + k.gone >= k.threads; });
  }
};

// n CTAs of two threads; the last CTA is late by far more than the others' polls, or what it sends to CTA 0 is lost
static int run(int n, bool late, bool lost) {
  const int polls = late || lost ? 20 : 20000;
  Cluster k(n, 2);
  for (int r = 0; r < n; ++r) k.cta[r].due = exchange_bytes_expected(n, r);
  std::vector<std::atomic<int>> left(n);
  for (auto& x : left) x = 2;
  std::vector<std::thread> threads;
  for (int r = 0; r < n; ++r)
    for (int half = 0; half < 2; ++half)
      threads.emplace_back([&, r, half] {
        if (late && r == n - 1) std::this_thread::sleep_for(std::chrono::milliseconds(300));
        for (int to = half; to < n; to += 2) {
          if (!k.cta[to].here) ++k.to_the_gone;
          if (lost && r == n - 1 && to == 0) continue;
          k.cta[to].due -= exchange_bytes_expected(n, to) / n;
        }
        if (!await_exchange(HostIo{k, r}, polls)) ++k.incomplete;
        if (--left[r] == 0) k.cta[r].here = false;
        std::lock_guard<std::mutex> lock(k.mu);
        ++k.gone;
        k.cv.notify_all();
      });
  for (auto& t : threads) t.join();
  std::printf("%d CTAs: sent to one that had left %d, reports %d, incomplete %d\n", n, k.to_the_gone.load(), k.reports.load(), k.incomplete.load());
  if (k.to_the_gone) return 1;
  return (k.reports > 0) == (late || lost) && k.incomplete == (lost ? 2 : 0) ? 0 : 2;
}

int main(int argc, char** argv) {
  if (!std::strcmp(argv[1], "geometry")) return geometry();
  int bad = 0;
  for (int n : {2, 3, 8}) bad |= run(n, !std::strcmp(argv[1], "late"), !std::strcmp(argv[1], "lost"));
  return bad;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")) or not shutil.which("g++"):
        pytest.skip("no compiler")
    d = tmp_path_factory.mktemp("exchange")
    src, exe = d / "exchange.cpp", d / "exchange"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", _build.CSRC, "-I", os.path.join(cuda, "include"), str(src), "-o", str(exe), "-lpthread"],
                   check=True)
    return str(exe)


@pytest.mark.parametrize("what", ["geometry", "on time", "late", "lost"])
def test_exchange_between_the_ctas_of_a_cluster(harness, what):
    r = subprocess.run([harness, what], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
