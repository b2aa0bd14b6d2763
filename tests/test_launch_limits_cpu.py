"""The shared-memory limit of a kernel is the kernel's on a device, not a launch's and not the process's.  Two host threads that make work lists (level plans)
of different sizes at once must both be able to launch, and every kernel on every device: here with the launch functions
linked against a small fake of the CUDA runtime that applies the threads' limits in the worst order, larger one first, and
refuses a launch above the limit as the runtime does."""
import os
import shutil
import subprocess

import pytest

from paper_2608_23599_b200 import build as _build

FAKE = r"""
#include <condition_variable>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <thread>
#include <vector>
#include "gkv_internal.h"
#include "gkv_mla.h"

static std::mutex mu;
static std::condition_variable cv;
static std::map<std::pair<int, const void*>, size_t> limit;      // by device and kernel
static thread_local int device = 0;
static thread_local cudaError_t last = cudaSuccess;
static int expected = 0;                                         // threads that meet in cudaFuncSetAttribute
static std::vector<int> asked;
static bool refuse_query = false;

static size_t& limit_of(const void* f) {
  auto it = limit.find({device, f});
  if (it == limit.end()) it = limit.insert({{device, f}, 48 * 1024}).first;
  return it->second;
}

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int value) {
  std::unique_lock<std::mutex> lock(mu);
  if (value > 232448) return cudaErrorInvalidValue;              // what an SM has for one block
  asked.push_back(value);
  cv.notify_all();
  if (expected > 1) cv.wait_for(lock, std::chrono::seconds(2), [] { return static_cast<int>(asked.size()) >= expected; });
  if (expected > 1)
    for (int v : asked) value = v < value ? v : value;           // whoever asked for least comes last
  limit_of(f) = static_cast<size_t>(value);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t bytes, cudaStream_t) {
  std::lock_guard<std::mutex> lock(mu);
  last = bytes > limit_of(f) ? cudaErrorInvalidValue : cudaSuccess;
  return last;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return cudaLaunchKernel(f, c->gridDim, c->blockDim, nullptr, c->dynamicSmemBytes, c->stream);
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) {
  *n = 18;
  if (refuse_query) return last = cudaErrorMemoryAllocation;
  return c->dynamicSmemBytes > limit_of(f) ? cudaErrorInvalidValue : cudaSuccess;
}
static thread_local struct { dim3 g, b; size_t s; cudaStream_t st; } pushed;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t st) { pushed = {g, b, s, st}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = pushed.g; *b = pushed.b; *s = pushed.s; std::memcpy(st, &pushed.st, sizeof(pushed.st));
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
}

static cudaError_t lists(int units) {
  gkv::UnitsParams p{};
  p.pad = 4096;
  return gkv::launch_units(p, 1, units, nullptr);
}
static cudaError_t plans(int blocks) {
  gkv::RdPlanParams p{};
  p.n = blocks;
  gkv::rd_plan_smem_bytes(blocks, &p.pad);
  return gkv::launch_rd_plan(p, 1, nullptr);
}

// every other kernel with a limit of its own, on two devices in turn
static int every_kernel() {
  using namespace gkv;
  int bad = 0, at = 0;
  auto check = [&](cudaError_t e) {
    bad += e != cudaSuccess;
    std::printf("device %d, kernel %d: %d\n", device, at++, e);
  };
  static int32_t some;
  for (int d = 0; d < 4; ++d) {
    device = d & 1;
    at = 0;
    DecodeParams read{};
    check(launch_decode(read, 1, true, nullptr));
    read.mass_raw = reinterpret_cast<float2*>(&some);
    check(launch_decode(read, 1, false, nullptr));
    read.mass_raw = nullptr;
    read.page_idx = &some;
    check(launch_decode(read, 1, true, nullptr));
    check(decode_max_clusters(2) == 18 ? cudaSuccess : cudaErrorInvalidValue);
    EncodeParams enc{};
    enc.n_jobs = 1;
    check(launch_encode(enc, nullptr));
    check(launch_ingest(enc, nullptr));
    MlaEncodeParams lat{};
    lat.n_jobs = 1;
    check(launch_mla_encode(lat, nullptr));
    check(launch_mla_ingest(lat, nullptr));
    check(launch_mla_decode(MlaDecodeParams{}, 1, nullptr, 1, nullptr, nullptr, nullptr));
    for (int group = 1; group <= kMaxHeadsPerKv; ++group)
      for (int streams : {1, 1024}) check(launch_quest_scores(nullptr, 4096, 4096, nullptr, streams, 1, group, 0, nullptr, 4096, nullptr));
  }
  return bad != 0;
}

int main(int argc, char** argv) {
  if (argc > 1 && !std::strcmp(argv[1], "kernels")) return every_kernel();
  if (argc > 1 && !std::strcmp(argv[1], "clusters")) {
    refuse_query = true;
    const int none = gkv::decode_max_clusters(4);
    const bool clean = cudaGetLastError() == cudaSuccess;      // the caller does not find the query's error
    refuse_query = false;
    const int some = gkv::decode_max_clusters(4);
    std::printf("%d %d %d\n", none, clean, some);
    return none == 0 && clean && some == 18 ? 0 : 1;
  }
  cudaError_t (*launch)(int) = argc > 1 && !std::strcmp(argv[1], "plans") ? plans : lists;
  const bool is_plans = launch == plans;
  const int small = is_plans ? 1700 : 2300, large = is_plans ? 4095 : 45056;
  int bad = 0;
  // two threads at once
  expected = 2;
  cudaError_t r[2];
  std::thread a([&] { r[0] = launch(large); }), b([&] { r[1] = launch(small); });
  a.join();
  b.join();
  for (cudaError_t e : r) bad += e != cudaSuccess;
  std::printf("two threads: %d %d\n", r[0], r[1]);
  // one after the other, on this device and on one that was not asked before
  expected = 0;
  for (int d = 0; d < 2; ++d) {
    device = d;
    asked.clear();
    for (int n : {large, small, large, small}) {
      const cudaError_t e = launch(n);
      bad += e != cudaSuccess;
      std::printf("device %d, size %d: %d\n", d, n, e);
    }
  }
  return bad != 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if not os.path.exists(os.path.join(cuda, "bin", "nvcc")) or not shutil.which("g++"):
        pytest.skip("no compiler")
    d = tmp_path_factory.mktemp("limits")
    src, exe = d / "fake.cpp", d / "fake"
    src.write_text(FAKE)
    names = [s[:-3] for s in _build.SOURCES if s != "gkv_api.cu"]
    objs = [str(d / f"{name}.o") for name in names]
    made = [subprocess.Popen([os.path.join(cuda, "bin", "nvcc"), *_build.NVCC_FLAGS, "-c", os.path.join(_build.CSRC, f"{name}.cu"), "-o", obj],
                             stdout=subprocess.DEVNULL, stderr=subprocess.DEVNULL) for name, obj in zip(names, objs)]
    assert [p.wait(600) for p in made] == [0] * len(made)
    subprocess.run(["g++", "-std=c++17", "-I", _build.CSRC, "-I", os.path.join(cuda, "include"), str(src), *objs, "-o", str(exe), "-lpthread"],
                   check=True)
    return str(exe)


@pytest.mark.parametrize("what", ["lists", "plans"])
def test_a_launch_is_not_refused_for_another_threads_smaller_one(harness, what):
    r = subprocess.run([harness, what], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_every_kernel_launches_on_every_device(harness):
    r = subprocess.run([harness, "kernels"], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_a_refused_query_of_cluster_room_is_asked_again(harness):
    r = subprocess.run([harness, "clusters"], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
