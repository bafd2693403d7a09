"""Host-side check of the persistent solve's launch set-up: two threads with
different batch sizes may interleave in any way, and every launch finds enough
shared memory allowed for its kernel.  A host program built with nvcc from the
launcher's own source, with stand-ins for the runtime calls that keep the
allowance as the driver does and hold one thread at a chosen call.  No GPU is
used."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include <cuda_runtime.h>
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <thread>
static std::mutex mu;
static std::condition_variable cv;
static std::map<const void*, int> allowed;  // dynamic shared memory per kernel, 48 KB unless raised
static int hold_at = -1, calls_of_big = 0;
static bool other_done = false;
static thread_local bool big = false;
// The thread with the large batch waits at its hold_at-th runtime call until
// the other one is through (or for half a second, if that one waits for it).
static void pause() {
  std::unique_lock<std::mutex> lk(mu);
  if (big && calls_of_big++ == hold_at) cv.wait_for(lk, std::chrono::milliseconds(500), [] { return other_done; });
}
template <typename K> static cudaError_t fake_set(K k, cudaFuncAttribute, int n) {
  pause();
  { std::lock_guard<std::mutex> lk(mu); allowed[(const void*)k] = n; }
  pause();
  return cudaSuccess;
}
template <typename K> static cudaError_t fake_fattr(cudaFuncAttributes* a, K) { pause(); *a = {}; a->sharedSizeBytes = 64; return cudaSuccess; }
static cudaError_t fake_get(int* d) { pause(); *d = 0; return cudaSuccess; }
static cudaError_t fake_attr(int* v, cudaDeviceAttr a, int) { pause(); *v = a == cudaDevAttrMultiProcessorCount ? 152 : 232448; return cudaSuccess; }
template <typename K> static cudaError_t fake_occ(int* n, K, int, size_t) { pause(); *n = 1; return cudaSuccess; }
static cudaError_t fake_memset(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
static cudaError_t fake_launch(const void* k, dim3, dim3, void**, size_t smem, cudaStream_t) {
  std::lock_guard<std::mutex> lk(mu);
  const auto it = allowed.find(k);
  // without an opt-in, 48 KB for static and dynamic shared memory together
  return smem <= (size_t)(it == allowed.end() ? 48 * 1024 - 64 : it->second) ? cudaSuccess : cudaErrorInvalidValue;
}
#define cudaFuncSetAttribute fake_set
#define cudaFuncGetAttributes fake_fattr
#define cudaGetDevice fake_get
#define cudaDeviceGetAttribute fake_attr
#define cudaOccupancyMaxActiveBlocksPerMultiprocessor fake_occ
#define cudaMemsetAsync fake_memset
#define cudaLaunchCooperativeKernel fake_launch
#include "paper_1307_7867_gb300/csrc/coarse_fused.cu"
#include "paper_1307_7867_gb300/csrc/persist.cu"
namespace h3d { void count_launch() {} }
using namespace h3d;
static cudaError_t solve(int B) {
  MgPersist<double> p{};
  p.nlev = 5;
  for (int k = 0, N = 31; k < 5; ++k, N = (N - 1) / 2) p.g[k] = make_grid(N);
  p.B = B;
  p.nu1 = 2;
  p.nu2 = 1;
  p.inner = p.max_cycles = 1;
  return launch_mg_persist<double>(2, p, 0);
}
int main(int argc, char** argv) {
  hold_at = atoi(argv[1]);
  const int small = atoi(argv[2]);
  int fails = 0;
  std::thread a([&] { big = true; fails += solve(15000) != cudaSuccess; });
  std::thread b([&] {
    std::this_thread::sleep_for(std::chrono::milliseconds(50));
    const cudaError_t e = solve(small);
    { std::lock_guard<std::mutex> lk(mu); fails += e != cudaSuccess; other_done = true; }
    cv.notify_all();
  });
  a.join();
  b.join();
  // afterwards, with nothing in between, from the same and from new threads
  fails += solve(15000) != cudaSuccess;
  fails += solve(small) != cudaSuccess;
  std::thread([&] { fails += solve(15000) != cudaSuccess; }).join();
  printf("%d\n", fails);
}
'''


def test_batches_of_different_size(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    (tmp_path / "p.cu").write_text(PROGRAM)
    exe = str(tmp_path / "p")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-Xptxas", "-O0", f"-I{ROOT}",
                    f"-I{ROOT}/include", "-o", exe, str(tmp_path / "p.cu")], check=True, capture_output=True)
    for small in (4, 10060, 12000):  # 9 KB, 8 bytes below 48 KB, 56 KB
        for hold_at in range(8):
            out = subprocess.run([exe, str(hold_at), str(small)], capture_output=True, text=True, check=True).stdout
            assert out.strip() == "0", (small, hold_at)
