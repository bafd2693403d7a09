"""Host-side check that what a kernel needs before its first launch on a device
(the shared-memory opt-in above all) is done on every device that is current at
a launch: host programs built with nvcc from the launchers' own source, with
the runtime calls replaced by stand-ins that count per device.  No GPU is used
(the launches themselves fail, which the programs ignore)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = r'''
#include <cuda_runtime.h>
#include <cstdio>
static int now = 0;          // the current device
static int optins[4] = {0};  // shared-memory opt-ins per device
template <typename K> static cudaError_t fake_set(K, cudaFuncAttribute, int) { optins[now] += 1; return cudaSuccess; }
static cudaError_t fake_get(int* d) { *d = now; return cudaSuccess; }
static cudaError_t fake_attr(int* v, cudaDeviceAttr, int) { *v = 100; return cudaSuccess; }
template <typename K> static cudaError_t fake_occ(int* n, K, int, size_t) { *n = 2; return cudaSuccess; }
#define cudaFuncSetAttribute fake_set
#define cudaGetDevice fake_get
#define cudaDeviceGetAttribute fake_attr
#define cudaOccupancyMaxActiveBlocksPerMultiprocessor fake_occ
'''

FUSED = HEAD + r'''
#include "paper_1307_7867_gb300/csrc/coarse_fused.cu"
namespace h3d { void count_launch() {} }
using namespace h3d;
int main() {
  const int Ns[4] = {15, 7, 3, 1};
  const Coef<double>* cf[4] = {nullptr, nullptr, nullptr, nullptr};
  for (int d : {0, 1, 0, 2, 1}) {
    now = d;
    launch_vcycle_small<double>(2, 4, Ns, cf, 1, nullptr, nullptr, make_grid(15), 2, 1, nullptr, 0);
  }
  printf("%d %d %d %d\n", optins[0], optins[1], optins[2], optins[3]);
}
'''

STENCIL = HEAD + r'''
#include "paper_1307_7867_gb300/csrc/stencil_impl.cuh"
namespace h3d { void count_launch() {} }
using namespace h3d;
int main() {
  for (int d : {0, 1, 0, 2, 1}) {
    now = d;
    OpLap<2, false> op{};
    run_stencil<2, false>(make_grid(127), 1, nullptr, nullptr, op, Shape{}, 0);
  }
  printf("%d %d %d %d\n", optins[0], optins[1], optins[2], optins[3]);
}
'''


@pytest.mark.parametrize("program", [FUSED, STENCIL], ids=["fused levels", "large FP64 stencil"])
def test_every_device_is_set_up_once(tmp_path, program):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    (tmp_path / "p.cu").write_text(program)
    exe = str(tmp_path / "p")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", f"-I{ROOT}",
                    f"-I{ROOT}/include", "-o", exe, str(tmp_path / "p.cu")], check=True, capture_output=True)
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")
    out = subprocess.run([exe], capture_output=True, text=True, env=env, check=True).stdout
    assert out.split() == ["1", "1", "1", "0"]
