"""Host-side check of the zero rule of the fixed-point format (csrc/fix.cuh): a
set of values counts as zeros only if it holds nothing else.  A host program
built with nvcc applies the conversions; Python checks them.  No GPU is used."""
import os
import shutil
import struct
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include "paper_1307_7867_gb300/csrc/fix.cuh"
#include <cstdio>
#include <cstring>
using namespace h3d;
// stdin: doubles; stdout per double, taken as a set of its own (a subnormal one
// with a high word of 0 has the key 1): the set's exponent, whether the format
// takes it, and its fixed-point value there
int main() {
  double x;
  while (std::fread(&x, 8, 1, stdin) == 1) {
    unsigned long long b;
    std::memcpy(&b, &x, 8);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    unsigned key = hi & 0x7fffffffu;
    if (key == 0u && lo != 0u) key = 1u;
    const int E = fix_set_exponent(key);
    const long long o[3] = {E, E <= kFixHi && (E >= kFixLo || E == kFixZero), fix_value<6>(hi, lo, E)};
    std::fwrite(o, sizeof(o), 1, stdout);
  }
}
'''


def test_only_zeros_count_as_zeros(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    (tmp_path / "p.cu").write_text(PROGRAM)
    exe = str(tmp_path / "p")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", f"-I{ROOT}", "-o", exe,
                    str(tmp_path / "p.cu")], check=True, capture_output=True)
    x = [0.0, -0.0] + [s * m * 2.0 ** k for k in range(-1074, 1024) for m in (1.0, 1.75) for s in (1, -1)]
    out = subprocess.run([exe], input=struct.pack(f"<{len(x)}d", *x), capture_output=True, check=True).stdout
    got = list(struct.iter_unpack("<3q", out))
    assert len(got) == len(x)
    for a, (E, fits, v) in zip(x, got):
        if a == 0.0:
            assert fits and E == 64 and v == 0, a
        elif fits:  # the value's own unit: nothing is lost
            assert v == int(abs(a) * 2.0 ** -(E - 1023)  * 2.0 ** 58) * (1 if a > 0 else -1), a
        else:  # left to FP64
            assert E != 64 and not 1e-157 < abs(a) < 1e143, a
