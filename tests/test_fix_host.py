"""Host-side check of the fixed-point conversions of the FP64 stencils
(fix_value, fix_exponent and fix_double_bits in csrc/stencil_fix.cuh, all
__host__ __device__): a small host program built with nvcc applies them, and
Python integers check them exactly.  No GPU is used."""
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include "paper_1307_7867_gb300/csrc/stencil_impl.cuh"
#include <cstdio>
#include <cstring>
namespace h3d { void count_launch() {} }
using namespace h3d;
// stdin: records of a double and an exponent; stdout per record: the exponent
// of the double's own plane, fix_value<6> and <5> at the given exponent, and
// fix_double_bits of the first
int main() {
  struct Rec { double x; long long E; } r;
  while (std::fread(&r, sizeof(r), 1, stdin) == 1) {
    unsigned long long b;
    std::memcpy(&b, &r.x, 8);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    long long o[4];
    o[0] = fix_exponent(hi & 0x7fffffffu);
    o[1] = fix_value<6>(hi, lo, (int)r.E);
    o[2] = fix_value<5>(hi, lo, (int)r.E);
    o[3] = (long long)fix_double_bits(o[1]);
    std::fwrite(o, sizeof(o), 1, stdout);
  }
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("fix")
    (d / "p.cu").write_text(PROGRAM)
    exe = str(d / "p")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", f"-I{ROOT}",
                    f"-I{ROOT}/include", "-o", exe, str(d / "p.cu")], check=True, capture_output=True)
    return exe


def test_conversions_are_exact(program):
    rng = np.random.default_rng(7)
    x = np.concatenate([rng.standard_normal(2000), rng.standard_normal(500) * 2.0 ** rng.integers(-80, 1, 500),
                        [0.0, -0.0, 1.0, -1.0, np.nextafter(2.0, 0), -np.nextafter(2.0, 0), 2.0 ** -1000, 5e-324]])
    E = np.full(x.size, 1023 + 3, dtype=np.int64)
    E[: 1000] = 1023 + 2 + rng.integers(0, 70, 1000)
    rec = b"".join(struct.pack("<dq", a, e) for a, e in zip(x, E))
    out = subprocess.run([program], input=rec, capture_output=True, check=True).stdout
    got = np.frombuffer(out, dtype=np.int64).reshape(-1, 4)
    for a, e, (own, v6, v5, bits) in zip(x.tolist(), E.tolist(), got.tolist()):
        raw = struct.unpack("<Q", struct.pack("<d", a))[0]
        ex = raw >> 52 & 0x7ff
        assert own == max(ex, 64)
        sig = (raw & (1 << 52) - 1) | 1 << 52
        for g, v in ((6, v6), (5, v5)):
            want = (sig << g) >> min(e - ex, 63)
            assert v == (-want if raw >> 63 else want), (a, e, g)
        # back to a double: half a unit of its 53 bits, and one unit of the
        # integer for negative values
        d = struct.unpack("<d", struct.pack("<Q", bits & (1 << 64) - 1))[0]
        assert d == int(d)
        assert abs(int(d) - v6) <= max(abs(v6) >> 53, 0) + (1 if v6 < 0 else 0) + (abs(v6) >> 52 > 0), (a, d, v6)
        assert (d == 0.0) == (v6 in (0, -1))
