"""Host-side check of the quadrature's sums of products (FixSum in csrc/fix.cuh)
against Python integers, with digits up to the ends of their range, and of the
rounding of fix_double_bits on numbers of up to 63 bits.  No GPU is used."""
import os
import random
import shutil
import struct
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TERMS = 6

PROGRAM = r'''
#include "paper_1307_7867_gb300/csrc/fix.cuh"
#include <cstdio>
#include <cstring>
using namespace h3d;
// stdin: records of six (h, l, x, y); stdout: kFixBits, then value() of their
// sums.  With an argument: records of one 64-bit integer; stdout:
// fix_double_bits.
int main(int argc, char**) {
  if (argc > 1) {
    long long v;
    while (std::fread(&v, 8, 1, stdin) == 1) {
      const unsigned long long b = fix_double_bits(v);
      std::fwrite(&b, 8, 1, stdout);
    }
    return 0;
  }
  const long long bits = kFixBits;
  std::fwrite(&bits, 8, 1, stdout);
  int r[6][4];
  while (std::fread(r, sizeof(r), 1, stdin) == 1) {
    FixSum s;
    for (auto& t : r) s.add(FixTerm{t[0], t[1]}, make_int2(t[2], t[3]));
    const long long v = s.value();
    std::fwrite(&v, 8, 1, stdout);
  }
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("fixsum")
    (d / "p.cu").write_text(PROGRAM)
    exe = str(d / "p")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", f"-I{ROOT}", "-o", exe,
                    str(d / "p.cu")], check=True, capture_output=True)
    return exe


def test_sums_of_products(program):
    """Each of the three parts is cut down once or per term: the value is the
    exact sum in its unit but for the lost fractions, below 1 + 2^-10 in all.
    Values are up to 2^bits, the coefficients' magnitudes add up to 2^bits."""
    rng = random.Random(3)
    bits = struct.unpack("<q", subprocess.run([program], input=b"", capture_output=True, check=True).stdout)[0]
    top, end = 1 << bits - 31, 1 << 30
    rows = []
    for n in range(4000):
        row = []
        for _ in range(TERMS):
            extreme = n % 2 == 0
            h, x = (rng.choice((-1, 1)) * (top if extreme else rng.randrange(top)) for _ in range(2))
            lo, y = (rng.choice((-end, end)) if extreme else rng.randrange(-end, end) for _ in range(2))
            row.append((h, lo, x // TERMS, y))
        rows.append(row)
    rows.append([(top, end, top // TERMS, end)] * TERMS)
    rows.append([(-top, -end, top // TERMS, end)] * TERMS)
    rows.append([(0, end, 0, end)] * TERMS)
    data = b"".join(struct.pack("<4i", *t) for row in rows for t in row)
    out = subprocess.run([program], input=data, capture_output=True, check=True).stdout
    got = [v for v, in struct.iter_unpack("<q", out)][1:]
    assert len(got) == len(rows)
    shift = 2 * bits - 62  # the unit: full scale is 2^62
    for row, v in zip(rows, got):
        exact = sum(((h << 31) + lo) * ((x << 31) + y) for h, lo, x, y in row)
        low = (exact >> shift) - v
        assert 0 <= low <= 1, (row, v, exact >> shift)


def test_rounding_to_a_double(program):
    """Positive numbers round to nearest, halves away from zero; a negative one
    counts as ~|v|, one unit less."""
    rng = random.Random(4)
    vals = [0, -1, 1, -2, (1 << 63) - 1, -(1 << 63) + 1, -(1 << 63)]
    for b in range(1, 63):
        for _ in range(60):
            vals.append(rng.getrandbits(b) | 1 << b - 1)
        if b > 53:  # ties, just below and above, and carries into the exponent
            half = 1 << b - 54
            for sig in (1 << 52, (1 << 53) - 1, rng.getrandbits(52) | 1 << 52):
                vals += [(sig << b - 53) + half + d for d in (-1, 0, 1)]
    vals += [-v for v in vals if 0 < v]
    vals = [v for v in vals if -(1 << 63) <= v < 1 << 63]
    out = subprocess.run([program, "double"], input=struct.pack(f"<{len(vals)}q", *vals), capture_output=True,
                         check=True).stdout
    got = [d for d, in struct.iter_unpack("<d", out)]
    assert len(got) == len(vals)
    for v, d in zip(vals, got):
        mag = v if v >= 0 else ~v
        drop = max(mag.bit_length() - 53, 0)
        want = ((mag + (1 << drop - 1 if drop else 0)) >> drop) << drop
        assert d == (want if v >= 0 else -want), (v, d, want)
