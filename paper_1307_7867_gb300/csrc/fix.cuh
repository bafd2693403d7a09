// fix.cuh -- doubles as 64-bit fixed-point numbers: the conversions that the
// stencils of large grids (stencil_fix.cuh, which describes the format) and
// the quadrature (sdc_kernels.cu) use in place of FP64 operations.
#pragma once
#include <cuda_runtime.h>

namespace h3d {

constexpr int kFixZero = 64;  // exponent of a set of zeros
constexpr int kFixLo = 500, kFixHi = 1500;

// Exponent of a set of values (a tile plane, the nodes of a point) from the
// largest high word (sign cleared) in it, the unit of fix_value.
__host__ __device__ __forceinline__ int fix_exponent(unsigned key) {
  const int e = (int)(key >> 20);
  return e > kFixZero ? e : kFixZero;
}

// As fix_exponent for a key in which 0 stands for a set of nothing but zeros:
// a set with any other value, subnormal ones included, lies above kFixZero
// (and below kFixLo when it is that small).
__host__ __device__ __forceinline__ int fix_set_exponent(unsigned key) {
  const int e = fix_exponent(key);
  return key != 0u && e == kFixZero ? kFixZero + 1 : e;
}

// The double with high word hi and low word lo in a set of exponent E.
template <int G>
__host__ __device__ __forceinline__ long long fix_value(unsigned hi, unsigned lo, int E) {
  const int e = (int)((hi >> 20) & 0x7ffu);
  unsigned long long m =
      (((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << G;
  const int s = E - e;
  m >>= s < 63 ? s : 63;
  return (int)hi < 0 ? -(long long)m : (long long)m;
}

// v as a double, in integer operations: |v| < 2^63 is rounded to nearest
// (halves away from zero); a negative v counts as ~|v|, one unit less, which
// saves the carry of a negation.
__host__ __device__ __forceinline__ unsigned long long fix_double_bits(long long v) {
  const unsigned sign = (unsigned)(v >> 63);
  const unsigned hi = (unsigned)(v >> 32) ^ sign, lo = (unsigned)v ^ sign;
  const unsigned top = hi ? hi : lo;
#ifdef __CUDA_ARCH__
  const int lz = __clz((int)top) + (hi ? 0 : 32);
#else
  const int lz = (top ? __builtin_clz(top) : 32) + (hi ? 0 : 32);
#endif
  // leading bit at 62, half a unit of the 53-bit significand added, then the
  // significand with its leading bit at 52; a carry moves into the exponent
  const unsigned long long m = (((((unsigned long long)hi << 32) | lo) << (lz - 1)) + 0x200ull) >> 10;
  const unsigned e = top ? (unsigned)(1085 - lz) << 20 : 0u;
  return m + (((unsigned long long)(e | (sign & 0x80000000u))) << 32);
}

__device__ __forceinline__ double fix_double(long long v) {
  return __longlong_as_double((long long)fix_double_bits(v));
}

// coef * 2^ke by its exponent field (zero stays; the caller has checked the range).
__device__ __forceinline__ double fix_scale(double coef, int ke) {
  const int hi = __double2hiint(coef);
  return __hiloint2double((hi & 0x7fffffff) == 0 ? hi : hi + ke * (1 << 20), __double2loint(coef));
}
__device__ __forceinline__ bool fix_coef_ok(double coef) {
  const int e = (__double2hiint(coef) >> 20) & 0x7ff;
  return coef == 0.0 || (e >= 823 && e <= 1223);
}

// The quadrature's numbers: a value v of kFixBits bits as two centred digits,
// v = 2^31 h + l, and a sum of products with coefficients (x, y) of two such
// digits in three parts, 2^62 hi + 2^31 mid + 2^32 lo.  The coefficients'
// magnitudes add up to 2^kFixBits at most; value() has full scale 2^62.
constexpr int kFixBits = 61;
struct FixTerm {
  int h, l;
};
__host__ __device__ __forceinline__ FixTerm fix_digits(long long v) {
  const int h = (int)((v + (1ll << 30)) >> 31);
  return FixTerm{h, (int)((unsigned)v - ((unsigned)h << 31))};
}
struct FixSum {
  long long hi = 0, mid = 0;
  int lo = 0;  // six terms below 2^28
  __host__ __device__ void add(FixTerm f, int2 c) {
    hi += (long long)f.h * c.x;
    mid += (long long)f.h * c.y;
    mid += (long long)f.l * c.x;
    lo += (int)(((long long)f.l * c.y) >> 32);
  }
  __host__ __device__ long long value() const {
    return (hi << (124 - 2 * kFixBits)) + ((mid + 2ll * lo) >> (2 * kFixBits - 93));
  }
};

}  // namespace h3d
