// sdc_kernels.cu -- spectral-quadrature and FAS kernels (Sec. 1.1), point by
// point; the quadrature sums in fixed point, everything else FP64.
#include <type_traits>

#include "fix.cuh"
#include "kernels.cuh"

namespace h3d {
namespace {

__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

__device__ __forceinline__ void warp_max_to(unsigned long long v, unsigned long long* dst) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  if ((threadIdx.x & 31) == 0 && v != 0ull) atomicMax(dst, v);
}

inline dim3 point_grid(const Grid& g, int B) {
  return dim3((g.N + 31) / 32, (g.N + 7) / 8, g.N * B);
}

// Planes per thread of the quadrature kernels: as many as leave several
// blocks for every SM.
inline int points_per_thread(int N) { return N >= 255 ? 8 : N >= 127 ? 4 : 1; }

// The F values of a point (node stride fs) and its forcing field in digits at
// their largest exponent E; an even number of terms.
template <int M>
struct FixPoint {
  static constexpr int C = (M + 2) / 2 * 2;
  FixTerm f[C];
  int E;
  bool low;  // every F is below 1/16 of the largest number
  __device__ void load(const double* Fb, long long fs, double psi) {
    double x[C];
    unsigned key = 0u, keyF = 0u;
#pragma unroll
    for (int q = 0; q < C; ++q) {
      x[q] = q < M ? Fb[q * fs] : q == M ? psi : 0.0;
      key = max(key, (unsigned)__double2hiint(x[q]) & 0x7fffffffu);
      if (q == M - 1) keyF = key;
    }
    if (key == 0u) {  // zeros, or subnormal values whose high words are 0
#pragma unroll
      for (int q = 0; q < C; ++q) key |= __double2loint(x[q]) != 0;
    }
    E = fix_set_exponent(key);
    low = (int)(keyF >> 20) < E - 4;
#pragma unroll
    for (int q = 0; q < C; ++q)
      f[q] = q <= M ? fix_digits(fix_value<kFixBits - 53>(__double2hiint(x[q]), __double2loint(x[q]), E))
                       : FixTerm{0, 0};
  }
  __device__ bool fits() const { return E <= kFixHi && (E >= kFixLo || E == kFixZero); }
  // the sum of row c (shared memory, 16-byte aligned) as a double
  __device__ double row(const int2* c, int fe) const {
    FixSum s;
#pragma unroll
    for (int q = 0; q < C; q += 2) {
      const int4 v = *reinterpret_cast<const int4*>(c + q);
      s.add(f[q], make_int2(v.x, v.y));
      if (q + 1 <= M) s.add(f[q + 1], make_int2(v.z, v.w));
    }
    return fix_scale(fix_double(s.value()), E - 1084 + fe);
  }
};

// The FP64 form of one point (also the reading of the sums: J_m, I_m, r_m).
template <int M>
__device__ __noinline__ unsigned long long integrals_plain(const ItemSDC& it, const double* Ub, const double* Fb,
                                                           const double* tb, double* Ib, long long fs, double phi,
                                                           bool res) {
  const double u0 = Ub[0];
  double cum = 0.0;
  unsigned long long mx = 0ull;
  for (int m = 0; m < M - 1; ++m) {
    double J = it.gS[m] * phi;
    for (int q = 0; q < M; ++q) J = fma(it.dtS[m][q], Fb[q * fs], J);
    if (tb) J += tb[m * fs];
    if (Ib) {
      double Im = fma(-it.dtm[m], Fb[(m + 1) * fs], J);
      if (m == 0) Im += u0;
      Ib[m * fs] = Im;
    }
    if (res) {
      cum += J;
      const unsigned long long bits = abs_bits((u0 + cum) - Ub[(m + 1) * fs]);
      mx = bits > mx ? bits : mx;
    }
  }
  return mx;
}

// Quadrature integrals of one sweep and (optionally) the collocation residual
// of the current iterate.  I == nullptr: residual only.
//
// With FP64 multiply-adds a point costs 43 FP64 operations (M = 5), 1.40 ms at
// 255^3 on a pipe of 2 per clock and SM, five times the memory time of its 10
// to 14 fields.  The sums run in fixed point instead: the F values of a point
// (and Phi, scaled by a power of two to the size of the forcing) are brought to
// the largest exponent among them, kFixBits bits of each multiplied with copies
// of the matrices of as many bits (ItemSDC::fI, fQ) as two centred 31-bit
// digits, and each sum becomes a double once.  Points whose exponents the
// format does not take go through FP64 (plain), and where a coefficient of the
// forcing is tiny (fix_coefficients) those whose F is small against it.  A
// thread takes a run of kz points along z, which shares the loads of the digits
// and phi_x phi_y; the rows of the two matrices are a loop, which keeps a
// thread at 64 registers (224 and twice the time without).  Error of a sum
// against exact arithmetic: 0.3-1.0 of the FP64 sums' (rms and largest, M = 2
// to 5, node values alike, spread over 2^40, one much larger than the others,
// all far below the forcing).  Measured, residual only: 1.25 -> 0.66 ms at
// 255^3 with M = 5, 0.17 -> 0.10 ms at 127^3, 0.56 -> 0.40 ms at 255^3 with M =
// 3; the smallest grids take a launch either way.
template <int M, bool TAU, bool RES>
__global__ void __launch_bounds__(256, 4) k_integrals(Grid g, const double* __restrict__ U,
                                                      const double* __restrict__ F,
                                                      const double* __restrict__ tauS,
                                                      double* __restrict__ I,
                                                      const ItemSDC* __restrict__ items,
                                                      const double* __restrict__ phi1d,
                                                      unsigned long long* res_bits, const int* active,
                                                      int kz) {
  constexpr int C = FixPoint<M>::C;
  __shared__ __align__(16) int2 cI[M - 1][C], cQ[M - 1][C];
  __shared__ int eI[M - 1], eQ[M - 1];
  const int nkz = (g.N + kz - 1) / kz;
  const int b = blockIdx.z / nkz;
  if (active && !active[b]) return;  // uniform over the block
  const ItemSDC& it = items[b];
  const int tid = threadIdx.y * 32 + threadIdx.x;
  if (tid < (M - 1) * C) {
    const int m = tid / C, j = tid - m * C;
    cI[m][j] = j <= M ? it.fI[m][j] : make_int2(0, 0);
    cQ[m][j] = j <= M ? it.fQ[m][j] : make_int2(0, 0);
    if (j == 0) {
      eI[m] = it.feI[m];
      eQ[m] = it.feQ[m];
    }
  }
  const int fp = it.fp;
  const bool forced = it.forced != 0, fok = it.fok != 0, weak = it.weak != 0;
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k0 = (blockIdx.z - b * nkz) * kz, k1 = min(g.N, k0 + kz);
  unsigned long long mx = 0ull;
  if (i < g.N && j < g.N) {
    const long long fs = g.fs;
    const double phixy = phi1d[i] * phi1d[j];
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
      const long long idx = (long long)k * g.plane + (long long)j * g.px + i;
      const double* Ub = U + (long long)b * M * fs + idx;
      const double* Fb = F + (long long)b * M * fs + idx;
      const double* tb = TAU ? tauS + (long long)b * (M - 1) * fs + idx : nullptr;
      double* Ib = I ? I + (long long)b * (M - 1) * fs + idx : nullptr;
      const double phi = phixy * phi1d[k];
      FixPoint<M> p;
      p.load(Fb, fs, forced ? fix_scale(phi, fp) : 0.0);
      if (!fok || !p.fits() || (weak && p.low)) {
        const unsigned long long bits = integrals_plain<M>(it, Ub, Fb, tb, Ib, fs, phi, RES);
        mx = bits > mx ? bits : mx;
        continue;
      }
      const double u0 = Ub[0];
      double ctau = 0.0;
      // row m; the one that adds U_0 stands apart (an FP64 addition under a
      // condition runs for every row)
      auto substep = [&](int m, auto first) {
        const double tau = TAU ? tb[m * fs] : 0.0;
        if (I) {
          double Im = p.row(cI[m], eI[m]);
          if (TAU) Im += tau;
          if (decltype(first)::value) Im += u0;
          Ib[m * fs] = Im;
        }
        if (RES) {
          double rv = (u0 - Ub[(m + 1) * fs]) + p.row(cQ[m], eQ[m]);
          if (TAU) rv += ctau += tau;
          const unsigned long long bits = abs_bits(rv);
          mx = bits > mx ? bits : mx;
        }
      };
      substep(0, std::true_type{});
#pragma unroll 1
      for (int m = 1; m < M - 1; ++m) substep(m, std::false_type{});
    }
  }
  if (RES) warp_max_to(mx, res_bits + b);
}

template <int M>
void start_integrals(dim3 grd, dim3 blk, cudaStream_t st, const Grid& g, const double* U, const double* F,
                     const double* tauS, double* I, const ItemSDC* items, const double* phi1d,
                     unsigned long long* res_bits, const int* active, int kz) {
  auto k = tauS ? (res_bits ? k_integrals<M, true, true> : k_integrals<M, true, false>)
                : (res_bits ? k_integrals<M, false, true> : k_integrals<M, false, false>);
  k<<<grd, blk, 0, st>>>(g, U, F, tauS, I, items, phi1d, res_bits, active, kz);
}

// Coarse point (I, J, K) (0-based) sits on fine point (2I+1, 2J+1, 2K+1), or on
// the same point when the two grids are equal.
// X (compact fine level): qF_m = R(U_jm - U_0 + X_{m-1}) with X_{m-1} = W^{-1} r
// of coarse node m >= 1 (field m-1 of each item at item stride xs), qF_0 = 0.
template <int MF, int MG>
__global__ void k_fas_inject(Grid gf, Grid gg, int same, const double* __restrict__ UF,
                             const double* __restrict__ FF, double* __restrict__ UG,
                             double* __restrict__ UGr, double* __restrict__ qF,
                             const ItemSDC* __restrict__ itF, const FasMap* __restrict__ map,
                             const double* __restrict__ phif1d, const double* __restrict__ X,
                             long long xs) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int b = blockIdx.z / gg.N;
  const int k = blockIdx.z - b * gg.N;
  if (i >= gg.N || j >= gg.N) return;
  const int fi = same ? i : 2 * i + 1, fj = same ? j : 2 * j + 1, fk = same ? k : 2 * k + 1;
  const long long fidx = (long long)fk * gf.plane + (long long)fj * gf.px + fi;
  const long long gidx = (long long)k * gg.plane + (long long)j * gg.px + i;
  const double* UFb = UF + (long long)b * MF * gf.fs + fidx;
  const double* FFb = FF + (long long)b * MF * gf.fs + fidx;
  const ItemSDC& it = itF[b];
  double Fq[MF];
#pragma unroll
  for (int q = 0; q < MF; ++q) Fq[q] = FFb[q * gf.fs];
  const double phi = phif1d[fi] * phif1d[fj] * phif1d[fk];
#pragma unroll
  for (int m = 0; m < MG; ++m) {
    const int jm = map->jm[m];
    const double v = UFb[jm * gf.fs];
    const long long o = ((long long)b * MG + m) * gg.fs + gidx;
    UG[o] = v;
    UGr[o] = v;
    if (X) {
      qF[o] = m == 0 ? 0.0 : (v - UFb[0]) + X[(long long)b * xs + (long long)(m - 1) * gf.fs + fidx];
      continue;
    }
    double q = it.gQ[jm] * phi;
#pragma unroll
    for (int p = 0; p < MF; ++p) q = fma(it.dtQ[jm][p], Fq[p], q);
    qF[o] = q;
  }
}

// Compact fine level, coarse node m (fine node jm): the weighted residual
// r = W U_0 + dt sum_p Q[jm][p] (F_p + W f_p) - W U_jm on the fine grid, into
// R (one field per item) and into X (the W-solve's start value, item stride
// xs); max |r| per item into res_bits.
template <int MF>
__global__ void __launch_bounds__(256, 4) k_fas_wresid(Grid gf, int jm, const double* __restrict__ WU,
                                                       const double* __restrict__ FF,
                                                       const ItemSDC* __restrict__ itF,
                                                       const double* __restrict__ phif1d,
                                                       double* __restrict__ R, double* __restrict__ X,
                                                       long long xs, unsigned long long* res_bits, int kz) {
  constexpr int C = FixPoint<MF>::C;
  __shared__ __align__(16) int2 cQ[C];  // row jm of dt Q in digits, as k_integrals
  const int nkz = (gf.N + kz - 1) / kz;
  const int b = blockIdx.z / nkz;
  const ItemSDC& it = itF[b];
  const int tid = threadIdx.y * 32 + threadIdx.x;
  if (tid < C) cQ[tid] = tid <= MF ? it.fQ[jm - 1][tid] : make_int2(0, 0);
  const int fe = it.feQ[jm - 1], fp = it.fp;
  const bool fok = it.fok != 0, forced = it.forced != 0, weak = it.weak != 0;
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k0 = (blockIdx.z - b * nkz) * kz, k1 = min(gf.N, k0 + kz);
  unsigned long long mx = 0ull;
  if (i < gf.N && j < gf.N) {
    const double phixy = phif1d[i] * phif1d[j];
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
      const long long idx = (long long)k * gf.plane + (long long)j * gf.px + i;
      const double* Wb = WU + (long long)b * MF * gf.fs + idx;
      const double* Fb = FF + (long long)b * MF * gf.fs + idx;
      const double phi = phixy * phif1d[k];
      const double w0 = Wb[0], wj = Wb[jm * gf.fs];
      FixPoint<MF> p;
      p.load(Fb, gf.fs, forced ? fix_scale(phi, fp) : 0.0);
      double q;
      if (fok && p.fits() && !(weak && p.low)) {
        q = p.row(cQ, fe);
      } else {
        q = it.gQ[jm] * phi;
#pragma unroll 1
        for (int t = 0; t < MF; ++t) q = fma(it.dtQ[jm][t], Fb[t * gf.fs], q);
      }
      const double r = (w0 + q) - wj;
      R[(long long)b * gf.fs + idx] = r;
      X[(long long)b * xs + idx] = r;
      const unsigned long long bits = abs_bits(r);
      mx = bits > mx ? bits : mx;
    }
  }
  warp_max_to(mx, res_bits + b);
}

template <int MG>
__global__ void k_fas_tau(Grid gg, const double* __restrict__ qF, const double* __restrict__ FG,
                          double* __restrict__ tauS, const ItemSDC* __restrict__ itG,
                          const double* __restrict__ phig1d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int b = blockIdx.z / gg.N;
  const int k = blockIdx.z - b * gg.N;
  if (i >= gg.N || j >= gg.N) return;
  const long long gidx = (long long)k * gg.plane + (long long)j * gg.px + i;
  const ItemSDC& it = itG[b];
  double Fg[MG];
#pragma unroll
  for (int q = 0; q < MG; ++q) Fg[q] = FG[((long long)b * MG + q) * gg.fs + gidx];
  const double phi = phig1d[i] * phig1d[j] * phig1d[k];
  double prev = 0.0;  // tauQ_0 = 0 (Q's first row is zero)
#pragma unroll
  for (int m = 1; m < MG; ++m) {
    double c = it.gQ[m] * phi;
#pragma unroll
    for (int q = 0; q < MG; ++q) c = fma(it.dtQ[m][q], Fg[q], c);
    const double tq = qF[((long long)b * MG + m) * gg.fs + gidx] - c;
    tauS[((long long)b * (MG - 1) + (m - 1)) * gg.fs + gidx] = tq - prev;
    prev = tq;
  }
}

template <int MF, int MG>
__global__ void k_fas_delta(Grid gg, const double* __restrict__ UG, const double* __restrict__ UGr,
                            double* __restrict__ D, const FasMap* __restrict__ map) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int b = blockIdx.z / gg.N;
  const int k = blockIdx.z - b * gg.N;
  if (i >= gg.N || j >= gg.N) return;
  const long long gidx = (long long)k * gg.plane + (long long)j * gg.px + i;
  double dl[MG];
#pragma unroll
  for (int m = 0; m < MG; ++m) {
    const long long o = ((long long)b * MG + m) * gg.fs + gidx;
    dl[m] = UG[o] - UGr[o];
  }
#pragma unroll
  for (int q = 0; q < MF; ++q) {
    double s = 0.0;
#pragma unroll
    for (int m = 0; m < MG; ++m) s += map->L[q][m] * dl[m];
    D[((long long)b * MF + q) * gg.fs + gidx] = s;
  }
}

}  // namespace

cudaError_t launch_integrals(int M, const Grid& g, int B, const double* U, const double* F,
                             const double* tauS, double* I, const ItemSDC* items,
                             const double* phi1d, unsigned long long* res_bits,
                             const int* active, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  const int kz = points_per_thread(g.N);
  const dim3 grd((g.N + 31) / 32, (g.N + 7) / 8, (g.N + kz - 1) / kz * B), blk(32, 8);
  switch (M) {
    case 2: start_integrals<2>(grd, blk, st, g, U, F, tauS, I, items, phi1d, res_bits, active, kz); break;
    case 3: start_integrals<3>(grd, blk, st, g, U, F, tauS, I, items, phi1d, res_bits, active, kz); break;
    case 4: start_integrals<4>(grd, blk, st, g, U, F, tauS, I, items, phi1d, res_bits, active, kz); break;
    case 5: start_integrals<5>(grd, blk, st, g, U, F, tauS, I, items, phi1d, res_bits, active, kz); break;
    default: return cudaErrorInvalidValue;
  }
  count_launch();
  return cudaGetLastError();
}

#define H3D_FAS_CASES(X) \
  X(5, 3) X(5, 2) X(5, 5) X(3, 3) X(3, 2) X(2, 2) X(4, 4) X(4, 2)

cudaError_t launch_fas_inject(int MF, int MG, const Grid& gf, const Grid& gg, int B,
                              const double* UF, const double* FF, double* UG, double* UGr,
                              double* qF, const ItemSDC* itF, const FasMap* map,
                              const double* phif1d, cudaStream_t st, const double* X,
                              long long xs) {
  if (B <= 0) return cudaSuccess;
  int same = gf.N == gg.N;
  dim3 grd = point_grid(gg, B), blk(32, 8);
#define X_(a, b)                                                                        \
  if (MF == a && MG == b) {                                                             \
    k_fas_inject<a, b><<<grd, blk, 0, st>>>(gf, gg, same, UF, FF, UG, UGr, qF, itF, map, \
                                            phif1d, X, xs);                             \
    count_launch();                                                                     \
    return cudaGetLastError();                                                          \
  }
  H3D_FAS_CASES(X_)
#undef X_
  return cudaErrorInvalidValue;
}

cudaError_t launch_fas_wresid(int MF, const Grid& gf, int B, int jm, const double* WU,
                              const double* FF, const ItemSDC* itF, const double* phif1d,
                              double* R, double* X, long long xs, unsigned long long* res_bits,
                              cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  const int kz = points_per_thread(gf.N);
  const dim3 grd((gf.N + 31) / 32, (gf.N + 7) / 8, (gf.N + kz - 1) / kz * B), blk(32, 8);
  switch (MF) {
    case 2: k_fas_wresid<2><<<grd, blk, 0, st>>>(gf, jm, WU, FF, itF, phif1d, R, X, xs, res_bits, kz); break;
    case 3: k_fas_wresid<3><<<grd, blk, 0, st>>>(gf, jm, WU, FF, itF, phif1d, R, X, xs, res_bits, kz); break;
    case 4: k_fas_wresid<4><<<grd, blk, 0, st>>>(gf, jm, WU, FF, itF, phif1d, R, X, xs, res_bits, kz); break;
    case 5: k_fas_wresid<5><<<grd, blk, 0, st>>>(gf, jm, WU, FF, itF, phif1d, R, X, xs, res_bits, kz); break;
    default: return cudaErrorInvalidValue;
  }
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_fas_tau(int MG, const Grid& gg, int B, const double* qF, const double* FG,
                           double* tauS, const ItemSDC* itG, const double* phig1d,
                           cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  dim3 grd = point_grid(gg, B), blk(32, 8);
  switch (MG) {
    case 2: k_fas_tau<2><<<grd, blk, 0, st>>>(gg, qF, FG, tauS, itG, phig1d); break;
    case 3: k_fas_tau<3><<<grd, blk, 0, st>>>(gg, qF, FG, tauS, itG, phig1d); break;
    case 4: k_fas_tau<4><<<grd, blk, 0, st>>>(gg, qF, FG, tauS, itG, phig1d); break;
    case 5: k_fas_tau<5><<<grd, blk, 0, st>>>(gg, qF, FG, tauS, itG, phig1d); break;
    default: return cudaErrorInvalidValue;
  }
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_fas_delta(int MF, int MG, const Grid& gg, int B, const double* UG,
                             const double* UGr, double* D, const FasMap* map, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  dim3 grd = point_grid(gg, B), blk(32, 8);
#define X(a, b)                                                      \
  if (MF == a && MG == b) {                                          \
    k_fas_delta<a, b><<<grd, blk, 0, st>>>(gg, UG, UGr, D, map);     \
    count_launch();                                                  \
    return cudaGetLastError();                                       \
  }
  H3D_FAS_CASES(X)
#undef X
  return cudaErrorInvalidValue;
}

}  // namespace h3d
