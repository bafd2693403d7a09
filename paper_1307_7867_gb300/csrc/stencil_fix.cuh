// stencil_fix.cuh -- the FP64 stencil kernels of large grids with the
// neighbour sums in 64-bit fixed point (included by stencil_impl.cuh).
//
// GB300 executes 2 FP64 operations per clock and SM but 64 to 128 integer
// ones, so a stencil formed with FP64 adds (7, 13 or 19 operations a point)
// is bound by the FP64 pipe at about seven times its memory time.  Here each
// field value is turned once per tile into a 64-bit fixed-point number (block
// floating point), the stencil is summed in integers, the sum is turned back
// into a double in integers too, and two or three FP64 operations per point
// remain.  The sums are of differences (neighbours minus their count times
// the centre), exact but for the bits that the alignment drops, so the result
// is closer to the exact value than that of the FP64 sums.
//
// The format.  The unit of exponents is one z plane of a tile: 64 x 16 points
// of x and y (from multiples of 64 and 16) with the two halo points around.
// With E the largest biased exponent in it, a value of exponent e and 53-bit
// significand s becomes s 2^G >> (E - e), truncated towards zero; its unit is
// 2^(E - 1075 - G).  A point takes the largest E of the planes its stencil
// touches and shifts each plane's partial sum to it.  All of this depends on
// the values and their coordinates only, never on the launch.  A value keeps
// all its 53 bits down to 2^-G of the largest one; a pair of points is summed
// in integers only if each point's stencil holds such a value (the pair's own
// two and the neighbours in y are looked at).  Its sums are then off by a few
// units of 2^-52 of a value that it reads, as FP64 sums are; against quad
// precision at 127^3 the operator is off by 1e-16 of its norm (FP64 sums:
// 1e-14 on sums of sine modes, 1e-16 on random values).  The other pairs
// (0.3-0.5 % of a sum of sine modes, 1 % with the compact stencil: near the
// boundary and where the field changes sign; two thirds of a narrow hot spot)
// are redone in FP64 from the field.  G guard bits
// keep the sums below 2^63:
//   7-point and wide: |s1 - 6 c| <= 12 2^(53 + G), G = 6;
//   compact: |S2 - 12 c| <= 24 2^(53 + G), G = 5.
// On planes whose E lies outside [kFixLo, kFixHi] (Inf, NaN, values beyond
// 1e143 or below 1e-157), or with coefficients outside 2^+-200, every pair is
// redone; a plane of nothing but zeros counts as zero.
//
// Measured at 255^3 (one item; FP64 tiles before, random values and sums of
// sine modes now): damped Jacobi 423 -> 161 and 167 us wide, 595 -> 197 and
// 222 us compact, 219 -> 135 and 138 us 7-point; refinement residual (wide)
// 487 -> 199 and 203 us; memory time 59 us.  A hot spot of width 0.1 takes
// 465 us (wide), the FP64 redo being two thirds of it.  What is left is issue
// slots: 192 warp instructions per 32 points (wide; 237 compact, 169
// 7-point), 54-59 % of the slots used, ALU 45-53 %, FP64 pipe 39-47 %.  The
// line (fix_min_n) lies at 127 for the 7-point and the wide stencil: 34 -> 29
// and 62 -> 38 us there; at 63 both kernels take a launch's latency, and the
// persistent solve repeats the FP64 sums bit for bit.  The compact stencil
// has no persistent solve and 19 operations: from 63 on (a sweep of four
// items at 127^3 41.0 -> 39.1 ms by its 63^3 level, against 1.19 -> 1.23 ms
// for five V-cycles on one 63^3 item alone).
#pragma once
#include "fix.cuh"

namespace h3d {

constexpr int kFixTX = 64, kFixTY = 16;  // tile: points of x and y

template <int ORDER>
__host__ __device__ constexpr int fix_guard() {
  return ORDER == kCompact ? 5 : 6;
}

namespace {

template <int ORDER>
__host__ __device__ constexpr int fix_radius() {
  return ORDER == 4 ? 2 : 1;
}
constexpr int kFixW = kFixTY;  // warps of a block, one row each
// planes in the ring, a multiple of the 2R + 1 that a stencil reads
template <int ORDER>
__host__ __device__ constexpr int fix_ring() {
  return ORDER == 4 ? 10 : 9;
}
template <int ORDER>
__host__ __device__ constexpr int fix_plane_size() {
  return (kFixTY + 2 * fix_radius<ORDER>()) * (kFixTX + 4);
}
constexpr int kFixBatch = 16;  // pairs that a warp redoes in FP64 at once, a point a lane
constexpr int kFixSpan = 60;   // planes between two such turns, a multiple of 2R + 1
template <int ORDER>
constexpr int fix_smem() {
  return fix_ring<ORDER>() * fix_plane_size<ORDER>() * 8;
}

struct FixCtl {
  double k1, k2;  // the operator's coefficients, scaled
  int same;       // the planes k - R .. k + R share one exponent (or are zero)
  int add, sh;    // a value v keeps its 53 bits: (v's high word + add) >> sh
  int shift[5];   // alignment of plane k + d, at d + R
};

// A block of 16 warps owns a tile and marches along z, a warp one row and a
// thread two x points of it.  Planes of doubles arrive by cp.async in a
// shared ring, in which cells outside the domain stay zero.  In iteration k
// the block
//   - takes the largest exponent of plane k + R + 2,
//   - turns plane k + R + 1 into fixed point where it stands,
//   - computes plane k from the planes k - R .. k + R of the ring,
// with one barrier per plane.  Thread 0 prepares what a plane's threads share
// (alignment, coefficients scaled to the sums' unit) one plane ahead.  The z
// loop is unrolled by the 2R + 1 planes of a stencil and the ring is a
// multiple of that, so that every plane is a constant offset from one of a
// few base offsets.  The blocks divide the z planes of all tiles of all items
// into equal runs (`run` planes each; a run may end one tile and begin the
// next), so that every SM has the same work.  One row per warp and 64
// registers keep 32 warps on an SM: two rows per warp (128 registers, the z
// neighbours in a register queue, 16 warps) took 157 us, two rows from the
// ring 175 us, tiles of 12 rows with 80 registers 174 us, against 148.
template <int ORDER, bool NORM, typename Op>
__global__ void __launch_bounds__(32 * kFixW, 2) k_fix(Grid g, int B, int run, const int* active,
                                                       unsigned long long* norm_bits, Op op) {
  constexpr int R = fix_radius<ORDER>(), G = fix_guard<ORDER>();
  constexpr bool CP = ORDER == kCompact;
  constexpr int W = kFixW, TY = kFixTY, NT = 32 * W;
  constexpr int SX = kFixTX + 4, SY = TY + 2 * R, PS = SX * SY;
  constexpr int QL = 2 * R + 1, NB = fix_ring<ORDER>(), H = NB / QL;
  constexpr int D = NB - QL - 2;                       // planes in flight
  constexpr int XR0 = CP ? 0 : R, XRN = CP ? SY : TY;  // rows with halo pairs
  static_assert(NB % QL == 0 && W >= 2 * R + 2 && 2 * XRN <= 64, "ring and halo layout");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* ring = reinterpret_cast<double*>(smem_raw);  // [NB][SY][SX], doubles or fixed point
  __shared__ unsigned keys[8];   // largest high word of plane p, slot p mod 8
  __shared__ __align__(16) FixCtl ctl[2];
  __shared__ unsigned lost[kFixSpan][W];              // pairs left to FP64: a word per plane and row
  __shared__ unsigned short list[W][kFixBatch + 32];  // plane << 9 | row << 5 | pair, a warp's own
  const int N = g.N, plane = (int)g.plane;
  const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
  const int ntx = (N + kFixTX - 1) / kFixTX, nty = (N + TY - 1) / TY;
  const unsigned ring_s = (unsigned)__cvta_generic_to_shared(ring);
  double* const own = ring + (R + warp) * SX + 2 + 2 * lane;  // the thread's pair in slot 0
  const unsigned own_s = ring_s + (unsigned)((R + warp) * SX + 2 + 2 * lane) * 8u;

  // runs: planes [w, w1) of the sequence (item, tile, z)
  const long long total = (long long)B * ntx * nty * N;
  long long w = (long long)blockIdx.x * run;
  const long long w1 = min(total, w + run);
  while (w < w1) {
    const int t = (int)(w / N);
    const int z0 = (int)(w - (long long)t * N), z1 = (int)min((long long)N, z0 + (w1 - w));
    w += z1 - z0;
    const int b = t / (ntx * nty), tile = t - b * ntx * nty;
    if (active && !active[b]) continue;  // uniform over the block
    const int x0 = (tile % ntx) * kFixTX, y0 = (tile / ntx) * TY;
    Op o = op;
    o.init(b);
    const bool coefs = o.fix_init();
    const double* __restrict__ u = o.src(b);
    const int i = x0 + 2 * lane, j = y0 + warp;
    const int zlast = min(N - 1, z1 - 1 + R);  // last plane that is read

    // The thread's share of a plane: its own pair and, in the warps 0 .. 2R+1,
    // a pair of the halo (2R rows, then the pairs left and right); at halo_at
    // in a slot and halo_idx in the field (halo_at < 0: none).  A thread copies,
    // scans and converts the pairs it holds.  Pairs outside the domain stay
    // zero in every slot.
    int halo_at = -1, halo_idx = 0, halo_fill = 16;
    auto halo_pair = [&](int& row, int& col) {  // row < 0: none
      row = -1;
      col = 2 + 2 * lane;
      if (warp < 2 * R) {
        row = warp < R ? warp : TY + warp;
      } else if (warp < 2 * R + 2) {
        const int q = (warp - 2 * R) * 32 + lane;
        if (q < 2 * XRN) {
          row = XR0 + (q >> 1);
          col = (q & 1) ? SX - 2 : 0;
        }
      }
    };
    {
      int row, col;
      halo_pair(row, col);
      const int x = x0 - 2 + col, y = y0 - R + row;
      if (row >= 0) {
        if (x >= 0 && x < N && y >= 0 && y < N) {
          halo_at = row * SX + col;
          halo_idx = y * g.px + x;
          halo_fill = x + 1 < N ? 16 : 8;
        } else {
#pragma unroll 1
          for (int s = 0; s < NB; ++s)
            *reinterpret_cast<double2*>(ring + s * PS + row * SX + col) = make_double2(0.0, 0.0);
        }
      }
      if (j >= N)
#pragma unroll 1
        for (int s = 0; s < NB; ++s) *reinterpret_cast<double2*>(own + s * PS) = make_double2(0.0, 0.0);
    }
    auto issue = [&](int z, int s) {  // plane z into the slot at offset s
      if (z >= 0 && z <= zlast) {
        const double* uz = u + (long long)z * plane;
        // the second point of a row's last pair is outside: zero
        if (j < N) cp_async16_fill(own_s + (unsigned)s * 8u, uz + j * g.px + i, i + 1 < N ? 16 : 8);
        if (halo_at >= 0)
          cp_async16_fill(ring_s + (unsigned)(halo_at + s) * 8u, uz + halo_idx, halo_fill);
      }
      cp_async_commit();
    };
    auto key_of = [](double2 v) {
      return max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
    };
    auto low_of = [](double2 v) { return (unsigned)(__double2loint(v.x) | __double2loint(v.y)); };
    // largest exponent of plane p (at ring offset s) into keys; 0 is kept for
    // zeros, subnormal values whose high words are 0 count as 1
    auto scan = [&](int p, int s) {
      unsigned m = key_of(*reinterpret_cast<const double2*>(own + s));
      if (halo_at >= 0) m = max(m, key_of(*reinterpret_cast<const double2*>(ring + halo_at + s)));
      m = __reduce_max_sync(0xffffffffu, m);
      if (m == 0u) {
        unsigned l = low_of(*reinterpret_cast<const double2*>(own + s));
        if (halo_at >= 0) l |= low_of(*reinterpret_cast<const double2*>(ring + halo_at + s));
        m = __any_sync(0xffffffffu, l != 0u) ? 1u : 0u;
      }
      if (lane == 0) atomicMax(&keys[p & 7], m);
    };
    // plane p (at ring offset s) into fixed point
    auto fix2 = [](double* p, int E) {
      const double2 v = *reinterpret_cast<const double2*>(p);
      *reinterpret_cast<longlong2*>(p) =
          make_longlong2(fix_value<G>(__double2hiint(v.x), __double2loint(v.x), E),
                         fix_value<G>(__double2hiint(v.y), __double2loint(v.y), E));
    };
    auto decode = [&](int p, int s) {
      const int E = fix_set_exponent(keys[p & 7]);
      fix2(own + s, E);
      if (halo_at >= 0) fix2(ring + halo_at + s, E);
    };
    // The boundary rule in the ring: planes -1 and N are zero, the wide
    // stencil's planes -2 and N + 1 minus planes 0 and N - 1 (at offset f),
    // and in every plane its cells -2 and N + 1 of x and y minus the cells 0
    // and N - 1 (those at -1 and N are zero as they are).
    auto negate = [&](const double* from, double* to) {
      const longlong2 v = *reinterpret_cast<const longlong2*>(from);
      *reinterpret_cast<longlong2*>(to) = make_longlong2(-v.x, -v.y);
    };
    auto ghost_plane = [&](int p, int s, int f) {
      if (R == 2 && (p == -2 || p == N + 1)) negate(own + f, own + s);
      else *reinterpret_cast<longlong2*>(own + s) = make_longlong2(0, 0);
      if (CP && halo_at >= 0) *reinterpret_cast<longlong2*>(ring + halo_at + s) = make_longlong2(0, 0);
    };
    const bool ghosts = R == 2 && (x0 == 0 || x0 + kFixTX >= N || y0 == 0 || y0 + TY >= N);
    auto ghost_cells = [&](int s) {
      int row, col;
      halo_pair(row, col);
      const int x = x0 - 2 + col, y = y0 - R + row;
      if (row < 0) return;
      double* at = ring + row * SX + col + s;
      if (y == -2) negate(at + 2 * SX, at);
      else if (y == N + 1) negate(at - 2 * SX, at);
      else if (x == -2) *reinterpret_cast<long long*>(at) = -*reinterpret_cast<const long long*>(at + 2);
      else if (x == N + 1) *reinterpret_cast<long long*>(at) = -*reinterpret_cast<const long long*>(at - 2);
    };
    // what plane k's threads share; planes outside the domain are zero, the
    // wide stencil's ghost planes have the exponent of their source
    auto prepare = [&](int k) {
      int e[QL], em = kFixZero;
#pragma unroll
      for (int q = 0; q < QL; ++q) {
        int p = k - R + q;
        if (R == 2) p = p == -2 ? 0 : p == N + 1 ? N - 1 : p;
        e[q] = p < 0 || p >= N ? kFixZero : fix_set_exponent(keys[p & 7]);
        em = max(em, e[q]);
      }
      FixCtl& c = ctl[k & 1];
      bool same = true;
#pragma unroll
      for (int q = 0; q < QL; ++q) {
        same = same && (e[q] == em || e[q] == kFixZero);
        c.shift[q] = min(em - e[q], 63);
      }
      const bool plain = !coefs || em > kFixHi || (em > kFixZero && em < kFixLo);
      const bool zero = em == kFixZero && !plain;  // sums and results 0
      c.same = same;
      // the line is 2^52 in the unit of em; on plain planes no value reaches
      // it, on planes of zeros every one counts as if
      const int lim = plain ? 30 : min(20 + em - e[R], 30);
      c.add = zero ? (int)0x80000000u : 1 << lim;
      c.sh = zero ? 31 : lim + 1;
      // exponent of the sums' unit
      o.fix_scales(zero || plain ? 0 : em - 1075 - G, c.k1, c.k2);
    };

    // ---- prologue: planes z0 - R .. z0 - R + NB - 2 under way, those up to
    // z0 + R in fixed point.  Plane p lies in slot (p - z0 + R) mod NB. ----
    if (tid < 8) keys[tid] = 0u;
    for (int q = tid; q < kFixSpan * W; q += NT) lost[0][q] = 0u;
#pragma unroll 1
    for (int q = 0; q < NB - 1; ++q) issue(z0 - R + q, q * PS);
    cp_async_wait<NB - 1 - (QL + 1)>();
    __syncthreads();
#pragma unroll 1
    for (int q = 0; q <= QL; ++q)
      if (const int p = z0 - R + q; p >= 0 && p <= zlast) scan(p, q * PS);
    __syncthreads();
#pragma unroll 1
    for (int q = 0; q < QL; ++q)
      if (const int p = z0 - R + q; p >= 0 && p < N) decode(p, q * PS);
#pragma unroll 1
    for (int q = 0; q < QL; ++q)
      if (const int p = z0 - R + q; p < 0 || p >= N) ghost_plane(p, q * PS, (p < 0 ? q + 2 : q - 2) * PS);
    if (tid == NT - 32) prepare(z0);
    if (ghosts) {
      __syncthreads();
      ghost_cells(R * PS);
    }

    unsigned long long mx = 0ull;
    int idx = z0 * plane + j * g.px + i;
    const int nx = N - i;       // points of the thread's two inside the grid
    const bool live = j < N;    // uniform over the warp
    int base[H];  // ring offsets of the slots QL h .. of the current turn
#pragma unroll
    for (int h = 0; h < H; ++h) base[h] = h * QL * PS;
#pragma unroll 1
    for (int kc = z0; kc < z1; kc += kFixSpan) {
      const int ke = min(z1, kc + kFixSpan);
#pragma unroll 1
      for (int kb = kc; kb < ke; kb += QL) {
#pragma unroll
        for (int uu = 0; uu < QL; ++uu) {
          const int k = kb + uu;
          if (k >= z1) break;  // uniform
          // ring offset of plane k + d
          auto off = [&](int d) { return base[((uu + d + R + NB) / QL) % H] + ((uu + d + R + NB) % QL) * PS; };
          typename Op::Ex2 ex;
          typename Op::Late late;
          double2 c0;
          if (live) {
            ex = o.load2(idx);
            late = o.late2(idx);
            if (Op::kFixCentre) c0 = *reinterpret_cast<const double2*>(u + idx);
          }
          cp_async_wait<D - 1>();  // plane k + R + 2 has arrived
          __syncthreads();
          issue(k - R - 1 + NB, off(-R - 1));
          if (tid == NT - 32) keys[(k + R + 3) & 7] = 0u;
          if (k + R + 2 <= zlast) scan(k + R + 2, off(R + 2));
          if (k + R + 1 <= zlast) decode(k + R + 1, off(R + 1));
          else if (k + 1 < z1) ghost_plane(k + R + 1, off(R + 1), off(R - 1));
          if (ghosts && k + 1 < z1) ghost_cells(off(1));
          if (live) {
            const FixCtl& cc = ctl[k & 1];
            auto at = [&](int d, int dy, int dx) {  // pair dx points to the right in row j + dy of plane k + d
              return *reinterpret_cast<const longlong2*>(own + off(d) + dy * SX + dx);
            };
            auto one = [&](int d, int dy, int dx) {
              return *reinterpret_cast<const long long*>(own + off(d) + dy * SX + dx);
            };
            // the pair's own values decide, each of which is in the other's
            // stencil, or else the neighbours in y of both
            auto top = [&](int dy, int x) {
              return (unsigned)reinterpret_cast<const int*>(own + off(0) + dy * SX + x)[1] + (unsigned)cc.add;
            };
            bool keep = (top(0, 0) | top(0, 1)) >> cc.sh;
            if (!keep) {  // seldom
              keep = (top(-1, 0) | top(1, 0)) >> cc.sh && (top(-1, 1) | top(1, 1)) >> cc.sh;
              if (!keep) atomicOr(&lost[k - kc][warp], 1u << lane);
            }
            longlong2 d1, d2 = make_longlong2(0, 0);
            // the sums; al(a, b, d) aligns the partial sums of plane k + d
            auto sums = [&](auto al) {
              const longlong2 cr = at(0, 0, 0);
              const longlong2 c = al(cr.x, cr.y, 0);
              const long long c60 = 6 * c.x, c61 = 6 * c.y;
              // n - 6 c and the pairs of the planes k -+ d
              auto add_z = [&](const longlong2& n, const longlong2& m, const longlong2& p, int d) {
                const longlong2 v = al(m.x, m.y, -d), w = al(p.x, p.y, d);
                return make_longlong2(n.x - c60 + (v.x + w.x), n.y - c61 + (v.y + w.y));
              };
              const longlong2 ym = at(0, -1, 0), yp = at(0, 1, 0);
              if constexpr (!CP) {
                const longlong2 l = at(0, 0, -2), h = at(0, 0, 2);
                d1 = add_z(al(l.y + cr.y + ym.x + yp.x, cr.x + h.x + ym.y + yp.y, 0), at(-1, 0, 0), at(1, 0, 0), 1);
                if constexpr (R == 2) {
                  const longlong2 ym2 = at(0, -2, 0), yp2 = at(0, 2, 0);
                  const longlong2 t = add_z(al(l.x + h.x + ym2.x + yp2.x, l.y + h.y + ym2.y + yp2.y, 0),
                                            at(-2, 0, 0), at(2, 0, 0), 2);
                  d1.x -= t.x >> 4;
                  d1.y -= t.y >> 4;
                }
              } else {
                const longlong2 zm = at(-1, 0, 0), zp = at(1, 0, 0);
                d1 = add_z(al(one(0, 0, -1) + cr.y + ym.x + yp.x, cr.x + one(0, 0, 2) + ym.y + yp.y, 0), zm, zp, 1);
                // edges: four of plane k, four of each plane next to it
                const longlong2 e0 = al((one(0, -1, -1) + ym.y) + (one(0, 1, -1) + yp.y),
                                        (ym.x + one(0, -1, 2)) + (yp.x + one(0, 1, 2)), 0);
                auto cross = [&](const longlong2& z, int d) {
                  const longlong2 a = at(d, -1, 0), q = at(d, 1, 0);
                  return al((one(d, 0, -1) + z.y) + (a.x + q.x), (z.x + one(d, 0, 2)) + (a.y + q.y), d);
                };
                const longlong2 em1 = cross(zm, -1), ep1 = cross(zp, 1);
                d2.x = e0.x + em1.x + ep1.x - 2 * c60;
                d2.y = e0.y + em1.y + ep1.y - 2 * c61;
              }
            };
            if (cc.same) {
              sums([](long long a, long long q, int) { return make_longlong2(a, q); });
            } else {
              sums([&](long long a, long long q, int d) {
                const int s = cc.shift[d + R];
                return make_longlong2(a >> s, q >> s);
              });
            }
            const typename Op::Out2 out = o.post2(o.pre2(c0, ex), c0, d1, d2, cc.k1, cc.k2);
            if (keep) o.template put2<NORM>(idx, nx, out, late, mx);
          }
          idx += plane;
          if (tid == NT - 32 && k + 1 < z1) prepare(k + 1);
        }
        const int first = base[0];  // the next turn begins QL slots further
#pragma unroll
        for (int h = 0; h + 1 < H; ++h) base[h] = base[h + 1];
        base[H - 1] = first;
      }
      // the pairs left to FP64 (no operator writes the field it reads, so their
      // order is free): a warp takes one row per plane, another one in the next
      __syncthreads();
      int n = 0;  // listed
#pragma unroll 1
      for (int k0 = kc; k0 < ke; k0 += 32) {
        const int kl = k0 + lane, row = (warp + kl) & (W - 1);
        unsigned m = kl < ke ? lost[kl - kc][row] : 0u;
        if (m) lost[kl - kc][row] = 0u;
        unsigned todo = __ballot_sync(0xffffffffu, m != 0u);
#pragma unroll 1
        for (bool more = true; more;) {
          const int src = __ffs(todo) - 1;
          if (todo) {
            const unsigned w = __shfl_sync(0xffffffffu, m, src);
            if (w >> lane & 1)
              list[warp][n + __popc(w & ((1u << lane) - 1))] =
                  (unsigned short)((k0 + src - kc) << 9 | ((warp + k0 + src) & (W - 1)) << 5 | lane);
            n += __popc(w);
            todo &= todo - 1;
            __syncwarp();
          }
          more = todo != 0u;
#pragma unroll 1
          while (n >= kFixBatch || (n > 0 && !more && k0 + 32 >= ke)) {
            const int take = min(n, kFixBatch);
            n -= take;
            const int code = list[warp][n + min(lane >> 1, take - 1)];
            const int x = x0 + 2 * (code & 31) + (lane & 1), y = y0 + (code >> 5 & (W - 1)), z = kc + (code >> 9);
            if (lane < 2 * take && x < N) {
              double cc, s1, s2;
              plain_sums<ORDER>(u, g, x, y, z, cc, s1, s2);
              const int p = z * plane + y * g.px + x;
              const double rv = o.apply(p, cc, s1, s2, o.load(p));
              if (NORM) mx = max(mx, abs_bits(rv));
            }
            __syncwarp();
          }
        }
      }
    }
    cp_async_wait<0>();
    if (NORM) warp_max_to(mx, norm_bits + b);
    __syncthreads();  // the next run's prologue reuses the shared memory
  }
}

// Equal runs over the whole GPU in one wave; up to four waves of shorter ones
// for a batch, whose converged items drop out and leave their share to the
// others, as long as a run has 24 planes (its prologue costs about five).
// `spare`: resident blocks left free for the kernels of other streams, which
// would otherwise wait for a whole wave.
template <int ORDER, bool NORM, typename Op>
cudaError_t launch_fix(const Grid& g, int B, int spare, const int* active, unsigned long long* norm_bits,
                       const Op& op, cudaStream_t st) {
  constexpr int smem = fix_smem<ORDER>();
  auto kern = k_fix<ORDER, NORM, Op>;
  static PerDevice once;
  int slots = 0;
  const cudaError_t e = once.get(&slots, [&](int dev, int* n) {
    const cudaError_t rc = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return rc == cudaSuccess ? resident_blocks(dev, kern, 32 * kFixW, smem, n) : rc;
  });
  if (e != cudaSuccess) return e;
  const long long total =
      (long long)((g.N + kFixTX - 1) / kFixTX) * ((g.N + kFixTY - 1) / kFixTY) * g.N * B;
  const long long one = std::max(1, slots - spare);
  const long long waves = B > 1 ? std::max<long long>(1, std::min<long long>(4, total / (one * 24))) : 1;
  const int run = (int)std::max<long long>(2, (total + waves * one - 1) / (waves * one));
  kern<<<(unsigned)((total + run - 1) / run), dim3(32, kFixW), smem, st>>>(g, B, run, active, norm_bits, op);
  return cudaSuccess;
}

}  // namespace
}  // namespace h3d
