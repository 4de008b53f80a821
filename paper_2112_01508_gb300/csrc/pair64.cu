// FP64 pair forces and their adjoint (one-sided: every receiver gathers).
//
// What bounds them: the FP64 pipe of this part retires about two lane operations per SM
// and clock, a warp instruction every 16 clocks, while everything else (FP32, integers,
// shared memory) runs 30-60 times faster.  So only the arithmetic that fixes the result
// is FP64, and FP64 instructions are issued for interacting pairs as far as possible:
//   * the supplier traversal and a first distance test run in FP32 in the chunk's frame,
//     with a margin far above its rounding.  The test leaves one bit per (receiver,
//     staged supplier); the set bits are dealt out to the lanes in equal runs, so that
//     every lane holds an interacting pair in every step, instead of all lanes meeting
//     one supplier with 0.39 of them in range;
//   * the bracket is a table of degree-6 polynomials in r^2 (pair_tables.cuh) held in
//     shared memory: one FMA for the offset in the interval and six for the value, in
//     place of erfc, exp, a square root and divisions.  The interval index comes from
//     the bits of r^2 by integer and FP32 operations, compares and selects are made on
//     the bits, so an interacting pair costs 16 FP64 instructions (adjoint: 32), at
//     126 (170) with the library functions;
//   * pairs that may be closer than r_sw (softened form) are walked in a second pass, so
//     that its longer evaluation is not paid by a warp of which one lane is that close;
//   * with few chunks the suppliers of a chunk are split between work items, the partial
//     sums added in a fixed order (the result stays bitwise reproducible).
// The cutoff and the pair count are decided on the FP64 r^2.
// Measured (B-spline): 262,144 clustered particles, 82.5 M pairs: forces 40.2 -> 3.03 ms
// (27 G pairs/s; the FP64 pipe 87% busy, 97% of its lanes on interacting pairs, 17.8 lane
// operations a pair), adjoint 5.6 ms; 9261 particles, 2.9 M pairs, Plummer: 0.19 and
// 0.35 ms (0.45 and 0.80 with chunks split by subtiles instead of equal supplier counts).
// Against 113-bit sums (relative RMS) the force error fell from 6.7e-16 to 2.3e-16 and the
// adjoint's from 1.6e-15 to 4.3e-16 (B-spline), from 5.8e-16 to 1.8e-16 and from 6.8e-16 to
// 3.3e-16 (Plummer).  A double evaluation of the closed forms shares the earlier kernel's
// rounding and stands further from this one than from that: it is no measure below 1e-15.
#include <algorithm>
#include <cmath>

#include "pair_tables.cuh"
#include "traverse.cuh"

namespace p3m {

constexpr int kBatch64 = 128;  // suppliers staged per walk: longer walks even out the lanes' hit counts
constexpr int kMaxWarps64 = 16;
constexpr int kMaxParts64 = 32;  // 9261 particles: 0.193 ms (16: 0.209, 64: 0.202)

struct Pair64Args {
  const double* tab;   // log f, log f', uniform h, uniform h'
  int row0, rows;      // logarithmic rows in use
  int urows;           // uniform rows in use
  double c;            // 1 / (2 x_s)^2: s = c r^2
  double len;          // 2^-k, k = the binary exponent of the box side: FP32 quantities are in units of 2^k
  unsigned bias;       // FP32 bits of r^2 in those units: (high word - bias) << 3
  float c_f;           // c in those units
  double ce2;          // Plummer: c eps^2
  float ce2_f;
  double xr2, rsw2;
  float cut2;          // FP32 test: r^2 below it may interact
  float near2;         // ... and below this may be softened (B-spline)
  double cb, cd, ieb;  // B-spline shape: 32 / eps_B^3, 32 / eps_B^5, 1 / eps_B
  double scale;        // -G m
};

template <bool VJP>
struct Warp64 {
  WarpListOf<kBatch64> L;
  union {
    struct {
      float4 sxy[kBatch64 / 2];  // (-x_a, -x_b, -y_a, -y_b) of suppliers 2p and 2p + 1, chunk frame
      float2 sz[kBatch64 / 2];
    };
    double part[3][2 * kWarp];  // during a walk (the FP32 coordinates are done with): sums of its segments
  };
  double x[kBatch64], y[kBatch64], z[kBatch64];  // absolute, nearest image
  double v[VJP ? 3 : 1][VJP ? kBatch64 : 1];     // masked abar
  double ri[VJP ? 6 : 3][kWarp];                 // the receivers: position and masked abar
  int j[kBatch64];
  unsigned mask[2][kBatch64];                    // hit bits, word q of receiver i at [q 32 + i]: main walk, near walk
};

// hs = c^{3/2} turns b, q and h into brackets, 2 c hs their s-derivatives into B'(r)/r.  hs
// is taken from the rounded c, in double-double, so that hs b(c r^2) carries no common
// error from the rounding of c (b ~ s^{-3/2} for close pairs).
__global__ void k_fill_tables(const __grid_constant__ SeriesDD t, double* tab, int plummer, int row0, int rows,
                              int urows, double c) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double* f = tab;
  double* fd = f + kTabLogRows * kTabRow;
  double* h = fd + kTabLogRows * kTabRow;
  double* hd = h + kTabUniRows * kTabRow;
  const DD hs = dd_div(DD{1.0, 0.0}, pow_m32(c));
  const double ds = 2.0 * c * hs.hi;
  if (i < rows) table_log_row(t, row0 + i, plummer != 0, hs, ds, f + (row0 + i) * kTabRow, fd + (row0 + i) * kTabRow);
  else if (i < rows + urows) table_uni_row(t, i - rows, hs, ds, h + (i - rows) * kTabRow, hd + (i - rows) * kTabRow);
}

int64_t pair_table_doubles() { return kTabDoubles; }

__device__ __forceinline__ double poly7(const double* __restrict__ c, double t) {
  double p = c[kTabDeg];
#pragma unroll
  for (int k = kTabDeg - 1; k >= 0; --k) p = __fma_rn(p, t, c[k]);
  return p;
}

// r^2 in FP32 (truncated) in the units that `bias` stands for, 0 below the normal range.
__device__ __forceinline__ float trunc_f32(double v, unsigned bias) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  return hi < bias + 0x00100000u ? 0.0f : __uint_as_float(__funnelshift_l(lo, hi - bias, 3));
}

// The middle of the table interval that holds s (a float with few mantissa bits) as a double.
__device__ __forceinline__ double widen_bits(unsigned fbits) {
  return __hiloint2double((int)((fbits >> 3) + 0x38000000u), (int)(fbits << 29));
}

struct Tables {
  const double *f, *fd, *h, *hd;  // shared memory
};

// b (or q) and optionally its s-derivative at s = c r2 + s_off, s_f ~ s in FP32; false
// outside the tabulated range.
template <bool D>
__device__ __forceinline__ bool log_lookup(const Pair64Args& p, const Tables& T, double r2, double s_off, float s_f,
                                           double& f, double& fd) {
  const unsigned bits = __float_as_uint(s_f);
  const int row = (int)(bits >> kTabLogShift) - (kTabLogFirst + p.row0);
  const bool in = (unsigned)row < (unsigned)p.rows;
  const int o = (in ? row : 0) * kTabRow;
  const unsigned mid = (bits >> kTabLogShift << kTabLogShift) | (1u << (kTabLogShift - 1));
  const double m = widen_bits(mid);
  const double t = __fma_rn(r2, p.c, s_off - m);
  f = poly7(T.f + o, t);
  if (D) fd = poly7(T.fd + o, t);
  return in;
}

template <bool D>
__device__ __forceinline__ bool uni_lookup(const Pair64Args& p, const Tables& T, double r2, float s_f, double& h,
                                           double& hd) {
  const int row = (int)(s_f * (float)kTabUniPerUnit);
  const bool in = row < p.urows;
  const int k = in ? row : 0;
  // the middle (2 k + 1) / 32 is exact in FP32
  const double m = widen_bits(__float_as_uint((float)(2 * k + 1) * (0.5f / kTabUniPerUnit)));
  const double t = __fma_rn(r2, p.c, -m);
  h = poly7(T.h + k * kTabRow, t);
  if (D) hd = poly7(T.hd + k * kTabRow, t);
  return in;
}

// Outside the tables: the closed forms.
template <int SOFT, bool VJP>
__device__ __noinline__ double2 bracket_direct(double r2, const ForceConsts& f, const SeriesConsts& sc) {
  double D = 0.0;
  const double B = bracket_f64<SOFT, VJP>(r2, f, sc, D);
  return make_double2(B, D);
}

// B-spline softened form, r < r_sw = eps_B (Section 2.1.1): shape minus h.  1/r: with a first
// value y and e = 1 - r^2 y^2, 1/r = y (1 - e)^(-1/2) = y (1 + e/2 + 3/8 e^2 + ...), the
// binomial series cut after e^2 (one third-order Householder step).  y, from the truncated FP32
// r^2 (2^-23) and the approximate root (2^-22.9), has |e| < 2^-21.3, so the rest of the series,
// 5/16 e^3, is below 2^-65 and what remains is the rounding of the step itself.
template <bool VJP>
__device__ __forceinline__ bool soft_bspline(const Pair64Args& p, const Tables& T, double r2, float r2_f, float s_f,
                                             double& b, double& d) {
  double h, hd;
  const bool in = uni_lookup<VJP>(p, T, r2, s_f, h, hd);
  double y = r2_f > 0.0f ? (double)rsqrt_approx(r2_f) * p.len : 0.0;
  const double e = __fma_rn(-(r2 * y), y, 1.0);
  y = __fma_rn(y * e, __fma_rn(0.375, e, 0.5), y);
  const double x = (r2 * y) * p.ieb, w = 1.0 - x, w2 = w * w;
  // x < 1/2: 32 / eps_B^3 (x^3 - 6/5 x^2 + 1/3).  Outer piece: r^-3 M with the mass fraction
  // M = 1 - (32/3) (1 - x)^4 (x^2 + 2/5 x + 1/10), M' = 64 x^2 (1 - x)^3: the polynomial of
  // Eq. bspline_force without its cancellation towards x = 1.
  const double s_in = __fma_rn(x * x, x - 1.2, 1.0 / 3.0);
  const double M = __fma_rn(w2 * w2 * (-32.0 / 3.0), __fma_rn(x, x + 0.4, 0.1), 1.0);
  const double y3 = y * y * y;
  const bool inner = x < 0.5;
  b = inner ? __fma_rn(p.cb, s_in, -h) : __fma_rn(y3, M, -h);
  if (VJP) {
    const double xw = x * w;
    const double d_in = __fma_rn(p.cd, __fma_rn(3.0, x, -2.4), -hd);
    const double d_out = __fma_rn(y3 * (y * y), __fma_rn(64.0 * xw, xw * xw, -3.0 * M), -hd);
    d = inner ? d_in : d_out;
  }
  return in && (r2_f > 1e-30f || r2 == 0.0);
}

template <bool VJP, int SOFT>
__global__ void __launch_bounds__(kMaxWarps64 * kWarp, 1) k_pair64(const __grid_constant__ TraversalArgs a,
                                                                  const __grid_constant__ Pair64Args p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Warp64<VJP>* warps = reinterpret_cast<Warp64<VJP>*>(smem_raw);
  const int n_warps = blockDim.x >> 5;
  double* tab = reinterpret_cast<double*>(warps + n_warps);
  Tables T64{};
  {  // the rows in use, into shared memory (even row counts: whole 16-byte pieces)
    auto rows = [&](int first, int count) {
      const double* dst = tab;
      const double* src = p.tab + (int64_t)first * kTabRow;
      for (int i = 2 * threadIdx.x; i < count * kTabRow; i += 2 * blockDim.x) cp_async16(tab + i, src + i);
      tab += count * kTabRow;
      return dst;
    };
    T64.f = rows(p.row0, p.rows);
    if (VJP) T64.fd = rows(kTabLogRows + p.row0, p.rows);
    if (SOFT != P3M_SOFT_NONE) {
      T64.h = rows(2 * kTabLogRows, p.urows);
      if (VJP) T64.hd = rows(2 * kTabLogRows + kTabUniRows, p.urows);
    }
    cp_async_commit();
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  Warp64<VJP>& S = warps[threadIdx.x >> 5];
  const Geometry& g = a.g;
  const int n_chunks = *a.n_chunks;
  const int nparts = a.part_acc ? parts_for(n_chunks, a.part_items, kMaxParts64) : 1;
  const int n_items = n_chunks * nparts;
  const Reach rc = make_reach<true>(a, p.len);
  // an FP32 distance is within ~1e-5 x_r of the exact one (a little more after long drifts)
  const float slack = 1e-6f * rc.delta;
  const float cut = sqrtf(p.cut2) + slack, nearr = sqrtf(p.near2) + slack;
  const float cut2 = cut * cut, near2 = SOFT == P3M_SOFT_BSPLINE ? nearr * nearr : 0.0f;
  unsigned long long pair_total = 0;
  for (;;) {
    const int w = next_chunk(a, lane);
    if (w >= n_items) break;
    const int ci = w / nparts, part = w - ci * nparts;
    const Chunk ch = chunk_at(a, ci);
    ChunkFrame F;
    load_chunk(a, rc, ch, lane, F);
    double xi = 0.0, yi = 0.0, zi = 0.0;
    double vxi = 0.0, vyi = 0.0, vzi = 0.0;
    if (F.valid) {
      xi = a.pos[F.pidx];
      yi = a.pos[a.n + F.pidx];
      zi = a.pos[2 * a.n + F.pidx];
      if (a.n_drift > 0) {  // drifted since the sort: the image nearest its sorted subtile
        xi += g.box * rint(((F.gi[0] + 0.5) * g.side64[0] - xi) / g.box);
        yi += g.box * rint(((F.gi[1] + 0.5) * g.side64[1] - yi) / g.box);
        zi += g.box * rint(((F.gi[2] + 0.5) * g.side64[2] - zi) / g.box);
      }
      if (VJP) {
        vxi = a.abar_d[F.pidx];
        vyi = a.abar_d[a.n + F.pidx];
        vzi = a.abar_d[2 * a.n + F.pidx];
      }
    }
    S.ri[0][lane] = xi;
    S.ri[1][lane] = yi;
    S.ri[2][lane] = zi;
    if (VJP) {
      S.ri[VJP ? 3 : 0][lane] = vxi;
      S.ri[VJP ? 4 : 0][lane] = vyi;
      S.ri[VJP ? 5 : 0][lane] = vzi;
    }
    const int own_lo = __reduce_min_sync(full, F.valid ? F.pidx : 0x7fffffff);
    const int own_hi = __reduce_max_sync(full, F.valid ? F.pidx : -1);
    const f2 px = pk(F.pi.x, F.pi.x), py = pk(F.pi.y, F.pi.y), pz = pk(F.pi.z, F.pi.z);
    double ax = 0.0, ay = 0.0, az = 0.0;
    int hits = 0;
    int cnt = 0;  // staged suppliers (warp-uniform)
    bool blk_near = false, blk_own = false;

    // Evaluate the pairs of the hit bits in S.mask[near].  The bits, in the order of the
    // receivers, are dealt out to the lanes in equal runs, so that every lane evaluates
    // the same number of pairs; a lane stores the sum of each receiver it passes through
    // (its segment; slot receiver + lane is unique) and the receivers add theirs in lane order.
    auto walk = [&](auto near_walk) {
      constexpr bool kNear = decltype(near_walk)::value;
      const unsigned* mask = S.mask[kNear ? 1 : 0];
      int c = 0;
#pragma unroll
      for (int q = 0; q < kBatch64 / kWarp; ++q) c += __popc(mask[q * kWarp + lane]);
      int inc = c;
#pragma unroll
      for (int o = 1; o < kWarp; o <<= 1) {
        const int u = __shfl_up_sync(full, inc, o);
        if (lane >= o) inc += u;
      }
      const int total = __shfl_sync(full, inc, kWarp - 1), first = inc - c;
      if (total == 0) return;
      const int T = (total + kWarp - 1) >> 5;
      const int e0 = lane * T, mine = min(T, total - e0);  // this lane's run (mine <= 0: none)
      int r = 0;                                            // its first receiver: the last with first <= e0
#pragma unroll
      for (int o = kWarp / 2; o > 0; o >>= 1)
        if (__shfl_sync(full, first, r + o) <= e0) r += o;
      int skip = e0 - __shfl_sync(full, first, r);
      int q = 0;
      unsigned word = 0;
      double rx = 0.0, ry = 0.0, rz = 0.0, rvx = 0.0, rvy = 0.0, rvz = 0.0;
      auto receiver = [&]() {
        rx = S.ri[0][r];
        ry = S.ri[1][r];
        rz = S.ri[2][r];
        if (VJP) {
          rvx = S.ri[VJP ? 3 : 0][r];
          rvy = S.ri[VJP ? 4 : 0][r];
          rvz = S.ri[VJP ? 5 : 0][r];
        }
      };
      if (mine > 0) {
        word = mask[r];
        for (int n; skip >= (n = __popc(word)); word = mask[q * kWarp + r]) {
          skip -= n;
          ++q;
        }
        for (; skip > 0; --skip) word &= word - 1;
        receiver();
      }
      double sx = 0.0, sy = 0.0, sz = 0.0;
      auto flush = [&]() {
        S.part[0][r + lane] = sx;
        S.part[1][r + lane] = sy;
        S.part[2][r + lane] = sz;
      };
      __syncwarp();
      for (int it = 0; it < T; ++it) {
        const bool act = it < mine;
        if (act && word == 0) {  // the next word with a hit, of this or a later receiver
          const int r0 = r;
          do {
            if (++q == kBatch64 / kWarp) {
              q = 0;
              if (r == r0) flush();
              ++r;
            }
            word = mask[q * kWarp + r];
          } while (word == 0);
          if (r != r0) {
            sx = sy = sz = 0.0;
            receiver();
          }
        }
        const int k = act ? q * kWarp + __ffs((int)word) - 1 : 0;
        word &= word - 1;
        const double dx = rx - S.x[k], dy = ry - S.y[k], dz = rz - S.z[k];
        const double r2 = __fma_rn(dz, dz, __fma_rn(dy, dy, dx * dx));
        const bool hit = act && __double_as_longlong(r2) < __double_as_longlong(p.xr2);
        const float r2f = trunc_f32(r2, p.bias);
        const float sf = r2f * p.c_f;
        double b = 0.0, d = 0.0;
        bool in;
        if (SOFT == P3M_SOFT_PLUMMER) {
          double h, hd;
          in = log_lookup<VJP>(p, T64, r2, p.ce2, sf + p.ce2_f, b, d);
          in = uni_lookup<VJP>(p, T64, r2, sf, h, hd) && in;
          b -= h;
          if (VJP) d -= hd;
        } else {
          const bool soft = SOFT == P3M_SOFT_BSPLINE && __double_as_longlong(r2) < __double_as_longlong(p.rsw2);
          in = !soft;
          if (!kNear || __any_sync(full, hit && !soft)) in = log_lookup<VJP>(p, T64, r2, 0.0, sf, b, d) && !soft;
          if (kNear && soft) in = soft_bspline<VJP>(p, T64, r2, r2f, sf, b, d);
        }
        if (__any_sync(full, hit && !in)) {  // outside the tables (rare)
          if (hit && !in) {
            const double2 v = bracket_direct<SOFT, VJP>(r2, a.f, a.sc);
            b = VJP || r2 > 0.0 ? v.x : 0.0;
            d = v.y;
          }
        }
        b = hit ? b : 0.0;
        hits += hit ? 1 : 0;
        if (VJP) {
          d = hit ? d : 0.0;
          const double vx = rvx - S.v[0][k], vy = rvy - S.v[VJP ? 1 : 0][k], vz = rvz - S.v[VJP ? 2 : 0][k];
          const double xv = __fma_rn(dz, vz, __fma_rn(dy, vy, dx * vx));
          const double cc = d * xv;
          sx = __fma_rn(b, vx, __fma_rn(cc, dx, sx));
          sy = __fma_rn(b, vy, __fma_rn(cc, dy, sy));
          sz = __fma_rn(b, vz, __fma_rn(cc, dz, sz));
        } else {
          sx = __fma_rn(b, dx, sx);
          sy = __fma_rn(b, dy, sy);
          sz = __fma_rn(b, dz, sz);
        }
      }
      if (mine > 0) flush();
      __syncwarp();
      if (c > 0) {
        const int last = (inc - 1) / T;
        for (int l = first / T; l <= last; ++l) {
          ax += S.part[0][lane + l];
          ay += S.part[1][lane + l];
          az += S.part[2][lane + l];
        }
      }
      __syncwarp();
    };

    // The staged suppliers against the chunk.
    auto eval_batch = [&](int nb) {
      for (int q = 0; q < kBatch64 / kWarp; ++q) {
        unsigned m = 0, mnear = 0;
        if (32 * q >= nb) {
          S.mask[0][q * kWarp + lane] = S.mask[1][q * kWarp + lane] = 0;
          continue;
        }
        const float n2 = blk_near ? near2 : -1.0f;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float4 s = S.sxy[16 * q + i];
          const float2 z = S.sz[16 * q + i];
          const f2 dx = add2(px, pk(s.x, s.y));
          const f2 dy = add2(py, pk(s.z, s.w));
          const f2 dz = add2(pz, pk(z.x, z.y));
          float q0, q1;
          upk(fma2(dx, dx, fma2(dy, dy, mul2(dz, dz))), q0, q1);
          if (q0 < cut2) m |= 1u << (2 * i);
          if (q1 < cut2) m |= 2u << (2 * i);
          if (SOFT == P3M_SOFT_BSPLINE) {
            if (q0 < n2) mnear |= 1u << (2 * i);
            if (q1 < n2) mnear |= 2u << (2 * i);
          }
        }
        const int left = nb - 32 * q;
        if (left < 32) m &= (1u << left) - 1u;
        if (blk_own) {  // a receiver does not meet itself
          for (int i = 0; i < 32; ++i)
            if (S.j[32 * q + i] == F.pidx) m &= ~(1u << i);
        }
        if (!F.valid) m = 0;
        S.mask[0][q * kWarp + lane] = m & ~mnear;
        S.mask[1][q * kWarp + lane] = m & mnear;
      }
      __syncwarp();
      walk(std::false_type{});
      if (SOFT == P3M_SOFT_BSPLINE && blk_near) walk(std::true_type{});
    };

    enumerate_suppliers(a, rc, F, S.L, lane, part, nparts, 0, [&](int nlist, int lo, int hi, bool last) {
      ListCursor<WarpListOf<kBatch64>> cur;
      cur.seek(S.L, nlist, lane, lo);
      for (int b = lo;; b += kWarp) {
        const bool more = b < hi;  // warp-uniform
        bool keep = false, near = false, own = false;
        Vec3<float> pj = {0.f, 0.f, 0.f};
        int j = 0, dx = 0, dy = 0, dz = 0, ns = 0;
        unsigned m = 0;
        if (more) {
          unsigned dpk;
          if (cur.locate(S.L, nlist, hi, lane, b, j, dpk)) {
            const float4 r = a.rel4[j];
            unpack_delta(dpk, dx, dy, dz);
            pj.x = fmaf((float)dx, g.side32[0], r.x * a.rel_scale);
            pj.y = fmaf((float)dy, g.side32[1], r.y * a.rel_scale);
            pj.z = fmaf((float)dz, g.side32[2], r.z * a.rel_scale);
            const float gap2 = box_gap2(F, pj);
            keep = gap2 < cut2;
            near = gap2 < near2;
            own = keep && j >= own_lo && j <= own_hi;
          }
          m = __ballot_sync(full, keep);
          ns = __popc(m);
        }
        if (more ? cnt + ns > kBatch64 : last && cnt > 0) {
          __syncwarp();
          eval_batch(cnt);
          cnt = 0;
          blk_near = blk_own = false;
        }
        if (!more) break;
        if (keep) {
          const int k = cnt + __popc(m & lt_mask);
          float* sxy = (float*)S.sxy;
          float* sz = (float*)S.sz;
          const int q = k >> 1, h = k & 1;
          sxy[4 * q + h] = -pj.x;
          sxy[4 * q + 2 + h] = -pj.y;
          sz[2 * q + h] = -pj.z;
          // absolute position, the image in the chunk's neighbourhood
          const int gx = F.g0[0] + dx, gy = F.g0[1] + dy, gz = F.g0[2] + dz;
          double x = a.pos[j], y = a.pos[a.n + j], z = a.pos[2 * a.n + j];
          if (gx < 0 || gx >= g.M[0]) x += gx < 0 ? -g.box : g.box;
          if (gy < 0 || gy >= g.M[1]) y += gy < 0 ? -g.box : g.box;
          if (gz < 0 || gz >= g.M[2]) z += gz < 0 ? -g.box : g.box;
          if (a.n_drift > 0) {  // drifted since the sort: the image nearest the candidate subtile
            x += g.box * rint(((gx + 0.5) * g.side64[0] - x) / g.box);
            y += g.box * rint(((gy + 0.5) * g.side64[1] - y) / g.box);
            z += g.box * rint(((gz + 0.5) * g.side64[2] - z) / g.box);
          }
          S.x[k] = x;
          S.y[k] = y;
          S.z[k] = z;
          S.j[k] = j;
          if (VJP) {
            S.v[0][k] = a.abar_d[j];
            S.v[VJP ? 1 : 0][k] = a.abar_d[a.n + j];
            S.v[VJP ? 2 : 0][k] = a.abar_d[2 * a.n + j];
          }
        }
        blk_near = blk_near || __any_sync(full, near);
        blk_own = blk_own || __any_sync(full, own);
        cnt += ns;
      }
    });
    if (nparts == 1) {
      if (F.valid) {
        double* o = (double*)a.out;
        o[F.pidx] = p.scale * ax;
        o[a.n + F.pidx] = p.scale * ay;
        o[2 * a.n + F.pidx] = p.scale * az;
      }
    } else {
      double* o = (double*)a.part_acc + (int64_t)w * (3 * kWarp) + lane;
      o[0] = ax;
      o[kWarp] = ay;
      o[2 * kWarp] = az;
    }
    pair_total += (unsigned long long)__reduce_add_sync(full, (unsigned)hits);
  }
  if (lane == 0 && pair_total) atomicAdd(a.pairs, pair_total);
}

// The parts of each chunk added in part order, when k_pair64 split its chunks.
__global__ void k_parts_finish64(TraversalArgs a, double scale) {
  const int n_chunks = *a.n_chunks;
  const int nparts = parts_for(n_chunks, a.part_items, kMaxParts64);
  if (nparts == 1) return;
  const int lane = threadIdx.x & 31;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  double* o = (double*)a.out;
  for (int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < n_chunks; c += nw) {
    const Chunk ch = chunk_at(a, c);
    if (lane >= ch.count) continue;
    const int pidx = a.active_idx ? a.active_idx[ch.start + lane] : ch.start + lane;
    double s[3] = {0.0, 0.0, 0.0};
    for (int k = 0; k < nparts; ++k) {
      const double* v = (const double*)a.part_acc + ((int64_t)c * nparts + k) * (3 * kWarp) + lane;
#pragma unroll
      for (int d = 0; d < 3; ++d) s[d] += v[d * kWarp];
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) o[d * a.n + pidx] = scale * s[d];
  }
}

// The FP32 records are in the units of the positions where floats hold the box and, as normal
// numbers, 2^-26 of it: nearly always.  Else in units of the box's binary exponent.
double rel_unit(double box) {
  const int k = std::ilogb(box);
  return k >= -100 && k <= 120 ? 1.0 : std::ldexp(1.0, -k);
}

static Pair64Args pair64_args(const p3m_sr_ctx* ctx) {
  const p3m_sr_params& q = ctx->prm;
  const ForceConsts& f = ctx->fc;
  Pair64Args p{};
  p.tab = ctx->tab64;
  p.c = 1.0 / (4.0 * q.x_s * q.x_s);
  const int k = std::ilogb(q.box);
  p.len = std::ldexp(1.0, -k);
  p.bias = 0x38000000u + ((unsigned)(2 * k) << 20);
  p.c_f = (float)std::ldexp(p.c, 2 * k);
  p.xr2 = f.xr2_d;
  p.scale = -q.G_m;
  const double cut = q.x_r * (1.0 + 5e-5) * p.len;
  p.cut2 = (float)(cut * cut);
  double s_lo = 0.0;
  const double s_hi = p.c * f.xr2_d;
  double log_hi = s_hi;
  if (q.softening == P3M_SOFT_BSPLINE) {
    p.rsw2 = f.rsw2_d;
    const double near = (f.r_sw + 2e-5 * q.x_r) * p.len;
    p.near2 = (float)(near * near);
    s_lo = p.c * f.rsw2_d;
    const double eb = f.eps_b;
    const DD e2 = dd_prod(eb, eb), e3 = dd_mul(e2, DD{eb, 0.0});
    p.cb = 32.0 * dd_div(DD{1.0, 0.0}, e3).hi;
    p.cd = 32.0 * dd_div(DD{1.0, 0.0}, dd_mul(e3, e2)).hi;
    p.ieb = 1.0 / eb;
  } else if (q.softening == P3M_SOFT_PLUMMER) {
    p.ce2 = p.c * q.eps * q.eps;
    p.ce2_f = (float)p.ce2;
    s_lo = p.ce2;
    log_hi = s_hi + p.ce2;
  }
  // rows of [s_lo, log_hi], one more on each side for the rounding of the FP32 index
  const double lo2 = std::ldexp(1.0, kTabLogMinExp), hi2 = std::ldexp(1.0, kTabLogMaxExp);
  auto row_of = [&](double s) {
    int e;
    const double m = 2.0 * std::frexp(s, &e);  // s = m 2^(e - 1), m in [1, 2)
    return ((e - 1 - kTabLogMinExp) << kTabLogBits) + (int)((m - 1.0) * (1 << kTabLogBits));
  };
  p.rows = 2;  // at least two rows are there: a lookup outside the tables reads row 0 and drops the value
  if (s_lo < hi2 && log_hi > lo2) {
    const int first = std::max(0, row_of(std::max(s_lo, lo2)) - 1);
    const int last = std::min(kTabLogRows - 1, log_hi < hi2 ? row_of(log_hi) + 1 : kTabLogRows - 1);
    p.row0 = first & ~1;  // even: the copy to shared memory moves 16 bytes at a time
    p.rows = (last - p.row0 + 2) & ~1;
  }
  if (q.softening != P3M_SOFT_NONE) {
    const double u_hi = q.softening == P3M_SOFT_BSPLINE ? s_lo : s_hi;
    p.urows = std::min<int>(kTabUniRows, ((int)(std::min(u_hi, 8.0) * kTabUniPerUnit) + 3) & ~1);
  }
  return p;
}

p3m_status fill_pair_tables(p3m_sr_ctx* ctx) {
  const Pair64Args p = pair64_args(ctx);
  const int threads = p.rows + p.urows;
  static const SeriesDD series = make_series_dd();
  k_fill_tables<<<(threads + 31) / 32, 32, 0, ctx->stream>>>(series, ctx->tab64, ctx->prm.softening == P3M_SOFT_PLUMMER, p.row0,
                                                            p.rows, p.urows, p.c);
  ++ctx->launches;
  return cuda_check(ctx, cudaGetLastError(), "pair table kernel");
}

template <bool VJP, int SOFT>
static cudaError_t launch_pair64_soft(p3m_sr_ctx* ctx, TraversalArgs a) {
  const Pair64Args p = pair64_args(ctx);
  const size_t table = sizeof(double) * kTabRow * (size_t)(p.rows + p.urows) * (VJP ? 2 : 1);
  constexpr size_t kMaxShared = 227 * 1024;
  const int warps = (int)std::min<size_t>(kMaxWarps64, (kMaxShared - table) / sizeof(Warp64<VJP>));
  const size_t shm = table + (size_t)warps * sizeof(Warp64<VJP>);
  cudaError_t e = cudaFuncSetAttribute(k_pair64<VJP, SOFT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxShared);
  if (e != cudaSuccess) return e;
  const int slot = VJP ? 1 : 0;
  a.rel_scale = rel_unit(ctx->prm.box) == 1.0 ? (float)p.len : 1.0f;
  for (int d = 0; d < 3; ++d) a.g.side32[d] = (float)(a.g.side64[d] * p.len);
  a.f.margin2_f = (float)(p.len * p.len * (ctx->prm.x_r * ctx->prm.x_r * (1.0 + 1e-4)));
  a.part_acc = ctx->part_acc;
  a.part_items = ctx->part_items * 2 / 3;  // three doubles per lane in place of one float4
  cudaStream_t s = ctx->stream;
  cudaEventRecord(ctx->kt_ev[2 * slot], s);
  k_pair64<VJP, SOFT><<<(unsigned)ctx->num_sms, warps * kWarp, shm, s>>>(a, p);
  ++ctx->launches;
  cudaEventRecord(ctx->kt_ev[2 * slot + 1], s);
  ctx->kt_pending[slot] = true;
  k_parts_finish64<<<(unsigned)(ctx->num_sms * 4), 256, 0, s>>>(a, p.scale);
  ++ctx->launches;
  return cudaGetLastError();
}

cudaError_t launch_pair64(p3m_sr_ctx* ctx, const TraversalArgs& a, bool vjp) {
  switch (ctx->prm.softening) {
    case P3M_SOFT_NONE:
      return vjp ? launch_pair64_soft<true, P3M_SOFT_NONE>(ctx, a) : launch_pair64_soft<false, P3M_SOFT_NONE>(ctx, a);
    case P3M_SOFT_PLUMMER:
      return vjp ? launch_pair64_soft<true, P3M_SOFT_PLUMMER>(ctx, a)
                 : launch_pair64_soft<false, P3M_SOFT_PLUMMER>(ctx, a);
    default:
      return vjp ? launch_pair64_soft<true, P3M_SOFT_BSPLINE>(ctx, a)
                 : launch_pair64_soft<false, P3M_SOFT_BSPLINE>(ctx, a);
  }
}

}  // namespace p3m
