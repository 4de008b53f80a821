// Receiver work lists, the FP32 short-range pair-force kernels and their adjoints
// (VJP); the FP64 ones are in pair64.cu, and the traversal they share in traverse.cuh.
//
// Paper design (Section 2.1.3): tiles of side >= x_r, subtiles inside them,
// precomputed subtile pairings inside a "blocky ball" of radius x_r, a
// squared-distance rejection r^2 >= x_r^2 before the force, image shift n'
// known per subtile pair, particles stored in tile -> subtile -> particle
// order.  Receivers are the particles on active rungs (Section 2.2.2).
//
// GB300 design: the work unit is a receiver chunk -- up to 32 consecutive
// receivers of one row of tiles (spanning at most four tiles along z), one per
// warp lane.  A warp owns a chunk and:
//   1. builds the chunk's frame (origin: the subtile of its first receiver)
//      and the receivers' tight bounding box;
//   2. enumerates, 32 candidates at a time across the lanes, the subtiles of
//      the blocky ball around the chunk's subtile block (the paper's subtile
//      pairing generalised to a block of subtiles), keeps those whose box gap
//      to the bounding box is below x_r, and appends their particle ranges to
//      a per-warp list in shared memory;
//   3. walks the concatenated supplier ranges 32 at a time: each lane loads
//      one supplier j (FP32 coordinates relative to its subtile origin, moved
//      into the chunk frame by the integer subtile offset) and tests it against
//      the bounding box.
// The one-sided kernels stage the survivors in shared memory as packed pairs,
// and every lane evaluates its own receiver with two suppliers per step in f32x2
// arithmetic.  With every particle a receiver, the forward and the adjoint
// evaluate each pair once instead (k_force_sym, below).  Chunks are
// handed out through an atomic counter to persistent warps, which balances the
// strongly varying cost of clustered regions.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include <type_traits>

#include "erfcx_fit.h"
#include "traverse.cuh"

namespace p3m {

// Supplier subtiles buffered per warp before their particles are walked: 256
// measured best on the 128^3 and 512^3 sets (the one-sided kernel 4-8% faster than
// with 128, the each-pair-once kernel unchanged; 64 slower).
#ifndef P3M_LISTCAP
#define P3M_LISTCAP 256
#endif
constexpr int kListCap = P3M_LISTCAP;

static unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// ---------------------------------------------------------------------------
// Prologue kernels.
// ---------------------------------------------------------------------------

// FP32 coordinates relative to the particle's subtile origin, plus the id bits.
// All lanes of a warp reach the vote: launched with whole warps, lanes past n only vote.
// SCALED: times `scale`, a power of two (FP64 pairs of a box beyond the range of floats).
template <bool SCALED>
__global__ void k_rel4(const double* __restrict__ pos, const int* __restrict__ cell, int64_t n, Geometry g, double scale,
                       float4* __restrict__ rel4) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = i < n;
  int id = 0, gx = 0, gy = 0, gz = 0;
  double x = 0.0, y = 0.0, z = 0.0;
  if (valid) {
    id = cell[i];
    decode_subtile(g, id, gx, gy, gz);
    x = pos[i];
    y = pos[n + i];
    z = pos[2 * n + i];
  }
  double r[3];
  rel_to_subtile(g, x, y, z, gx, gy, gz, r);
  if constexpr (SCALED) {
#pragma unroll
    for (int d = 0; d < 3; ++d) r[d] *= scale;
    g.box *= scale;
  }
  float f[3] = {narrow(r[0]), narrow(r[1]), narrow(r[2])};
  // relative to the origin of the subtile of the last sort; a particle that drifted
  // across the periodic boundary since then takes its nearest image.  Its offset is
  // then near +-L, every other one far below L/2, so the test is made in FP32, and
  // only warps that hold such a particle spend FP64 operations on it.
  const float half = 0.5f * (float)g.box;
  const bool far = fabsf(f[0]) > half || fabsf(f[1]) > half || fabsf(f[2]) > half;
  if (__any_sync(0xffffffffu, far)) {
#pragma unroll
    for (int d = 0; d < 3; ++d)
      if (fabsf(f[d]) > half) {
        r[d] = f[d] > 0.0f ? __dsub_rn(r[d], g.box) : __dadd_rn(r[d], g.box);
        f[d] = (float)r[d];
      }
  }
  if (valid) rel4[i] = make_float4(f[0], f[1], f[2], __int_as_float(id));
}

// The receiver set in two passes over tiles of kActTile sorted particles: the number
// of receivers (rung >= rung_min) per tile, then (after a scan of those counts) each
// tile's flags, its exclusive scan act_scan[0..n] and the compacted receiver list.
constexpr int kActThreads = 256;
constexpr int kActItems = 16;
constexpr int kActTile = kActThreads * kActItems;

__global__ void __launch_bounds__(kActThreads) k_active_count(const int8_t* __restrict__ rung, int64_t n, int rung_min,
                                                              int* __restrict__ tile_count) {
  __shared__ int warp_sums[kActThreads / kWarp];
  const int64_t base = (int64_t)blockIdx.x * kActTile;
  int c = 0;
  for (int k = 0; k < kActItems; ++k) {
    const int64_t i = base + (int64_t)k * kActThreads + threadIdx.x;
    if (i < n) c += rung[i] >= rung_min ? 1 : 0;
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < kActThreads / kWarp; ++w) t += warp_sums[w];
    tile_count[blockIdx.x] = t;
  }
}

// flag and act_scan are 16-byte aligned (context arrays); rung is read as 16-byte
// vectors when it is too.
__global__ void __launch_bounds__(kActThreads) k_active_scan_compact(const int8_t* __restrict__ rung, int64_t n,
                                                                     int rung_min, const int* __restrict__ tile_base,
                                                                     int8_t* __restrict__ flag, int* __restrict__ act_scan,
                                                                     int* __restrict__ active_idx) {
  static_assert(kActItems == 16, "one 16-byte vector of rungs and flags per thread");
  __shared__ int warp_tot[kActThreads / kWarp];
  const int64_t base = (int64_t)blockIdx.x * kActTile + (int64_t)threadIdx.x * kActItems;  // 16 consecutive items
  const bool whole = base + kActItems <= n;
  int f[kActItems];
  int tot = 0;
  if (whole && ((reinterpret_cast<uintptr_t>(rung) & 15) == 0)) {
    const int4 v = *reinterpret_cast<const int4*>(rung + base);
    const int w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < kActItems; ++k) {
      const int r = (int)(int8_t)((w[k >> 2] >> (8 * (k & 3))) & 0xff);
      f[k] = r >= rung_min ? 1 : 0;
      tot += f[k];
    }
  } else {
#pragma unroll
    for (int k = 0; k < kActItems; ++k) {
      const int64_t i = base + k;
      f[k] = (i < n && rung[i] >= rung_min) ? 1 : 0;
      tot += f[k];
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = tot;
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  int run = inc - tot + tile_base[blockIdx.x];
  for (int w = 0; w < warp; ++w) run += warp_tot[w];
  if (whole) {  // vector stores: 16 flags, then 16 scan values as four int4
    int fw[4] = {0, 0, 0, 0};
    int sc[kActItems];
#pragma unroll
    for (int k = 0; k < kActItems; ++k) {
      fw[k >> 2] |= f[k] << (8 * (k & 3));
      sc[k] = run;
      if (f[k]) active_idx[run] = (int)(base + k);
      run += f[k];
    }
    *reinterpret_cast<int4*>(flag + base) = make_int4(fw[0], fw[1], fw[2], fw[3]);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      reinterpret_cast<int4*>(act_scan + base)[q] = make_int4(sc[4 * q], sc[4 * q + 1], sc[4 * q + 2], sc[4 * q + 3]);
  } else {
#pragma unroll
    for (int k = 0; k < kActItems; ++k) {
      const int64_t i = base + k;
      if (i <= n) act_scan[i] = run;
      if (i < n) {
        flag[i] = (int8_t)f[k];
        if (f[k]) active_idx[run] = (int)i;
      }
      run += f[k];
    }
  }
}

// Receiver chunks.  The receivers of one row of tiles (fixed tile x, y) are
// consecutive in the sorted order.  Each row is cut into segments of
// kChunkSpan consecutive tiles along z, and the receivers of a segment into
// ceil(count / 32) chunks, so that sparse tiles share a warp while every chunk
// stays spatially compact.  One thread per segment: no sequential walk.
#ifndef P3M_CHUNK_SPAN
#define P3M_CHUNK_SPAN 4
#endif
constexpr int kChunkSpan = P3M_CHUNK_SPAN;

__device__ __forceinline__ int tile_start(const int* __restrict__ offsets, const int* __restrict__ act_scan, int nsub3,
                                          int64_t T) {
  int p = offsets[T * nsub3];
  return act_scan ? act_scan[p] : p;
}

// Receiver range [a0, a1) of segment `seg` (row-major over rows, then segments).
__device__ __forceinline__ void segment_range(const int* __restrict__ offsets, const int* __restrict__ act_scan,
                                              int nsub3, int n_t, int64_t seg, int& a0, int& a1) {
  const int nseg = (n_t + kChunkSpan - 1) / kChunkSpan;
  const int64_t row = seg / nseg;
  const int k = (int)(seg - row * nseg);
  const int64_t t0 = row * n_t + (int64_t)k * kChunkSpan;
  const int64_t t1 = row * n_t + min(n_t, (k + 1) * kChunkSpan);
  a0 = tile_start(offsets, act_scan, nsub3, t0);
  a1 = tile_start(offsets, act_scan, nsub3, t1);
}

// The chunk list in one launch: each block takes 256 segments, scans their chunk counts and
// reserves its part of the list with one atomic, so blocks follow one another in the order in
// which they finish counting.  That is nearly the order of the segments (neighbouring chunks
// share suppliers in L2), and nothing but that locality depends on it.  The last block to
// finish publishes the count and clears the two work words, which are zero between launches.
// (Counts, their scan in one or two launches and the list took 4 launches, 17 us at 128^3.)
constexpr int kSegThreads = 256;
__global__ void __launch_bounds__(kSegThreads) k_build_chunks(const int* __restrict__ offsets,
                                                              const int* __restrict__ act_scan, int n_t, int nsub3,
                                                              Chunk* __restrict__ chunks, int* work,
                                                              int* __restrict__ n_chunks_out,
                                                              int* __restrict__ n_active_out, int64_t n) {
  __shared__ int warp_tot[kSegThreads / kWarp];
  __shared__ int base;
  const int64_t seg = (int64_t)blockIdx.x * kSegThreads + threadIdx.x;
  const int64_t nsegs = (int64_t)n_t * n_t * ((n_t + kChunkSpan - 1) / kChunkSpan);
  int a0 = 0, a1 = 0;
  if (seg < nsegs) segment_range(offsets, act_scan, nsub3, n_t, seg, a0, a1);
  const int c = (a1 - a0 + kChunk - 1) / kChunk;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = c;
  for (int o = 1; o < kWarp; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == kWarp - 1) warp_tot[warp] = inc;
  __syncthreads();
  int at = inc - c;
  for (int w = 0; w < warp; ++w) at += warp_tot[w];
  if (threadIdx.x == kSegThreads - 1) {
    base = atomicAdd(&work[0], at + c);
    __threadfence();
    if (atomicAdd(&work[1], 1) == (int)gridDim.x - 1) {
      __threadfence();
      *n_chunks_out = atomicExch(&work[0], 0);
      work[1] = 0;
      if (n_active_out) *n_active_out = act_scan ? act_scan[n] : (int)n;
    }
  }
  __syncthreads();
  Chunk* out = chunks + base + at;
  for (int k = 0; k < c; ++k) {
    const int s0 = a0 + k * kChunk;
    out[k] = Chunk{s0, min(kChunk, a1 - s0)};
  }
}

// Masked abar for the VJP: abar_i * [i active].
__global__ void k_abar_f32(const float* __restrict__ abar, const int8_t* __restrict__ flag, int all_active,
                           int64_t n, float4* __restrict__ out) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float m = (all_active || flag[i]) ? 1.0f : 0.0f;
  out[i] = make_float4(abar[i] * m, abar[n + i] * m, abar[2 * n + i] * m, 0.0f);
}

__global__ void k_abar_f64(const double* __restrict__ abar, const int8_t* __restrict__ flag, int all_active,
                           int64_t n, double* __restrict__ out) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double m = (all_active || flag[i]) ? 1.0 : 0.0;
  out[i] = abar[i] * m;
  out[n + i] = abar[n + i] * m;
  out[2 * n + i] = abar[2 * n + i] * m;
}

// ---------------------------------------------------------------------------
// FP32 kernels (the traversal they share with the FP64 ones is in traverse.cuh).
// ---------------------------------------------------------------------------

using WarpList = WarpListOf<kListCap>;

// Supplier number f of the list (lane-parallel): its position in the chunk frame and
// its masked abar.  Returns whether it can reach the receivers' bounding box.
__device__ __forceinline__ bool load_supplier(const TraversalArgs& a, const WarpList& L, int nlist, int f,
                                              const ChunkFrame& F, Vec3<float>& pj, Vec3<float>& aj, float* gap2_out) {
  int lo_e = 0, hi_e = nlist - 1;  // last entry with pre <= f
  while (lo_e < hi_e) {
    int mid = (lo_e + hi_e + 1) >> 1;
    if (L.pre[mid] <= f) lo_e = mid; else hi_e = mid - 1;
  }
  int j = L.start[lo_e] + (f - L.pre[lo_e]);
  int dx, dy, dz;
  unpack_delta(L.delta[lo_e], dx, dy, dz);
  float4 r = a.rel4[j];
  pj.x = fmaf((float)dx, a.g.side32[0], r.x);
  pj.y = fmaf((float)dy, a.g.side32[1], r.y);
  pj.z = fmaf((float)dz, a.g.side32[2], r.z);
  float4 q = a.abar4[j];
  aj.x = q.x; aj.y = q.y; aj.z = q.z;
  const float gap2 = box_gap2(F, pj);
  *gap2_out = gap2;
  return gap2 < a.f.margin2_f;
}

__device__ __forceinline__ void store_result(const TraversalArgs& a, const ChunkFrame& F, const Vec3<float>& acc) {
  if (!F.valid) return;
  const float s = -(float)a.f.G_m;
  float* o = (float*)a.out;
  o[F.pidx] = s * acc.x;
  o[a.n + F.pidx] = s * acc.y;
  o[2 * a.n + F.pidx] = s * acc.z;
}

// ---------------------------------------------------------------------------
// FP32 forward, one-sided: 32 receivers per warp, every surviving supplier tested
// by all lanes; the survivors of a batch are staged, compacted and negated, in shared memory
// as packed pairs, read back with broadcast loads, and two suppliers are
// evaluated per step in f32x2 arithmetic.
// ---------------------------------------------------------------------------

constexpr int kPThreads = 128;
constexpr int kPWarps = kPThreads / kWarp;
constexpr float kR2Floor = 1e-24f;    // added to r^2 in the packed forward kernel
constexpr float kR2Self = 1e-23f;     // r^2 below this: a zero displacement
constexpr float kCutScale = 0x1p64f;  // cutoff mask: sat((x_r^2 - r^2) 2^64)

// saturate(a * b + c) in one FP32 instruction
__device__ __forceinline__ float fma_sat(float a, float b, float c) {
  float d;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Survivors staged before they are evaluated: more than one batch of 32, so that the loop is
// entered, and its last pair padded, half as often (against 32: 2 M particles all active 1.794
// -> 1.773 ms, a third 0.917 -> 0.907, tabulated 1.474 -> 1.432; 96: no more).
constexpr int kGpStage = 64;
struct PackedSmem {
  WarpList L;
  float4 sxy[kGpStage / 2 + 1];  // (-xa, -xb, -ya, -yb)
  float2 sz[kGpStage / 2 + 1];   // (-za, -zb)
  float4 rec[2][kWarp];          // records of the current and the next batch, by cp.async as in k_force_sym
};

// 7 resident blocks of 4 warps per SM bound the kernel to 70 registers (no
// spills); with the cp.async staging measured best among 5 to 8 on the state of the
// 128^3 set after 25 benchmark steps (deep-rung substep 3% faster than with 6).
#ifndef P3M_GP_UNROLL
#define P3M_GP_UNROLL 2  // supplier pairs per loop iteration (2: 2-3% faster than 1 on the 128^3 set)
#endif
constexpr int kGpUnroll = P3M_GP_UNROLL;
#ifndef P3M_GP_MINBLOCKS
#define P3M_GP_MINBLOCKS 7
#endif

template <int SOFT, bool TABLE = false>
__global__ void __launch_bounds__(kPThreads, P3M_GP_MINBLOCKS) k_force_packed(TraversalArgs a) {
  __shared__ PackedSmem smem[kPWarps];
  extern __shared__ float tab[];  // TABLE: the bracket table (n_table floats)
  if (TABLE) {
    for (int i = threadIdx.x; i < a.n_table; i += blockDim.x) tab[i] = a.table[i];
    __syncthreads();
  }

  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  PackedSmem& S = smem[threadIdx.x >> 5];
  const int n_chunks = *a.n_chunks;
  const int nparts = a.part_acc ? parts_for(n_chunks, a.part_items, kMaxParts) : 1;
  const int n_items = n_chunks * nparts;
  const Reach rc = make_reach(a);
  const float xr2 = a.f.xr2_f;
  const float xr2s = xr2 * kCutScale;
  unsigned long long pair_total = 0;
  for (;;) {
    const int w = next_chunk(a, lane);
    if (w >= n_items) break;
    const int c = w / nparts, part = w - c * nparts;
    ChunkFrame F;
    load_chunk(a, rc, chunk_at(a, c), lane, F);
    const f2 px = pk(F.pi.x, F.pi.x), py = pk(F.pi.y, F.pi.y), pz = pk(F.pi.z, F.pi.z);
    f2 ax = pk(0.f, 0.f), ay = pk(0.f, 0.f), az = pk(0.f, 0.f);
    f2 hitsf = pk(0.f, 0.f);  // interacting pairs of this lane (exact integers in FP32)
    float* sxy = (float*)S.sxy;
    float* sz = (float*)S.sz;
    int cnt = 0;            // staged survivors (warp-uniform)
    bool blk_near = false;  // one of them is near the box
    auto evaluate = [&] {
        if (lane == 0 && (cnt & 1)) {  // pad the last pair far from every receiver (finite B there)
          const int p = cnt >> 1;
          sxy[4 * p + 1] = 1e10f;
          sxy[4 * p + 3] = 1e10f;
          sz[2 * p + 1] = 1e10f;
        }
        __syncwarp();
        const int npairs = (cnt + 1) >> 1;
        // Batches with no supplier within r_sw of the receivers' box run a loop
        // without the softened-branch test (a vote and a branch per step).
        auto run_pairs = [&](auto check_soft) {
          constexpr bool kCheckSoft = decltype(check_soft)::value;
#pragma unroll kGpUnroll
        for (int p = 0; p < npairs; ++p) {
          const float4 s = S.sxy[p];
          const float2 z = S.sz[p];
          const f2 dx = add2(px, pk(s.x, s.y));
          const f2 dy = add2(py, pk(s.z, s.w));
          const f2 dz = add2(pz, pk(z.x, z.y));
          // r^2 + 1e-24: a zero displacement (the receiver itself, coincident
          // particles) gets a large but finite B and contributes B * 0 = 0; the
          // offset is far below one ulp of the r^2 near the cutoff, and below the
          // square of the smallest non-zero displacement of subtile-relative FP32
          // coordinates, so no cutoff decision changes
          const f2 r2 = fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, pk(kR2Floor, kR2Floor))));
          float q0, q1;
          upk(r2, q0, q1);
          const bool h0 = q0 < xr2, h1 = q1 < xr2;
          if (__any_sync(full, h0 || h1)) {
            // cutoff mask in the FP32 pipe: 1 iff r^2 < x_r^2 (exact: the scale is a power of two)
            const f2 c = pk(fma_sat(q0, -kCutScale, xr2s), fma_sat(q1, -kCutScale, xr2s));
            hitsf = add2(hitsf, c);
            f2 B;
            if (TABLE) {  // nearest-grid-point lookup in r^2 (softening included)
              const int i0 = min((int)(fminf(q0, a.f.xr2_f) * a.table_scale), a.n_table - 1);
              const int i1 = min((int)(fminf(q1, a.f.xr2_f) * a.table_scale), a.n_table - 1);
              B = pk(tab[max(i0, 0)], tab[max(i1, 0)]);
            } else {
              B = bracket_main_f32x2<SOFT>(r2, a.f);
              if (kCheckSoft) {
                const bool rare0 = h0 && (q0 < a.f.rsw2_f) && (q0 > kR2Self);
                const bool rare1 = h1 && (q1 < a.f.rsw2_f) && (q1 > kR2Self);
                if (__any_sync(full, rare0 || rare1)) {
                  float b0, b1, s0, s1;
                  upk(B, b0, b1);
                  upk(bracket_soft_f32x2<SOFT>(r2, a.f, a.sc), s0, s1);
                  if (rare0) b0 = s0;
                  if (rare1) b1 = s1;
                  B = pk(b0, b1);
                }
              }
            }
            B = mul2(B, c);
            ax = fma2(B, dx, ax);
            ay = fma2(B, dy, ay);
            az = fma2(B, dz, az);
          }
        }
        };
        if (TABLE || blk_near) run_pairs(std::true_type{});
        else run_pairs(std::false_type{});
        __syncwarp();
        cnt = 0;
        blk_near = false;
    };
    enumerate_strided(a, rc, F, S.L, lane, part, nparts, [&](int nlist, int total) {
      const WarpList& L = S.L;
      ListCursor<WarpList> cur;
      auto locate = [&](int b, int& j, unsigned& dpk) { return cur.locate(L, nlist, total, lane, b, j, dpk); };
      // software pipeline: the record of batch b + 32 is loaded while batch b is evaluated
      int jn;
      unsigned dn;
      bool vn = locate(0, jn, dn);
      int buf = 0;
      if (vn) cp_async16(&S.rec[0][lane], a.rel4 + jn);
      cp_async_commit();
      for (int b = 0; b < total; b += kWarp) {
        const bool have = vn;
        const unsigned dpk = dn;
        vn = (b + kWarp < total) ? locate(b + kWarp, jn, dn) : false;
        if (vn) cp_async16(&S.rec[buf ^ 1][lane], a.rel4 + jn);
        cp_async_commit();
        cp_async_wait_prev();  // this lane's copy of batch b has landed
        const float4 r = have ? S.rec[buf][lane] : make_float4(0.f, 0.f, 0.f, 0.f);
        buf ^= 1;
        bool keep = false, near = false;
        Vec3<float> pj = {0.f, 0.f, 0.f};
        if (have) {
          int dx, dy, dz;
          unpack_delta(dpk, dx, dy, dz);
          pj.x = fmaf((float)dx, a.g.side32[0], r.x);
          pj.y = fmaf((float)dy, a.g.side32[1], r.y);
          pj.z = fmaf((float)dz, a.g.side32[2], r.z);
          const float tx = fmaxf(fmaxf(F.lo.x - pj.x, pj.x - F.hi.x), 0.f);
          const float ty = fmaxf(fmaxf(F.lo.y - pj.y, pj.y - F.hi.y), 0.f);
          const float tz = fmaxf(fmaxf(F.lo.z - pj.z, pj.z - F.hi.z), 0.f);
          const float gap2 = fmaf(tx, tx, fmaf(ty, ty, tz * tz));
          keep = gap2 < a.f.margin2_f;
          // can this supplier come closer than r_sw to some receiver?  (the box gap
          // is a lower bound of every receiver distance)
          near = keep && gap2 < a.f.rsw2_f;
        }
        const unsigned m = __ballot_sync(full, keep);
        const int nsurv = __popc(m);
        if (keep) {
          const int k = cnt + __popc(m & ((1u << lane) - 1u));
          const int p = k >> 1, h = k & 1;
          sxy[4 * p + h] = -pj.x;
          sxy[4 * p + 2 + h] = -pj.y;
          sz[2 * p + h] = -pj.z;
        }
        cnt += nsurv;
        blk_near |= __any_sync(full, near);
        if (cnt > kGpStage - kWarp) evaluate();  // the next batch might not fit
      }
    });
    if (cnt > 0) evaluate();
    Vec3<float> acc;
    float l, h;
    upk(ax, l, h);
    acc.x = l + h;
    upk(ay, l, h);
    acc.y = l + h;
    upk(az, l, h);
    acc.z = l + h;
    if (nparts == 1) store_result(a, F, acc);
    else a.part_acc[(int64_t)w * kWarp + lane] = make_float4(acc.x, acc.y, acc.z, 0.f);
    upk(hitsf, l, h);
    // the receiver met itself once (r = 0), in the part that holds its own subtile; every
    // part counts its hits, and part 0 takes off one per receiver
    const int hits = F.valid ? (int)(l + h) - (part == 0 ? 1 : 0) : 0;
    // signed: a part-0 lane whose own subtile lies in another part counts -1; the sum
    // over a chunk's parts is exact, and the 64-bit total wraps back
    pair_total += (unsigned long long)(long long)__reduce_add_sync(full, hits);
  }
  if (lane == 0 && pair_total) atomicAdd(a.pairs, pair_total);
}

// acc = -G m (sum of the parts of each chunk, in part order), when k_force_packed
// split its chunks (nothing to do otherwise).  One warp per chunk position.
__global__ void k_parts_finish(TraversalArgs a) {
  const int n_chunks = *a.n_chunks;
  const int nparts = parts_for(n_chunks, a.part_items, kMaxParts);
  if (nparts == 1) return;
  const int lane = threadIdx.x & 31;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  const float s = -(float)a.f.G_m;
  float* o = (float*)a.out;
  for (int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < n_chunks; c += nw) {
    const Chunk ch = chunk_at(a, c);
    if (lane >= ch.count) continue;
    const int pidx = a.active_idx ? a.active_idx[ch.start + lane] : ch.start + lane;
    float x = 0.f, y = 0.f, z = 0.f;
    for (int k = 0; k < nparts; ++k) {
      const float4 v = a.part_acc[((int64_t)c * nparts + k) * kWarp + lane];
      x += v.x;
      y += v.y;
      z += v.z;
    }
    o[pidx] = s * x;
    o[a.n + pidx] = s * y;
    o[2 * a.n + pidx] = s * z;
  }
}

// ---------------------------------------------------------------------------
// FP32 kernel with Newton's third law: the forward of calls in which every particle
// is a receiver, and the adjoint (VJP).  The paper pairs two neighbouring tiles only
// once and updates the particles of both (Section 2.1.3); here each unordered pair
// {i, j} of sorted indices i < j is evaluated once, by the chunk that holds i, and
// both particles receive their share.  The chunk's own pairs come first, in a
// triangular pass (lane l with lanes l + k and l + k + 8); its supplier ranges are
// then cut to the indices past its last receiver.
//
// The survivors of the box test are staged 64 at a time as 32 packed pairs.  Each half
// of the warp holds all 32 receivers, two per lane (l and l + 16), and takes half of
// the pairs: P of them (a power of two <= 16) in P steps.  At step k lane l of a group
// of P lanes evaluates its two receivers against pair (l + k) mod P, so that every
// receiver meets every pair once and no two lanes of a group touch one supplier at the
// same time; each pair's accumulator travels with it from lane to lane by warp
// shuffles.  At the end of the block the groups' partial sums are reduced and added,
// like the receivers' own sums at the end of the chunk, into an FP32 float4 array with
// vector atomics.  k_sym_finish scales that array into the caller's 3 x n output.
// Pairs closer than r_sw (the softened form) are evaluated in the step: when some lane
// holds one, one packed softened evaluation serves both halves of a pair and each half
// selects its form.
//
// Bound: issue slots and the FP32 pipe (0.385 of the evaluated slots interact).  The
// rotation's fixed cost, 6 shuffles, 2 shared loads and the loop, is paid per step, so a
// step carries four (receiver, supplier) slots per lane instead of two: at 128^3 (654 M
// ordered pairs) the forward took 1.28 instead of 1.36 ms and the adjoint 1.82 instead of
// 1.96, and with the tile columns before the chunk's own cut off 1.25 and 1.79 ms (1.05 G
// warp instructions instead of 1.22, the FP32 pipe 60% busy).
// ---------------------------------------------------------------------------

constexpr float kSymPad = 1e10f;  // padding supplier at -1e10, invalid receiver at +1e10: finite B, no hit

struct SymSmem {
  WarpList L;
  float4 sxy[kWarp];  // pair q: (-x_a, -x_b, -y_a, -y_b) of suppliers a and b
  float2 sz[kWarp];   // (-z_a, -z_b)
  int2 sj[kWarp];     // (j_a, j_b): sorted indices, -1 for padding
  // records of the current and the next batch, copied with cp.async while the current
  // batch is staged (measured at 128^3 against a register prefetch: 1.551 -> 1.518 ms)
  float4 rec[2][kWarp];
};

struct SymVjpSmem : SymSmem {
  float4 vxy[kWarp];  // adjoint: the suppliers' masked abar, negated, in the layout of sxy / sz
  float2 vz[kWarp];
};

// Resident blocks of 4 warps per SM: 5 for the forward (94 to 96 registers; 4 or 6 are 1-2%
// slower at 128^3), 4 for the adjoint (122 to 128 registers; 5: 1% slower).
constexpr int kSymMinBlocks = 5;
constexpr int kSymVjpMinBlocks = 4;
// Chunks are split into parts (slices of equal supplier counts) up to about three work items
// per resident warp: forward of 4096 particles (155 chunks) 0.090 ms unsplit, 0.026 in 16
// parts; 32,768 (1181) 0.115 -> 0.055 in 8 (13: 0.067); 110,000 (4161) 0.139 -> 0.118 in 3;
// from 262,144 (9562) on no gain, each part enumerating the chunk's candidates again.
constexpr int kSymItems = 9120;
constexpr int kSymMaxParts = 16;

__device__ __forceinline__ f2 shfl2(f2 v, int src) {
  f2 r;
  r.v = __shfl_sync(0xffffffffu, v.v, src);
  return r;
}
__device__ __forceinline__ f2 shfl_xor2(f2 v, int o) {
  f2 r;
  r.v = __shfl_xor_sync(0xffffffffu, v.v, o);
  return r;
}

struct F2x3 {
  f2 x, y, z;
};
__device__ __forceinline__ F2x3 dup3(float x, float y, float z) { return F2x3{pk(x, x), pk(y, y), pk(z, z)}; }
__device__ __forceinline__ F2x3 sub3(const F2x3& p, const float4& xy, const float2& z) {  // p - s, s stored negated
  return F2x3{add2(p.x, pk(xy.x, xy.y)), add2(p.y, pk(xy.z, xy.w)), add2(p.z, pk(z.x, z.y))};
}
// The force term B d, or the adjoint's B v + D (d . v) d, added to a.
template <bool VJP>
__device__ __forceinline__ void add_term(F2x3& a, f2 B, const F2x3& d, const F2x3& v, f2 cc) {
  if constexpr (!VJP) {
    a.x = fma2(B, d.x, a.x);
    a.y = fma2(B, d.y, a.y);
    a.z = fma2(B, d.z, a.z);
  } else {
    a.x = fma2(B, v.x, fma2(cc, d.x, a.x));
    a.y = fma2(B, v.y, fma2(cc, d.y, a.y));
    a.z = fma2(B, v.z, fma2(cc, d.z, a.z));
  }
}

// Bracket (VJP: with D = B'(r)/r) of the packed pair at squared distances r2, 0 unless its
// cutoff mask c is 1 and where `coincident` pairs do not count; check: test for close pairs.
template <int SOFT, bool VJP>
__device__ __forceinline__ f2 masked_bracket(f2 r2, f2 c, bool check, const TraversalArgs& a, f2& D) {
  f2 B;
  if constexpr (VJP) B = bracket_main_vjp_f32x2<SOFT>(r2, a.f, D);
  else B = bracket_main_f32x2<SOFT>(r2, a.f);
  float q0, q1, c0, c1;
  upk(r2, q0, q1);
  upk(c, c0, c1);
  if (check) {
    // the softened form; in the forward a zero displacement contributes nothing (its
    // floored r^2 gives a finite B, times 0), in the adjoint coincident particles take B(0)
    const bool rare0 = c0 > 0.f && q0 < a.f.rsw2_f && (VJP || q0 > kR2Self);
    const bool rare1 = c1 > 0.f && q1 < a.f.rsw2_f && (VJP || q1 > kR2Self);
    if (__any_sync(0xffffffffu, rare0 || rare1)) {
      float b0, b1, s0, s1;
      upk(B, b0, b1);
      if constexpr (VJP) {
        f2 Ds;
        float d0, d1, e0, e1;
        upk(D, d0, d1);
        upk(bracket_soft_vjp_f32x2<SOFT>(r2, a.f, a.sc, Ds), s0, s1);
        upk(Ds, e0, e1);
        D = pk(rare0 ? e0 : d0, rare1 ? e1 : d1);
      } else {
        upk(bracket_soft_f32x2<SOFT>(r2, a.f, a.sc), s0, s1);
      }
      B = pk(rare0 ? s0 : b0, rare1 ? s1 : b1);
    }
  }
  if constexpr (VJP) D = mul2(D, c);
  return mul2(B, c);
}

// VJP = true: the adjoint with the same traversal.  Its pair term J_ij (v_i - v_j),
// v the masked abar, is antisymmetric in (i, j) like the force, so the partner
// receives the negated term; every particle is a receiver.
template <int SOFT, bool VJP = false>
__global__ void __launch_bounds__(kPThreads, VJP ? kSymVjpMinBlocks : kSymMinBlocks)
    k_force_sym(TraversalArgs a, float4* __restrict__ acc4) {
  using Smem = typename std::conditional<VJP, SymVjpSmem, SymSmem>::type;
  __shared__ Smem smem[kPWarps];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  Smem& S = smem[threadIdx.x >> 5];
  float* sxy = (float*)S.sxy;
  float* szf = (float*)S.sz;
  int* sjf = (int*)S.sj;
  float* vxy = nullptr;
  float* vzf = nullptr;
  if constexpr (VJP) {
    vxy = (float*)S.vxy;
    vzf = (float*)S.vz;
  }
  const int n_chunks = *a.n_chunks;
  const int nparts = parts_for(n_chunks, kSymItems + n_chunks - 1, kSymMaxParts);
  const int n_items = n_chunks * nparts;
  const Reach rc = make_reach(a);
  const float xr2 = a.f.xr2_f;
  const float xr2s = xr2 * kCutScale;
  unsigned long long pair_total = 0;
  for (;;) {
    const int w = next_chunk(a, lane);
    if (w >= n_items) break;
    const int ci = w / nparts, part = w - ci * nparts;
    const Chunk ch = chunk_at(a, ci);
    ChunkFrame F;
    load_chunk(a, rc, ch, lane, F);
    {  // subtile planes along x that hold only smaller indices: the tile columns before the chunk's own
      const int below = quot_small(F.g0[0], a.g.ns[0], a.g.inv_ns[0]) * a.g.ns[0] - F.g0[0] - F.elo[0];
      if (below > 0 && F.g0[0] + F.elo[0] >= 0) {  // (those before column 0 wrap round to the last ones)
        F.elo[0] += below;
        F.ext[0] -= below;
      }
    }
    const float rx = F.valid ? F.pi.x : kSymPad, ry = F.valid ? F.pi.y : kSymPad, rz = F.valid ? F.pi.z : kSymPad;
    float4 ab = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (VJP) {
      if (F.valid) ab = a.abar4[F.pidx];
    }
    const f2 zero = pk(0.f, 0.f);
    F2x3 own = {zero, zero, zero};  // sums of this lane's own receiver
    f2 hitsf = zero;
    const f2 floor2 = VJP ? zero : pk(kR2Floor, kR2Floor);

    // The chunk's own pairs: lane l with lanes l + k and l + k + 8, k = 1 ... 8 (l + 16 from
    // the lower half only), each pair {i, j} of the chunk once; the partner's share comes
    // back by a shuffle.
    if (part == 0) {
      const F2x3 p = dup3(rx, ry, rz);
#pragma unroll 1
      for (int k = 1; k <= 8; ++k) {
        const int m = (lane + k) & (kWarp - 1), m2 = (lane + k + 8) & (kWarp - 1);
        const F2x3 d = {add2(p.x, pk(-__shfl_sync(full, rx, m), -__shfl_sync(full, rx, m2))),
                        add2(p.y, pk(-__shfl_sync(full, ry, m), -__shfl_sync(full, ry, m2))),
                        add2(p.z, pk(-__shfl_sync(full, rz, m), -__shfl_sync(full, rz, m2)))};
        const f2 r2 = fma2(d.x, d.x, fma2(d.y, d.y, fma2(d.z, d.z, floor2)));
        float q0, q1;
        upk(r2, q0, q1);
        const bool t0 = F.valid && m < ch.count, t1 = F.valid && m2 < ch.count && (k < 8 || lane < kWarp / 2);
        const float c0 = t0 ? fma_sat(q0, -kCutScale, xr2s) : 0.f, c1 = t1 ? fma_sat(q1, -kCutScale, xr2s) : 0.f;
        hitsf = add2(hitsf, pk(c0, c1));
        f2 D = zero;
        f2 B = masked_bracket<SOFT, VJP>(r2, pk(c0, c1), true, a, D);
        float b0, b1;
        upk(B, b0, b1);
        B = pk(c0 > 0.f ? b0 : 0.f, c1 > 0.f ? b1 : 0.f);  // selects: a padded lane's B may not be finite
        F2x3 v = {zero, zero, zero};
        f2 cc = zero;
        if constexpr (VJP) {
          float d0, d1;
          upk(D, d0, d1);
          D = pk(c0 > 0.f ? d0 : 0.f, c1 > 0.f ? d1 : 0.f);
          v = {pk(ab.x - __shfl_sync(full, ab.x, m), ab.x - __shfl_sync(full, ab.x, m2)),
               pk(ab.y - __shfl_sync(full, ab.y, m), ab.y - __shfl_sync(full, ab.y, m2)),
               pk(ab.z - __shfl_sync(full, ab.z, m), ab.z - __shfl_sync(full, ab.z, m2))};
          cc = mul2(D, fma2(d.x, v.x, fma2(d.y, v.y, mul2(d.z, v.z))));
        }
        F2x3 t = {zero, zero, zero};
        add_term<VJP>(t, B, d, v, cc);
        const int from = (lane - k) & (kWarp - 1), from2 = (lane - k - 8) & (kWarp - 1);
        auto give = [&](f2& o, f2 u) {
          float lo, hi;
          upk(u, lo, hi);
          o = add2(o, add2(u, pk(-__shfl_sync(full, lo, from), -__shfl_sync(full, hi, from2))));
        };
        give(own.x, t.x);
        give(own.y, t.y);
        give(own.z, t.z);
      }
    }

    // Receivers of the rotation: l and l + 16 of the chunk, in both halves of the warp.
    const int l16 = lane & 15;
    const F2x3 pA = dup3(__shfl_sync(full, rx, l16), __shfl_sync(full, ry, l16), __shfl_sync(full, rz, l16));
    const F2x3 pB = dup3(__shfl_sync(full, rx, l16 + 16), __shfl_sync(full, ry, l16 + 16), __shfl_sync(full, rz, l16 + 16));
    F2x3 vA = {zero, zero, zero}, vB = vA;
    if constexpr (VJP) {
      vA = dup3(__shfl_sync(full, ab.x, l16), __shfl_sync(full, ab.y, l16), __shfl_sync(full, ab.z, l16));
      vB = dup3(__shfl_sync(full, ab.x, l16 + 16), __shfl_sync(full, ab.y, l16 + 16), __shfl_sync(full, ab.z, l16 + 16));
    }
    F2x3 aA = {zero, zero, zero}, aB = aA;
    int cnt = 0;            // staged suppliers (warp-uniform)
    bool blk_near = false;  // the staged block holds a supplier near the box

    auto stage = [&](int rank, const Vec3<float>& pj, int j, const float4& aj) {
      const int q = rank & (kWarp - 1), h = rank >> 5;
      sxy[4 * q + h] = -pj.x;
      sxy[4 * q + 2 + h] = -pj.y;
      szf[2 * q + h] = -pj.z;
      sjf[2 * q + h] = j;
      if constexpr (VJP) {
        vxy[4 * q + h] = -aj.x;
        vxy[4 * q + 2 + h] = -aj.y;
        vzf[2 * q + h] = -aj.z;
      }
    };
    auto pad = [&](int q, int h) {
      sxy[4 * q + h] = kSymPad;
      sxy[4 * q + 2 + h] = kSymPad;
      szf[2 * q + h] = kSymPad;
      sjf[2 * q + h] = -1;
      if constexpr (VJP) {
        vxy[4 * q + h] = 0.f;
        vxy[4 * q + 2 + h] = 0.f;
        vzf[2 * q + h] = 0.f;
      }
    };

    // Evaluate the staged block of nsup suppliers (1 <= nsup <= 64) against the chunk.
    auto eval_block = [&](int nsup) {
      int P = kWarp / 2;  // pairs of each half of the warp
      if (nsup < 2 * kWarp) {
        const int pairs = (nsup + 1) >> 1;
        P = 1;
        while (2 * P < pairs) P <<= 1;
        // pair q = (supplier q, supplier q + 2 P): move q + 2 P < 32 from the a halves to the b halves
        if (nsup <= kWarp && lane >= 2 * P && lane < nsup) {
          const int q = lane - 2 * P;
          sxy[4 * q + 1] = sxy[4 * lane];
          sxy[4 * q + 3] = sxy[4 * lane + 2];
          szf[2 * q + 1] = szf[2 * lane];
          sjf[2 * q + 1] = sjf[2 * lane];
          if constexpr (VJP) {
            vxy[4 * q + 1] = vxy[4 * lane];
            vxy[4 * q + 3] = vxy[4 * lane + 2];
            vzf[2 * q + 1] = vzf[2 * lane];
          }
        }
        if (lane < 2 * P && lane + 2 * P >= nsup) pad(lane, 1);
        if (lane < 2 * P && lane >= nsup) pad(lane, 0);
        __syncwarp();
      }
      const int pmask = P - 1, base = (lane >> 4) * P;
      const int src = (lane & ~pmask) | ((lane + 1) & pmask);
      F2x3 sa = {zero, zero, zero};
      int q = lane & pmask;
      auto run = [&](auto check_soft) {
        constexpr bool kCheckSoft = decltype(check_soft)::value;
#pragma unroll 1
        for (int k = 0; k < P; ++k) {
          const float4 s = S.sxy[base + q];
          const float2 z = S.sz[base + q];
          const F2x3 dA = sub3(pA, s, z), dB = sub3(pB, s, z);
          const f2 rA = fma2(dA.x, dA.x, fma2(dA.y, dA.y, fma2(dA.z, dA.z, floor2)));
          const f2 rB = fma2(dB.x, dB.x, fma2(dB.y, dB.y, fma2(dB.z, dB.z, floor2)));
          float qa0, qa1, qb0, qb1;
          upk(rA, qa0, qa1);
          upk(rB, qb0, qb1);
          // cutoff masks in the FP32 pipe; no skip of steps without a hit (almost every one has one)
          const f2 cA = pk(fma_sat(qa0, -kCutScale, xr2s), fma_sat(qa1, -kCutScale, xr2s));
          const f2 cB = pk(fma_sat(qb0, -kCutScale, xr2s), fma_sat(qb1, -kCutScale, xr2s));
          hitsf = add2(hitsf, add2(cA, cB));
          bool near = false;  // warp-uniform: some slot is closer than r_sw
          if (kCheckSoft) near = __any_sync(full, fminf(fminf(qa0, qa1), fminf(qb0, qb1)) < a.f.rsw2_f);
          f2 DA = zero, DB = zero;
          const f2 BA = masked_bracket<SOFT, VJP>(rA, cA, kCheckSoft && near, a, DA);
          const f2 BB = masked_bracket<SOFT, VJP>(rB, cB, kCheckSoft && near, a, DB);
          F2x3 wA = {zero, zero, zero}, wB = wA;
          f2 ccA = zero, ccB = zero;
          if constexpr (VJP) {
            const float4 vs = S.vxy[base + q];
            const float2 vz = S.vz[base + q];
            wA = sub3(vA, vs, vz);
            wB = sub3(vB, vs, vz);
            ccA = mul2(DA, fma2(dA.x, wA.x, fma2(dA.y, wA.y, mul2(dA.z, wA.z))));
            ccB = mul2(DB, fma2(dB.x, wB.x, fma2(dB.y, wB.y, mul2(dB.z, wB.z))));
          }
          add_term<VJP>(aA, BA, dA, wA, ccA);
          add_term<VJP>(sa, BA, dA, wA, ccA);
          add_term<VJP>(aB, BB, dB, wB, ccB);
          add_term<VJP>(sa, BB, dB, wB, ccB);
          // the pair of lane l + 1 comes to lane l, with its accumulator
          sa.x = shfl2(sa.x, src);
          sa.y = shfl2(sa.y, src);
          sa.z = shfl2(sa.z, src);
          q = (q + 1) & pmask;
        }
      };
      if (blk_near) run(std::true_type{});
      else run(std::false_type{});
      // after P steps lane l holds the sum of its group for pair l mod P of its half
      for (int o = P; o < kWarp / 2; o <<= 1) {
        sa.x = add2(sa.x, shfl_xor2(sa.x, o));
        sa.y = add2(sa.y, shfl_xor2(sa.y, o));
        sa.z = add2(sa.z, shfl_xor2(sa.z, o));
      }
      if (l16 < P) {
        const int2 jj = S.sj[base + l16];
        float xa, xb, ya, yb, za, zb;
        upk(sa.x, xa, xb);
        upk(sa.y, ya, yb);
        upk(sa.z, za, zb);
        if (jj.x >= 0) atomicAdd(acc4 + jj.x, make_float4(-xa, -ya, -za, 0.f));
        if (jj.y >= 0) atomicAdd(acc4 + jj.y, make_float4(-xb, -yb, -zb, 0.f));
      }
      __syncwarp();
    };

    // Stage the survivors of each batch of 32 list positions; evaluate a block
    // whenever 64 are staged, and the rest once the enumeration is done (one
    // call site of eval_block, so its loops are inlined once).
    enumerate_suppliers(
        a, rc, F, S.L, lane, part, nparts, ch.start + ch.count, [&](int nlist, int lo, int hi, bool last) {
          const WarpList& L = S.L;
          ListCursor<WarpList> cur;
          cur.seek(L, nlist, lane, lo);
          auto locate = [&](int b, int& j, unsigned& dpk) { return cur.locate(L, nlist, hi, lane, b, j, dpk); };
          int jn;
          unsigned dn;
          bool vn = locate(lo, jn, dn);
          int buf = 0;
          if (vn) cp_async16(&S.rec[0][lane], a.rel4 + jn);
          cp_async_commit();
          float4 an = make_float4(0.f, 0.f, 0.f, 0.f);
          if (VJP && vn) an = a.abar4[jn];
          for (int b = lo;; b += kWarp) {
            const bool more = b < hi;  // warp-uniform
            bool keep = false, near = false;
            Vec3<float> pj = {0.f, 0.f, 0.f};
            int j = 0, rank = 0, ns = 0;
            float4 aj = make_float4(0.f, 0.f, 0.f, 0.f);
            if (more) {
              const bool have = vn;
              const unsigned dpk = dn;
              j = jn;
              if (VJP) aj = an;
              vn = (b + kWarp < hi) ? locate(b + kWarp, jn, dn) : false;
              if (vn) cp_async16(&S.rec[buf ^ 1][lane], a.rel4 + jn);
              cp_async_commit();
              cp_async_wait_prev();  // this lane's copy of batch b has landed
              const float4 r = have ? S.rec[buf][lane] : make_float4(0.f, 0.f, 0.f, 0.f);
              buf ^= 1;
              if (VJP && vn) an = a.abar4[jn];
              if (have) {
                int ddx, ddy, ddz;
                unpack_delta(dpk, ddx, ddy, ddz);
                pj.x = fmaf((float)ddx, a.g.side32[0], r.x);
                pj.y = fmaf((float)ddy, a.g.side32[1], r.y);
                pj.z = fmaf((float)ddz, a.g.side32[2], r.z);
                const float gap2 = box_gap2(F, pj);
                keep = gap2 < a.f.margin2_f;
                near = keep && gap2 < a.f.rsw2_f;
              }
              const unsigned m = __ballot_sync(full, keep);
              ns = __popc(m);
              rank = cnt + __popc(m & lt_mask);
              if (keep && rank < 2 * kWarp) stage(rank, pj, j, aj);
              blk_near = blk_near || __any_sync(full, near && rank < 2 * kWarp);
            }
            const bool flush = more ? (cnt + ns >= 2 * kWarp) : (last && cnt > 0);
            if (flush) {
              __syncwarp();
              eval_block(more ? 2 * kWarp : cnt);
              if (more) {
                blk_near = __any_sync(full, near && rank >= 2 * kWarp);
                if (keep && rank >= 2 * kWarp) stage(rank - 2 * kWarp, pj, j, aj);
                cnt += ns - 2 * kWarp;
              } else {
                cnt = 0;
              }
            } else {
              cnt += ns;
            }
            if (!more) break;
          }
        });
    // lane l keeps receiver l: the lower half's A sums and the upper half's B sums are its
    // own, the other half of the warp holds the rest of each
    auto total = [&](f2 o, f2 A, f2 B) {
      const bool upper = lane >= 16;
      const f2 mine = upper ? B : A, other = shfl_xor2(upper ? A : B, 16);
      float lo, hi;
      upk(add2(o, add2(mine, other)), lo, hi);
      return lo + hi;
    };
    const float4 mine = make_float4(total(own.x, aA.x, aB.x), total(own.y, aA.y, aB.y), total(own.z, aA.z, aB.z), 0.f);
    if (F.valid) atomicAdd(acc4 + F.pidx, mine);
    float l, h;
    upk(hitsf, l, h);
    pair_total += 2ull * (unsigned long long)__reduce_add_sync(full, (unsigned)(int)(l + h));  // ordered pairs
  }
  if (lane == 0 && pair_total) atomicAdd(a.pairs, pair_total);
}

// acc = -G m * (sum over partners of B(r) (x_i - x_j)) (or the adjoint's sum), from
// the float4 sums of k_force_sym.
__global__ void k_sym_finish(const float4* __restrict__ acc4, int64_t n, float scale, float* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 v = acc4[i];
    out[i] = scale * v.x;
    out[n + i] = scale * v.y;
    out[2 * n + i] = scale * v.z;
  }
}

// ---------------------------------------------------------------------------
// FP32 adjoint, packed broadcast: as k_force_packed, with every particle a
// receiver and the masked abar of each supplier staged beside its position.
//   xbar_k = -G m sum_j [ B v + (B'/r) (x_kj . v) x_kj ],  v = abar_k - abar_j.
// ---------------------------------------------------------------------------

struct PackedVjpSmem {
  WarpList L;
  float4 sxy[kWarp / 2 + 1];  // (-xa, -xb, -ya, -yb)
  float2 sz[kWarp / 2 + 1];   // (-za, -zb)
  float4 vxy[kWarp / 2 + 1];  // (-abar_xa, -abar_xb, -abar_ya, -abar_yb)
  float2 vz[kWarp / 2 + 1];   // (-abar_za, -abar_zb)
};

template <int SOFT>
__global__ void __launch_bounds__(kPThreads, P3M_GP_MINBLOCKS) k_vjp_packed(TraversalArgs a) {
  __shared__ PackedVjpSmem smem[kPWarps];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  PackedVjpSmem& S = smem[threadIdx.x >> 5];
  const int n_chunks = *a.n_chunks;
  const Reach rc = make_reach(a);
  const float xr2 = a.f.xr2_f;
  unsigned long long pair_total = 0;
  for (;;) {
    const int c = next_chunk(a, lane);
    if (c >= n_chunks) break;
    ChunkFrame F;
    load_chunk(a, rc, chunk_at(a, c), lane, F);
    const f2 px = pk(F.pi.x, F.pi.x), py = pk(F.pi.y, F.pi.y), pz = pk(F.pi.z, F.pi.z);
    float4 ab = make_float4(0.f, 0.f, 0.f, 0.f);
    if (F.valid) ab = a.abar4[F.pidx];
    const f2 vix = pk(ab.x, ab.x), viy = pk(ab.y, ab.y), viz = pk(ab.z, ab.z);
    f2 gx = pk(0.f, 0.f), gy = pk(0.f, 0.f), gz = pk(0.f, 0.f);
    int hits = 0;
    enumerate_strided(a, rc, F, S.L, lane, 0, 1, [&](int nlist, int total) {
      float* sxy = (float*)S.sxy;
      float* sz = (float*)S.sz;
      float* vxy = (float*)S.vxy;
      float* vz = (float*)S.vz;
      for (int b = 0; b < total; b += kWarp) {
        const int f = b + lane;
        Vec3<float> pj = {0.f, 0.f, 0.f}, aj = {0.f, 0.f, 0.f};
        bool keep = false, near = false;
        if (f < total) {
          float gap2;
          keep = load_supplier(a, S.L, nlist, f, F, pj, aj, &gap2);
          near = keep && gap2 < a.f.rsw2_f;  // may come within r_sw of a receiver (or coincide)
        }
        const unsigned m = __ballot_sync(full, keep);
        const int nsurv = __popc(m);
        if (keep) {
          const int k = __popc(m & ((1u << lane) - 1u));
          const int p = k >> 1, h = k & 1;
          sxy[4 * p + h] = -pj.x;
          sxy[4 * p + 2 + h] = -pj.y;
          sz[2 * p + h] = -pj.z;
          vxy[4 * p + h] = -aj.x;
          vxy[4 * p + 2 + h] = -aj.y;
          vz[2 * p + h] = -aj.z;
        }
        if (lane == 0 && (nsurv & 1)) {  // pad the last pair far from every receiver
          const int p = nsurv >> 1;
          sxy[4 * p + 1] = 1e30f;
          sxy[4 * p + 3] = 1e30f;
          sz[2 * p + 1] = 1e30f;
          vxy[4 * p + 1] = 0.f;
          vxy[4 * p + 3] = 0.f;
          vz[2 * p + 1] = 0.f;
        }
        __syncwarp();
        const int npairs = (nsurv + 1) >> 1;
        // as in the forward kernel: batches with no supplier within r_sw of the
        // receivers' box skip the softened-branch test
        auto run_pairs = [&](auto check_soft) {
          constexpr bool kCheckSoft = decltype(check_soft)::value;
#pragma unroll kGpUnroll
        for (int p = 0; p < npairs; ++p) {
          const float4 s = S.sxy[p];
          const float2 z = S.sz[p];
          const f2 dx = add2(px, pk(s.x, s.y));
          const f2 dy = add2(py, pk(s.z, s.w));
          const f2 dz = add2(pz, pk(z.x, z.y));
          const f2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
          float q0, q1;
          upk(r2, q0, q1);
          const bool h0 = q0 < xr2, h1 = q1 < xr2;
          if (__any_sync(full, h0 || h1)) {
            hits += (int)h0 + (int)h1;
            const float4 w = S.vxy[p];
            const float2 wz = S.vz[p];
            const f2 vx = add2(vix, pk(w.x, w.y));
            const f2 vy = add2(viy, pk(w.z, w.w));
            const f2 vz2 = add2(viz, pk(wz.x, wz.y));
            // r = 0 in the adjoint: the receiver itself has v = 0; coincident distinct
            // particles take the softened value B(0) (zero for point particles)
            f2 D;
            f2 B = bracket_main_vjp_f32x2<SOFT>(r2, a.f, D);
            float b0, b1, d0, d1;
            upk(B, b0, b1);
            upk(D, d0, d1);
            if (kCheckSoft) {
              const bool rare0 = h0 && (q0 < a.f.rsw2_f), rare1 = h1 && (q1 < a.f.rsw2_f);
              if (__any_sync(full, rare0 || rare1)) {
                f2 Dsp;
                float s0, s1, Ds0, Ds1;
                upk(bracket_soft_vjp_f32x2<SOFT>(r2, a.f, a.sc, Dsp), s0, s1);
                upk(Dsp, Ds0, Ds1);
                if (rare0) { b0 = s0; d0 = Ds0; }
                if (rare1) { b1 = s1; d1 = Ds1; }
              }
            }
            B = pk(h0 ? b0 : 0.0f, h1 ? b1 : 0.0f);
            D = pk(h0 ? d0 : 0.0f, h1 ? d1 : 0.0f);
            const f2 xv = fma2(dx, vx, fma2(dy, vy, mul2(dz, vz2)));
            const f2 cc = mul2(D, xv);
            gx = fma2(B, vx, fma2(cc, dx, gx));
            gy = fma2(B, vy, fma2(cc, dy, gy));
            gz = fma2(B, vz2, fma2(cc, dz, gz));
          }
        }
        };
        if (__any_sync(full, near)) run_pairs(std::true_type{});
        else run_pairs(std::false_type{});
        __syncwarp();
      }
    });
    Vec3<float> acc;
    float l, h;
    upk(gx, l, h);
    acc.x = l + h;
    upk(gy, l, h);
    acc.y = l + h;
    upk(gz, l, h);
    acc.z = l + h;
    store_result(a, F, acc);
    hits = F.valid ? hits - 1 : 0;  // the receiver met itself once (r = 0)
    pair_total += (unsigned long long)__reduce_add_sync(full, (unsigned)hits);
  }
  if (lane == 0 && pair_total) atomicAdd(a.pairs, pair_total);
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------

static SeriesConsts make_series() {
  SeriesConsts s{};
  const double two_over_sqrt_pi = 1.12837916709551257390;
  // h(u) = sum_m H_m u^{2m},  H_m = (2/sqrt(pi)) (-1)^m 2(m+1) / ((m+1)! (2m+3))
  double H[kHTermsD + 1];
  double fact = 1.0;
  for (int m = 0; m <= kHTermsD; ++m) {
    fact *= (double)(m + 1);
    H[m] = two_over_sqrt_pi * ((m & 1) ? -1.0 : 1.0) * 2.0 * (m + 1) / (fact * (2.0 * m + 3.0));
  }
  for (int m = 0; m < kHTermsD; ++m) {
    s.h_d[m] = H[m];
    s.hd_d[m] = 2.0 * (m + 1) * H[m + 1];  // h'(u)/u
  }
  for (int m = 0; m < kHTermsF; ++m) {
    s.h_f[m] = (float)s.h_d[m];
    s.hd_f[m] = (float)s.hd_d[m];
  }
  return s;
}

// One-sided FP32 kernels.
template <bool VJP, int SOFT>
static cudaError_t launch_packed(p3m_sr_ctx* ctx, const TraversalArgs& a) {
  static int blocks_per_sm = 0;
  if (blocks_per_sm == 0) {
    if (VJP) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, k_vjp_packed<SOFT>, kPThreads, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, k_force_packed<SOFT>, kPThreads, 0);
    if (blocks_per_sm < 1) blocks_per_sm = 1;
  }
  unsigned grid = (unsigned)(ctx->num_sms * blocks_per_sm);
  const int slot = VJP ? 1 : 0;
  TraversalArgs ap = a;
  if (!VJP) {  // sparse receivers: chunks split into parts
    ap.part_acc = ctx->part_acc;
    ap.part_items = ctx->part_items;
  }
  cudaEventRecord(ctx->kt_ev[2 * slot], ctx->stream);
  if (VJP) k_vjp_packed<SOFT><<<grid, kPThreads, 0, ctx->stream>>>(ap);
  else k_force_packed<SOFT><<<grid, kPThreads, 0, ctx->stream>>>(ap);
  ++ctx->launches;
  cudaEventRecord(ctx->kt_ev[2 * slot + 1], ctx->stream);
  ctx->kt_pending[slot] = true;
  if (!VJP) {
    k_parts_finish<<<(unsigned)(ctx->num_sms * 4), 256, 0, ctx->stream>>>(ap);
    ++ctx->launches;
  }
  return cudaGetLastError();
}

// Newton-III FP32 forward (all particles receivers) or adjoint: zero the float4
// sums, run k_force_sym, scale the sums into a.out.
template <int SOFT, bool VJP>
static cudaError_t launch_sym_soft(p3m_sr_ctx* ctx, const TraversalArgs& a, float4* acc4) {
  static int blocks_per_sm = 0;
  if (blocks_per_sm == 0) {
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, k_force_sym<SOFT, VJP>, kPThreads, 0);
    if (blocks_per_sm < 1) blocks_per_sm = 1;
  }
  cudaStream_t s = ctx->stream;
  cudaError_t e = cudaMemsetAsync(acc4, 0, sizeof(float4) * (size_t)ctx->n, s);
  if (e != cudaSuccess) return e;
  const int slot = VJP ? 1 : 0;
  cudaEventRecord(ctx->kt_ev[2 * slot], s);
  k_force_sym<SOFT, VJP><<<(unsigned)(ctx->num_sms * blocks_per_sm), kPThreads, 0, s>>>(a, acc4);
  ++ctx->launches;
  cudaEventRecord(ctx->kt_ev[2 * slot + 1], s);
  ctx->kt_pending[slot] = true;
  const unsigned fin = (unsigned)std::min<int64_t>((ctx->n + 255) / 256, (int64_t)ctx->num_sms * 16);
  k_sym_finish<<<fin, 256, 0, s>>>(acc4, ctx->n, -(float)a.f.G_m, (float*)a.out);
  ++ctx->launches;
  return cudaGetLastError();
}

template <bool VJP>
static cudaError_t launch_sym(p3m_sr_ctx* ctx, const TraversalArgs& a) {
  float4* acc4 = (float4*)ctx->gather_tmp;  // 32 n bytes, idle outside the sort
  switch (ctx->prm.softening) {
    case P3M_SOFT_NONE: return launch_sym_soft<P3M_SOFT_NONE, VJP>(ctx, a, acc4);
    case P3M_SOFT_PLUMMER: return launch_sym_soft<P3M_SOFT_PLUMMER, VJP>(ctx, a, acc4);
    default: return launch_sym_soft<P3M_SOFT_BSPLINE, VJP>(ctx, a, acc4);
  }
}

template <bool VJP>
static cudaError_t dispatch_packed(p3m_sr_ctx* ctx, const TraversalArgs& a) {
  switch (ctx->prm.softening) {
    case P3M_SOFT_NONE: return launch_packed<VJP, P3M_SOFT_NONE>(ctx, a);
    case P3M_SOFT_PLUMMER: return launch_packed<VJP, P3M_SOFT_PLUMMER>(ctx, a);
    default: return launch_packed<VJP, P3M_SOFT_BSPLINE>(ctx, a);
  }
}

// Receiver chunks of the row segments.
static p3m_status build_chunks(p3m_sr_ctx* ctx, const int* act_scan, Chunk* chunks, int* n_chunks_dev,
                               int* n_active_dev) {
  cudaStream_t s = ctx->stream;
  const int n_t = ctx->geo.n_t;
  const int64_t rows = (int64_t)n_t * n_t * ((n_t + kChunkSpan - 1) / kChunkSpan);  // segments
  k_build_chunks<<<blocks_for(rows, kSegThreads), kSegThreads, 0, s>>>(
      ctx->offsets, act_scan, n_t, ctx->geo.nsub3, chunks, ctx->dev_small + 8, n_chunks_dev, n_active_dev, ctx->n);
  ++ctx->launches;
  return cuda_check(ctx, cudaGetLastError(), "chunk kernel");
}

p3m_status ensure_all_chunks(p3m_sr_ctx* ctx) {
  if (ctx->all_chunks_built) return P3M_OK;
  p3m_status st = build_chunks(ctx, nullptr, ctx->chunks_all, ctx->dev_small + 1, nullptr);
  if (st == P3M_OK) ctx->all_chunks_built = true;
  return st;
}

static TraversalArgs base_args(p3m_sr_ctx* ctx) {
  static SeriesConsts series = make_series();
  TraversalArgs a{};
  a.g = ctx->geo;
  a.f = ctx->fc;
  a.sc = series;
  a.offsets = ctx->offsets;
  a.n = ctx->n;
  a.rel4 = ctx->rel4;
  a.rel_scale = 1.0f;
  a.pairs = ctx->pair_count;
  a.drift_slots = ctx->drift_slots;
  a.n_drift = ctx->n_drift;
  a.err = ctx->err_dev;
  return a;
}

// The work counters of the traversals and the pair count, in one memset.
static p3m_status clear_counters(p3m_sr_ctx* ctx) {
  return cuda_check(ctx, cudaMemsetAsync(ctx->dev_small + 3, 0, 5 * sizeof(int), ctx->stream), "memset");
}

// Records of pos.  ctx->rel4 holds those of sorted_pos unless rel4_stale says otherwise, so
// building another array's leaves it stale: every pair kernel, the FP64 ones included, finds
// its candidates from these records.
// For the FP64 kernels of a box whose records would leave the range of floats (rel_unit) they
// are built in its units, each time: for other calls they are stale too.
static p3m_status prepare_rel4(p3m_sr_ctx* ctx, const double* pos, int precision) {
  if (ctx->n == 0) return P3M_OK;
  const double unit = precision == 64 ? rel_unit(ctx->prm.box) : 1.0;
  if (unit == 1.0 && pos == ctx->sorted_pos && !ctx->rel4_stale) return P3M_OK;  // written by the sort or an earlier call
  auto kernel = unit == 1.0 ? k_rel4<false> : k_rel4<true>;
  kernel<<<blocks_for(ctx->n, 256), 256, 0, ctx->stream>>>(pos, ctx->cell, ctx->n, ctx->geo, unit, ctx->rel4);
  ++ctx->launches;
  ctx->rel4_stale = unit != 1.0 || pos != ctx->sorted_pos;
  return cuda_check(ctx, cudaGetLastError(), "rel4 kernel");
}

}  // namespace p3m

using namespace p3m;

extern "C" p3m_status p3m_sr_build_pairs(p3m_sr_ctx* ctx, const int8_t* rung, int rung_min) {
  if (!ctx) return P3M_ERR_INVALID;
  if (!ctx->sorted) return fail(ctx, P3M_ERR_STATE, "build_pairs: call p3m_sr_sort first");
  p3m_status st = poll_latched(ctx);
  if (st != P3M_OK) return st;
  cudaStream_t s = ctx->stream;
  const int64_t n = ctx->n;
  ctx->all_active = (rung == nullptr);
  const int* act_scan = nullptr;
  if (!ctx->all_active) {
    // receivers per tile of sorted particles, scanned, then flags + act_scan + list in one pass
    const int64_t tiles = (n + 1 + kActTile - 1) / kActTile;  // act_scan has n + 1 entries
    int* tile_count = ctx->hist;                                // idle outside the sort (>= 1024 per radix tile)
    k_active_count<<<(unsigned)tiles, kActThreads, 0, s>>>(rung, n, rung_min, tile_count);
    ++ctx->launches;
    if ((st = cuda_check(ctx, cudaGetLastError(), "active count")) != P3M_OK) return st;
    st = cuda_check(ctx, scan_exclusive_i32(tile_count, tile_count, tiles, ctx->scan_scratch, ctx->scan_scratch_ints, s,
                                            &ctx->launches), "scan");
    if (st != P3M_OK) return st;
    k_active_scan_compact<<<(unsigned)tiles, kActThreads, 0, s>>>(rung, n, rung_min, tile_count, ctx->active_flag,
                                                                   ctx->act_scan, ctx->active_idx);
    ++ctx->launches;
    if ((st = cuda_check(ctx, cudaGetLastError(), "active scan")) != P3M_OK) return st;
    act_scan = ctx->act_scan;
  }
  st = build_chunks(ctx, act_scan, ctx->chunks, ctx->dev_small + 0, ctx->dev_small + 2);
  if (st != P3M_OK) return st;
  ctx->pairs_built = true;
  return P3M_OK;
}

extern "C" p3m_status p3m_sr_forces(p3m_sr_ctx* ctx, const double* pos, int precision, void* acc_out) {
  if (!ctx) return P3M_ERR_INVALID;
  if (precision != 32 && precision != 64) return fail(ctx, P3M_ERR_INVALID, "forces: precision must be 32 or 64");
  if (ctx->n > 0 && (!pos || !acc_out)) return fail(ctx, P3M_ERR_INVALID, "forces: null pointer");
  if (!ctx->sorted || !ctx->pairs_built)
    return fail(ctx, P3M_ERR_STATE, "forces: call p3m_sr_sort and p3m_sr_build_pairs first");
  if (precision == 32 && ctx->prm.x_r > 2.0 * P3M_ERFCX_UMAX * ctx->prm.x_s)
    return fail(ctx, P3M_ERR_INVALID, "forces: the FP32 path needs x_r <= 4.6 x_s");
  p3m_status st = poll_latched(ctx);
  if (st != P3M_OK) return st;
  cudaStream_t s = ctx->stream;
  if ((st = clear_counters(ctx)) != P3M_OK) return st;
  if (ctx->n == 0) return P3M_OK;
  if ((st = prepare_rel4(ctx, pos, precision)) != P3M_OK) return st;
  TraversalArgs a = base_args(ctx);
  a.pos = pos;
  a.chunks = ctx->chunks;
  a.n_chunks = ctx->dev_small + 0;
  a.counter = ctx->dev_small + 3;
  a.active_idx = ctx->all_active ? nullptr : ctx->active_idx;
  a.out = acc_out;
  cudaError_t e;
  if (precision == 64) e = launch_pair64(ctx, a, false);
  else e = ctx->all_active && ctx->symmetric ? launch_sym<false>(ctx, a) : dispatch_packed<false>(ctx, a);
  if ((st = cuda_check(ctx, e, "force kernel")) != P3M_OK) return st;
  report_latched(ctx);
  return P3M_OK;
}

// B(r) in double on the host, for the table of p3m_sr_forces_tabulated.
static double bracket_host(double r, const ForceConsts& f, const SeriesConsts& sc) {
  const double inv_sqrt_pi = 0.56418958354775628695;
  const double r2 = r * r;
  if (r < f.r_sw) {
    if (f.softening == P3M_SOFT_NONE) return 0.0;
    const double u = r / (2.0 * f.x_s), u2 = u * u, w = 2.0 * f.x_s;
    double h = sc.h_d[kHTermsD - 1];
    for (int k = kHTermsD - 2; k >= 0; --k) h = h * u2 + sc.h_d[k];
    double s3;
    if (f.softening == P3M_SOFT_BSPLINE) {
      const double x = r / f.eps_b, c = 32.0 / (f.eps_b * f.eps_b * f.eps_b);
      s3 = (x < 0.5) ? c * (x * x * x - 1.2 * x * x + 1.0 / 3.0)
                     : c * (-x * x * x / 3.0 + 1.2 * x * x - 1.5 * x + 2.0 / 3.0 - 1.0 / (480.0 * x * x * x));
    } else {
      const double p = 1.0 / std::sqrt(r2 + f.eps * f.eps);
      s3 = p * p * p;
    }
    return s3 - h / (w * w * w);
  }
  const double u = r / (2.0 * f.x_s);
  double B = (std::erfc(u) + 2.0 * inv_sqrt_pi * u * std::exp(-u * u)) / (r2 * r);
  if (f.softening == P3M_SOFT_PLUMMER) {
    const double p = 1.0 / std::sqrt(r2 + f.eps * f.eps);
    B += p * p * p - 1.0 / (r2 * r);
  }
  return B;
}

extern "C" p3m_status p3m_sr_forces_tabulated(p3m_sr_ctx* ctx, const double* pos, int table_bits, float* acc_out) {
  if (!ctx) return P3M_ERR_INVALID;
  if (table_bits < 4 || table_bits > 14) return fail(ctx, P3M_ERR_INVALID, "forces_tabulated: table_bits must be 4..14");
  if (ctx->n > 0 && (!pos || !acc_out)) return fail(ctx, P3M_ERR_INVALID, "forces_tabulated: null pointer");
  if (!ctx->sorted || !ctx->pairs_built)
    return fail(ctx, P3M_ERR_STATE, "forces_tabulated: call p3m_sr_sort and p3m_sr_build_pairs first");
  p3m_status st = poll_latched(ctx);
  if (st != P3M_OK) return st;
  cudaStream_t s = ctx->stream;
  const int nt = 1 << table_bits;
  if (ctx->table_bits != table_bits) {
    static SeriesConsts series = make_series();
    std::vector<float> h(nt);
    for (int i = 0; i < nt; ++i) {
      const double r2c = (i + 0.5) * ctx->prm.x_r * ctx->prm.x_r / nt;  // bin centre in r^2
      h[i] = (float)bracket_host(std::sqrt(r2c), ctx->fc, series);
    }
    if (ctx->table) {
      cudaStreamSynchronize(s);
      cudaFree(ctx->table);
      ctx->table = nullptr;
    }
    if ((st = cuda_check(ctx, cudaMalloc((void**)&ctx->table, sizeof(float) * nt), "cudaMalloc(table)")) != P3M_OK)
      return st;
    if ((st = cuda_check(ctx, cudaMemcpy(ctx->table, h.data(), sizeof(float) * nt, cudaMemcpyHostToDevice),
                         "table copy")) != P3M_OK)
      return st;
    ctx->table_bits = table_bits;
  }
  if ((st = clear_counters(ctx)) != P3M_OK) return st;
  if (ctx->n == 0) return P3M_OK;
  if ((st = prepare_rel4(ctx, pos, 32)) != P3M_OK) return st;
  TraversalArgs a = base_args(ctx);
  a.pos = pos;
  a.chunks = ctx->chunks;
  a.n_chunks = ctx->dev_small + 0;
  a.counter = ctx->dev_small + 3;
  a.active_idx = ctx->all_active ? nullptr : ctx->active_idx;
  a.out = acc_out;
  a.table = ctx->table;
  a.part_acc = ctx->part_acc;
  a.part_items = ctx->part_items;
  a.n_table = nt;
  a.table_scale = (float)(nt / (ctx->prm.x_r * ctx->prm.x_r));
  const size_t shm = sizeof(float) * nt;
  auto launch = [&](auto kern) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
    int bps = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, kPThreads, shm);
    const unsigned grid = (unsigned)(ctx->num_sms * (bps > 0 ? bps : 1));
    cudaEventRecord(ctx->kt_ev[0], s);
    kern<<<grid, kPThreads, shm, s>>>(a);
    ++ctx->launches;
    cudaEventRecord(ctx->kt_ev[1], s);
    ctx->kt_pending[0] = true;
    k_parts_finish<<<(unsigned)(ctx->num_sms * 4), 256, 0, s>>>(a);
    ++ctx->launches;
  };
  switch (ctx->prm.softening) {
    case P3M_SOFT_NONE: launch(k_force_packed<P3M_SOFT_NONE, true>); break;
    case P3M_SOFT_PLUMMER: launch(k_force_packed<P3M_SOFT_PLUMMER, true>); break;
    default: launch(k_force_packed<P3M_SOFT_BSPLINE, true>); break;
  }
  if ((st = cuda_check(ctx, cudaGetLastError(), "tabulated force kernel")) != P3M_OK) return st;
  report_latched(ctx);
  return P3M_OK;
}

extern "C" p3m_status p3m_sr_vjp(p3m_sr_ctx* ctx, const double* pos, int precision, const void* acc_bar,
                                 void* pos_bar_out) {
  if (!ctx) return P3M_ERR_INVALID;
  if (precision != 32 && precision != 64) return fail(ctx, P3M_ERR_INVALID, "vjp: precision must be 32 or 64");
  if (ctx->n > 0 && (!pos || !acc_bar || !pos_bar_out)) return fail(ctx, P3M_ERR_INVALID, "vjp: null pointer");
  if (!ctx->sorted || !ctx->pairs_built)
    return fail(ctx, P3M_ERR_STATE, "vjp: call p3m_sr_sort and p3m_sr_build_pairs first");
  if (precision == 32 && ctx->prm.x_r > 2.0 * P3M_ERFCX_UMAX * ctx->prm.x_s)
    return fail(ctx, P3M_ERR_INVALID, "vjp: the FP32 path needs x_r <= 4.6 x_s");
  p3m_status st = poll_latched(ctx);
  if (st != P3M_OK) return st;
  cudaStream_t s = ctx->stream;
  const int64_t n = ctx->n;
  if ((st = clear_counters(ctx)) != P3M_OK) return st;
  if (n == 0) return P3M_OK;
  if (precision == 32 && !ctx->abar4) {
    if ((st = cuda_check(ctx, cudaMalloc((void**)&ctx->abar4, sizeof(float4) * ctx->cap), "cudaMalloc(abar4)")) != P3M_OK)
      return st;
  }
  if (precision == 64 && !ctx->abar_d) {
    if ((st = cuda_check(ctx, cudaMalloc((void**)&ctx->abar_d, sizeof(double) * 3 * ctx->cap), "cudaMalloc(abar_d)")) != P3M_OK)
      return st;
  }
  if ((st = ensure_all_chunks(ctx)) != P3M_OK) return st;
  if ((st = prepare_rel4(ctx, pos, precision)) != P3M_OK) return st;
  if (precision == 32)
    k_abar_f32<<<blocks_for(n, 256), 256, 0, s>>>((const float*)acc_bar, ctx->active_flag, ctx->all_active, n,
                                                   ctx->abar4);
  else
    k_abar_f64<<<blocks_for(n, 256), 256, 0, s>>>((const double*)acc_bar, ctx->active_flag, ctx->all_active, n,
                                                   ctx->abar_d);
  ++ctx->launches;
  if ((st = cuda_check(ctx, cudaGetLastError(), "abar kernel")) != P3M_OK) return st;
  TraversalArgs a = base_args(ctx);
  a.pos = pos;
  a.chunks = ctx->chunks_all;
  a.n_chunks = ctx->dev_small + 1;
  a.counter = ctx->dev_small + 4;
  a.active_idx = nullptr;
  a.out = pos_bar_out;
  a.abar4 = ctx->abar4;
  a.abar_d = ctx->abar_d;
  cudaError_t e;
  if (precision == 64) e = launch_pair64(ctx, a, true);
  else e = ctx->symmetric ? launch_sym<true>(ctx, a) : dispatch_packed<true>(ctx, a);  // each pair once (any active set)
  if ((st = cuda_check(ctx, e, "vjp kernel")) != P3M_OK) return st;
  report_latched(ctx);
  return P3M_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free entry point.
//
// Some callers cannot allocate device memory at all: code that runs under a
// memory pool or arena owned by a host application, a plugin that is handed
// only its input and output buffers, or a pipeline that forbids cudaMalloc
// after start-up.  p3m_sr_forces_noalloc serves them: it sorts a small
// particle set, builds its receiver chunks and evaluates the FP32 forces with
// the same kernels as the context-based path, but every intermediate array
// lives in one file-scope device array of fixed size.  That array belongs to
// every GPU that loads the library, for as long as the process lives.
// ---------------------------------------------------------------------------

namespace p3m {

constexpr int64_t kNoallocMaxN = 1 << 16;         // particles
constexpr int64_t kNoallocMaxSubtiles = 1 << 18;  // subtiles (n_t n_sub)^3
constexpr int64_t kNoallocMaxRows = 1 << 14;      // chunk segments n_t^2 ceil(n_t / 4)
constexpr int64_t kNoallocRadixBlocks = (kNoallocMaxN + kRadixTilePublic - 1) / kRadixTilePublic;
constexpr int64_t kNoallocMaxChunks = kNoallocMaxN + kNoallocMaxN / kChunk + 1;

constexpr int64_t noalloc_align(int64_t b) { return (b + 255) / 256 * 256; }
constexpr int64_t kNoallocScanInts = 4096;  // scan scratch; its last int is the scan's ticket

// Byte layout of the scratch array (each part 256-byte aligned).
struct NoallocLayout {
  static constexpr int64_t keys0 = 0;
  static constexpr int64_t keys1 = keys0 + noalloc_align(4 * kNoallocMaxN);
  static constexpr int64_t vals0 = keys1 + noalloc_align(4 * kNoallocMaxN);
  static constexpr int64_t vals1 = vals0 + noalloc_align(4 * kNoallocMaxN);
  static constexpr int64_t offsets = vals1 + noalloc_align(4 * kNoallocMaxN);
  static constexpr int64_t hist = offsets + noalloc_align(4 * (kNoallocMaxSubtiles + 1));
  static constexpr int64_t scan = hist + noalloc_align(4 * 1024 * kNoallocRadixBlocks);
  static constexpr int64_t wpos = scan + noalloc_align(4 * kNoallocScanInts);
  static constexpr int64_t bad = wpos + noalloc_align(8 * 3 * kNoallocMaxN);
  static constexpr int64_t pos = bad + noalloc_align(kNoallocMaxN);
  static constexpr int64_t rel4 = pos + noalloc_align(8 * 3 * kNoallocMaxN);
  static constexpr int64_t chunks = rel4 + noalloc_align(16 * kNoallocMaxN);
  static constexpr int64_t acc = chunks + noalloc_align(8 * kNoallocMaxChunks);
  static constexpr int64_t small = acc + noalloc_align(4 * 3 * kNoallocMaxN);
  static constexpr int64_t total = small + noalloc_align(64);
};

static __device__ __align__(256) unsigned char g_noalloc_scratch[NoallocLayout::total];

constexpr int kNoallocMaxDevices = 64;
static void* g_noalloc_addr[kNoallocMaxDevices];
static std::mutex g_noalloc_mutex;

// The caller's positions brought into the periodic box: x - L floor(x / L) for a
// finite coordinate outside [0, L) (the same point of the periodic box), 0 with
// bad[i] = 1 for a non-finite one.
__global__ void k_noalloc_wrap(const double* __restrict__ pos, int64_t n, double box, double* __restrict__ wpos,
                               unsigned char* __restrict__ bad) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  bool finite = true;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    double v = pos[d * n + i];
    if (!isfinite(v)) {
      finite = false;
      v = 0.0;
    } else if (!(v >= 0.0 && v < box)) {
      v = __dsub_rn(v, __dmul_rn(box, floor(__ddiv_rn(v, box))));
      if (!(v >= 0.0 && v < box)) v = 0.0;  // rounded up to L: the same point as 0
    }
    if (v == 0.0) v = 0.0;  // -0 as +0 (the binning compares bit patterns)
    wpos[d * n + i] = v;
  }
  bad[i] = finite ? 0 : 1;
}

// Sorted positions and FP32 subtile-relative records; a particle with a
// non-finite coordinate gets a record far outside the box, so that no receiver
// ever meets it (its own row is overwritten with NaN by k_noalloc_unsort).
__global__ void k_noalloc_gather(const double* __restrict__ wpos, const unsigned char* __restrict__ bad,
                                 const int* __restrict__ perm, const int* __restrict__ cell, int64_t n, Geometry g,
                                 double* __restrict__ spos, float4* __restrict__ rel4) {
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int64_t j = perm[k];
  const double x = wpos[j], y = wpos[n + j], z = wpos[2 * n + j];
  spos[k] = x;
  spos[n + k] = y;
  spos[2 * n + k] = z;
  const int id = cell[k];
  if (bad[j]) {
    rel4[k] = make_float4(1e10f, 1e10f, 1e10f, __int_as_float(id));
    return;
  }
  int gx, gy, gz;
  decode_subtile(g, id, gx, gy, gz);
  rel4[k] = make_float4((float)__fma_rn(-(double)gx, g.side64[0], x), (float)__fma_rn(-(double)gy, g.side64[1], y),
                        (float)__fma_rn(-(double)gz, g.side64[2], z), __int_as_float(id));
}

// acc_out[d][perm[k]] = acc[d][k], NaN for a particle with a non-finite coordinate
__global__ void k_noalloc_unsort(const float* __restrict__ acc, const int* __restrict__ perm,
                                 const unsigned char* __restrict__ bad, int64_t n, float* __restrict__ out) {
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  int64_t j = perm[k];
  const float nan = __int_as_float(0x7fc00000);
  const bool b = bad[j] != 0;
  out[j] = b ? nan : acc[k];
  out[n + j] = b ? nan : acc[n + k];
  out[2 * n + j] = b ? nan : acc[2 * n + k];
}

}  // namespace p3m

extern "C" p3m_status p3m_sr_forces_noalloc(const p3m_sr_params* params, void* cuda_stream, const double* pos,
                                            float* acc_out) {
  if (!params) return P3M_ERR_INVALID;
  p3m_sr_ctx c;  // host-side bookkeeping only: no device memory, no events
  p3m_status st = validate_params(&c, *params);
  if (st != P3M_OK) return st;
  const int64_t n = params->n;
  if (n > kNoallocMaxN) return P3M_ERR_INVALID;
  c.prm = *params;
  c.n = n;
  setup_geometry(&c);
  setup_force_consts(&c);
  const Geometry& g = c.geo;
  if (g.S > kNoallocMaxSubtiles ||
      (int64_t)g.n_t * g.n_t * ((g.n_t + kChunkSpan - 1) / kChunkSpan) > kNoallocMaxRows)
    return P3M_ERR_INVALID;
  if (params->x_r > 2.0 * P3M_ERFCX_UMAX * params->x_s) return P3M_ERR_INVALID;
  if (n == 0) return P3M_OK;
  if (!pos || !acc_out) return P3M_ERR_INVALID;

  // once per device: the device address of the scratch array
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoallocMaxDevices) return P3M_ERR_CUDA;
  unsigned char* base = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_addr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
        cudaGetLastError();
        return P3M_ERR_CUDA;
      }
      g_noalloc_addr[dev] = p;
    }
    base = (unsigned char*)g_noalloc_addr[dev];
  }
  using Lay = NoallocLayout;
  int* keys[2] = {(int*)(base + Lay::keys0), (int*)(base + Lay::keys1)};
  int* vals[2] = {(int*)(base + Lay::vals0), (int*)(base + Lay::vals1)};
  int* offsets = (int*)(base + Lay::offsets);
  int* hist = (int*)(base + Lay::hist);
  int* scan = (int*)(base + Lay::scan);
  double* wpos = (double*)(base + Lay::wpos);
  unsigned char* bad = base + Lay::bad;
  double* spos = (double*)(base + Lay::pos);
  float4* rel4 = (float4*)(base + Lay::rel4);
  Chunk* chunks = (Chunk*)(base + Lay::chunks);
  float* acc = (float*)(base + Lay::acc);
  int* small = (int*)(base + Lay::small);  // [0] n_chunks, [1] counter, [2] k_bin's error word (unused: the
                                           // positions are wrapped first), [4..5] pair count
  cudaStream_t s = (cudaStream_t)cuda_stream;
  int64_t launches = 0;
  auto ok = [&](cudaError_t e) { return e == cudaSuccess; };

  // periodic wrap, then bin + subtile offsets (histogram, exclusive scan)
  if (!ok(cudaMemsetAsync(offsets, 0, sizeof(int) * (g.S + 1), s))) return P3M_ERR_CUDA;
  if (!ok(cudaMemsetAsync(small, 0, 64, s))) return P3M_ERR_CUDA;
  if (!ok(cudaMemsetAsync(scan + kNoallocScanInts - 1, 0, sizeof(int), s))) return P3M_ERR_CUDA;
  k_noalloc_wrap<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pos, n, g.box, wpos, bad);
  if (!ok(cudaGetLastError())) return P3M_ERR_CUDA;
  k_bin<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(wpos, n, g, keys[0], vals[0], offsets, small + 2);
  if (!ok(cudaGetLastError())) return P3M_ERR_CUDA;
  if (!ok(scan_exclusive_i32(offsets, offsets, g.S + 1, scan, kNoallocScanInts, s, &launches))) return P3M_ERR_CUDA;
  // stable LSD radix sort of the subtile ids
  int key_bits = 1;
  while (key_bits < 31 && ((int64_t)1 << key_bits) < g.S) ++key_bits;
  const int passes = (key_bits + 9) / 10;
  const int nblocks = (int)((n + kRadixTilePublic - 1) / kRadixTilePublic);
  int cur = 0, shift = 0;
  for (int p = 0, left = key_bits; p < passes; ++p) {
    const int bits = (left + (passes - p) - 1) / (passes - p);
    left -= bits;
    k_radix_hist<<<nblocks, kRadixThreadsPublic, 0, s>>>(keys[cur], n, shift, bits, hist, nblocks);
    if (!ok(cudaGetLastError())) return P3M_ERR_CUDA;
    if (!ok(scan_exclusive_i32(hist, hist, (int64_t)nblocks << bits, scan, kNoallocScanInts, s, &launches))) return P3M_ERR_CUDA;
    launch_radix_scatter(nblocks, s, keys[cur], vals[cur], keys[cur ^ 1], vals[cur ^ 1], n, shift, bits, hist);
    if (!ok(cudaGetLastError())) return P3M_ERR_CUDA;
    cur ^= 1;
    shift += bits;
  }
  const int* cell = keys[cur];
  const int* perm = vals[cur];
  // sorted positions and their FP32 subtile-relative records
  k_noalloc_gather<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(wpos, bad, perm, cell, n, g, spos, rel4);
  if (!ok(cudaGetLastError())) return P3M_ERR_CUDA;
  // receiver chunks (all particles active)
  const int64_t nrows = (int64_t)g.n_t * g.n_t * ((g.n_t + kChunkSpan - 1) / kChunkSpan);  // segments
  k_build_chunks<<<(unsigned)((nrows + kSegThreads - 1) / kSegThreads), kSegThreads, 0, s>>>(
      offsets, nullptr, g.n_t, g.nsub3, chunks, small + 8, small + 0, nullptr, n);
  if (!ok(cudaGetLastError())) return P3M_ERR_CUDA;
  // pair forces in the sorted order, then back to the caller's order
  static SeriesConsts series = make_series();
  TraversalArgs a{};
  a.g = g;
  a.f = c.fc;
  a.sc = series;
  a.pos = spos;
  a.rel4 = rel4;
  a.rel_scale = 1.0f;
  a.offsets = offsets;
  a.chunks = chunks;
  a.n_chunks = small + 0;
  a.counter = small + 1;
  a.active_idx = nullptr;
  a.n = n;
  a.out = acc;
  a.pairs = (unsigned long long*)(small + 4);
  int num_sms = 0;
  cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
  const unsigned grid = (unsigned)(num_sms > 0 ? num_sms : 1) * 4;
  switch (params->softening) {
    case P3M_SOFT_NONE: k_force_packed<P3M_SOFT_NONE><<<grid, kPThreads, 0, s>>>(a); break;
    case P3M_SOFT_PLUMMER: k_force_packed<P3M_SOFT_PLUMMER><<<grid, kPThreads, 0, s>>>(a); break;
    default: k_force_packed<P3M_SOFT_BSPLINE><<<grid, kPThreads, 0, s>>>(a); break;
  }
  if (!ok(cudaGetLastError())) return P3M_ERR_CUDA;
  k_noalloc_unsort<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(acc, perm, bad, n, acc_out);
  if (!ok(cudaGetLastError())) return P3M_ERR_CUDA;
  return P3M_OK;
}
