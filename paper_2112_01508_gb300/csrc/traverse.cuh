// The supplier traversal shared by the pair kernels (force.cu, pair64.cu): a receiver
// chunk's frame, the candidate subtiles around it and the per-warp supplier list.
//
// All of it is FP32 in the frame of the chunk's first subtile, for both precisions:
// the FP64 kernels take their exact displacements afterwards, and the margins of the
// box tests are far above the FP32 rounding.
#pragma once

#include "ctx.cuh"
#include "pair_math.cuh"

namespace p3m {

struct TraversalArgs {
  Geometry g;
  ForceConsts f;
  SeriesConsts sc;
  const double* pos;          // FP64 path positions
  const float4* rel4;         // FP32 coordinates relative to the subtile, and its id
  float rel_scale;            // power of two that brings rel4 into the units of g.side32 and f.margin2_f
  const int* offsets;         // S + 1 subtile offsets
  const Chunk* chunks;
  float4* part_acc;           // per (work item, lane) partial sums when chunks are split, or nullptr
  int part_items;             // work items part_acc holds
  const float* drift_slots;   // displacement bounds of the drifts since the sort (device)
  int n_drift;                // how many of them
  int* err;                   // device error bits (kErrDrift), or nullptr
  const int* n_chunks;        // device count
  int* counter;               // dynamic chunk counter (zeroed before launch)
  const int* active_idx;      // receiver list (nullptr: chunk ranges are particle indices)
  int64_t n;
  void* out;                  // acc (forward) or xbar (vjp), 3 x n
  // vjp only
  const float4* abar4;        // masked abar FP32
  const double* abar_d;       // masked abar FP64, 3 x n
  unsigned long long* pairs;  // interacting ordered pairs
  // tabulated bracket (p3m_sr_forces_tabulated): B at the centres of n_table
  // equal bins of r^2 in [0, x_r^2)
  const float* table;
  int n_table;
  float table_scale;          // n_table / x_r^2
};

template <class Real>
struct Vec3 {
  Real x, y, z;
};

__device__ __forceinline__ float warp_min(float v) {
  float r;
  asm("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float warp_max(float v) {
  float r;
  asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

__device__ __forceinline__ unsigned pack_delta(int dx, int dy, int dz) {
  return ((unsigned)(dx + 512) << 20) | ((unsigned)(dy + 512) << 10) | (unsigned)(dz + 512);
}
__device__ __forceinline__ void unpack_delta(unsigned p, int& dx, int& dy, int& dz) {
  dx = (int)(p >> 20) - 512;
  dy = (int)((p >> 10) & 1023u) - 512;
  dz = (int)(p & 1023u) - 512;
}

// Supplier ranges buffered per warp before their particles are walked.
template <int CAP>
struct WarpListOf {
  static constexpr int kCap = CAP;
  int start[CAP];
  int pre[CAP];       // exclusive prefix of the supplier counts
  unsigned delta[CAP];
};

// Reach of the traversal.  Right after a sort: the block R of subtiles around the
// receivers' subtiles and the pruning bound x_r on the gap between a candidate
// subtile box and the receivers' box.  After drifts of total length delta since
// the sort, a particle may lie up to delta outside the subtile it was sorted into:
// the gap bound grows to x_r + delta and the block to x_r + 2 delta (receivers and
// suppliers both moved).  F64: lengths are multiplied by unit64, whatever the records' scale,
// and a saturated bound is an error (in FP32 no box is that large).
struct Reach {
  int R[3];
  float sub2;   // squared gap bound
  float delta;  // total drift bound
};

template <bool F64 = false>
__device__ __forceinline__ Reach make_reach(const TraversalArgs& a, double unit64 = 1.0) {
  Reach r;
  float delta = 0.0f;
  for (int k = 0; k < a.n_drift; ++k) delta += a.drift_slots[k];
  if (!(delta > 0.0f)) {
#pragma unroll
    for (int d = 0; d < 3; ++d) r.R[d] = a.g.R[d];
    r.sub2 = a.f.margin2_f;
    r.delta = 0.0f;
    return r;
  }
  const auto unit = [&] {
    if constexpr (F64) return unit64;
    else return a.rel_scale;
  }();
  r.delta = (float)(delta * unit);
  const double dl = (double)delta * (1.0 + 1e-5) * unit;  // the float sum may round down
  const double reach = sqrt((double)a.f.margin2_f) + dl;
  const double half = 0.5 * a.g.box * unit;
  if (!(reach + dl < half) || (F64 && delta >= 3.0e38f)) {  // (disp_bound saturates there)
    if ((threadIdx.x & 31) == 0 && a.err) atomicOr(a.err, kErrDrift);
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double rr = fmin(reach + dl, half);
    r.R[d] = (int)ceil(rr / (a.g.side64[d] * unit) * (1.0 + 1e-12));
  }
  r.sub2 = (float)(reach * reach * (1.0 + 1e-6));
  return r;
}

// The receivers of one chunk in its frame: positions, bounding box, subtile block.
struct ChunkFrame {
  bool valid;          // this lane holds a receiver
  int pidx;            // its sorted particle index
  int gi[3];           // its subtile
  int g0[3];           // subtile of lane 0 (frame origin)
  Vec3<float> pi;      // receiver position in the frame (1e30 on an empty lane)
  Vec3<float> lo, hi;  // bounding box of the receivers
  int elo[3], ext[3];  // candidate subtile block (offsets from g0) and its extent
  float inv_ext[2];    // 1 / ext[2], 1 / ext[1], for decoding candidate indices
};

__device__ __forceinline__ void load_chunk(const TraversalArgs& a, const Reach& rc, const Chunk& ch, int lane,
                                           ChunkFrame& F) {
  const unsigned full = 0xffffffffu;
  const Geometry& g = a.g;
  F.valid = lane < ch.count;
  F.pidx = 0;
  if (F.valid) F.pidx = a.active_idx ? a.active_idx[ch.start + lane] : ch.start + lane;
  F.gi[0] = F.gi[1] = F.gi[2] = 0;
  float4 ri = make_float4(0.f, 0.f, 0.f, 0.f);
  if (F.valid) {
    ri = a.rel4[F.pidx];
    decode_subtile(g, __float_as_int(ri.w), F.gi[0], F.gi[1], F.gi[2]);
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) F.g0[d] = __shfl_sync(full, F.gi[d], 0);
  const int e[3] = {F.gi[0] - F.g0[0], F.gi[1] - F.g0[1], F.gi[2] - F.g0[2]};
  F.pi.x = fmaf((float)e[0], g.side32[0], ri.x * a.rel_scale);
  F.pi.y = fmaf((float)e[1], g.side32[1], ri.y * a.rel_scale);
  F.pi.z = fmaf((float)e[2], g.side32[2], ri.z * a.rel_scale);
  const float big = 1e30f;
  F.lo.x = warp_min(F.valid ? F.pi.x : big);
  F.lo.y = warp_min(F.valid ? F.pi.y : big);
  F.lo.z = warp_min(F.valid ? F.pi.z : big);
  F.hi.x = warp_max(F.valid ? F.pi.x : -big);
  F.hi.y = warp_max(F.valid ? F.pi.y : -big);
  F.hi.z = warp_max(F.valid ? F.pi.z : -big);
  if (!F.valid) { F.pi.x = big; F.pi.y = big; F.pi.z = big; }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    F.elo[d] = __reduce_min_sync(full, F.valid ? e[d] : 1 << 20) - rc.R[d];
    int ehi = __reduce_max_sync(full, F.valid ? e[d] : -(1 << 20)) + rc.R[d];
    F.ext[d] = ehi - F.elo[d] + 1;
  }
  F.inv_ext[0] = 1.0f / (float)F.ext[2];
  F.inv_ext[1] = 1.0f / (float)F.ext[1];
}

// Candidate subtile cc (of ncand) of the blocky ball around the chunk's subtile
// block: whether its box gap to the receivers' bounding box is below the reach
// and it holds particles at indices >= clip_from; if so their range and the
// subtile offset.
__device__ __forceinline__ bool candidate_range(const TraversalArgs& a, const Reach& rc, const ChunkFrame& F, int cc,
                                                int ncand, int clip_from, int& start, int& cnt, unsigned& dpk) {
  const Geometry& g = a.g;
  start = 0;
  cnt = 0;
  dpk = 0;
  if (cc >= ncand) return false;
  int t, dx;
  if (ncand < (1 << 22)) {  // always, unless a drift has widened the block enormously
    t = quot_small(cc, F.ext[2], F.inv_ext[0]);
    dx = quot_small(t, F.ext[1], F.inv_ext[1]);
  } else {
    t = cc / F.ext[2];
    dx = t / F.ext[1];
  }
  int dz = cc - t * F.ext[2];
  int dy = t - dx * F.ext[1];
  dx += F.elo[0]; dy += F.elo[1]; dz += F.elo[2];
  const int dd[3] = {dx, dy, dz};
  const float blo[3] = {F.lo.x, F.lo.y, F.lo.z}, bhi[3] = {F.hi.x, F.hi.y, F.hi.z};
  float gap2 = 0.f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float side = g.side32[d];
    const float jlo = (float)dd[d] * side;
    const float jhi = jlo + side;
    const float gp = fmaxf(fmaxf(blo[d] - jhi, jlo - bhi[d]), 0.f);
    gap2 += gp * gp;
  }
  if (!(gap2 < rc.sub2)) return false;
  int gx = F.g0[0] + dx, gy = F.g0[1] + dy, gz = F.g0[2] + dz;
  gx += gx < 0 ? g.M[0] : (gx >= g.M[0] ? -g.M[0] : 0);
  gy += gy < 0 ? g.M[1] : (gy >= g.M[1] ? -g.M[1] : 0);
  gz += gz < 0 ? g.M[2] : (gz >= g.M[2] ? -g.M[2] : 0);
  const int sid = encode_subtile_fast(g, gx, gy, gz);
  start = max(a.offsets[sid], clip_from);
  cnt = a.offsets[sid + 1] - start;
  dpk = pack_delta(dx, dy, dz);
  return cnt > 0;
}

// Append the taken candidates of one round (ballot tm) to the warp's list.
template <class List>
__device__ __forceinline__ void append_round(List& L, int lane, bool take, int start, int cnt, unsigned dpk,
                                             unsigned tm, int& nlist, int& total) {
  const unsigned full = 0xffffffffu;
  int v = take ? cnt : 0;  // inclusive scan of the taken counts
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int u = __shfl_up_sync(full, v, o);
    if (lane >= o) v += u;
  }
  const int round_total = __shfl_sync(full, v, 31);
  if (take) {
    const int slot = nlist + __popc(tm & ((1u << lane) - 1u));
    L.start[slot] = start;
    L.pre[slot] = total + v - cnt;
    L.delta[slot] = dpk;
  }
  nlist += __popc(tm);
  total += round_total;
}

// The slice of `total` list positions that belongs to part `part` of a chunk split between
// nparts work items: equal numbers of suppliers, whatever the subtiles hold.
__device__ __forceinline__ int slice_start(int total, int part, int nparts) {
  return nparts == 1 ? (part ? total : 0) : (int)((long long)total * part / nparts);
}

// Enumerate the subtiles of the blocky ball around the chunk's subtile block
// (32 candidates per round, one per lane), keep those whose box gap to the
// receivers' bounding box is below x_r and that hold particles at indices >=
// clip_from, and append their particle ranges to the warp's list.
// `proc(nlist, lo, hi, last)` consumes the list positions [lo, hi), this part's slice:
// called from one place, each time the list fills up and once more at the end (last =
// true, possibly with nothing), so that a large consumer is inlined once.
template <class List, class Proc>
__device__ __forceinline__ void enumerate_suppliers(const TraversalArgs& a, const Reach& rc, const ChunkFrame& F,
                                                    List& L, int lane, int part, int nparts, int clip_from,
                                                    Proc&& proc) {
  const unsigned full = 0xffffffffu;
  const int ncand = F.ext[0] * F.ext[1] * F.ext[2];
  int nlist = 0, total = 0;
  int cb = 0;
  bool take = false;
  int start = 0, cnt = 0;
  unsigned dpk = 0, tm = 0;
  for (;;) {
    bool overflow = false;
    for (; cb < ncand; cb += kWarp) {
      take = candidate_range(a, rc, F, cb + lane, ncand, clip_from, start, cnt, dpk);
      tm = __ballot_sync(full, take);
      if (tm == 0) continue;
      if (nlist + __popc(tm) > List::kCap) {  // flush first; this batch of candidates is appended after
        overflow = true;
        break;
      }
      append_round(L, lane, take, start, cnt, dpk, tm, nlist, total);
    }
    __syncwarp();
    proc(nlist, slice_start(total, part, nparts), slice_start(total, part + 1, nparts), !overflow);
    __syncwarp();
    if (!overflow) break;
    nlist = 0;
    total = 0;
    append_round(L, lane, take, start, cnt, dpk, tm, nlist, total);
    cb += kWarp;
  }
}

// The same, with only every nparts-th candidate subtile, starting at `part`, enumerated:
// the parts of a chunk split its subtiles.  `proc(nlist, total)` consumes a full list and
// the last one.  The one-sided FP32 kernels take this form: with the sliced one above they
// run 14% slower on a full set (1.80 -> 2.06 ms at 128^3, 66 -> 72 registers).
template <class List, class Proc>
__device__ __forceinline__ void enumerate_strided(const TraversalArgs& a, const Reach& rc, const ChunkFrame& F,
                                                  List& L, int lane, int part, int nparts, Proc&& proc) {
  const unsigned full = 0xffffffffu;
  const int ncand_all = F.ext[0] * F.ext[1] * F.ext[2];
  const int ncand = (ncand_all - part + nparts - 1) / nparts;  // candidates of this part
  int nlist = 0, total = 0;
  for (int cb = 0; cb < ncand; cb += kWarp) {
    int start, cnt;
    unsigned dpk;
    const bool take = candidate_range(a, rc, F, (cb + lane) * nparts + part, ncand_all, 0, start, cnt, dpk);
    const unsigned tm = __ballot_sync(full, take);
    if (tm == 0) continue;
    if (nlist + __popc(tm) > List::kCap) {
      __syncwarp();
      proc(nlist, total);
      __syncwarp();
      nlist = 0;
      total = 0;
    }
    append_round(L, lane, take, start, cnt, dpk, tm, nlist, total);
  }
  __syncwarp();
  if (nlist > 0) proc(nlist, total);
  __syncwarp();
}

// Positions b + lane of the list (b advances by 32 per call, from `lo` given to seek, up
// to `hi`): supplier f lies in entry e_cur + (number of entries starting in (b, b + lane]);
// the start positions of the next 32 entries are gathered into one bit mask with a warp
// OR-reduction.
template <class List>
struct ListCursor {
  int e_cur = 0;  // entry holding position b
  __device__ __forceinline__ void seek(const List& L, int nlist, int lane, int lo) {
    if (lo == 0) return;
    int n = 0;  // entries starting at or before lo
    for (int e = 0; e < nlist; e += kWarp) {
      const unsigned m = __ballot_sync(0xffffffffu, e + lane < nlist && L.pre[e + lane] <= lo);
      n += __popc(m);
      if (m != 0xffffffffu) break;
    }
    e_cur = max(n - 1, 0);
  }
  __device__ __forceinline__ bool locate(const List& L, int nlist, int hi, int lane, int b, int& j, unsigned& dpk) {
    const unsigned full = 0xffffffffu;
    const int ek = e_cur + 1 + lane;
    const int pos = (ek < nlist) ? L.pre[ek] - b : 64;
    const unsigned bit = (pos > 0 && pos < kWarp) ? (1u << pos) : 0u;
    const unsigned starts = __reduce_or_sync(full, bit);
    const bool at_end = __any_sync(full, pos == kWarp);
    const unsigned upto = (lane == kWarp - 1) ? 0xffffffffu : ((2u << lane) - 1u);
    const int e = e_cur + __popc(starts & upto);
    e_cur += __popc(starts) + (at_end ? 1 : 0);
    const bool have = b + lane < hi;
    j = have ? L.start[e] + (b + lane - L.pre[e]) : 0;
    dpk = have ? L.delta[e] : 0u;
    return have;
  }
};

// Squared gap between a point of the chunk frame and the receivers' bounding box.
__device__ __forceinline__ float box_gap2(const ChunkFrame& F, const Vec3<float>& p) {
  const float tx = fmaxf(fmaxf(F.lo.x - p.x, p.x - F.hi.x), 0.f);
  const float ty = fmaxf(fmaxf(F.lo.y - p.y, p.y - F.hi.y), 0.f);
  const float tz = fmaxf(fmaxf(F.lo.z - p.z, p.z - F.hi.z), 0.f);
  return fmaf(tx, tx, fmaf(ty, ty, tz * tz));
}

// cp.async of 16 bytes into shared memory (completion per thread, by commit groups)
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

__device__ __forceinline__ int next_chunk(const TraversalArgs& a, int lane) {
  int c = 0;
  if (lane == 0) c = atomicAdd(a.counter, 1);
  return __shfl_sync(0xffffffffu, c, 0);
}

// The c-th chunk to process (c < n_chunks): the chunk list is in the sorted, spatial
// order, which keeps neighbouring chunks, and the suppliers they share, together in L2.
__device__ __forceinline__ Chunk chunk_at(const TraversalArgs& a, int c) { return a.chunks[c]; }

// Work items per chunk: with few chunks (sparse receivers, small sets) each chunk's
// suppliers are split between up to max_parts work items so that every resident
// warp has work, `items` in all.
__host__ __device__ __forceinline__ int parts_for(int n_chunks, int items, int max_parts) {
  if (n_chunks <= 0) return 1;
  const int k = items / n_chunks;
  return k < 1 ? 1 : (k > max_parts ? max_parts : k);
}

}  // namespace p3m
