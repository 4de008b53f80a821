// Sorting particles into tiles and subtiles (Section 2.1.3, "Tiles": an O(N)
// sort into the box tiling, with the particles reordered in memory in the
// tile -> subtile -> particle walk order of the short-range computation).
//
// GPU design: one pass bins every particle (subtile id from one correctly
// rounded multiply per dimension) and builds the subtile histogram; an
// exclusive scan turns it into the subtile offsets.  The permutation itself
// comes from a stable LSD radix sort of the subtile ids (digits of at most
// 10 bits, warp-level ranking with ballots so that equal ids keep their input
// order), after which positions and any carried arrays are gathered.
#include <algorithm>
#include <string>

#include "ctx.cuh"

namespace p3m {

constexpr int kRadixThreads = 256;
constexpr int kRadixWarps = kRadixThreads / kWarp;
static_assert(kRadixThreads == kRadixThreadsPublic, "radix tiling");
// Items per lane of a radix block: a serial chain of rounds, which is what a small set waits
// for, so up to kRadixSmallN particles (one long tile per SM) the tiles are a quarter as
// long.  A whole nearly sorted sort with long -> short tiles: 32,768 particles 62 -> 55 us,
// 131,072 73 -> 62, 311,296 71 -> 66, 524,288 75 -> 78, 1,048,576 99 -> 112.
template <int STEPS>
constexpr int kTileOf = kRadixThreads * STEPS;

// Subtile id of particle i: g_d = min(floor(x_d M_d / L), M_d - 1) with one correctly
// rounded multiply; a coordinate outside [0, L) (or NaN) is binned as 0 and sets *bad.
__device__ __forceinline__ int bin_one(const double (&x)[3], const Geometry& g, bool& bad) {
  int gc[3];
  const long long box_bits = __double_as_longlong(g.box);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double v = x[d];
    // 0 <= v < L on the bit patterns (non-negative doubles order like integers;
    // NaN, negative values and v >= L all fail)
    const long long vb = __double_as_longlong(v);
    bool ok = (vb >= 0) && (vb < box_bits);
    bad |= !ok;
    double p = __dmul_rn(ok ? v : 0.0, g.scale64[d]);
    // floor(p) for 0 <= p < 2^31 from the exponent and mantissa bits
    const long long pb = __double_as_longlong(p);
    const int e = (int)(pb >> 52) - 1023;
    int q = 0;
    if (e >= 0) q = (int)((((pb & 0xfffffffffffffLL) | (1LL << 52)) >> (52 - e)));
    gc[d] = q < g.M[d] - 1 ? q : g.M[d] - 1;
  }
  return encode_subtile_fast(g, gc[0], gc[1], gc[2]);  // 0 <= gc < M < 2^22
}

__global__ void k_bin(const double* __restrict__ pos, int64_t n, Geometry g, int* __restrict__ keys,
                      int* __restrict__ vals, int* __restrict__ counts, int* __restrict__ err) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = i < n;  // every lane stays for the warp-wide match below
  int id = 0;
  if (valid) {
    bool bad = false;
    const double x[3] = {pos[i], pos[n + i], pos[2 * n + i]};
    id = bin_one(x, g, bad);
    if (bad) atomicOr(err, kErrPosition);
    keys[i] = id;
    vals[i] = (int)i;
  }
  // one atomic per distinct subtile in the warp (sorted input repeats ids)
  const int lane = threadIdx.x & 31;
  const unsigned peers = __match_any_sync(0xffffffffu, valid ? id : -1 - lane);
  if (valid && lane == __ffs(peers) - 1) atomicAdd(&counts[id], __popc(peers));
}

// Staging of the gather.  Reading the particles of a set in random order costs one 32-byte
// sector per array and particle, about 20 us each at 128^3 and 300 us at 15.4 M, whatever the
// element size.  The binning kernel therefore copies the positions of such tiles, and up to 8
// bytes of what is carried, into records of one sector (32 n bytes of scratch); a tile of an
// input that is already spatially ordered, where the gather's reads are nearly sequential and
// the copy would be wasted, is left alone.  A tile counts as unordered if a quarter of its
// first particles have a neighbour kStageTiles tiles away in walk order.  Sets whose arrays
// fit half of L2 are not staged at all: there the sectors cost less than the copy (128^3,
// nothing carried: 202 us unstaged, 217 staged).
// Out-of-place sort in random order, by this step alone: 15.4 M particles with 12 carried bytes
// 2540 -> 1505 us, with 45 4174 -> 3064 us; 128^3 with 12 265 -> 259 us, with 45 405 -> 371 us;
// in nearly sorted order faster (15.4 M, 45 bytes: 1060 -> 948 us, from the loads issued
// together).
constexpr int kStageTiles = 4;
constexpr int64_t kStageBytes = 64 << 20;
struct StageArgs {
  double2* rec;             // 2 per particle: (x, y), (z, words); nullptr: no staging
  unsigned char* staged;    // per radix tile: its particles are in rec
  const void* word[2];      // carried arrays in the record: one of 8 bytes, or up to two of 4
  int n8, n4;
  int always;               // stage every tile (in-place sorts)
  int* unordered;           // number of staged tiles (zero before the sort)
  int nblocks;              // radix tiles
  float* drift_slots;       // cleared by the binning kernel
  int phased;               // the other one-word arrays of an unordered input go to k_gather_phases
};

__device__ __forceinline__ void stage_record(const StageArgs& st, int64_t i, const double (&x)[3]) {
  unsigned long long w = 0;
  if (st.n8) w = ((const unsigned long long*)st.word[0])[i];
  if (st.n4 > 0) w = ((const unsigned*)st.word[0])[i];
  if (st.n4 > 1) w |= (unsigned long long)((const unsigned*)st.word[1])[i] << 32;
  st.rec[2 * i] = make_double2(x[0], x[1]);
  st.rec[2 * i + 1] = make_double2(x[2], __longlong_as_double((long long)w));
}

// One atomic per run of consecutive lanes with the same index (at: a negative one takes no
// part).  The lanes hold nearly sorted items, whose equal indices are mostly neighbours, and a
// shuffle and a ballot cost a fraction of __match_any_sync.
__device__ __forceinline__ void count_runs(int* counts, int at, int lane) {
  const int before = __shfl_up_sync(0xffffffffu, at, 1);
  const bool head = lane == 0 || before != at;
  const unsigned heads = __ballot_sync(0xffffffffu, head);
  if (head && at >= 0) {
    const unsigned after = heads & (0xfffffffeu << lane);
    atomicAdd(&counts[at], (after ? __ffs(after) - 1 : 32) - lane);
  }
}

// k_bin over radix tiles of kTileOf<STEPS> particles, which also counts the digits of
// the first radix pass (bits low bits of the id) per tile: hist[d nblocks + tile].  Latency
// bound (44 us at 128^3, 31% of the issue slots); loading the next round's positions a round
// ahead changed nothing.
template <int STEPS>
__global__ void __launch_bounds__(256) k_bin_tile(const double* __restrict__ pos, int64_t n, Geometry g,
                                                  int* __restrict__ keys, int* __restrict__ counts,
                                                  int* __restrict__ err, int* __restrict__ hist, int bits, int nblocks,
                                                  int* __restrict__ hist_next, int next_ints,
                                                  const __grid_constant__ StageArgs st) {
  __shared__ int cnt[1024];
  for (int d = threadIdx.x; d < next_ints; d += blockDim.x)  // the next pass's counts, cleared
    hist_next[(int64_t)blockIdx.x * next_ints + d] = 0;
  if (blockIdx.x == 0 && threadIdx.x < kMaxDrifts) st.drift_slots[threadIdx.x] = 0.0f;  // no displacement since this sort
  const int radix = 1 << bits, mask = radix - 1;
  for (int d = threadIdx.x; d < radix; d += blockDim.x) cnt[d] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t base = (int64_t)blockIdx.x * kTileOf<STEPS>;
  bool any_bad = false, staged = false;
  for (int k = 0; k < STEPS; ++k) {
    const int64_t i = base + (int64_t)k * kRadixThreads + threadIdx.x;
    const bool valid = i < n;
    int id = 0;
    double x[3] = {0.0, 0.0, 0.0};
    if (valid) {
#pragma unroll
      for (int d = 0; d < 3; ++d) x[d] = pos[d * n + i];
      id = bin_one(x, g, any_bad);
      keys[i] = id;
      atomicAdd(&cnt[id & mask], 1);
    }
    if (k == 0) {
      const int next = __shfl_down_sync(0xffffffffu, id, 1);
      const bool far = valid && lane < 31 && abs(next - id) > kStageTiles * g.nsub3;
      staged = st.rec && (__syncthreads_count(far) > kRadixThreads / 4 || st.always);
      constexpr int kFlags = STEPS / kRadixSmallSteps;  // one per kRadixSmallSteps rounds
      if (threadIdx.x < kFlags) st.staged[blockIdx.x * kFlags + threadIdx.x] = staged ? 1 : 0;
      if (threadIdx.x == 0 && staged && st.phased) atomicAdd(st.unordered, 1);
    }
    if (staged && valid) stage_record(st, i, x);
    count_runs(counts, valid ? id : -1, lane);
  }
  if (any_bad) atomicOr(err, kErrPosition);
  __syncthreads();
  for (int d = threadIdx.x; d < radix; d += blockDim.x) hist[(int64_t)d * nblocks + blockIdx.x] = cnt[d];
}

constexpr int kMaxRadix = 1024;  // digits of at most 10 bits

__global__ void k_radix_hist(const int* __restrict__ keys, int64_t n, int shift, int bits,
                             int* __restrict__ hist, int nblocks) {
  __shared__ int cnt[kMaxRadix];
  const int radix = 1 << bits;
  for (int d = threadIdx.x; d < radix; d += blockDim.x) cnt[d] = 0;
  __syncthreads();
  int64_t base = (int64_t)blockIdx.x * kRadixTilePublic;
  const int mask = radix - 1;
  for (int k = 0; k < kRadixTilePublic / kRadixThreads; ++k) {
    int64_t i = base + (int64_t)k * kRadixThreads + threadIdx.x;
    if (i < n) atomicAdd(&cnt[(keys[i] >> shift) & mask], 1);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < radix; d += blockDim.x) hist[(int64_t)d * nblocks + blockIdx.x] = cnt[d];
}

// Stable scatter of one radix pass.  Warp w of a block owns the contiguous
// items [32 STEPS w, 32 STEPS (w + 1)) of the block's tile and walks them in STEPS rounds
// of 32 consecutive items, so ranks follow the input order; the lanes with the same digit
// are found by one ballot per digit bit.  The block then puts
// its tile in digit order in shared memory and writes it out from there, so that
// consecutive threads write consecutive positions of each digit's run.
// hist_next (nullable, zeroed before the launch): the digit counts of the next pass
// (bits_next bits from shift_next) per output tile, accumulated here with one atomic
// per run of equal (digit, tile) in a warp, so that pass needs no histogram kernel (with one,
// a nearly sorted sort at 128^3 takes 150 us, with the atomics 138).
// What bounds it is latency: the serial rounds and the barriers.  Counts in 16 bits, loads
// issued before the rounds and the digits' output positions read once per block let 6 blocks
// be resident (7 or 8 spill: 138 -> 160 us); ballots cost the same in every order, where
// __match_any_sync took longer the more different digits a warp held.  Whole sorts before and
// after: 15.4 M particles, nothing carried, nearly sorted 702 -> 651 us; 12 bytes carried,
// nearly sorted 801 -> 754, in random order 1522 -> 1268; 128^3 in random order 250 -> 224.
constexpr int kScatterBlocks = 6;
template <int STEPS>
__global__ void __launch_bounds__(kRadixThreads, kScatterBlocks) k_radix_scatter(
    const int* __restrict__ keys_in, const int* __restrict__ vals_in, int* __restrict__ keys_out,
    int* __restrict__ vals_out, int64_t n, int shift, int bits, const int* __restrict__ hist, int nblocks,
    int* __restrict__ hist_next, int shift_next, int bits_next) {
  constexpr int kTile = kTileOf<STEPS>;
  constexpr int kCounts = kRadixWarps * kMaxRadix * (int)sizeof(unsigned short), kStage = 2 * kTile * (int)sizeof(int);
  __shared__ __align__(16) unsigned char area[kCounts > kStage ? kCounts : kStage];
  unsigned short(*wcnt)[kMaxRadix] = (unsigned short(*)[kMaxRadix])area;  // per-warp digit counts (at most kTile)
  int* sk = (int*)area;                                                   // later the staged tile
  int* sv = sk + kTile;
  __shared__ int bstart[kMaxRadix];  // first position of each digit in the block's tile
  __shared__ int gstart[kMaxRadix];  // ... and its position in the output, less that
  __shared__ int wtot[kRadixWarps];
  const int radix = 1 << bits;
  const int mask = radix - 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t tile0 = (int64_t)blockIdx.x * kTile;
  const int64_t wbase = tile0 + (int64_t)warp * (STEPS * kWarp);
  const unsigned lt = (1u << lane) - 1u;
  int key[STEPS], rank[STEPS];
#pragma unroll
  for (int k = 0; k < STEPS; ++k) {  // all loads in flight before the serial rounds
    const int64_t i = wbase + k * kWarp + lane;
    key[k] = i < n ? keys_in[i] : 0;
  }
  for (int d = threadIdx.x; d < radix; d += kRadixThreads) gstart[d] = hist[(int64_t)d * nblocks + blockIdx.x];
  for (int d = lane; d < radix; d += 32) wcnt[warp][d] = 0;
  __syncwarp();
#pragma unroll
  for (int k = 0; k < STEPS; ++k) {
    const bool valid = wbase + k * kWarp + lane < n;
    const int d = (key[k] >> shift) & mask;
    unsigned peers = __ballot_sync(0xffffffffu, valid);  // the lanes with the same digit
    for (int b = 0; b < bits; ++b) {
      const bool one = (d >> b) & 1;
      const unsigned m = __ballot_sync(0xffffffffu, one);
      peers &= one ? m : ~m;
    }
    const int r = __popc(peers & lt);
    const int base = valid ? wcnt[warp][d] : 0;
    __syncwarp();
    if (valid && r == 0) wcnt[warp][d] = (unsigned short)(base + __popc(peers));
    __syncwarp();
    rank[k] = base + r;
  }
  __syncthreads();
  // exclusive prefix over the warps of the block, per digit; the digit totals
  for (int d = threadIdx.x; d < radix; d += kRadixThreads) {
    int run = 0;
#pragma unroll
    for (int w = 0; w < kRadixWarps; ++w) {
      const int t = wcnt[w][d];
      wcnt[w][d] = (unsigned short)run;
      run += t;
    }
    bstart[d] = run;
  }
  __syncthreads();
  // exclusive scan of the digit totals: thread t holds digits [4t, 4t + 4)
  {
    int v[4], tot = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int d = 4 * threadIdx.x + q;
      v[q] = d < radix ? bstart[d] : 0;
      tot += v[q];
    }
    int inc = tot;
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += u;
    }
    if (lane == 31) wtot[warp] = inc;
    __syncthreads();
    int run = inc - tot;
    for (int w = 0; w < warp; ++w) run += wtot[w];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int d = 4 * threadIdx.x + q;
      if (d < radix) {
        bstart[d] = run;
        gstart[d] -= run;
      }
      run += v[q];
    }
  }
  __syncthreads();
  // position of each item in the block's digit-ordered tile
#pragma unroll
  for (int k = 0; k < STEPS; ++k) {
    const int d = (key[k] >> shift) & mask;
    rank[k] += bstart[d] + wcnt[warp][d];
  }
  int val[STEPS];
#pragma unroll
  for (int k = 0; k < STEPS; ++k) {
    const int64_t i = wbase + k * kWarp + lane;
    val[k] = vals_in && i < n ? vals_in[i] : (int)i;  // first pass: the values are the positions
  }
  __syncthreads();  // every warp has read wcnt
  const int64_t left = n - tile0;
  const int nvalid = left < kTile ? (int)left : kTile;
#pragma unroll
  for (int k = 0; k < STEPS; ++k) {
    if (wbase + k * kWarp + lane < n) {
      sk[rank[k]] = key[k];
      sv[rank[k]] = val[k];
    }
  }
  __syncthreads();
  const int mask_next = (1 << bits_next) - 1;
  for (int p = threadIdx.x; p < kTile; p += kRadixThreads) {
    const bool valid = p < nvalid;
    int tag = -1;
    if (valid) {
      const int kk = sk[p];
      const int dst = gstart[(kk >> shift) & mask] + p;  // n < 2^31 - 64
      keys_out[dst] = kk;
      vals_out[dst] = sv[p];
      tag = ((kk >> shift_next) & mask_next) * nblocks + (int)((unsigned)dst / kTile);
    }
    if (hist_next) count_runs(hist_next, tag, lane);  // uniform over the launch
  }
}

void launch_radix_scatter(int nblocks, cudaStream_t s, const int* keys_in, const int* vals_in, int* keys_out, int* vals_out,
                          int64_t n, int shift, int bits, const int* hist) {
  k_radix_scatter<kRadixStepsPublic><<<nblocks, kRadixThreads, 0, s>>>(keys_in, vals_in, keys_out, vals_out, n, shift, bits,
                                                                       hist, nblocks, nullptr, 0, 0);
}

// Gather the positions into walk order from the staged records and write the FP32 record of
// each particle: its coordinates relative to the origin of its subtile and the id.
__global__ void k_gather_pos_rel4(const double2* __restrict__ rec, const int* __restrict__ perm,
                                  const int* __restrict__ cell, int64_t n, Geometry g, double* __restrict__ dst,
                                  float4* __restrict__ rel4) {
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  int64_t j = perm[k];
  const double2 xy = __ldg(rec + 2 * j);
  const double x = xy.x, y = xy.y, z = __ldg(&rec[2 * j + 1].x);
  dst[k] = x;
  dst[n + k] = y;
  dst[2 * n + k] = z;
  const int id = cell[k];
  int gx, gy, gz;
  decode_subtile(g, id, gx, gy, gz);
  double r[3];
  rel_to_subtile(g, x, y, z, gx, gy, gz, r);
  rel4[k] = make_float4(narrow(r[0]), narrow(r[1]), narrow(r[2]), __int_as_float(id));
}

// Carried arrays of an out-of-place sort: element bytes as `words` words of `wbytes` (8, 4,
// 2 or 1) bytes, chosen from the size and alignment.  Arrays of one 8-byte, 4-byte or
// 1-byte word come first, in this order (n8, n4, n1 of them); the rest follow.
constexpr int kMaxCarry = 8;
struct CarrySet {
  const void* src[kMaxCarry];
  void* dst[kMaxCarry];
  int words[kMaxCarry];
  int wbytes[kMaxCarry];
  int n8, n4, n1, count;
};

template <class T>
__device__ __forceinline__ void copy_words(const void* src, void* dst, int64_t j, int64_t k, int words) {
  const T* s = (const T*)src + j * words;
  T* d = (T*)dst + k * words;
  for (int w = 0; w < words; ++w) d[w] = s[w];
}

// Up to N arrays of one-word elements, from index `at` of the set: all loads, then (store) all stores.
template <class T, int N>
struct WordGroup {
  T v[N];
  __device__ __forceinline__ void load(const CarrySet& cs, int at, int from, int count, int64_t j) {
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (i >= from && i < count) v[i] = __ldg((const T*)cs.src[at + i] + j);
  }
  __device__ __forceinline__ void store(const CarrySet& cs, int at, int count, int64_t k) const {
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (i < count) ((T*)cs.dst[at + i])[k] = v[i];
  }
};

// The sorted positions, their FP32 records and every carried array: element k of each output
// is element perm[k] of the input (of the staged record where its tile has one).  All loads
// of a particle are issued before its first store.
//
// When the input is mostly unordered and its arrays together exceed half of L2, though each
// fits it with room for its output, this kernel takes the positions and the record words
// only and k_gather_phases the other one-word arrays, 16 bytes per particle at a time, so
// that the sectors of an array stay in L2 until its other particles have been read: 128^3 in
// random order with 45 carried bytes moved 694 MB from DRAM in one pass (27% L2 hits).
// Sort of 2.1 M in random order with 45 bytes 371 -> 334 us (404 before either), of 4.1 M
// 916 -> 582 us; nearly sorted 246 -> 236 and 387 -> 357 us.  PHASED is a parameter, and
// the two cases have code of their own, because counts that are not uniform constants cost a
// nearly sorted input 10%.  Without carried arrays the kernel is the lighter one.
constexpr int kPhase8 = 2, kPhase4 = 4;
template <bool CARRY, bool PHASED>
__global__ void __launch_bounds__(256) k_gather_all(const double* __restrict__ src, const int* __restrict__ perm,
                                                    const int* __restrict__ cell, int64_t n, Geometry g,
                                                    double* __restrict__ dst, float4* __restrict__ rel4,
                                                    const __grid_constant__ CarrySet cs,
                                                    const __grid_constant__ StageArgs st) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int64_t j = perm[k];
  const int at4 = cs.n8, at1 = at4 + cs.n4;
  const int id = cell[k];
  const bool split = PHASED && __ldg(st.unordered) > st.nblocks / 2;  // uniform over the launch
  const bool staged = st.rec && __ldg(st.staged + j / kTileOf<kRadixSmallSteps>) != 0;
  double x, y, z;
  WordGroup<unsigned long long, 4> w8;
  WordGroup<unsigned, 4> w4;
  WordGroup<unsigned char, 2> w1;
  if (staged) {
    const double2 xy = __ldg(st.rec + 2 * j), zw = __ldg(st.rec + 2 * j + 1);
    const unsigned long long w = (unsigned long long)__double_as_longlong(zw.y);
    x = xy.x;
    y = xy.y;
    z = zw.x;
    w8.v[0] = w;
    w4.v[0] = (unsigned)w;
    w4.v[1] = (unsigned)(w >> 32);
  } else {
    x = __ldg(src + j);
    y = __ldg(src + n + j);
    z = __ldg(src + 2 * n + j);
  }
  if constexpr (CARRY) {
    if (split) {
      w8.load(cs, 0, staged ? st.n8 : 0, st.n8, j);
      w4.load(cs, at4, staged ? st.n4 : 0, st.n4, j);
    } else {
      w8.load(cs, 0, staged ? st.n8 : 0, cs.n8, j);
      w4.load(cs, at4, staged ? st.n4 : 0, cs.n4, j);
    }
    w1.load(cs, at1, 0, cs.n1, j);
  }
  dst[k] = x;
  dst[n + k] = y;
  dst[2 * n + k] = z;
  int gx, gy, gz;
  decode_subtile(g, id, gx, gy, gz);
  double r[3];
  rel_to_subtile(g, x, y, z, gx, gy, gz, r);
  rel4[k] = make_float4(narrow(r[0]), narrow(r[1]), narrow(r[2]), __int_as_float(id));
  if constexpr (!CARRY) return;
  if (split) {
    w8.store(cs, 0, st.n8, k);
    w4.store(cs, at4, st.n4, k);
  } else {
    w8.store(cs, 0, cs.n8, k);
    w4.store(cs, at4, cs.n4, k);
  }
  w1.store(cs, at1, cs.n1, k);
  for (int c = at1 + cs.n1; c < cs.count; ++c) {
    switch (cs.wbytes[c]) {
      case 8: copy_words<unsigned long long>(cs.src[c], cs.dst[c], j, k, cs.words[c]); break;
      case 4: copy_words<unsigned>(cs.src[c], cs.dst[c], j, k, cs.words[c]); break;
      case 2: copy_words<unsigned short>(cs.src[c], cs.dst[c], j, k, cs.words[c]); break;
      default: copy_words<unsigned char>(cs.src[c], cs.dst[c], j, k, cs.words[c]); break;
    }
  }
}

// blockIdx.y: the phase.  In phase order by the order in which blocks start.
__global__ void __launch_bounds__(256) k_gather_phases(const int* __restrict__ perm, int64_t n,
                                                       const __grid_constant__ CarrySet cs,
                                                       const __grid_constant__ StageArgs st) {
  if (__ldg(st.unordered) <= st.nblocks / 2) return;  // k_gather_all has copied everything
  const int g8 = (cs.n8 - st.n8 + kPhase8 - 1) / kPhase8, y = (int)blockIdx.y;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = perm[k];
    if (y < g8) {
      const int at = st.n8 + y * kPhase8, m = min(kPhase8, cs.n8 - at);
      WordGroup<unsigned long long, kPhase8> w;
      w.load(cs, at, 0, m, j);
      w.store(cs, at, m, k);
    } else {
      const int at = st.n4 + (y - g8) * kPhase4, m = min(kPhase4, cs.n4 - at);
      WordGroup<unsigned, kPhase4> w;
      w.load(cs, cs.n8 + at, 0, m, j);
      w.store(cs, cs.n8 + at, m, k);
    }
  }
}

template <class T>
__global__ void k_gather_words(const T* __restrict__ src, const int* __restrict__ perm, int64_t n, int words,
                               T* __restrict__ dst) {
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  int64_t j = perm[k];
  for (int w = 0; w < words; ++w) dst[k * words + w] = src[j * words + w];
}

__global__ void k_fill_origins(Geometry g, double* __restrict__ org) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int d = i < g.M[0] ? 0 : (i < g.M[0] + g.M[1] ? 1 : 2);
  const int j = i - (d > 0 ? g.M[0] : 0) - (d > 1 ? g.M[1] : 0);
  if (d == 2 && j >= g.M[2]) return;
  org[i] = __dmul_rn((double)j, g.side64[d]);
}

static unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// dst[r n + k] = src[r n + perm[k]] (to sorted order) or dst[r n + perm[k]] = src[r n + k] (back).
template <class T>
__global__ void k_permute_rows(const T* __restrict__ src, T* __restrict__ dst, const int* __restrict__ perm, int64_t n,
                               int rows, int to_sorted) {
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  int64_t j = perm[k];
  for (int r = 0; r < rows; ++r) {
    if (to_sorted) dst[(int64_t)r * n + k] = src[(int64_t)r * n + j];
    else dst[(int64_t)r * n + j] = src[(int64_t)r * n + k];
  }
}

static p3m_status gather_carry(p3m_sr_ctx* ctx, void* arr, int bytes) {
  const int64_t n = ctx->n;
  const int t = 256;
  cudaStream_t s = ctx->stream;
  uintptr_t a = (uintptr_t)arr;
  if (bytes % 8 == 0 && a % 8 == 0)
    k_gather_words<uint64_t><<<blocks_for(n, t), t, 0, s>>>((const uint64_t*)arr, ctx->perm, n, bytes / 8,
                                                             (uint64_t*)ctx->gather_tmp);
  else if (bytes % 4 == 0 && a % 4 == 0)
    k_gather_words<uint32_t><<<blocks_for(n, t), t, 0, s>>>((const uint32_t*)arr, ctx->perm, n, bytes / 4,
                                                             (uint32_t*)ctx->gather_tmp);
  else if (bytes % 2 == 0 && a % 2 == 0)
    k_gather_words<uint16_t><<<blocks_for(n, t), t, 0, s>>>((const uint16_t*)arr, ctx->perm, n, bytes / 2,
                                                             (uint16_t*)ctx->gather_tmp);
  else
    k_gather_words<uint8_t><<<blocks_for(n, t), t, 0, s>>>((const uint8_t*)arr, ctx->perm, n, bytes,
                                                            (uint8_t*)ctx->gather_tmp);
  ++ctx->launches;
  p3m_status st = cuda_check(ctx, cudaGetLastError(), "gather kernel");
  if (st != P3M_OK) return st;
  return cuda_check(ctx, cudaMemcpyAsync(arr, ctx->gather_tmp, (size_t)bytes * n, cudaMemcpyDeviceToDevice, s),
                    "carry copy");
}

}  // namespace p3m

using namespace p3m;

// Bin the particles of pos and sort their subtile ids (Section 2.1.3: an O(N)
// sort into tiles): fills the subtile offsets, ctx->cell (sorted ids) and
// ctx->perm (sorted -> input index).  The first radix pass's digit histogram is
// counted by the binning kernel and each later pass's by the scatter before it.
static p3m_status bin_and_sort_ids(p3m_sr_ctx* ctx, const double* pos, StageArgs& stage) {
  const int64_t n = ctx->n;
  cudaStream_t s = ctx->stream;
  const Geometry& g = ctx->geo;
  // the subtile counts and, in front of them, the count of unordered tiles
  p3m_status st = cuda_check(ctx, cudaMemsetAsync(ctx->offsets - kOffsetsLead, 0, sizeof(int) * (g.S + 1 + kOffsetsLead), s),
                             "memset offsets");
  if (st != P3M_OK) return st;
  const bool small = n <= kRadixSmallN;
  const int tile = kRadixThreads * (small ? kRadixSmallSteps : kRadixStepsPublic);
  const int nblocks = (int)((n + tile - 1) / tile);
  int* hist[2] = {ctx->hist, ctx->hist + ctx->hist_ints};  // this pass's and the next pass's digit counts
  const int passes = ctx->radix_passes;
  stage.staged = ctx->staged;
  stage.unordered = ctx->offsets - kOffsetsLead;
  stage.nblocks = nblocks;
  stage.drift_slots = ctx->drift_slots;
  if (n > 0) {
    auto bin = small ? k_bin_tile<kRadixSmallSteps> : k_bin_tile<kRadixStepsPublic>;
    bin<<<nblocks, kRadixThreads, 0, s>>>(pos, n, g, ctx->keys[0], ctx->offsets, ctx->err_dev, hist[0],
                                          ctx->radix_bits[0], nblocks, hist[1], passes > 1 ? 1 << ctx->radix_bits[1] : 0,
                                          stage);
    ++ctx->launches;
    if ((st = cuda_check(ctx, cudaGetLastError(), "bin kernel")) != P3M_OK) return st;
  }
  // the subtile offsets and the first pass's digit positions
  st = cuda_check(ctx, scan_exclusive_i32_pair(ctx->offsets, g.S + 1, hist[0], n > 0 ? (int64_t)nblocks << ctx->radix_bits[0] : 0,
                                               ctx->scan_scratch, ctx->scan_scratch_ints, s, &ctx->launches),
                  "scan");
  if (st != P3M_OK) return st;
  int cur = 0;
  if (n > 0) {
    auto scatter = small ? k_radix_scatter<kRadixSmallSteps> : k_radix_scatter<kRadixStepsPublic>;
    int shift = 0;
    for (int p = 0; p < passes; ++p) {
      const int bits = ctx->radix_bits[p];
      const bool more = p + 1 < passes;
      if (p > 0) {
        st = cuda_check(ctx, scan_exclusive_i32(hist[p & 1], hist[p & 1], (int64_t)nblocks << bits, ctx->scan_scratch,
                                                ctx->scan_scratch_ints, s, &ctx->launches), "radix scan");
        if (st != P3M_OK) return st;
      }
      int* next = more ? hist[(p + 1) & 1] : nullptr;
      if (more && p > 0 &&  // the second pass's were cleared by the binning kernel
          (st = cuda_check(ctx, cudaMemsetAsync(next, 0, sizeof(int) * ((int64_t)nblocks << ctx->radix_bits[p + 1]), s),
                           "memset hist")) != P3M_OK)
        return st;
      scatter<<<nblocks, kRadixThreads, 0, s>>>(ctx->keys[cur], p > 0 ? ctx->vals[cur] : nullptr, ctx->keys[cur ^ 1],
                                                ctx->vals[cur ^ 1], n, shift, bits, hist[p & 1], nblocks, next,
                                                shift + bits, more ? ctx->radix_bits[p + 1] : 0);
      ++ctx->launches;
      if ((st = cuda_check(ctx, cudaGetLastError(), "radix scatter")) != P3M_OK) return st;
      cur ^= 1;
      shift += bits;
    }
  }
  ctx->cell = ctx->keys[cur];
  ctx->perm = ctx->vals[cur];
  return P3M_OK;
}

static p3m_status sort_outputs(p3m_sr_ctx* ctx, int32_t* perm_out, int32_t* subtile_id_out) {
  const int64_t n = ctx->n;
  p3m_status st = P3M_OK;
  if (n > 0 && perm_out)
    if ((st = cuda_check(ctx, cudaMemcpyAsync(perm_out, ctx->perm, sizeof(int) * n, cudaMemcpyDeviceToDevice,
                                              ctx->stream), "perm copy")) != P3M_OK)
      return st;
  if (n > 0 && subtile_id_out)
    if ((st = cuda_check(ctx, cudaMemcpyAsync(subtile_id_out, ctx->cell, sizeof(int) * n, cudaMemcpyDeviceToDevice,
                                              ctx->stream), "id copy")) != P3M_OK)
      return st;
  return P3M_OK;
}

static p3m_status sort_done(p3m_sr_ctx* ctx, const double* sorted_pos) {
  report_latched(ctx);
  ctx->sorted = true;
  ctx->sorted_pos = sorted_pos;  // the FP32 records in ctx->rel4 describe these positions
  ctx->n_drift = 0;              // no displacement since this sort
  ctx->rel4_stale = false;
  if (ctx->n > 0) return P3M_OK;  // the binning kernel cleared the drift slots
  return cuda_check(ctx, cudaMemsetAsync(ctx->drift_slots, 0, sizeof(float) * kMaxDrifts, ctx->stream), "memset");
}

static p3m_status check_carry(p3m_sr_ctx* ctx, void* const* carry, const int* carry_bytes, int n_carry,
                              const char* name) {
  if (n_carry < 0 || (n_carry > 0 && (!carry || !carry_bytes)))
    return fail(ctx, P3M_ERR_INVALID, std::string(name) + ": bad carry arguments");
  for (int c = 0; c < n_carry; ++c) {
    if (carry_bytes[c] < 1 || carry_bytes[c] > 32)
      return fail(ctx, P3M_ERR_INVALID, std::string(name) + ": carry_bytes must be 1..32");
    if (!carry[c] && ctx->n > 0) return fail(ctx, P3M_ERR_INVALID, std::string(name) + ": null carry array");
  }
  return P3M_OK;
}

extern "C" p3m_status p3m_sr_sort(p3m_sr_ctx* ctx, double* pos, void* const* carry, const int* carry_bytes,
                                  int n_carry, int32_t* perm_out, int32_t* subtile_id_out) {
  if (!ctx) return P3M_ERR_INVALID;
  const int64_t n = ctx->n;
  p3m_status st = check_carry(ctx, carry, carry_bytes, n_carry, "sort");
  if (st != P3M_OK) return st;
  if (!pos && n > 0) return fail(ctx, P3M_ERR_INVALID, "sort: null positions");
  if ((st = poll_latched(ctx)) != P3M_OK) return st;
  cudaStream_t s = ctx->stream;
  ctx->pairs_built = false;
  ctx->all_chunks_built = false;
  StageArgs stage{};  // every position staged: the gather then writes them back in place
  stage.rec = (double2*)ctx->gather_tmp;
  stage.always = 1;
  if ((st = bin_and_sort_ids(ctx, pos, stage)) != P3M_OK) return st;
  if (n > 0) {
    k_gather_pos_rel4<<<blocks_for(n, 256), 256, 0, s>>>(stage.rec, ctx->perm, ctx->cell, n, ctx->geo, pos, ctx->rel4);
    ++ctx->launches;
    if ((st = cuda_check(ctx, cudaGetLastError(), "gather positions")) != P3M_OK) return st;
    for (int c = 0; c < n_carry; ++c)
      if ((st = gather_carry(ctx, carry[c], carry_bytes[c])) != P3M_OK) return st;
  }
  if ((st = sort_outputs(ctx, perm_out, subtile_id_out)) != P3M_OK) return st;
  return sort_done(ctx, pos);
}

extern "C" p3m_status p3m_sr_sort_into(p3m_sr_ctx* ctx, const double* pos_in, double* pos_out,
                                       const void* const* carry_in, void* const* carry_out, const int* carry_bytes,
                                       int n_carry, int32_t* perm_out, int32_t* subtile_id_out) {
  if (!ctx) return P3M_ERR_INVALID;
  const int64_t n = ctx->n;
  if (n_carry > kMaxCarry) return fail(ctx, P3M_ERR_INVALID, "sort_into: at most 8 carried arrays");
  p3m_status st = check_carry(ctx, carry_out, carry_bytes, n_carry, "sort_into");
  if (st != P3M_OK) return st;
  if (n > 0 && (!pos_in || !pos_out)) return fail(ctx, P3M_ERR_INVALID, "sort_into: null positions");
  if (n > 0 && pos_in == pos_out) return fail(ctx, P3M_ERR_INVALID, "sort_into: pos_in and pos_out must differ");
  CarrySet cs{};
  int wbytes[kMaxCarry];
  for (int c = 0; c < n_carry; ++c) {
    if (n > 0 && (!carry_in || !carry_in[c] || carry_in[c] == carry_out[c]))
      return fail(ctx, P3M_ERR_INVALID, "sort_into: carried inputs must be non-null and differ from the outputs");
    const int b = carry_bytes[c];
    const uintptr_t al = (uintptr_t)(n > 0 ? carry_in[c] : nullptr) | (uintptr_t)carry_out[c];
    wbytes[c] = (b % 8 == 0 && al % 8 == 0) ? 8 : (b % 4 == 0 && al % 4 == 0) ? 4 : (b % 2 == 0 && al % 2 == 0) ? 2 : 1;
  }
  bool placed[kMaxCarry] = {};
  auto add = [&](int c) {
    const int i = cs.count++;
    cs.src[i] = n > 0 ? carry_in[c] : nullptr;
    cs.dst[i] = carry_out[c];
    cs.wbytes[i] = wbytes[c];
    cs.words[i] = carry_bytes[c] / wbytes[c];
    placed[c] = true;
  };
  auto add_single = [&](int bytes, int most) {  // arrays of one word of `bytes`
    int m = 0;
    for (int c = 0; c < n_carry && m < most; ++c)
      if (!placed[c] && carry_bytes[c] == bytes && wbytes[c] == bytes) {
        add(c);
        ++m;
      }
    return m;
  };
  cs.n8 = add_single(8, 4);
  cs.n4 = add_single(4, 4);
  cs.n1 = add_single(1, 2);
  for (int c = 0; c < n_carry; ++c)
    if (!placed[c]) add(c);
  if ((st = poll_latched(ctx)) != P3M_OK) return st;
  ctx->pairs_built = false;
  ctx->all_chunks_built = false;
  StageArgs stage{};
  int64_t bytes = 24;
  for (int c = 0; c < n_carry; ++c) bytes += carry_bytes[c];
  if (n * bytes > kStageBytes) stage.rec = (double2*)ctx->gather_tmp;
  stage.n8 = std::min(cs.n8, 1);
  stage.n4 = stage.n8 ? 0 : std::min(cs.n4, 2);
  for (int i = 0; i < stage.n8 + stage.n4; ++i) stage.word[i] = cs.src[i];  // n8 = 0: the 4-byte arrays come first
  const int rest = 8 * (cs.n8 - stage.n8) + 4 * (cs.n4 - stage.n4);  // one-word bytes outside the record
  stage.phased = stage.rec && 16 * n <= kStageBytes && rest >= 16;
  if ((st = bin_and_sort_ids(ctx, pos_in, stage)) != P3M_OK) return st;
  if (n > 0) {
    auto gather = n_carry == 0 ? k_gather_all<false, false> : stage.phased ? k_gather_all<true, true> : k_gather_all<true, false>;
    gather<<<blocks_for(n, 256), 256, 0, ctx->stream>>>(pos_in, ctx->perm, ctx->cell, n, ctx->geo, pos_out, ctx->rel4,
                                                        cs, stage);
    if (stage.phased) {
      const int phases = (cs.n8 - stage.n8 + kPhase8 - 1) / kPhase8 + (cs.n4 - stage.n4 + kPhase4 - 1) / kPhase4;
      k_gather_phases<<<dim3((unsigned)ctx->num_sms * 8, phases), 256, 0, ctx->stream>>>(ctx->perm, n, cs, stage);
      ++ctx->launches;
    }
    ++ctx->launches;
    if ((st = cuda_check(ctx, cudaGetLastError(), "gather kernel")) != P3M_OK) return st;
  }
  if ((st = sort_outputs(ctx, perm_out, subtile_id_out)) != P3M_OK) return st;
  return sort_done(ctx, pos_out);
}

// out[T] = first sorted index of tile T (T = (t_x n_t + t_y) n_t + t_z), out[n_tiles] = n.
__global__ void k_tile_offsets(const int* __restrict__ offsets, int64_t n_tiles, int nsub3, int* __restrict__ out) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t <= n_tiles) out[t] = offsets[t * nsub3];
}

extern "C" p3m_status p3m_sr_tile_offsets(p3m_sr_ctx* ctx, int32_t* offsets_out) {
  if (!ctx) return P3M_ERR_INVALID;
  if (!offsets_out) return fail(ctx, P3M_ERR_INVALID, "tile_offsets: null output");
  if (!ctx->sorted) return fail(ctx, P3M_ERR_STATE, "tile_offsets: call p3m_sr_sort first");
  const int64_t nt = ctx->n_tiles;
  k_tile_offsets<<<blocks_for(nt + 1, 256), 256, 0, ctx->stream>>>(ctx->offsets, nt, ctx->geo.nsub3, offsets_out);
  ++ctx->launches;
  return cuda_check(ctx, cudaGetLastError(), "tile offsets kernel");
}

static p3m_status permute_rows(p3m_sr_ctx* ctx, const void* src, void* dst, int elem_bytes, int rows, int to_sorted,
                               const char* name) {
  if (!ctx) return P3M_ERR_INVALID;
  if (!ctx->sorted && !ctx->perm) return fail(ctx, P3M_ERR_STATE, std::string(name) + ": call p3m_sr_sort first");
  if (!ctx->perm) return fail(ctx, P3M_ERR_STATE, std::string(name) + ": call p3m_sr_sort first");
  if (rows < 1 || (elem_bytes != 1 && elem_bytes != 2 && elem_bytes != 4 && elem_bytes != 8))
    return fail(ctx, P3M_ERR_INVALID, std::string(name) + ": elem_bytes must be 1, 2, 4 or 8 and rows >= 1");
  const int64_t n = ctx->n;
  if (n == 0) return P3M_OK;
  if (!src || !dst || src == dst) return fail(ctx, P3M_ERR_INVALID, std::string(name) + ": need distinct non-null arrays");
  const unsigned b = blocks_for(n, 256);
  cudaStream_t s = ctx->stream;
  switch (elem_bytes) {
    case 1: k_permute_rows<uint8_t><<<b, 256, 0, s>>>((const uint8_t*)src, (uint8_t*)dst, ctx->perm, n, rows, to_sorted); break;
    case 2: k_permute_rows<uint16_t><<<b, 256, 0, s>>>((const uint16_t*)src, (uint16_t*)dst, ctx->perm, n, rows, to_sorted); break;
    case 4: k_permute_rows<uint32_t><<<b, 256, 0, s>>>((const uint32_t*)src, (uint32_t*)dst, ctx->perm, n, rows, to_sorted); break;
    default: k_permute_rows<uint64_t><<<b, 256, 0, s>>>((const uint64_t*)src, (uint64_t*)dst, ctx->perm, n, rows, to_sorted); break;
  }
  ++ctx->launches;
  return cuda_check(ctx, cudaGetLastError(), name);
}

extern "C" p3m_status p3m_sr_permute(p3m_sr_ctx* ctx, const void* src, void* dst, int elem_bytes, int rows) {
  return permute_rows(ctx, src, dst, elem_bytes, rows, 1, "permute");
}

extern "C" p3m_status p3m_sr_unpermute(p3m_sr_ctx* ctx, const void* src, void* dst, int elem_bytes, int rows) {
  return permute_rows(ctx, src, dst, elem_bytes, rows, 0, "unpermute");
}
