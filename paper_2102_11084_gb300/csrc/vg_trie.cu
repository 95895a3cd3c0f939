// Steps a1-a5 by an occupancy trie: one cooperative launch, no sort.
//
// arXiv 2102.11084 Sec. II-C classifies every point into a cell of an ordered subdivision of
// space and keeps one point per occupied cell, in the order of the cells.  A sort orders all
// points to get there; the occupied cells alone give the order: the rank of a cell's key
// among the occupied keys is its row, and the points add their offsets at the row (exact
// integers, so in any order).  The ranks come from a trie of bitmaps over the keys:
//   level 1   one bit per prefix of up to 26 key bits (28 for large clouds), grouped in slots
//             of 2^7 bits;
//   level j   one slot of 2^7 bits per occupied prefix of level j - 1, numbered by its rank
//             there, for the next 7 key bits.
// Each level is marked by a pass over the points, its set bits counted per block and, after a
// barrier, ranked: a slot's record holds the set bits before the slot and, as bytes, before
// each of its words.  Keys of up to 26 bits take one level, each 7 bits more another one.
// The points are read twice, for the extents and for the first level; that second pass also
// merges runs of equal keys among 32 consecutive points (neighbouring pixels of a camera
// frame often share a cell) and writes each run, 16 bytes, to a dense list of its block
// (L2-resident scratch), which every later pass reads instead, its lanes evenly filled.  A
// 1280x720 frame at 0.05 m: 44 us; with every point's run kept in shared memory, undensed, 50
// us; computing the keys again in every pass 63 us.  A lane takes 2 or 4 consecutive points, so
// that it merges within itself and the warp's shuffles, ballots and scans run once for 64 or
// 128 points: 64 frames of 20k to 920k points 905 -> 771 us with 4; calls of at most
// kTrMaxPoints points, bound by latency and L2, take 2 (one frame's runs are added in 28,900
// cycles, not 40,000; with 4 a shuffled cloud's first pass took 91,000 cycles, not 79,000).
//
// Passes, with a grid barrier after each:
//   extents   per-frame min and max; the first level's bits cleared;
//   mark      (per level) the bit of every run's prefix, and no atomic where the bit is seen
//             set already; the lanes of a warp that set bits of one word merge while that
//             merges anything (a camera frame's warp meets few words, a shuffled cloud's many);
//   count, rank
//   add       a run's points and sums at its row, with two 64-bit atomics whose returned
//             values tell the carries out of their 32-bit halves (rows that many runs meet
//             first in the block's shared memory); attribute sums and, through the runs,
//             point_to_voxel here too;
//   rows      one thread a row: the centroid, by the formula and from the integer sums of every
//             other grouping, so the rows are theirs bit for bit.
// Bound by the latency of the passes and barriers (1.2 us each) for a camera frame, by
// instruction issue in the first mark pass for several, and by L2's random accesses (80 to 115
// sectors a cycle) for a shuffled cloud; HBM is idle.  A 640x480 frame at 0.05 m: 33 us, where
// the radix sort's 15 launches take 105; 1M shuffled points: 110 us against 156.
// Every wait is bounded (kErrTimeout after the limit, and the block returns), and every index
// read back from scratch is checked against its buffer.
#include <cstddef>

#include "vg_device.cuh"
#include "vg_device_int.h"
#include "vg_internal.h"
#include "vg_rows.cuh"
#include "vg_stream.cuh"
#include "vg_trie.h"

namespace vg {
namespace {

// Consecutive points of a lane in the marking pass: calls of up to kTrMaxPoints points, larger
// ones.
constexpr int kTrLane = 2, kTrLaneLarge = 4;

struct TrArgs {
  const float* xyz;
  FramesArg fr;
  State* st;
  FrameState* fs;
  uint32_t* root;      // first level: bits, then records (below)
  uint2* rootrec;
  char* x;             // buffers of the further levels
  char* y;
  uint4* run;          // a block's runs: {key, sum x, sum y, sum z | points << 26}
  uint32_t* runhi;     // the upper key words (keys of more than 32 bits)
  uint2* runatt;       // the runs' attribute sums, 16 bits a channel
  unsigned long long* rowatt;  // the rows', two words a row
  uint32_t* pslot;     // the slot of a run's prefix, then its row
  uint2* mask;         // per warp's points of one place in their lanes: ends of runs, valid points
  uint32_t* first;     // per warp's points: its first run (both for point_to_voxel)
  uint32_t* stat;      // per level (8): the blocks' totals
  SegOut out;
  int64_t slots;       // slots and rows the buffers hold
  uint32_t hot;        // entries of a block's table of hot rows (a power of two)
  uint32_t chunks;     // chunks of points at most
  int root_bits;
  int large;           // after the extent kernel; the call may be left to the sort path
  uint32_t spin_limit;
  int* err;
};

struct TrSmem {
  uint32_t tmp[kTrThreads / 32];
  uint32_t bits[kTrThreads / 32];
  uint32_t first;
  uint32_t nruns;
  uint32_t hot;     // some entry of the table of hot rows is taken
  uint32_t look;    // rows that the block's runs meet again are looked for
  uint32_t single;  // its runs are hardly more than points
};

// Tables of a call's frames (dynamic shared memory).
struct TrFrames {
  float4* pose;      // [F][4]: the rows of [R|t], then the height limits (posed calls)
  int64_t* off;      // [F + 1]
  float* org;        // [F][3]
  float* leaf;       // [F]
  float* rleaf;
  float* inv_unit;
  uint32_t* cstart;  // [F + 1]
  uint32_t* ext;     // [F][6]: the block's extents, as the frames' (ord_min_inv, ord_max)
};
constexpr size_t tr_frames_bytes(int frames, bool posed) {
  return align_up(size_t(frames + 1) * 12 + size_t(frames) * (posed ? 112 : 48), 16);
}
__device__ __forceinline__ TrFrames tr_frames(unsigned char* mem, int F, bool posed) {
  TrFrames t;
  t.pose = reinterpret_cast<float4*>(mem);
  t.off = reinterpret_cast<int64_t*>(t.pose + (posed ? 4 * F : 0));
  t.org = reinterpret_cast<float*>(t.off + F + 1);
  t.leaf = t.org + 3 * F;
  t.rleaf = t.leaf + F;
  t.inv_unit = t.rleaf + F;
  t.cstart = reinterpret_cast<uint32_t*>(t.inv_unit + F);
  t.ext = t.cstart + F + 1;
  return t;
}

__device__ __forceinline__ Pose tr_pose(const TrArgs& a, const TrFrames& fm, int f) {
  const float4* t = fm.pose + 4 * f;
  const float4 r0 = t[0], r1 = t[1], r2 = t[2], z = t[3];
  Pose P;
  P.r[0] = r0.x, P.r[1] = r0.y, P.r[2] = r0.z, P.r[3] = r0.w;
  P.r[4] = r1.x, P.r[5] = r1.y, P.r[6] = r1.z, P.r[7] = r1.w;
  P.r[8] = r2.x, P.r[9] = r2.y, P.r[10] = r2.z, P.r[11] = r2.w;
  P.zlo = z.x;
  P.zhi = z.y;
  P.rigid = a.fr.poses != nullptr;
  return P;
}

// A lane's points: K consecutive ones from p on, m of them in frame f (NaN past them).
// Chunk k of the block is the cloud's k * grid + blockIdx.x; kChunk / 32K warps take it.
template <int K>
struct TrLanePoints {
  int f, m;
  int64_t p;
  float q[K][3];
};
template <int K>
constexpr uint32_t tr_chunk_warps() {
  return kChunk / (32 * K);
}
template <int K>
__device__ __forceinline__ void tr_lane_load(const TrArgs& a, TrLanePoints<K>& t) {
  const float* src = a.xyz + 3 * t.p;
  const uint32_t low = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(src));
  if (K == 4 && t.m == K && (low & 15u) == 0u) {
    const float4* v = reinterpret_cast<const float4*>(src);
#pragma unroll
    for (int i = 0; i < 3 * K / 4; ++i) {
      const float4 x = __ldg(v + i);
      t.q[(4 * i) / 3][(4 * i) % 3] = x.x;
      t.q[(4 * i + 1) / 3][(4 * i + 1) % 3] = x.y;
      t.q[(4 * i + 2) / 3][(4 * i + 2) % 3] = x.z;
      t.q[(4 * i + 3) / 3][(4 * i + 3) % 3] = x.w;
    }
  } else if (K == 2 && t.m == K && (low & 7u) == 0u) {
    const float2* v = reinterpret_cast<const float2*>(src);
#pragma unroll
    for (int i = 0; i < 3 * K / 2; ++i) {
      const float2 x = __ldg(v + i);
      t.q[(2 * i) / 3][(2 * i) % 3] = x.x;
      t.q[(2 * i + 1) / 3][(2 * i + 1) % 3] = x.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < K; ++j)
#pragma unroll
      for (int c = 0; c < 3; ++c)
        t.q[j][c] = j < t.m ? __ldg(src + 3 * j + c) : __int_as_float(0x7fc00000);
  }
}
// fn(part, points) for every part of this block's chunks that this warp takes; with kLoad the
// coordinates too (one step ahead where a lane has few), posed in a posed call.
template <bool kPosed, int K, bool kLoad, typename Fn>
__device__ __forceinline__ void tr_lanes(const TrArgs& a, const TrFrames& fm, uint32_t T, Fn fn) {
  constexpr uint32_t kWarps = tr_chunk_warps<K>();
  constexpr bool kAhead = kLoad && K <= 2;
  static_assert(kTrThreads / 32 % kWarps == 0, "whole chunks of points");
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  const int nf = a.fr.nframes;
  TrLanePoints<K> next;
  auto find = [&](uint32_t k) {
    const uint64_t c = uint64_t(k) * gridDim.x + blockIdx.x;
    if (c >= T) return false;
    next.f = nf > 1 ? chunk_frame(fm.cstart, nf, uint32_t(c)) : 0;
    next.p = fm.off[next.f] + (int64_t(c) - fm.cstart[next.f]) * kChunk +
             ((warp % kWarps) * 32u + lane) * K;
    const int64_t left = fm.off[next.f + 1] - next.p;
    next.m = left < K ? (left < 0 ? 0 : static_cast<int>(left)) : K;
    if (kAhead) tr_lane_load<K>(a, next);
    return true;
  };
  uint32_t k = warp / kWarps;
  bool more = find(k);
  while (more) {
    TrLanePoints<K> t = next;
    const uint32_t part = k * kWarps + warp % kWarps;
    k += kTrThreads / 32 / kWarps;
    if (kAhead) more = find(k);
    if (kAhead || __any_sync(kFullMask, t.m != 0)) {
      if (kLoad && !kAhead) tr_lane_load<K>(a, t);
      if (kLoad && kPosed) {
        const Pose P = tr_pose(a, fm, t.f);
#pragma unroll
        for (int j = 0; j < K; ++j) pose_point(P, t.q[j][0], t.q[j][1], t.q[j][2]);
      }
      fn(part, t);
    }
    if (!kAhead) more = find(k);
  }
}

// The sort key of a point of frame f (its indices as floats in fi); false for an invalid point or one out
// of range (*range_bad set).
__device__ __forceinline__ bool tr_key(const TrFrames& fm, int f, float x, float y, float z,
                                       bool wide, uint32_t key_shift, uint64_t* key,
                                       float fi[3], bool* range_bad) {
  uint32_t ijk[3];
  const float o[3] = {fm.org[3 * f], fm.org[3 * f + 1], fm.org[3 * f + 2]};
  if (!point_index(x, y, z, o, fm.leaf[f], fm.rleaf[f], ijk, fi, range_bad)) return false;
  if (wide)
    *key = key_compose(uint32_t(f), morton3(ijk[0], ijk[1], ijk[2]), key_shift);
  else  // per-frame keys of at most 32 bits
    *key = key_compose(uint32_t(f),
                       spread3_32(ijk[0]) | (spread3_32(ijk[1]) << 1) | (spread3_32(ijk[2]) << 2),
                       key_shift);
  return true;
}

// Place of the lane's first run among the warp's, in the points' order, from the ballots of the
// points that end one.
template <int K>
__device__ __forceinline__ uint32_t tr_place(const uint32_t tails[K]) {
  uint32_t i = 0u;
#pragma unroll
  for (int j = 0; j < K; ++j) i += __popc(tails[j] & ((1u << (threadIdx.x & 31u)) - 1u));
  return i;
}

// Sets the bits `bit` of a word for every lane that has some (those it did not see set in the
// word as loaded before; a stale one can only lack bits).  Up to half a warp of
// lanes (a camera frame's runs, which meet a few words) merges them word by word: the
// atomics of all warps on the few words took 8,500 cycles more of a 640x480 frame.  More
// lanes (a shuffled cloud's points, a word each) merge the first two words' only: match.any
// and a redux a group cost a full warp 2,000 cycles.
__device__ __forceinline__ void tr_set(uint32_t* bits, uint32_t word, uint32_t bit) {
  const uint32_t lane = threadIdx.x & 31u;
  bool need = bit != 0u;
  uint32_t m = __ballot_sync(kFullMask, need);
  if (__popc(m) <= 16) {
    if (need) {
      const uint32_t peers = __match_any_sync(m, word);
      const uint32_t v = __reduce_or_sync(peers, bit);
      if (int(lane) == __ffs(peers) - 1) atomicOr(bits + word, v);
    }
    return;
  }
#pragma unroll 1
  for (int k = 0; k < 2 && m; ++k) {
    const uint32_t w = __shfl_sync(kFullMask, word, __ffs(m) - 1);
    const bool mine = need && word == w;
    const uint32_t same = __ballot_sync(kFullMask, mine);
    const uint32_t v = __reduce_or_sync(kFullMask, mine ? bit : 0u);
    if (mine) {
      if (int(lane) == __ffs(same) - 1) atomicOr(bits + w, v);
      need = false;
    }
    m &= ~same;
  }
  if (need) atomicOr(bits + word, bit);
}

// Rank of bit d of a slot, from its record r and the word v that holds the bit.
__device__ __forceinline__ uint32_t tr_rank(uint2 r, uint32_t v, uint32_t d) {
  const uint32_t w = d >> 5;
  const uint32_t before = (r.y >> (8u * w)) & 255u;
  return r.x + before + __popc(v & ((1u << (d & 31u)) - 1u));
}

__device__ __forceinline__ uint4 tr_slot_words(const uint32_t* bits, uint32_t s) {
  return __ldcg(reinterpret_cast<const uint4*>(bits) + s);
}

// Ranking the set bits of slots [0, ns) takes two steps around a grid barrier: block b takes a
// contiguous slice of the slots and publishes its set bits in agg[b]; then every block sums
// its predecessors' totals (a thread each) and ranks its slice, a thread a slot.
__device__ __forceinline__ void tr_slice(uint32_t ns, uint32_t* s0, uint32_t* s1) {
  const uint32_t q = (ns + gridDim.x - 1u) / gridDim.x;
  *s0 = min(ns, blockIdx.x * q);
  *s1 = min(ns, *s0 + q);
}
__device__ __forceinline__ void tr_count(const uint32_t* bits, uint32_t ns, uint32_t* agg,
                                         uint32_t* tmp) {
  uint32_t s0, s1, mine = 0;
  tr_slice(ns, &s0, &s1);
  for (uint32_t s = s0 + threadIdx.x; s < s1; s += kTrThreads) {
    const uint4 v = tr_slot_words(bits, s);
    mine += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
  }
  uint32_t total;
  (void)block_excl_scan(mine, &total, tmp);
  if (threadIdx.x == 0) agg[blockIdx.x] = total;
}
// Returns the grand total (the same in every block).  Contains __syncthreads.
__device__ __forceinline__ uint32_t tr_rank_slots(const uint32_t* bits, uint2* rec, uint32_t ns,
                                                  const uint32_t* agg, TrSmem& sm) {
  uint32_t s0, s1;
  tr_slice(ns, &s0, &s1);
  const uint32_t g = threadIdx.x < gridDim.x ? __ldcg(agg + threadIdx.x) : 0u;
  uint32_t all;
  const uint32_t pre = block_excl_scan(g, &all, sm.tmp);
  if (threadIdx.x == blockIdx.x) sm.first = pre;
  __syncthreads();
  uint32_t base = sm.first;
  for (uint32_t t0 = s0; t0 < s1; t0 += kTrThreads) {  // (the same trips in every thread)
    const uint32_t s = t0 + threadIdx.x;
    const uint4 v = s < s1 ? tr_slot_words(bits, s) : make_uint4(0u, 0u, 0u, 0u);
    // set bits before each word: at most 96
    const uint32_t b1 = __popc(v.x), b2 = b1 + __popc(v.y), b3 = b2 + __popc(v.z);
    const uint32_t run = b3 + __popc(v.w);
    uint32_t tot;
    const uint32_t r = base + block_excl_scan(run, &tot, sm.tmp);
    if (s < s1) rec[s] = make_uint2(r, (b1 << 8) | (b2 << 16) | (b3 << 24));
    base += tot;
  }
  return all;
}

// Folds the warp's min and max of the valid points of a frame into the block's (no barrier: a
// block meets every frame of a call, and folding the block's six values in two barriers a frame
// took a third of the pass over 8 posed frames).
__device__ __forceinline__ void tr_fold_extent(float mn[3], float mx[3], uint32_t* ext) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const uint32_t lo =
        __reduce_max_sync(kFullMask, mn[c] == INFINITY ? 0u : ~float_to_ordered(mn[c]));
    const uint32_t hi =
        __reduce_max_sync(kFullMask, mx[c] == -INFINITY ? 0u : float_to_ordered(mx[c]));
    if (lane == 0 && lo) {
      atomicMax(ext + c, lo);
      atomicMax(ext + 3 + c, hi);
    }
    mn[c] = INFINITY;
    mx[c] = -INFINITY;
  }
}

// Biased corner offsets of a point, in the form of a run's sums: z carries the number of points
// above its 26 bits (32 offsets of 21 bits fit them).
__device__ __forceinline__ void tr_offsets(const TrFrames& fm, int f, const float q[3],
                                           const float fi[3], uint32_t w[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c)
    w[c] = quant_biased(q[c], voxel_corner(fi[c], fm.org[3 * f + c], fm.leaf[f]), fm.inv_unit[f]);
  w[2] |= 1u << 26;
}
// A level in use: its slots' bits and records.
struct TrLevel {
  uint32_t* bits;
  uint2* rec;
  uint32_t ns;  // slots
};

// The rows' sums (arrays of `cap` entries): A = x + y 2^32 and B = z + points 2^32 (mod 2^64),
// C = the carries out of A's and B's low halves and out of A, 21 bits each (a cell of n < 2^30
// points carries at most n / 2^11 times); the row's key; attribute sums of channels 0, 1 and
// 2, 3 in 32 bits each.
struct TrRows {
  unsigned long long *A, *B, *C, *key, *att;
  int64_t cap;
  uint32_t rows;
};

// A run's sums at a row: x + y 2^32 and z + points 2^32, and the carries that the old values
// tell (and those the sums themselves hold beyond 64 and 32 bits).
__device__ __forceinline__ void tr_add(const TrRows& R, uint32_t row, unsigned long long va,
                                       unsigned long long vb, uint32_t hx = 0u, uint32_t hy = 0u,
                                       uint32_t hz = 0u) {
  const unsigned long long oa = atomicAdd(R.A + row, va), ob = atomicAdd(R.B + row, vb);
  // carries out of a 32-bit half: x into y, A out of 64 bits, z into the points
  const unsigned long long cx = hx + (((oa & 0xffffffffull) + (va & 0xffffffffull)) >> 32);
  const unsigned long long cy = hy + (oa + va < oa ? 1ull : 0ull);
  const unsigned long long cz = hz + (((ob & 0xffffffffull) + (vb & 0xffffffffull)) >> 32);
  if (cx | cy | cz) atomicAdd(R.C + row, cx | (cy << 21) | (cz << 42));
}

// Rows that many of a block's runs meet, summed in its shared memory before the rows are
// touched: in a crowded cloud without order the atomics of all blocks meet on a few sectors of
// L2.  Entry `row` mod the entries, first come, first kept.  Where there are fewer rows than
// entries, and runs for them, every row has its own; else a row takes one once a warp has met
// it again, or eight times in 32 runs.  Shuffled points, before -> after (and the radix sort): 2.5M
// of 10 cells 1255 -> 102 us (289), of 1000 cells 351 -> 118 (258), a quarter in one of 100,000
// cells 551 -> 156 (362); 4M of 100 cells 879 -> 190 (302).  The tests of a run cost clouds that
// are not crowded nothing that shows (2.5M points of 2.16M cells 216 and 217 us).
struct TrHot {
  uint32_t *tag, *x, *y, *z, *n, *carry;  // (carries of the sums, 10 bits each)
  uint32_t* att;                          // sums of 4 channels an entry
  uint32_t mask;
};
constexpr uint32_t kTrHotWords = 6, kTrHotAttWords = 4;
constexpr uint32_t kTrNoRow = 0xffffffffu;
constexpr uint32_t kTrHotPlaces = 1u << 21;  // points of a block whose carries fit 10 bits
static_assert((uint64_t(kTrHotPlaces) * 0x1fffffu) >> 32 < 1024, "10-bit carries");
__device__ __forceinline__ TrHot tr_hot(uint32_t* mem, uint32_t entries) {
  TrHot h;
  h.tag = mem;
  h.x = h.tag + entries;
  h.y = h.x + entries;
  h.z = h.y + entries;
  h.n = h.z + entries;
  h.carry = h.n + entries;
  h.att = h.carry + entries;
  h.mask = entries - 1u;
  return h;
}
// Adds to an entry; true for the entry's first run.
__device__ __forceinline__ bool tr_hot_add(const TrHot& h, uint32_t e, uint32_t x, uint32_t y,
                                           uint32_t z, uint32_t n) {
  const uint32_t ox = atomicAdd(h.x + e, x), oy = atomicAdd(h.y + e, y), oz = atomicAdd(h.z + e, z);
  const uint32_t c = (ox + x < x ? 1u : 0u) | (oy + y < y ? 1u << 10 : 0u) |
                     (oz + z < z ? 1u << 20 : 0u);
  if (c) atomicAdd(h.carry + e, c);
  return atomicAdd(h.n + e, n) == 0u;
}

template <bool kPosed, int K>
__global__ __launch_bounds__(kTrThreads, 1) void trie_kernel(const TrArgs a) {
  extern __shared__ __align__(16) unsigned char tr_smem[];
  __shared__ TrSmem sm;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t gt = blockIdx.x * kTrThreads + threadIdx.x, gthreads = gridDim.x * kTrThreads;
  const int F = a.fr.nframes;
  const TrFrames fm = tr_frames(tr_smem, F, kPosed);
  // this block's places (for its chunks at most) and runs in them
  const uint32_t cq = a.chunks / gridDim.x, cr = a.chunks % gridDim.x;
  const uint32_t places = (cq + (blockIdx.x < cr ? 1u : 0u)) * kChunk;
  const size_t w0 = size_t(blockIdx.x * cq + min(blockIdx.x, cr)) * kChunk;
  uint4* run = a.run + w0;
  uint32_t* runhi = a.runhi + w0;
  uint2* runatt = a.runatt + w0;
  uint32_t* pslot = a.pslot + w0;
  uint2* mask = a.mask + w0 / 32;
  uint32_t* firsts = a.first + w0 / (32 * K);
  int* err = a.err;
  uint32_t* bar = &a.st->fz_bar;
  uint32_t target = 0;
  const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);

  // (barriers below come before their first use)
  if (threadIdx.x == 0) {
    sm.nruns = 0u;
    sm.look = 1u;
  }
  for (int i = threadIdx.x; i < 6 * F; i += kTrThreads) fm.ext[i] = 0u;
  bool few = true, ordered = true;  // (the same in every block)
  if (a.large) {
    const unsigned long long smp = a.st->smp;
    const uint32_t pairs = uint32_t(smp) & 0x1fffffu;
    few = kTrSameOf * (uint32_t(smp >> 21) & 0x1fffffu) >= kTrSame * pairs;
    ordered = 2u * uint32_t(smp >> 42) >= pairs;
    // (camera frames: the ballots took 64 of them 0.6 % longer)
    if (few && threadIdx.x == 0) sm.look = 0u;
    if (!few && a.fr.n > kTrMidPoints) return;
  }
  // ---- extents; the first level's bits cleared ----
  if (!a.large)
    for (uint32_t i = gt; i < (1u << (kTrRootClear - 7)); i += gthreads)
      reinterpret_cast<uint4*>(a.root)[i] = zero4;
  if (kPosed)
    for (int f = threadIdx.x; f < F; f += kTrThreads) {
      Pose P;
      load_pose(a.fr, f, P);
      for (int r = 0; r < 3; ++r)
        fm.pose[4 * f + r] = make_float4(P.r[4 * r], P.r[4 * r + 1], P.r[4 * r + 2], P.r[4 * r + 3]);
      fm.pose[4 * f + 3] = make_float4(P.zlo, P.zhi, 0.0f, 0.0f);
    }
  uint32_t T;
  if (F > 1) {
    T = build_chunk_map(a.fr, fm.off, fm.cstart, sm.tmp, err);
  } else {
    const bool bad =
        a.fr.offsets && (__ldg(a.fr.offsets) != 0 || __ldg(a.fr.offsets + 1) != a.fr.n);
    T = bad ? 0u : static_cast<uint32_t>(ceil_div(a.fr.n, kChunk));
    if (threadIdx.x == 0) {
      fm.off[0] = 0;
      fm.off[1] = a.fr.n;
      fm.cstart[0] = 0u;
      fm.cstart[1] = T;
      if (bad && blockIdx.x == 0) set_error(err, kErrInvalidArg);
    }
    __syncthreads();
  }
  if (!a.large) {
    // four points a lane: 48 bytes in flight a lane, and a frame looked up for 128 points, not
    // 32 (8 posed frames: 40,500 -> 20,300 cycles, a 1280x720 frame 7,300 -> 5,600)
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    int cur = 0;
    tr_lanes<kPosed, 4, true>(a, fm, T, [&](uint32_t, const TrLanePoints<4>& t) {
      if (t.f != cur) {
        tr_fold_extent(mn, mx, fm.ext + 6 * cur);
        cur = t.f;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (!point_valid(t.q[j][0], t.q[j][1], t.q[j][2])) continue;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          mn[c] = fminf(mn[c], t.q[j][c]);
          mx[c] = fmaxf(mx[c], t.q[j][c]);
        }
      }
    });
    tr_fold_extent(mn, mx, fm.ext + 6 * cur);
    __syncthreads();
    for (int i = threadIdx.x; i < 6 * F; i += kTrThreads) {
      const uint32_t v = fm.ext[i];
      const int c = i % 6;
      FrameState& f = a.fs[i / 6];
      if (v) atomicMax(c < 3 ? &f.ord_min_inv[c] : &f.ord_max[c - 3], v);
    }
    if (!grid_barrier(bar, target, a.spin_limit, err)) return;
  }

  // ---- every frame's origin and leaf, the width of the keys (the same in every block) ----
  uint32_t key_shift = 64, kb, local_bits;
  bool go;
  {
    uint32_t bits = 0;
    bool bad_leaf = false;
    for (int f = threadIdx.x; f < F; f += kTrThreads) {
      const float leaf = a.fr.leaves ? __ldg(a.fr.leaves + f) : a.fr.leaf;
      const bool bad = !(leaf > 0.0f) || !isfinite(leaf);
      bad_leaf = bad_leaf || bad;
      const bool any = __ldcg(&a.fs[f].ord_min_inv[0]) != 0u;
      float o[3];
      for (int c = 0; c < 3; ++c) {
        if (a.fr.origin_in) {
          o[c] = __ldg(a.fr.origin_in + 3 * f + c);
        } else {
          const uint32_t u = __ldcg(&a.fs[f].ord_min_inv[c]);
          o[c] = u == 0u ? 0.0f : ordered_to_float(~u);
        }
        fm.org[3 * f + c] = o[c];
      }
      fm.leaf[f] = leaf;
      fm.rleaf[f] = fast_leaf(leaf) ? __fdiv_rn(1.0f, leaf) : 0.0f;
      fm.inv_unit[f] = quant_inv_unit(leaf);
      if (blockIdx.x == 0) {
        for (int c = 0; c < 3; ++c) {
          a.fs[f].origin[c] = o[c];
          if (!a.fr.origin_in && a.fr.origin_out) a.fr.origin_out[3 * f + c] = o[c];
        }
        a.fs[f].leaf = leaf;
      }
      if (any && !bad) {
        uint32_t ii[3];
        bool ok = true;
        for (int c = 0; c < 3; ++c)
          ok = ok && axis_index(ordered_to_float(__ldcg(&a.fs[f].ord_max[c])), o[c], leaf, &ii[c]);
        const uint64_t m = ok ? morton3(ii[0], ii[1], ii[2]) : ~0ull >> 1;
        bits = max(bits, m ? 64u - __clzll(static_cast<long long>(m)) : 0u);
      }
    }
    bits = __reduce_max_sync(kFullMask, bits);
    if (lane == 0) sm.bits[warp] = bits;
    const bool any_bad = __syncthreads_or(bad_leaf) != 0;
    local_bits = __reduce_max_sync(kFullMask, sm.bits[lane]);
    kb = local_bits;
    if (F > 1) {
      key_shift = local_bits;
      kb = local_bits + (32u - __clz(F - 1));
    }
    // (points out of range are invalid, whatever the width: their frame's bound is 63 bits)
    go = !any_bad && kb <= 63u && T > 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      a.st->key_shift = key_shift;
      a.st->nframes = F;
      if (any_bad) set_error(err, kErrInvalidArg);
      else if (kb > 63u) set_error(err, kErrRange);
    }
  }
  if (!go) {  // (the same in every block)
    if (blockIdx.x == 0 && !a.large) {
      if (a.out.frame_offsets)
        for (int f = threadIdx.x; f <= F; f += kTrThreads) a.out.frame_offsets[f] = 0;
      if (threadIdx.x == 0) *a.out.num_voxels = 0;
    }
    return;
  }
  if (!few && kb > kTrMidBits && (kb <= 32u || !ordered)) return;
  const bool wide = local_bits > 32u;
  // levels, and the key bits below level 1
  const uint32_t root_bits = static_cast<uint32_t>(a.root_bits);
  const int levels =
      kb <= root_bits ? 1 : 1 + int((kb - root_bits + kTrDigitBits - 1) / kTrDigitBits);
  const uint32_t below = uint32_t(levels - 1) * kTrDigitBits;
  const uint32_t top = max(kb - below, uint32_t(kTrDigitBits));
  TrLevel lv{a.root, a.rootrec, 1u << (top - kTrDigitBits)};
  const int64_t cap = a.slots;
  const bool with_attrs = a.out.attrs_in != nullptr;

  // the bits of the first level not cleared yet
  const uint32_t clean = a.large ? 0u : 1u << (kTrRootClear - kTrDigitBits);
  if (lv.ns > clean) {  // (the same in every block)
    for (uint32_t i = clean + gt; i < lv.ns; i += gthreads)
      reinterpret_cast<uint4*>(a.root)[i] = zero4;
    if (!grid_barrier(bar, target, a.spin_limit, err)) return;
  }

  // ---- runs; level 1 marked ----
  bool range_bad = false;
  tr_lanes<kPosed, K, true>(a, fm, T, [&](uint32_t part, const TrLanePoints<K>& t) {
    uint64_t key[K];
    uint32_t w[K][3];
#pragma unroll
    for (int j = 0; j < K; ++j) {
      float fi[3];
      key[j] = kNoKey;
      w[j][0] = w[j][1] = w[j][2] = 0u;
      if (tr_key(fm, t.f, t.q[j][0], t.q[j][1], t.q[j][2], wide, key_shift, &key[j], fi,
                 &range_bad))
        tr_offsets(fm, t.f, t.q[j], fi, w[j]);
    }
    const LaneRuns r = lane_runs<K>(key);
    run_sums<K, 3>(w, r);
    uint32_t tails[K], total = 0u, base = 0u;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      tails[j] = __ballot_sync(kFullMask, (r.tail >> j) & 1u);
      total += __popc(tails[j]);
    }
    if (lane == 0) base = atomicAdd(&sm.nruns, total);
    base = __shfl_sync(kFullMask, base, 0);
    const uint32_t place = tr_place<K>(tails);
    if (a.out.p2v) {
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const uint32_t valid = __ballot_sync(kFullMask, key[j] != kNoKey);
        if (lane == 0) mask[part * K + j] = make_uint2(tails[j], valid);
      }
      if (lane == 0) firsts[part] = base;
    }
    uint32_t word[K], bit[K], seen[K];
    uint32_t i = base + place;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const bool tail = (r.tail >> j) & 1u;
      const uint32_t id = static_cast<uint32_t>(key[j] >> below);  // (at most 28 bits)
      word[j] = id >> 5;
      bit[j] = seen[j] = 0u;
      if (tail) {
        run[i] = make_uint4(uint32_t(key[j]), w[j][0], w[j][1], w[j][2]);
        if (wide || kb > 32u) runhi[i] = static_cast<uint32_t>(key[j] >> 32);
        ++i;
      }
      if (tail && (id >> kTrDigitBits) < lv.ns) {
        bit[j] = 1u << (id & 31u);
        seen[j] = __ldca(a.root + word[j]);
      }
    }
    if (with_attrs) {
      uint32_t at[K][2];
#pragma unroll
      for (int j = 0; j < K; ++j) {
        at[j][0] = at[j][1] = 0u;
        if (key[j] == kNoKey) continue;
        const uint8_t* b = a.out.attrs_in + size_t(t.p + j) * a.out.channels;
#pragma unroll
        for (int c = 0; c < 4; ++c)  // two 16-bit sums a word (32 x 255 fit)
          if (c < a.out.channels) at[j][c >> 1] |= uint32_t(__ldg(b + c)) << (16 * (c & 1));
      }
      run_sums<K, 2>(at, r);
      uint32_t i = base + place;
#pragma unroll
      for (int j = 0; j < K; ++j)
        if ((r.tail >> j) & 1u) runatt[i++] = make_uint2(at[j][0], at[j][1]);
    }
    // the bits not seen set; of two points a lane's in one word together (a scan of 1M points,
    // whose runs are single points: 10 us less; large calls mostly see them set)
#pragma unroll
    for (int j = 0; j < K; ++j) bit[j] &= ~seen[j];
    if (K == 2 && word[0] == word[K - 1]) {
      bit[K - 1] |= bit[0];
      bit[0] = 0u;
    }
#pragma unroll
    for (int j = 0; j < K; ++j)
      if (__any_sync(kFullMask, bit[j] != 0u)) tr_set(a.root, word[j], bit[j]);
  });
  if (__any_sync(kFullMask, range_bad) && lane == 0) set_error(err, kErrRange);
  if (!grid_barrier(bar, target, a.spin_limit, err)) return;
  const uint32_t nruns = min(sm.nruns, places);
  if (threadIdx.x == 0) sm.single = nruns >= places - places / 4u ? 1u : 0u;

  // ---- every level ranked, the next one marked ----
  uint32_t rows = 0;
  for (int j = 1;; ++j) {
    uint32_t* agg = a.stat + size_t(j - 1) * kTrMaxGrid;
    tr_count(lv.bits, lv.ns, agg, sm.tmp);
    if (!grid_barrier(bar, target, a.spin_limit, err)) return;
    const uint32_t set = tr_rank_slots(lv.bits, lv.rec, lv.ns, agg, sm);
    const uint32_t n1 = static_cast<uint32_t>(min(int64_t(set), cap));
    if (set > n1) {  // (the same in every block)
      if (a.large) return;  // more cells than the buffers hold: the sort path
      if (blockIdx.x == 0 && threadIdx.x == 0) set_error(err, kErrInvalidArg);
    }
    if (j == levels) {
      rows = n1;
      break;
    }
    // the buffers alternate so that the last level lies in x
    char* nb = ((levels - j - 1) & 1) ? a.y : a.x;
    uint32_t* nbits = reinterpret_cast<uint32_t*>(nb);
    for (uint32_t i = gt; i < n1; i += gthreads) reinterpret_cast<uint4*>(nbits)[i] = zero4;
    if (!grid_barrier(bar, target, a.spin_limit, err)) return;
    const uint32_t sh = below - uint32_t(j) * kTrDigitBits;  // key bits below the next level
    // Where the prefixes are many for the points, and the runs hardly more than points, few runs
    // would see their bit set: it is not looked for, one of four accesses a run (2.5M shuffled
    // points of 60-bit keys 738 -> 631 us, of 45 bits 425 -> 390; 1M points of a scan in its
    // order 2 % less; a 1280x720 frame at 0.01 m, whose runs meet again, would take 3 % more).
    const bool sparse = int64_t(n1) * kTrSparse >= a.fr.n && sm.single;  // (a block's own)
    for (uint32_t i0 = 0; i0 < nruns; i0 += 2 * kTrThreads) {
      uint32_t id[2], seen[2], v[2];
      uint2 r[2];
      bool in[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t i = i0 + kTrThreads * u + threadIdx.x;
        in[u] = i < nruns;
        id[u] = 0u;
        v[u] = 0u;
        r[u] = make_uint2(~0u, 0u);
        if (!in[u]) continue;
        uint64_t key = run[i].x;
        if (kb > 32u) key |= uint64_t(runhi[i]) << 32;
        id[u] = static_cast<uint32_t>(key >> sh) & ((kTrDigit << kTrDigitBits) | kTrDigit);  // two digits
        const uint32_t s0 =
            j == 1 ? static_cast<uint32_t>(key >> (sh + 2 * kTrDigitBits)) : pslot[i];
        if (s0 < lv.ns) {
          v[u] = __ldcg(lv.bits + trie_word(s0, id[u] >> kTrDigitBits));
          r[u] = __ldcg(lv.rec + s0);
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        seen[u] = 0u;
        if (!in[u]) continue;
        const uint32_t s = r[u].x == ~0u ? ~0u : tr_rank(r[u], v[u], id[u] >> kTrDigitBits);
        pslot[i0 + kTrThreads * u + threadIdx.x] = s;
        if (s >= n1) {
          set_error(err, kErrInvalidArg);
          in[u] = false;
          continue;
        }
        v[u] = 1u << (id[u] & 31u);  // (the bit and, below, its word)
        id[u] = trie_word(s, id[u] & kTrDigit);
        if (!sparse) seen[u] = __ldcg(nbits + id[u]);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u)
        tr_set(nbits, id[u], in[u] ? v[u] & ~seen[u] : 0u);
    }
    if (!grid_barrier(bar, target, a.spin_limit, err)) return;
    lv = TrLevel{nbits, reinterpret_cast<uint2*>(nb + size_t(cap) * (kTrWords * 4)), n1};
  }

  // ---- the rows' sums cleared ----
  TrRows R;
  R.A = reinterpret_cast<unsigned long long*>(a.y);
  R.B = R.A + cap;
  R.C = R.B + cap;
  R.key = R.C + cap;
  R.att = a.rowatt;
  R.cap = cap;
  R.rows = rows;
  for (uint32_t i = gt; i < rows; i += gthreads) {
    R.A[i] = 0ull;
    R.B[i] = 0ull;
    R.C[i] = 0ull;
    if (with_attrs) {
      R.att[i] = 0ull;
      R.att[i + cap] = 0ull;
    }
  }
  // (the same in every thread of the block; few runs are not worth clearing the table)
  const uint32_t hot_entries = places <= kTrHotPlaces && nruns >= kTrThreads ? a.hot : 0u;
  const TrHot hot = tr_hot(reinterpret_cast<uint32_t*>(tr_smem + tr_frames_bytes(F, kPosed)), a.hot);
  const bool all_hot = rows <= hot_entries && nruns / 2u >= rows;
  for (uint32_t e = threadIdx.x; e < hot_entries; e += kTrThreads) {
    hot.tag[e] = all_hot && e < rows ? e : kTrNoRow;
    hot.x[e] = hot.y[e] = hot.z[e] = hot.n[e] = hot.carry[e] = 0u;
  }
  if (with_attrs)
    for (uint32_t e = threadIdx.x; e < kTrHotAttWords * hot_entries; e += kTrThreads)
      hot.att[e] = 0u;
  if (threadIdx.x == 0) sm.hot = all_hot ? 1u : 0u;
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) {
      // more cells than output rows: recorded once, here; the first cap rows are written
      if (int64_t(rows) > a.out.cap) set_error(err, kErrCapacity);
      *a.out.num_voxels = rows;
      if (a.large) {
        a.st->narrow = 1u;
        a.st->msd = kRowsWritten;
      }
    }
    if (a.out.frame_offsets && (F == 1 || rows == 0))
      for (int f = threadIdx.x; f <= F; f += kTrThreads)
        a.out.frame_offsets[f] = f == F ? rows : 0;
  }
  if (!grid_barrier(bar, target, a.spin_limit, err)) return;

  // ---- every run's points and sums at its row ----
  uint32_t met = kTrNoRow;  // a row that the warp has met, looked for again
  for (uint32_t i0 = 0; i0 < nruns; i0 += kTrThreads) {
    const uint32_t i = i0 + threadIdx.x;
    uint4 e = zero4;
    uint32_t row = kTrNoRow;
    if (i < nruns) {
      e = run[i];
      const uint32_t s0 = levels == 1 ? e.x >> kTrDigitBits : pslot[i];
      if (s0 < lv.ns) {
        const uint32_t v = __ldcg(lv.bits + trie_word(s0, e.x & kTrDigit));
        row = tr_rank(__ldcg(lv.rec + s0), v, e.x & kTrDigit);
      }
      if (row >= rows) {
        set_error(err, kErrInvalidArg);
        row = kTrNoRow;
      }
      if (a.out.p2v) pslot[i] = row;
    }
    bool in_hot = false;
    if (hot_entries) {
      if (!all_hot && sm.look) {
        const uint32_t lead = __shfl_sync(kFullMask, row, 0);
        const uint32_t again = __ballot_sync(kFullMask, row == met && row != kTrNoRow);
        const bool many = __popc(__ballot_sync(kFullMask, row == lead)) >= 8;
        if (many || __popc(again) >= 2) {
          const uint32_t r = many ? lead : met;
          if (lane == 0 && r != kTrNoRow &&
              atomicCAS(hot.tag + (r & hot.mask), kTrNoRow, r) == kTrNoRow)
            sm.hot = 1u;
        } else if (again == 0u) {
          met = lead;
        }
      }
      in_hot = row != kTrNoRow && *reinterpret_cast<volatile uint32_t*>(&sm.hot) != 0u &&
               *reinterpret_cast<volatile uint32_t*>(hot.tag + (row & hot.mask)) == row;
    }
    if (row == kTrNoRow) continue;
    const uint2 at = with_attrs ? runatt[i] : make_uint2(0u, 0u);
    bool first = true;
    if (in_hot) {
      const uint32_t h = row & hot.mask;
      first = tr_hot_add(hot, h, e.y, e.z, e.w & 0x3ffffffu, e.w >> 26);
      if (with_attrs) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c < a.out.channels)
            atomicAdd(hot.att + kTrHotAttWords * h + c, ((c >> 1 ? at.y : at.x) >> (16 * (c & 1))) & 0xffffu);
      }
    } else {
      tr_add(R, row, e.y | ((unsigned long long)e.z << 32),
             (e.w & 0x3ffffffu) | ((unsigned long long)(e.w >> 26) << 32));
      if (with_attrs) {
        atomicAdd(R.att + row,
                  (unsigned long long)(at.x & 0xffffu) | ((unsigned long long)(at.x >> 16) << 32));
        if (a.out.channels > 2)
          atomicAdd(R.att + cap + row, (unsigned long long)(at.y & 0xffffu) |
                                           ((unsigned long long)(at.y >> 16) << 32));
      }
    }
    if (first) {
      uint64_t key = e.x;
      if (kb > 32u) key |= uint64_t(runhi[i]) << 32;
      R.key[row] = key;  // (every run of the row stores the same key)
    }
  }
  __syncthreads();
  if (sm.hot)
    for (uint32_t h = threadIdx.x; h < hot_entries; h += kTrThreads) {
      const uint32_t n = hot.n[h], row = hot.tag[h];
      if (n == 0u) continue;
      const uint32_t c = hot.carry[h], cx = c & 1023u, cy = (c >> 10) & 1023u, cz = c >> 20;
      // x + y 2^32 of sums beyond 32 bits: the carries of x add to y
      const unsigned long long y = hot.y[h] + (unsigned long long)cx;
      tr_add(R, row, hot.x[h] | (y << 32), hot.z[h] | ((unsigned long long)(n + cz) << 32), cx,
             cy + uint32_t(y >> 32), cz);
      if (with_attrs) {
        const uint32_t* t = hot.att + kTrHotAttWords * h;
        atomicAdd(R.att + row, t[0] | ((unsigned long long)t[1] << 32));
        if (a.out.channels > 2) atomicAdd(R.att + cap + row, t[2] | ((unsigned long long)t[3] << 32));
      }
    }
  if (a.out.p2v) {  // a point's row is its run's: that of the next point to end one
    tr_lanes<kPosed, K, false>(a, fm, T, [&](uint32_t part, const TrLanePoints<K>& t) {
      uint32_t row[K], tails[K], m = 0u, valid = 0u, first = ~0u;
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const uint2 b = mask[part * K + j];
        tails[j] = b.x;
        m |= ((b.x >> lane) & 1u) << j;
        valid |= ((b.y >> lane) & 1u) << j;
      }
      const uint32_t place = firsts[part] + tr_place<K>(tails);
#pragma unroll
      for (int j = K - 1; j >= 0; --j) {
        row[j] = ~0u;
        if (!((m >> j) & 1u)) continue;
        const uint32_t i = place + __popc(m & ((1u << j) - 1u));
        first = row[j] = i < nruns ? pslot[i] : ~0u;
      }
      const uint32_t later = (__ballot_sync(kFullMask, m != 0u) >> 1) >> lane;
      uint32_t cur = __shfl_sync(kFullMask, first, later ? int(lane) + __ffs(later) : int(lane));
#pragma unroll
      for (int j = K - 1; j >= 0; --j) {
        if ((m >> j) & 1u) cur = row[j];
        row[j] = (valid >> j) & 1u ? cur : ~0u;
      }
      int32_t* dst = a.out.p2v + t.p;
      if (K == 4 && t.m == K && (reinterpret_cast<uintptr_t>(dst) & 15u) == 0u) {
        *reinterpret_cast<uint4*>(dst) = make_uint4(row[0], row[1 % K], row[2 % K], row[3 % K]);
      } else {
#pragma unroll
        for (int j = 0; j < K; ++j)
          if (j < t.m) dst[j] = static_cast<int32_t>(row[j]);
      }
    });
  }
  if (!grid_barrier(bar, target, a.spin_limit, err)) return;

  // ---- rows (a thread a row), the first out.cap of them ----
  // (every error but the capacity one stops it; none is set from here on)
  if (__syncthreads_or(threadIdx.x == 0 && error_raised(err) &&
                       *reinterpret_cast<const volatile int*>(err) != kErrCapacity))
    return;
  const bool small = kb <= 32u;
  RowCtx rc;
  rc.fs = a.fs;
  rc.key_shift = key_shift;
  rc.o1[0] = fm.org[0];
  rc.o1[1] = fm.org[1];
  rc.o1[2] = fm.org[2];
  rc.leaf1 = fm.leaf[0];
  for (uint32_t row = gt; row < rows; row += gthreads) {
    const unsigned long long key = __ldcg(R.key + row);
    if (F > 1 && a.out.frame_offsets) {
      const uint32_t fk = key_frame(key, key_shift);
      const uint32_t f0 = row > 0 ? key_frame(__ldcg(R.key + row - 1), key_shift) + 1u : 0u;
      for (uint32_t f = f0; f <= fk; ++f) a.out.frame_offsets[f] = row;
      if (row + 1u == rows)
        for (uint32_t f = fk + 1u; f <= uint32_t(F); ++f) a.out.frame_offsets[f] = rows;
    }
    if (int64_t(row) >= a.out.cap) continue;
    const unsigned long long A = __ldcg(R.A + row), B = __ldcg(R.B + row), C = __ldcg(R.C + row);
    const unsigned long long cx = C & 0x1fffffull, cy = (C >> 21) & 0x1fffffull, cz = C >> 42;
    // x = low(A) + cx 2^32; y = high(A) + cy 2^32 - cx; z = low(B) + cz 2^32;
    // points = high(B) - cz
    const unsigned long long sb[3] = {(A & 0xffffffffull) + (cx << 32),
                                      (A >> 32) + (cy << 32) - cx,
                                      (B & 0xffffffffull) + (cz << 32)};
    Acc r;
    r.n = static_cast<uint32_t>((B >> 32) - cz);
    float sf[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      r.s[c] = static_cast<long long>(sb[c]) + static_cast<long long>(r.n) * kQMin;
      sf[c] = __ll2float_rn(r.s[c]);
    }
    if (small)
      put_row32(rc, a.out, row, static_cast<uint32_t>(key), r.n, sf, r.s, err);
    else
      put_row(rc, a.out, row, key, r, err);
    if (with_attrs) {
      const unsigned long long t[2] = {__ldcg(R.att + row), __ldcg(R.att + cap + row)};
      // The exact sum over the points, divided in FP64 and rounded to float32.  Where both are
      // exact in binary32 its own division gives the same bits (FP64 has more than twice its
      // digits, so rounding a quotient twice changes nothing), without the few FP64 units: 2.5M
      // shuffled points with 4 channels 584 -> 398 us (the radix sort 487).
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c < a.out.channels) {
          const uint32_t sum = uint32_t(t[c >> 1] >> (32 * (c & 1)));
          a.out.attrs_out[size_t(row) * a.out.channels + c] =
              (sum | r.n) < (1u << 24)
                  ? __fdiv_rn(__uint2float_rn(sum), __uint2float_rn(r.n))
                  : __double2float_rn(
                        __ddiv_rn(static_cast<double>(sum), static_cast<double>(r.n)));
        }
    }
  }
}

// What the launch reads before writing: the state (the pyramid's tile counters among it), the
// frames' extent words and the error word.
__global__ __launch_bounds__(1024) void trie_clear_kernel(uint32_t* st, uint32_t words, int* err) {
  for (uint32_t i = threadIdx.x; i < words; i += 1024) st[i] = 0u;
  if (threadIdx.x == 0) *err = 0;
}

// Entries of the table of hot rows, and their bytes.  Smaller calls have none: clearing and
// looking costs them 0.4 us, and even ten cells of 100,000 points take 81 us without (38 with,
// the radix sort 116).
constexpr int64_t kTrHotPoints = int64_t(1) << 17;
constexpr uint32_t tr_hot_entries(bool attrs, int64_t n) {
  return n < kTrHotPoints ? 0u : (attrs ? 2048u : 4096u);
}
constexpr size_t tr_hot_bytes(bool attrs, int64_t n) {
  return size_t(tr_hot_entries(attrs, n)) * (kTrHotWords + (attrs ? kTrHotAttWords : 0u)) * 4u;
}
// Dynamic shared memory of a block at most: the tables of kMaxFrames frames and the hot rows.
constexpr size_t kTrSmem = tr_frames_bytes(kMaxFrames, true) + tr_hot_bytes(false, kMaxPoints);
static_assert(tr_hot_bytes(true, kMaxPoints) <= tr_hot_bytes(false, kMaxPoints), "the larger table");
static_assert(kTrSmem + sizeof(TrSmem) <= 227 * 1024, "block shared memory");

// Blocks an SM holds of the kernel (0: it cannot run there), per device.
using TrKernel = void (*)(const TrArgs);
TrKernel trie_kernel_of(bool posed, bool large) {
  if (posed) return large ? trie_kernel<true, kTrLaneLarge> : trie_kernel<true, kTrLane>;
  return large ? trie_kernel<false, kTrLaneLarge> : trie_kernel<false, kTrLane>;
}
int trie_blocks_per_sm(bool posed, bool large) {
  static DeviceInt cache[2][2];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  return cache[posed ? 1 : 0][large ? 1 : 0].get(dev, [posed, large] {
    const void* fn = reinterpret_cast<const void*>(trie_kernel_of(posed, large));
    int v = 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kTrSmem)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, fn, kTrThreads, kTrSmem) != cudaSuccess)
      v = 0;
    (void)cudaGetLastError();
    return v;
  });
}

}  // namespace

bool trie_available(bool posed) {
  return trie_blocks_per_sm(posed, false) > 0 && trie_blocks_per_sm(posed, true) > 0;
}

void warm_trie_config() {
  for (int i = 0; i < 4; ++i) (void)trie_blocks_per_sm((i & 1) != 0, (i & 2) != 0);
}

cudaError_t launch_trie(const float* xyz, const FramesArg& fr, State* st, FrameState* fs, char* ws,
                        const TrieLayout& L, const SegOut& out, uint32_t spin_limit, int* err,
                        cudaStream_t stream) {
  TrArgs a;
  a.xyz = xyz;
  a.fr = fr;
  a.st = st;
  a.fs = fs;
  a.root = reinterpret_cast<uint32_t*>(ws + L.root);
  a.rootrec = reinterpret_cast<uint2*>(ws + L.rootrec);
  a.x = ws + L.x;
  a.y = ws + L.y;
  a.run = reinterpret_cast<uint4*>(ws + L.run);
  a.runhi = reinterpret_cast<uint32_t*>(ws + L.runhi);
  a.runatt = reinterpret_cast<uint2*>(ws + L.runatt);
  a.rowatt = reinterpret_cast<unsigned long long*>(ws + L.rowatt);
  a.pslot = reinterpret_cast<uint32_t*>(ws + L.pslot);
  a.mask = reinterpret_cast<uint2*>(ws + L.mask);
  a.first = reinterpret_cast<uint32_t*>(ws + L.first);
  a.stat = reinterpret_cast<uint32_t*>(ws + L.stat);
  a.out = out;
  const bool attrs = out.attrs_in != nullptr;
  a.hot = tr_hot_entries(attrs, fr.n);
  a.slots = L.slots;
  a.spin_limit = spin_limit;
  a.err = err;
  // one block a chunk of points, but enough of them to clear and rank the first level
  const int64_t chunks = max_chunks(fr.n, fr.nframes);
  const int64_t g = trie_grid(chunks, num_sms());
  a.chunks = static_cast<uint32_t>(chunks);
  a.large = fr.n > kTrMaxPoints ? 1 : 0;
  a.root_bits = trie_root_bits(fr.n);
  if (!a.large) {
    const size_t head = reinterpret_cast<char*>(fs + fr.nframes) - reinterpret_cast<char*>(st);
    trie_clear_kernel<<<1, 1024, 0, stream>>>(reinterpret_cast<uint32_t*>(st),
                                             static_cast<uint32_t>(head / sizeof(uint32_t)), err);
  }
  void* args[] = {&a};
  const void* fn = reinterpret_cast<const void*>(trie_kernel_of(posed(fr), a.large != 0));
  return launch_cooperative(fn, g, kTrThreads, args,
                            tr_frames_bytes(fr.nframes, posed(fr)) + tr_hot_bytes(attrs, fr.n),
                            stream);
}

}  // namespace vg
