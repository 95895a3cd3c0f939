// Steps a1-a5 by an occupancy trie: one cooperative launch, no sort.
//
// arXiv 2102.11084 Sec. II-C classifies every point into a cell of an ordered subdivision of
// space and keeps one point per occupied cell, in the order of the cells.  A sort orders all
// points to get there; the occupied cells alone give the order: the rank of a cell's key
// among the occupied keys is its row, and the points add their offsets at the row (exact
// integers, so in any order).  The ranks come from a trie of bitmaps over the keys:
//   level 1   one bit per prefix of up to 24 key bits (28 for large clouds), grouped in slots
//             of 2^8 bits;
//   level j   one slot of 2^8 bits per occupied prefix of level j - 1, numbered by its rank
//             there, for the next 8 key bits.
// Each level is marked by a pass over the points, its set bits counted per block and, after a
// barrier, ranked: a slot's record holds the set bits before the slot and, as bytes, before
// each of its 8 words.  Keys of up to 24 bits take one level, each 8 bits more another one.
// The points are read again by every pass (from L2 for the clouds this is made for) and
// their keys computed again: that costs less than keeping them.
//
// Passes, with a grid barrier after each:
//   extents   per-frame min and max; the first level's bits cleared;
//   mark      (per level) the bit of every point's prefix: lanes of a warp with the same
//             word merged, and no atomic where the bit is seen set already;
//   count, rank
//   add       runs of equal keys among a warp's 32 consecutive points (neighbouring pixels of a
//             camera frame often share a cell) summed by a segmented scan; a run adds its points
//             and sums at its row with two 64-bit atomics whose returned values tell the
//             carries out of their 32-bit halves; point_to_voxel and attribute sums here too;
//   rows      one thread a row: the centroid, by the formula and from the integer sums of every
//             other grouping, so the rows are theirs bit for bit.
// Bound by the latency of the passes and barriers for a camera frame and by instruction issue
// for several (every pass computes keys), not by HBM: TRIE_NUMBERS
// Every wait is bounded (kErrTimeout after the limit, and the block returns), and every index
// read back from scratch is checked against its buffer.
#include <cstddef>

#include "vg_device.cuh"
#include "vg_internal.h"
#include "vg_rows.cuh"
#include "vg_stream.cuh"
#include "vg_trie.h"

namespace vg {
namespace {

struct TrArgs {
  const float* xyz;
  FramesArg fr;
  State* st;
  FrameState* fs;
  uint32_t* root;      // first level: bits, then records (below)
  uint4* rootrec;
  char* x;             // buffers of the further levels
  char* y;
  uint32_t* pslot;     // per point: the slot of its prefix (at the last point of its run)
  uint32_t* stat;      // per level (8): the blocks' totals
  SegOut out;
  int64_t slots;       // slots and rows the buffers hold
  int root_bits;
  uint32_t spin_limit;
  int* err;
};

struct TrSmem {
  int64_t off[kMaxFrames + 1];
  uint32_t cstart[kMaxFrames + 1];
  float org[kMaxFrames][3];
  float leaf[kMaxFrames];
  float rleaf[kMaxFrames];
  float inv_unit[kMaxFrames];
  uint32_t tmp[kTrThreads / 32];
  float red[kTrThreads / 32][6];
  unsigned long long kmax[kTrThreads / 32];
  uint32_t bits[kTrThreads / 32];
  uint32_t first;
};
static_assert(sizeof(TrSmem) <= 48 * 1024, "static shared memory");

// f(frame, point index, inside, x, y, z) for every point of chunks [c0, c1) (1024 points of
// one frame each, a thread a point; all threads call f, `inside` false past the frame's end,
// where the coordinates are NaN).  The next chunk's points are loaded one step ahead.
template <bool kPosed, typename F>
__device__ __forceinline__ void tr_points(const TrArgs& a, const TrSmem& sm, uint32_t c0,
                                          uint32_t c1, F f) {
  const int nf = a.fr.nframes;
  const float nan = __int_as_float(0x7fc00000);
  int fn = 0;
  int64_t pn = 0;
  bool inn = false;
  float nx = nan, ny = nan, nz = nan;
  auto load = [&](uint32_t c) {
    fn = nf > 1 ? chunk_frame(sm.cstart, nf, c) : 0;
    pn = sm.off[fn] + int64_t(c - sm.cstart[fn]) * kChunk + threadIdx.x;
    inn = pn < sm.off[fn + 1];
    const float* q = a.xyz + 3 * pn;
    nx = inn ? __ldg(q) : nan;
    ny = inn ? __ldg(q + 1) : nan;
    nz = inn ? __ldg(q + 2) : nan;
  };
  if (c0 < c1) load(c0);
  Pose P;
  int pose_f = -1;
  for (uint32_t c = c0; c < c1; ++c) {
    float x = nx, y = ny, z = nz;
    const int fr = fn;
    const int64_t p = pn;
    const bool in = inn;
    if (c + 1 < c1) load(c + 1);
    if (kPosed) {
      if (fr != pose_f) {
        load_pose(a.fr, fr, P);
        pose_f = fr;
      }
      pose_point(P, x, y, z);
    }
    f(fr, p, in, x, y, z);
  }
}

// The sort key of a point of frame f (indices in ijk); false for an invalid point or one out
// of range (*range_bad set).
__device__ __forceinline__ bool tr_key(const TrSmem& sm, int f, float x, float y, float z,
                                       bool wide, uint32_t key_shift, uint64_t* key,
                                       uint32_t ijk[3], bool* range_bad) {
  const float o[3] = {sm.org[f][0], sm.org[f][1], sm.org[f][2]};
  if (!point_index(x, y, z, o, sm.leaf[f], sm.rleaf[f], ijk, range_bad)) return false;
  if (wide)
    *key = key_compose(uint32_t(f), morton3(ijk[0], ijk[1], ijk[2]), key_shift);
  else  // per-frame keys of at most 32 bits
    *key = key_compose(uint32_t(f),
                       spread3_32(ijk[0]) | (spread3_32(ijk[1]) << 1) | (spread3_32(ijk[2]) << 2),
                       key_shift);
  return true;
}

// Last lane of the calling lane's run of equal keys among the valid lanes of the warp; the
// run's first lane in *head.
__device__ __forceinline__ uint32_t tr_run(uint64_t key, bool ok, uint32_t* head) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t prev = __shfl_up_sync(kFullMask, key, 1);
  const uint32_t okm = __ballot_sync(kFullMask, ok);
  const uint32_t heads =
      __ballot_sync(kFullMask, lane == 0 || !ok || !((okm >> (lane - 1u)) & 1u) || key != prev);
  *head = 31u - __clz(heads & (kFullMask >> (31u - lane)));
  const uint32_t later = lane == 31u ? 0u : heads >> (lane + 1u);
  return later ? lane + __ffs(later) - 1u : 31u;
}

// Sets bit d (0..255) of slot s for the lanes of `em`: one atomic a word among the warp's
// lanes that do not see their bit set (kCached: through L1, where a stale line can only
// lack bits).
template <bool kCached>
__device__ __forceinline__ void tr_mark(uint32_t* bits, uint32_t s, uint32_t d, bool emit) {
  const uint32_t word = s * kTrWords + (d >> 5);
  const uint32_t bit = 1u << (d & 31u);
  bool need = false;
  if (emit) need = ((kCached ? __ldca(bits + word) : __ldcg(bits + word)) & bit) == 0u;
  const uint32_t m = __ballot_sync(kFullMask, need);
  if (need) {
    const uint32_t peers = __match_any_sync(m, word);
    const uint32_t v = __reduce_or_sync(peers, bit);
    if (int(threadIdx.x & 31u) == __ffs(peers) - 1) atomicOr(bits + word, v);
  }
}

// Rank of bit d of slot s (the slots' records and bits).
__device__ __forceinline__ uint32_t tr_rank(const uint4* rec, const uint32_t* bits, uint32_t s,
                                            uint32_t d) {
  const uint32_t w = d >> 5;
  const uint32_t v = __ldcg(bits + s * kTrWords + w);
  const uint4 r = __ldcg(rec + s);
  const uint32_t before = ((w & 4u ? r.z : r.y) >> (8u * (w & 3u))) & 255u;
  return r.x + before + __popc(v & ((1u << (d & 31u)) - 1u));
}

__device__ __forceinline__ void tr_slot_words(const uint32_t* bits, uint32_t s, uint4 v[2]) {
  const uint4* q = reinterpret_cast<const uint4*>(bits) + 2 * size_t(s);
  v[0] = __ldcg(q);
  v[1] = __ldcg(q + 1);
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
    uint4 v[2];
    tr_slot_words(bits, s, v);
    mine += __popc(v[0].x) + __popc(v[0].y) + __popc(v[0].z) + __popc(v[0].w) + __popc(v[1].x) +
            __popc(v[1].y) + __popc(v[1].z) + __popc(v[1].w);
  }
  uint32_t total;
  (void)block_excl_scan(mine, &total, tmp);
  if (threadIdx.x == 0) agg[blockIdx.x] = total;
}
// Returns the grand total (the same in every block).  Contains __syncthreads.
__device__ __forceinline__ uint32_t tr_rank_slots(const uint32_t* bits, uint4* rec, uint32_t ns,
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
    uint4 v[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
    if (s < s1) tr_slot_words(bits, s, v);
    const uint32_t w[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
    uint32_t run = 0, lo = 0, hi = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {  // set bits before word i: at most 224
      if (i < 4) lo |= run << (8 * i);
      else hi |= run << (8 * (i - 4));
      run += __popc(w[i]);
    }
    uint32_t tot;
    const uint32_t r = base + block_excl_scan(run, &tot, sm.tmp);
    if (s < s1) rec[s] = make_uint4(r, lo, hi, 0u);
    base += tot;
  }
  return all;
}

// Folds the block's min and max of the valid points of frame f into its state.  Contains
// __syncthreads.
__device__ __forceinline__ void tr_flush_extent(float mn[3], float mx[3], FrameState* fs, int f,
                                                TrSmem& sm) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int off = 16; off; off >>= 1) {
      mn[c] = fminf(mn[c], __shfl_xor_sync(kFullMask, mn[c], off));
      mx[c] = fmaxf(mx[c], __shfl_xor_sync(kFullMask, mx[c], off));
    }
  __syncthreads();
  if (lane == 0)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      sm.red[warp][c] = mn[c];
      sm.red[warp][3 + c] = mx[c];
    }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float m = sm.red[lane][c], M = sm.red[lane][3 + c];
#pragma unroll
      for (int off = 16; off; off >>= 1) {
        m = fminf(m, __shfl_xor_sync(kFullMask, m, off));
        M = fmaxf(M, __shfl_xor_sync(kFullMask, M, off));
      }
      if (lane == 0 && m != INFINITY) {
        atomicMax(&fs[f].ord_min_inv[c], ~float_to_ordered(m));
        atomicMax(&fs[f].ord_max[c], float_to_ordered(M));
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    mn[c] = INFINITY;
    mx[c] = -INFINITY;
  }
}

template <bool kPosed>
__global__ __launch_bounds__(kTrThreads, 1) void trie_kernel(const TrArgs a) {
  __shared__ TrSmem sm;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t gt = blockIdx.x * kTrThreads + threadIdx.x, gthreads = gridDim.x * kTrThreads;
  const int F = a.fr.nframes;
  int* err = a.err;
  uint32_t* bar = &a.st->fz_bar;
  uint32_t target = 0;
  const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);

  // ---- extents; the first level's bits cleared ----
  for (uint32_t i = gt; i < (1u << (a.root_bits - 7)); i += gthreads)
    reinterpret_cast<uint4*>(a.root)[i] = zero4;
  const uint32_t T = build_chunk_map(a.fr, sm.off, sm.cstart, sm.tmp, err);
  uint32_t c0, c1;
  block_range(T, &c0, &c1);
  {
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    int cur = -1;
    tr_points<kPosed>(a, sm, c0, c1, [&](int f, int64_t, bool, float x, float y, float z) {
      if (f != cur) {
        if (cur >= 0) tr_flush_extent(mn, mx, a.fs, cur, sm);
        cur = f;
      }
      if (point_valid(x, y, z)) {
        mn[0] = fminf(mn[0], x), mx[0] = fmaxf(mx[0], x);
        mn[1] = fminf(mn[1], y), mx[1] = fmaxf(mx[1], y);
        mn[2] = fminf(mn[2], z), mx[2] = fmaxf(mx[2], z);
      }
    });
    if (cur >= 0) tr_flush_extent(mn, mx, a.fs, cur, sm);
  }
  if (!grid_barrier(bar, target, a.spin_limit, err)) return;

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
        sm.org[f][c] = o[c];
      }
      sm.leaf[f] = leaf;
      sm.rleaf[f] = fast_leaf(leaf) ? __fdiv_rn(1.0f, leaf) : 0.0f;
      sm.inv_unit[f] = quant_inv_unit(leaf);
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
    if (blockIdx.x == 0) {
      if (a.out.frame_offsets)
        for (int f = threadIdx.x; f <= F; f += kTrThreads) a.out.frame_offsets[f] = 0;
      if (threadIdx.x == 0) *a.out.num_voxels = 0;
    }
    return;
  }
  const bool wide = local_bits > 32u;
  // levels, and the key bits below level 1
  const uint32_t root_bits = static_cast<uint32_t>(a.root_bits);
  const int levels =
      kb <= root_bits ? 1 : 1 + int((kb - root_bits + kTrDigitBits - 1) / kTrDigitBits);
  const uint32_t below = uint32_t(levels - 1) * kTrDigitBits;
  const uint32_t top = max(kb - below, uint32_t(kTrDigitBits));
  uint32_t ns = 1u << (top - kTrDigitBits);  // slots of the level
  const int64_t cap = a.slots;

  // ---- level 1 marked ----
  bool range_bad = false;
  tr_points<kPosed>(a, sm, c0, c1, [&](int f, int64_t, bool, float x, float y, float z) {
    uint64_t key = 0;
    uint32_t ijk[3];
    const bool ok = tr_key(sm, f, x, y, z, wide, key_shift, &key, ijk, &range_bad);
    const uint64_t pre = key >> below;
    const uint32_t s = static_cast<uint32_t>(pre >> kTrDigitBits);
    tr_mark<true>(a.root, s, uint32_t(pre) & 255u, ok && s < ns);
  });
  if (__any_sync(kFullMask, range_bad) && lane == 0) set_error(err, kErrRange);
  if (!grid_barrier(bar, target, a.spin_limit, err)) return;

  // ---- every level ranked, the next one marked ----
  uint32_t* bits = a.root;
  uint4* rec = a.rootrec;
  uint32_t rows = 0;
  for (int j = 1;; ++j) {
    uint32_t* agg = a.stat + size_t(j - 1) * kTrMaxGrid;
    tr_count(bits, ns, agg, sm.tmp);
    if (!grid_barrier(bar, target, a.spin_limit, err)) return;
    const uint32_t set = tr_rank_slots(bits, rec, ns, agg, sm);
    const uint32_t n1 = static_cast<uint32_t>(min(int64_t(set), cap));
    if (set > n1 && blockIdx.x == 0 && threadIdx.x == 0) set_error(err, kErrInvalidArg);
    if (j == levels) {
      rows = n1;
      break;
    }
    // the buffers alternate so that the last level lies in x
    char* nb = ((levels - j - 1) & 1) ? a.y : a.x;
    uint32_t* nbits = reinterpret_cast<uint32_t*>(nb);
    uint4* nrec = reinterpret_cast<uint4*>(nb + size_t(cap) * 32);
    for (uint32_t i = gt; i < n1 * 2u; i += gthreads) reinterpret_cast<uint4*>(nbits)[i] = zero4;
    if (!grid_barrier(bar, target, a.spin_limit, err)) return;
    const uint32_t sh = below - uint32_t(j) * kTrDigitBits;  // key bits below the next level
    tr_points<kPosed>(a, sm, c0, c1, [&](int f, int64_t p, bool, float x, float y, float z) {
      uint64_t key = 0;
      uint32_t ijk[3], head;
      bool bad = false;
      const bool ok = tr_key(sm, f, x, y, z, wide, key_shift, &key, ijk, &bad);
      const bool tail = tr_run(key, ok, &head) == lane && ok;
      uint32_t s = 0;
      bool good = false;
      if (tail) {
        const uint64_t pre = key >> (sh + kTrDigitBits);
        const uint32_t s0 = j == 1 ? static_cast<uint32_t>(pre >> kTrDigitBits) : a.pslot[p];
        if (s0 < ns) {
          s = tr_rank(rec, bits, s0, uint32_t(pre) & 255u);
          good = s < n1;
        }
        a.pslot[p] = good ? s : ~0u;
        if (!good) set_error(err, kErrInvalidArg);
      }
      tr_mark<false>(nbits, s, uint32_t(key >> sh) & 255u, good);
    });
    if (!grid_barrier(bar, target, a.spin_limit, err)) return;
    bits = nbits;
    rec = nrec;
    ns = n1;
  }

  // ---- the rows' sums cleared ----
  unsigned long long* accA = reinterpret_cast<unsigned long long*>(a.y);
  unsigned long long* accB = accA + cap;
  unsigned long long* accC = accB + cap;
  unsigned long long* rowkey = accC + cap;
  unsigned long long* att = rowkey + cap;  // two a row: channels 0, 1 and 2, 3 in 32 bits each
  const bool with_attrs = a.out.attrs_in != nullptr;
  for (uint32_t i = gt; i < rows; i += gthreads) {
    accA[i] = 0ull;
    accB[i] = 0ull;
    accC[i] = 0ull;
    if (with_attrs) {
      att[i] = 0ull;
      att[i + cap] = 0ull;
    }
  }
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) {
      // more cells than output rows: recorded once, here; the first cap rows are written
      if (int64_t(rows) > a.out.cap) set_error(err, kErrCapacity);
      *a.out.num_voxels = rows;
    }
    if (a.out.frame_offsets && (F == 1 || rows == 0))
      for (int f = threadIdx.x; f <= F; f += kTrThreads)
        a.out.frame_offsets[f] = f == F ? rows : 0;
  }
  if (!grid_barrier(bar, target, a.spin_limit, err)) return;

  // ---- every run's points and sums at its row ----
  tr_points<kPosed>(a, sm, c0, c1, [&](int f, int64_t p, bool in, float x, float y, float z) {
    uint64_t key = 0;
    uint32_t ijk[3], head;
    bool bad = false;
    const bool ok = tr_key(sm, f, x, y, z, wide, key_shift, &key, ijk, &bad);
    const uint32_t last = tr_run(key, ok, &head);
    const bool tail = ok && last == lane;
    uint32_t row = ~0u;
    if (tail) {
      const uint32_t s0 = levels == 1 ? static_cast<uint32_t>(key >> kTrDigitBits) : a.pslot[p];
      if (s0 < ns) row = tr_rank(rec, bits, s0, uint32_t(key) & 255u);
      if (row >= rows) {
        set_error(err, kErrInvalidArg);
        row = ~0u;
      }
    }
    // biased offsets, summed over the run (32 offsets of 21 bits fit 32 bits)
    uint32_t v[3] = {0u, 0u, 0u}, at[2] = {0u, 0u};
    if (ok) {
      const float q[3] = {x, y, z};
#pragma unroll
      for (int c = 0; c < 3; ++c)
        v[c] = uint32_t(quant_offset(q[c], voxel_corner(ijk[c], sm.org[f][c], sm.leaf[f]),
                                     sm.inv_unit[f]) -
                        kQMin);
      if (with_attrs) {
        const uint8_t* b = a.out.attrs_in + size_t(p) * a.out.channels;
#pragma unroll
        for (int c = 0; c < 4; ++c)  // two 16-bit sums a word (32 x 255 fit)
          if (c < a.out.channels) at[c >> 1] |= uint32_t(__ldg(b + c)) << (16 * (c & 1));
      }
    }
#pragma unroll
    for (uint32_t d = 1; d < 32; d <<= 1) {
      if (!__any_sync(kFullMask, lane >= head + d)) break;  // no run is longer
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const uint32_t u = __shfl_up_sync(kFullMask, v[c], d);
        if (lane >= head + d) v[c] += u;
      }
      if (with_attrs) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const uint32_t u = __shfl_up_sync(kFullMask, at[c], d);
          if (lane >= head + d) at[c] += u;
        }
      }
    }
    if (row != ~0u) {
      rowkey[row] = key;  // (every run of the row stores the same key)
      const unsigned long long va = v[0] | ((unsigned long long)v[1] << 32);
      const unsigned long long vb = v[2] | ((unsigned long long)(lane - head + 1u) << 32);
      const unsigned long long oa = atomicAdd(accA + row, va);
      const unsigned long long ob = atomicAdd(accB + row, vb);
      if (with_attrs) {
        atomicAdd(att + row, (unsigned long long)(at[0] & 0xffffu) |
                                 ((unsigned long long)(at[0] >> 16) << 32));
        if (a.out.channels > 2)
          atomicAdd(att + cap + row, (unsigned long long)(at[1] & 0xffffu) |
                                         ((unsigned long long)(at[1] >> 16) << 32));
      }
      // carries out of a 32-bit half: x into y, A out of 64 bits, z into the points
      const unsigned long long cx = ((oa & 0xffffffffull) + (va & 0xffffffffull)) >> 32;
      const unsigned long long cy = oa + va < oa ? 1ull : 0ull;
      const unsigned long long cz = ((ob & 0xffffffffull) + (vb & 0xffffffffull)) >> 32;
      if (cx | cy | cz) atomicAdd(accC + row, cx | (cy << 21) | (cz << 42));
    }
    if (a.out.p2v) {
      const uint32_t r = __shfl_sync(kFullMask, row, last);
      if (in) a.out.p2v[p] = ok && r != ~0u ? static_cast<int32_t>(r) : -1;
    }
  });
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
  rc.o1[0] = sm.org[0][0];
  rc.o1[1] = sm.org[0][1];
  rc.o1[2] = sm.org[0][2];
  rc.leaf1 = sm.leaf[0];
  for (uint32_t row = gt; row < rows; row += gthreads) {
    const unsigned long long key = __ldcg(rowkey + row);
    if (F > 1 && a.out.frame_offsets) {
      const uint32_t fk = key_frame(key, key_shift);
      const uint32_t f0 = row > 0 ? key_frame(__ldcg(rowkey + row - 1), key_shift) + 1u : 0u;
      for (uint32_t f = f0; f <= fk; ++f) a.out.frame_offsets[f] = row;
      if (row + 1u == rows)
        for (uint32_t f = fk + 1u; f <= uint32_t(F); ++f) a.out.frame_offsets[f] = rows;
    }
    if (int64_t(row) >= a.out.cap) continue;
    const unsigned long long A = __ldcg(accA + row), B = __ldcg(accB + row),
                             C = __ldcg(accC + row);
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
      const unsigned long long w[2] = {__ldcg(att + row), __ldcg(att + cap + row)};
#pragma unroll
      for (int c = 0; c < 4; ++c)  // exact sums, one FP64 division each
        if (c < a.out.channels)
          a.out.attrs_out[size_t(row) * a.out.channels + c] = __double2float_rn(
              __ddiv_rn(static_cast<double>(uint32_t(w[c >> 1] >> (32 * (c & 1)))),
                        static_cast<double>(r.n)));
    }
  }
}

// What the launch reads before writing: the state (the pyramid's tile counters among it), the
// frames' extent words and the error word.
__global__ __launch_bounds__(1024) void trie_clear_kernel(uint32_t* st, uint32_t words, int* err) {
  for (uint32_t i = threadIdx.x; i < words; i += 1024) st[i] = 0u;
  if (threadIdx.x == 0) *err = 0;
}

// Blocks an SM holds of the kernel (0: it cannot run there), per device.
int trie_blocks_per_sm(bool posed) {
  static int cache[64][2];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int& b = cache[dev][posed ? 1 : 0];
  if (b == 0) {
    const void* fn = posed ? reinterpret_cast<const void*>(trie_kernel<true>)
                           : reinterpret_cast<const void*>(trie_kernel<false>);
    int v = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, fn, kTrThreads, 0) != cudaSuccess) v = 0;
    (void)cudaGetLastError();
    b = v > 0 ? v : -1;
  }
  return b > 0 ? b : 0;
}

}  // namespace

bool trie_available(bool posed) { return trie_blocks_per_sm(posed) > 0; }

void warm_trie_config() {
  (void)trie_blocks_per_sm(false);
  (void)trie_blocks_per_sm(true);
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
  a.rootrec = reinterpret_cast<uint4*>(ws + L.rootrec);
  a.x = ws + L.x;
  a.y = ws + L.y;
  a.pslot = reinterpret_cast<uint32_t*>(ws + L.pslot);
  a.stat = reinterpret_cast<uint32_t*>(ws + L.stat);
  a.out = out;
  a.slots = L.slots;
  a.root_bits = trie_root_bits(fr.n);
  a.spin_limit = spin_limit;
  a.err = err;
  // one block a chunk of points, but enough of them to clear and rank the first level
  const int64_t sms = num_sms() < kTrMaxGrid ? num_sms() : kTrMaxGrid;
  const int64_t chunks = max_chunks(fr.n, fr.nframes);
  const int64_t half = sms > 1 ? sms / 2 : 1;
  const int64_t g = chunks < half ? half : (chunks < sms ? chunks : sms);
  const size_t head = reinterpret_cast<char*>(fs + fr.nframes) - reinterpret_cast<char*>(st);
  trie_clear_kernel<<<1, 1024, 0, stream>>>(reinterpret_cast<uint32_t*>(st),
                                           static_cast<uint32_t>(head / sizeof(uint32_t)), err);
  void* args[] = {&a};
  const void* fn = posed(fr) ? reinterpret_cast<const void*>(trie_kernel<true>)
                             : reinterpret_cast<const void*>(trie_kernel<false>);
  return cudaLaunchCooperativeKernel(fn, dim3(static_cast<unsigned>(g)), dim3(kTrThreads), args, 0,
                                     stream);
}

}  // namespace vg
