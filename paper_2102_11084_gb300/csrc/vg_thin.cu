// Neighbour-count thinning (vg_thin): the paper's own filter loop.
//
// arXiv 2102.11084 Sec. II-C, Algorithm 1: every point is placed in a cell of a regular
// grid, the (cell, point) table is radix-sorted, and then, pass after pass, every point
// counts its neighbours in its own and the 26 surrounding cells (Euclidean distance,
// Eq. 1), is marked when the count exceeds a threshold, and a batch of the marked points
// is deleted; when no more than a batch is marked, all of them are deleted and the loop
// ends.  The paper deletes a random batch; here the batch is the marked points of lowest
// caller-given priority (ties by point index), so the result is reproducible.
//
// GPU layout of the loop:
//   grouping   the sort path (wide layout, point_to_voxel on) gives the occupied cells
//              in key order and the points in cell order;
//   setup      per entry of the sorted table: its coordinates and index in one 16-byte
//              word; per cell: its first entry and the rows of its 26 neighbour cells
//              (binary search in the sorted cell keys, once), and how many (point,
//              candidate) pairs the 27 cells of all points hold.
// Then one of two forms of the same loop:
//   counts kept (the usual one)   every point's neighbours are counted once, the points
//              that start marked are sorted by (priority, index), and one cooperative
//              launch runs every pass.  A point's count only falls, so the marked set only
//              shrinks and the batch of every pass is the next `batch` points of the sorted
//              list that are still marked; the pass then takes one from the count of every
//              neighbour of a deleted point.  No pass reads the other points again and none
//              goes through the host.
//   recounted  where the points are so dense, or the batch so large, that the deleted points
//              meet more candidates than a fresh count (which stops at the threshold), or the
//              device cannot hold the cooperative launch:
//              thin_count_kernel counts and marks every pass, the host reads the number
//              marked and finds the batch by a radix select on 256-bin histograms
//              (thin_hist_kernel), thin_delete_kernel removes it.
//   output     keep flag per input point and the number kept.
#include <algorithm>
#include <cmath>

#include "../../include/vg.h"
#include "vg_api_internal.h"
#include "vg_device.cuh"
#include "vg_internal.h"

namespace vg {
namespace {

constexpr int kNb = 27;
constexpr uint32_t kLoopGroup = 128;  // entries a warp takes at a time (4 a lane)
constexpr uint32_t kNoCell = 0xffffffffu;
constexpr uint8_t kAlive = 1, kMarked = 2;
// Words of the loop: marked points (recounted form), kept points, grid-barrier arrivals, passes
// run, the candidate pairs (one 64-bit word), groups of entries (at most kLoopGroup of one cell:
// how many there are, and how many are listed).
constexpr int kCtrMarked = 0, kCtrKept = 1, kCtrBar = 2, kCtrPasses = 3, kCtrPairs = 4,
              kCtrAll = 6, kCtrGroups = 7;
constexpr int kCtrWords = 8;

struct ThinLayout {
  size_t base, vkeys, pos, cnt, vcnt, vnum, p2v, cstart, nb, sprio, sidx, state, ctr, hist, st2,
      total;
};

ThinLayout thin_layout(int64_t n) {
  ThinLayout L{};
  const int64_t nn = n < 1 ? 1 : n;
  size_t off = frames_workspace_bytes(n, 1, VG_METHOD_SORT);
  L.base = 0;
  auto take = [&](size_t* at, size_t bytes) {
    *at = off;
    off = align_up(off + bytes, 256);
  };
  take(&L.vkeys, size_t(nn) * sizeof(uint64_t));
  take(&L.pos, size_t(nn) * sizeof(float4));  // the grouping's centroids first, then the entries
  take(&L.cnt, size_t(nn) * sizeof(uint32_t));
  take(&L.vcnt, size_t(nn) * sizeof(uint32_t));
  take(&L.vnum, sizeof(int64_t));
  take(&L.p2v, size_t(nn) * sizeof(int32_t));
  take(&L.cstart, size_t(nn) * sizeof(uint32_t));
  take(&L.nb, size_t(nn) * kNb * sizeof(uint32_t));
  take(&L.sprio, size_t(nn) * sizeof(uint32_t));
  take(&L.sidx, size_t(nn) * sizeof(uint32_t));
  take(&L.state, size_t(nn));
  take(&L.ctr, kCtrWords * sizeof(uint32_t));
  take(&L.hist, 256 * sizeof(uint32_t));
  take(&L.st2, sizeof(State));  // of the sort of the marked points by priority
  L.total = off;
  return L;
}

__device__ __forceinline__ const uint32_t* sorted_idx(const State* st, const uint32_t* idx0,
                                                      const uint32_t* idx1) {
  return (max(1, sort_passes(st->maxkey)) & 1) ? idx1 : idx0;
}

// Per sorted entry: gather coordinates, priority and index; mark cell starts; each valid
// point's entry.
__global__ void thin_setup_kernel(const State* st, const uint32_t* idx0, const uint32_t* idx1,
                                  const float* __restrict__ xyz, const uint32_t* __restrict__ prio,
                                  const int32_t* __restrict__ p2v, uint32_t* cstart, float4* pos,
                                  float* sx, float* sy, float* sz, uint32_t* sprio,
                                  uint32_t* sidx, uint32_t* entry, uint8_t* state,
                                  const int* err) {
  if (error_raised(err)) return;  // the grouping failed: point_to_voxel is unwritten
  const int64_t m = st->nitems;
  const uint32_t* I = sorted_idx(st, idx0, idx1);
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < m;
       i += int64_t(gridDim.x) * blockDim.x) {
    const uint32_t p = I[i];
    const int32_t row = p2v[p];
    const int32_t prev = i > 0 ? p2v[I[i - 1]] : -1;
    if (row != prev) cstart[row] = static_cast<uint32_t>(i);
    const float x = xyz[3 * size_t(p)], y = xyz[3 * size_t(p) + 1], z = xyz[3 * size_t(p) + 2];
    pos[i] = make_float4(x, y, z, __uint_as_float(p));
    sx[i] = x;
    sy[i] = y;
    sz[i] = z;
    sprio[i] = prio[p];
    sidx[i] = p;
    entry[p] = static_cast<uint32_t>(i);
    state[i] = kAlive;
  }
}

// Per cell and neighbour offset: the row of that cell (kNoCell where empty), and the pairs
// of points the two hold.  A thread a (cell, offset) pair, not a cell: the 27 searches of a
// cell are independent chains of dependent loads (11,489 cells: 25.8 us one thread a cell).
__global__ __launch_bounds__(256) void thin_neighbors_kernel(
    const int64_t* __restrict__ num_cells, const uint64_t* __restrict__ vkeys,
    const uint32_t* __restrict__ vcnt, uint32_t* nb, uint32_t* ctr, const int* err) {
  if (error_raised(err)) return;
  const int64_t V = *num_cells;
  unsigned long long mine = 0;
  uint32_t groups = 0;
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < V * kNb;
       t += int64_t(gridDim.x) * blockDim.x) {
    const int64_t v = t / kNb;
    const int o = static_cast<int>(t - v * kNb);
    const uint64_t key = vkeys[v];
    const int64_t a = int64_t(compact3(key)) + o / 9 - 1;
    const int64_t b = int64_t(compact3(key >> 1)) + o / 3 % 3 - 1;
    const int64_t d = int64_t(compact3(key >> 2)) + o % 3 - 1;
    uint32_t row = kNoCell;
    const int64_t lim = int64_t(1) << 21;
    if (a >= 0 && b >= 0 && d >= 0 && a < lim && b < lim && d < lim) {
      const uint64_t want = morton3(uint32_t(a), uint32_t(b), uint32_t(d));
      int64_t lo = 0, hi = V;  // first key >= want
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (vkeys[mid] < want) lo = mid + 1; else hi = mid;
      }
      if (lo < V && vkeys[lo] == want) row = static_cast<uint32_t>(lo);
    }
    nb[t] = row;
    if (o == 0) groups += (vcnt[v] + kLoopGroup - 1) / kLoopGroup;
    if (row != kNoCell) mine += (unsigned long long)vcnt[v] * vcnt[row];
  }
  for (int off = 16; off; off >>= 1) mine += __shfl_xor_sync(kFullMask, mine, off);
  groups = __reduce_add_sync(kFullMask, groups);
  if ((threadIdx.x & 31) == 0 && mine)
    atomicAdd(reinterpret_cast<unsigned long long*>(ctr + kCtrPairs), mine);
  if ((threadIdx.x & 31) == 0 && groups) atomicAdd(ctr + kCtrAll, groups);
}

// Squared distance of the definition: binary32, ((dx*dx + dy*dy) + dz*dz), one rounding an
// operation.  The same value for either point of a pair.
__device__ __forceinline__ float dist2(const float4& q, float x, float y, float z) {
  const float ex = __fsub_rn(q.x, x), ey = __fsub_rn(q.y, y), ez = __fsub_rn(q.z, z);
  return __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
}

// ---- counts kept ------------------------------------------------------------------------

constexpr int kFullThreads = 128;
constexpr int kLoopThreads = 1024;
constexpr int kLoopItems = 2;   // list entries a thread tests per step of the batch search
constexpr int kLoopSplit = 8;   // warps that share the candidates of one deleted point

// Two binary32 operations in one instruction, each with its own rounding.
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long both(float v) {
  const unsigned long long b = __float_as_uint(v);
  return b | (b << 32);
}

// Every entry's neighbours, all of them, and its cell; the groups of kLoopGroup entries that
// the cells are cut into (their first entries, in any order).  A thread an entry, entries in
// cell order: the lanes of a warp mostly share a cell, so a candidate's load is a broadcast.
// Bound by FP32 issue: candidates are tested two to an instruction (dist2's operations, q + (-x)
// being q - x), four to three 16-byte loads of the coordinates' own arrays, where a candidate a
// time from 16-byte entries took 705 us of a 640x480 frame (1e9 pairs); 507 us.
__global__ __launch_bounds__(kFullThreads) void thin_full_count_kernel(
    const State* st, const int32_t* __restrict__ p2v, const uint32_t* __restrict__ cstart,
    const uint32_t* __restrict__ vcnt, const uint32_t* __restrict__ nb,
    const float4* __restrict__ pos, const float* __restrict__ sx, const float* __restrict__ sy,
    const float* __restrict__ sz, uint32_t* __restrict__ cnt, uint32_t* __restrict__ ecell,
    uint32_t* __restrict__ group, uint32_t* ctr, float r2, const int* err) {
  if (error_raised(err)) return;
  const int64_t i = blockIdx.x * int64_t(kFullThreads) + threadIdx.x;
  if (i >= int64_t(st->nitems)) return;
  const float4 me = __ldg(pos + i);
  const uint32_t cell = static_cast<uint32_t>(p2v[__float_as_uint(me.w)]);
  const uint32_t* row = nb + size_t(cell) * kNb;
  ecell[i] = cell;
  if ((uint32_t(i) - __ldg(cstart + cell)) % kLoopGroup == 0)
    group[atomicAdd(ctr + kCtrGroups, 1u)] = uint32_t(i);
  const unsigned long long mx = both(-me.x), my = both(-me.y), mz = both(-me.z);
  uint32_t n = 0;
  for (int o = 0; o < kNb; ++o) {
    const uint32_t c = __ldg(row + o);
    if (c == kNoCell) continue;
    uint32_t j = __ldg(cstart + c);
    const uint32_t end = j + __ldg(vcnt + c);
    auto one = [&](uint32_t k) {
      const float4 q = make_float4(__ldg(sx + k), __ldg(sy + k), __ldg(sz + k), 0.0f);
      n += dist2(q, me.x, me.y, me.z) <= r2;
    };
    for (; j < end && (j & 3u) != 0; ++j) one(j);  // up to a 16-byte boundary
#pragma unroll 2
    for (; j + 4 <= end; j += 4) {
      const ulonglong2 x = __ldg(reinterpret_cast<const ulonglong2*>(sx + j));
      const ulonglong2 y = __ldg(reinterpret_cast<const ulonglong2*>(sy + j));
      const ulonglong2 z = __ldg(reinterpret_cast<const ulonglong2*>(sz + j));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const unsigned long long ex = add2(h ? x.y : x.x, mx), ey = add2(h ? y.y : y.x, my),
                                 ez = add2(h ? z.y : z.x, mz);
        const unsigned long long d = add2(add2(mul2(ex, ex), mul2(ey, ey)), mul2(ez, ez));
        n += __uint_as_float(uint32_t(d)) <= r2;
        n += __uint_as_float(uint32_t(d >> 32)) <= r2;
      }
    }
    for (; j < end; ++j) one(j);
  }
  cnt[i] = n - 1u;  // (the point itself is at distance 0)
}

// Sort keys of the points that start marked, in point order: their priority (the pass that
// reads them drops the sentinel rows and keeps equal keys in point order); the first digit's
// histogram, the number of marked points and the largest key.
__global__ __launch_bounds__(256) void thin_prio_kernel(int64_t n, const int32_t* __restrict__ p2v,
                                                        const uint32_t* __restrict__ entry,
                                                        const uint32_t* __restrict__ cnt,
                                                        const uint32_t* __restrict__ prio,
                                                        uint32_t thr, uint64_t* keys, State* st2,
                                                        const int* err) {
  __shared__ uint32_t h[kRadix];
  if (block_error_raised(err)) return;
  h[threadIdx.x] = 0;
  __syncthreads();
  uint32_t mine = 0, big = 0;
  for (int64_t p = blockIdx.x * int64_t(256) + threadIdx.x; p < n; p += int64_t(gridDim.x) * 256) {
    const bool in = p2v[p] >= 0 && cnt[entry[p]] > thr;
    const uint32_t k = in ? prio[p] : 0u;
    keys[p] = in ? uint64_t(k) : kKeySentinel;
    if (in) {
      ++mine;
      big = max(big, k);
      atomicAdd(&h[k & (kRadix - 1)], 1u);
    }
  }
  // (the lanes of a warp may leave the loop after different numbers of trips)
  __syncwarp();
  mine = __reduce_add_sync(kFullMask, mine);
  big = __reduce_max_sync(kFullMask, big);
  if ((threadIdx.x & 31) == 0 && mine) {
    atomicAdd(&st2->nitems, mine);
    atomicMax(&st2->maxkey, (unsigned long long)big);
  }
  __syncthreads();
  if (h[threadIdx.x]) atomicAdd(&st2->hist[0][threadIdx.x], h[threadIdx.x]);
}

// The sorted points as entries.
__global__ __launch_bounds__(256) void thin_list_kernel(const State* st2, const uint32_t* idx0,
                                                        const uint32_t* idx1,
                                                        const uint32_t* __restrict__ entry,
                                                        uint32_t* __restrict__ list,
                                                        const int* err) {
  if (error_raised(err)) return;
  const uint32_t* I = sorted_idx(st2, idx0, idx1);
  const int64_t m = st2->nitems;
  for (int64_t k = blockIdx.x * int64_t(256) + threadIdx.x; k < m; k += int64_t(gridDim.x) * 256)
    list[k] = entry[I[k]];
}

struct LoopArgs {
  const State* st2;
  const uint32_t* list;  // entries that start marked, by (priority, point index)
  const uint32_t* ecell;
  const uint32_t* cstart;
  const uint32_t* vcnt;
  const uint32_t* nb;
  const float4* pos;
  const uint32_t* group;
  uint32_t* cnt;
  uint8_t* dead;
  uint32_t* sel;            // scattered: the entries a pass deletes
  unsigned long long* head;  // gathered: pass << 32 | the cell's last deleted entry's rank
  float4* node;             // gathered: place of the entry of each rank; w = the next rank
  // in the block's own memory: per list position its place (negated; w = its cell), the pass
  // that unmarked it (0: none yet) and whether a pass deleted it; per entry its position
  float4* lnode;
  uint32_t* off;
  uint8_t* gone;
  uint32_t* rank;
  uint32_t* ctr;
  float r2;
  uint32_t thr;
  uint32_t batch;
  double pairs_per_point;
  int64_t max_passes;
  uint32_t spin_limit;
  int* err;
};
constexpr uint32_t kListEnd = 0xffffffffu;

// Scattered: kLoopSplit warps a deleted entry share the candidates of its 27 cells, in groups
// of kLoopGroup, and take one from the count of every one within r.  Counts lie in entry
// order, so the 32 candidates of a warp step are consecutive words and their decrements
// (which return nothing) a few sectors.
__device__ __forceinline__ void thin_scatter(const LoopArgs& a, uint32_t taken, uint64_t gw,
                                             uint64_t gwarps) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t units = uint64_t(taken) * kLoopSplit;
  for (uint64_t u = gw; u < units; u += gwarps) {
    const uint32_t part = uint32_t(u % kLoopSplit);
    const uint32_t i = __ldcg(a.sel + u / kLoopSplit);
    const float4 me = __ldg(a.pos + i);
    uint32_t j0 = 0, mm = 0;
    if (lane < uint32_t(kNb)) {
      const uint32_t c = __ldg(a.nb + size_t(__ldg(a.ecell + i)) * kNb + lane);
      if (c != kNoCell) {
        j0 = __ldg(a.cstart + c);
        mm = __ldg(a.vcnt + c);
      }
    }
    const uint32_t ng = (mm + kLoopGroup - 1) / kLoopGroup;
    uint32_t inc = ng;  // groups of the cells up to this one
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(kFullMask, inc, off);
      if (lane >= uint32_t(off)) inc += y;
    }
    const uint32_t groups = __shfl_sync(kFullMask, inc, 31);
    for (uint32_t gi = part; gi < groups; gi += kLoopSplit) {
      const int l = __popc(__ballot_sync(kFullMask, inc <= gi));  // the group's cell
      const uint32_t off = (gi - __shfl_sync(kFullMask, inc - ng, l)) * kLoopGroup + lane;
      const uint32_t n = __shfl_sync(kFullMask, mm, l);
      const uint32_t j = __shfl_sync(kFullMask, j0, l) + off;
      float4 w[4];
#pragma unroll
      for (uint32_t v = 0; v < 4; ++v)
        if (off + 32u * v < n) w[v] = __ldg(a.pos + j + 32u * v);
#pragma unroll
      for (uint32_t v = 0; v < 4; ++v)  // (the counts of dead entries fall too: never read)
        if (off + 32u * v < n && j + 32u * v != i && dist2(w[v], me.x, me.y, me.z) <= a.r2)
          atomicSub(a.cnt + j + 32u * v, 1u);
    }
  }
}

// Gathered: a warp a group of entries of one cell walks the lists of this pass's deleted
// entries in the 27 cells around it (lane l the list of cell l) and counts, for the entries
// still marked (no other count is read again), the ones within r.
struct ThinGroup {
  uint32_t i0;       // first entry
  uint32_t nb;       // lane l: the l-th cell around, or kNoCell
  float x[4], y[4], z[4];  // the lane's entries
  uint32_t n[4];           // and their counts (0 past the cell's end)
};
__device__ __forceinline__ void thin_group_load(const LoopArgs& a, uint64_t u, ThinGroup& g) {
  const uint32_t lane = threadIdx.x & 31u;
  g.i0 = __ldg(a.group + u);
  const uint32_t cell = __ldg(a.ecell + g.i0);
  const uint32_t end = __ldg(a.cstart + cell) + __ldg(a.vcnt + cell);
  g.nb = lane < uint32_t(kNb) ? __ldg(a.nb + size_t(cell) * kNb + lane) : kNoCell;
#pragma unroll
  for (uint32_t v = 0; v < 4; ++v) {
    const uint32_t i = g.i0 + 32u * v + lane;
    g.n[v] = i < end ? __ldcg(a.cnt + i) : 0u;
    const float4 w = i < end ? __ldg(a.pos + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    g.x[v] = w.x;
    g.y[v] = w.y;
    g.z[v] = w.z;
  }
}
__device__ __forceinline__ void thin_gather(const LoopArgs& a, uint32_t pass, ThinGroup& g) {
  const uint32_t lane = threadIdx.x & 31u;
  if (!__any_sync(kFullMask, g.n[0] > a.thr || g.n[1] > a.thr || g.n[2] > a.thr || g.n[3] > a.thr))
    return;
  uint32_t r = kListEnd;
  if (g.nb != kNoCell) {
    const unsigned long long h = __ldcg(a.head + g.nb);
    if (uint32_t(h >> 32) == pass) r = uint32_t(h);
  }
  uint32_t hit[4] = {0u, 0u, 0u, 0u};
  for (uint32_t some; (some = __ballot_sync(kFullMask, r != kListEnd)) != 0u;) {
    float4 q = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (r != kListEnd) {
      q = __ldcg(a.node + r);
      r = __float_as_uint(q.w);
    }
    for (; some; some &= some - 1) {
      const int l = __ffs(some) - 1;
      const float x = __shfl_sync(kFullMask, q.x, l), y = __shfl_sync(kFullMask, q.y, l),
                  z = __shfl_sync(kFullMask, q.z, l);
#pragma unroll
      for (int v = 0; v < 4; ++v)
        hit[v] += dist2(make_float4(g.x[v], g.y[v], g.z[v], 0.0f), x, y, z) <= a.r2;
    }
  }
#pragma unroll
  for (uint32_t v = 0; v < 4; ++v)  // (a marked entry's count covers every neighbour left)
    if (g.n[v] > a.thr && hit[v]) {
      g.n[v] -= hit[v];
      a.cnt[g.i0 + 32u * v + lane] = g.n[v];
    }
}

// Every pass of the loop where local_lists leaves it (few candidates, or a batch of more than
// kLocalBatch), one cooperative launch (a block an SM), two grid barriers a pass:
//   1. the batch: every block walks the sorted list from where the last pass stopped, tests
//      kLoopItems entries a thread, and finds the same `batch` entries still marked (one more
//      tells that this is not the last pass); the block that a list entry belongs to writes it.
//      The list's next entries are loaded before the barrier;
//   2. the counts, by the deleted entries (thin_scatter) or by the marked ones (thin_gather: a
//      warp keeps its first group in registers through all passes).
// Bound by the latency of the steps and the barriers.  640x480 frame, cell 0.05 m, threshold
// 20, batches of 1000 (277K points of 3600 candidates each, 2008 cells, 271 passes): a pass
// takes 23 us scattered (the drain of its 1.8M decrements is 3/4 of it), 12 us gathered
// (thin_local_kernel, which takes it for batches of this size, 7.0 us),
// against 570 us for a fresh count and 500 us of host round trips (recounted).  The gathered
// form touches every group of entries each pass, 9000 cycles a round of the grid's warps; the
// scattered form 8000 cycles and one per 90 candidates.
__global__ __launch_bounds__(kLoopThreads, 1) void thin_loop_kernel(const LoopArgs a) {
  __shared__ uint32_t tmp[kLoopThreads / 32];
  __shared__ uint32_t s_next;
  if (block_error_raised(a.err)) {
    if (blockIdx.x == 0 && threadIdx.x == 0) a.ctr[kCtrPasses] = 1u;
    return;
  }
  const uint32_t m = a.st2->nitems;
  const uint32_t groups = a.ctr[kCtrGroups];
  const uint64_t gwarps = uint64_t(gridDim.x) * (kLoopThreads / 32);
  const uint64_t gw = uint64_t(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const bool gather = 9000.0 * ceil(double(groups) / double(gwarps)) <=
                      8000.0 + double(a.batch) * a.pairs_per_point / 90.0;
  uint32_t target = 0, first = 0;
  int64_t passes = 0;
  ThinGroup mine{};  // (no entries: no count is above the threshold)
  mine.nb = kNoCell;
  if (gather && gw < groups) thin_group_load(a, gw, mine);
  uint32_t e[kLoopItems];  // the list entries this thread tests next
  auto fetch = [&](uint32_t k0) {
#pragma unroll
    for (int q = 0; q < kLoopItems; ++q) {
      const uint32_t k = k0 + kLoopItems * threadIdx.x + q;
      e[q] = k < m ? __ldg(a.list + k) : kListEnd;
    }
  };
  fetch(0);
  while (passes < a.max_passes) {
    ++passes;
    // 1. the next `batch` marked entries of the list
    uint32_t found = 0;
    for (uint32_t k0 = first;;) {
      uint32_t some = 0, cell[kLoopItems];
      float4 w[kLoopItems];
      bool in[kLoopItems], own[kLoopItems];
#pragma unroll
      for (int q = 0; q < kLoopItems; ++q) {
        in[q] = e[q] != kListEnd && __ldcg(a.cnt + e[q]) > a.thr;
        // (its place and cell beside its count: one latency)
        own[q] = e[q] != kListEnd &&
                 ((k0 + kLoopItems * threadIdx.x + q) >> 5) % gridDim.x == blockIdx.x;
        if (gather && own[q]) {
          cell[q] = __ldg(a.ecell + e[q]);
          w[q] = __ldg(a.pos + e[q]);
        }
        some += in[q];
      }
      uint32_t total;
      uint32_t r = found + block_excl_scan(some, &total, tmp);
#pragma unroll
      for (int q = 0; q < kLoopItems; ++q) {
        if (!in[q]) continue;
        if (r < a.batch) {
          if (own[q]) {
            a.dead[e[q]] = 1;
            if (gather) {
              const unsigned long long tag = (unsigned long long)uint32_t(passes) << 32;
              const unsigned long long old = atomicExch(a.head + cell[q], tag | r);
              w[q].w = __uint_as_float((old ^ tag) >> 32 == 0 ? uint32_t(old) : kListEnd);
              a.node[r] = w[q];
            } else {
              a.sel[r] = e[q];
            }
          }
          if (r + 1 == a.batch) s_next = k0 + kLoopItems * threadIdx.x + q + 1;
        }
        ++r;
      }
      found += total;
      if (found > a.batch || m - k0 <= uint32_t(kLoopItems * kLoopThreads)) break;
      k0 += kLoopItems * kLoopThreads;  // (stays below m)
      fetch(k0);
    }
    // (the same in every block) the last pass: every marked point goes, by its count, in
    // the output
    if (found <= a.batch) break;
    __syncthreads();
    first = s_next;
    fetch(first);
    if (!grid_barrier(a.ctr + kCtrBar, target, a.spin_limit, a.err)) return;
    // 2. the counts
    if (gather) {
      thin_gather(a, uint32_t(passes), mine);
      for (uint64_t u = gw + gwarps; u < groups; u += gwarps) {
        ThinGroup more;
        thin_group_load(a, u, more);
        thin_gather(a, uint32_t(passes), more);
      }
    } else {
      thin_scatter(a, a.batch, gw, gwarps);
    }
    if (!grid_barrier(a.ctr + kCtrBar, target, a.spin_limit, a.err)) return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) a.ctr[kCtrPasses] = static_cast<uint32_t>(passes);
}

// The same loop for batches of at most kLocalBatch points, one grid barrier a pass: every block
// finds the same batch by itself and keeps its own copy, in lists by cell in shared memory, for
// thin_gather's walk.  What a pass reads to find its batch lies in list order, and a thread's
// first place is loaded ahead of the barrier.  A marked entry whose count falls to the
// threshold records the pass; one that a faster block records in this pass still counts as
// marked, so that no barrier is needed between finding the batch and counting.
// Bound by the walk of the densest groups (8000 of a pass's 14,500 cycles in the frame of
// thin_loop_kernel's comment; the barrier 2500, finding the batch 3000): 7.0 us a pass, where
// gathering from lists in global memory, two barriers a pass, took 12.  Three or four points at
// a time, or fewer warps with more registers, were no faster.
constexpr uint32_t kLocalBatch = 4096;
constexpr uint32_t kLocalHeads = 4096;  // lists (a power of two): a cell's by its low bits
constexpr int kLocalAtOnce = 2;  // deleted points a warp tests at a time
struct LocalSmem {
  float4 node[kLocalBatch + 1];  // place (negated); w = the next rank of the list; last, a NaN
  uint32_t cell[kLocalBatch];
  uint32_t head[kLocalHeads];
};
struct LocalGroup {
  uint32_t i0, nb;                         // as ThinGroup
  unsigned long long x[2], y[2], z[2];     // the lane's entries, two to a word
  uint32_t n[4];
  uint32_t changed;                        // bit v: n[v] is not the one in memory
};
__device__ __forceinline__ void local_group_load(const LoopArgs& a, uint64_t u, LocalGroup& g) {
  ThinGroup t;
  thin_group_load(a, u, t);
  g.i0 = t.i0;
  g.nb = t.nb;
  g.changed = 0u;
  auto two = [](float lo, float hi) {
    return __float_as_uint(lo) | ((unsigned long long)__float_as_uint(hi) << 32);
  };
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    g.x[h] = two(t.x[2 * h], t.x[2 * h + 1]);
    g.y[h] = two(t.y[2 * h], t.y[2 * h + 1]);
    g.z[h] = two(t.z[2 * h], t.z[2 * h + 1]);
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) g.n[v] = t.n[v];
}
__device__ __forceinline__ void local_gather(const LoopArgs& a, const LocalSmem& sm, uint32_t pass,
                                             LocalGroup& g) {
  const uint32_t lane = threadIdx.x & 31u;
  if (!__any_sync(kFullMask, g.n[0] > a.thr || g.n[1] > a.thr || g.n[2] > a.thr || g.n[3] > a.thr))
    return;
  uint32_t r = g.nb != kNoCell ? sm.head[g.nb & (kLocalHeads - 1u)] : kListEnd;
  uint32_t hit[4] = {0u, 0u, 0u, 0u};
  for (;;) {
    while (r != kListEnd && sm.cell[r] != g.nb) r = __float_as_uint(sm.node[r].w);
    uint32_t some = __ballot_sync(kFullMask, r != kListEnd);
    if (some == 0u) break;
    while (some) {
      float4 q[kLocalAtOnce];
#pragma unroll
      for (int b = 0; b < kLocalAtOnce; ++b) {
        const uint32_t at = __shfl_sync(kFullMask, r, (__ffs(some) - 1) & 31);
        q[b] = sm.node[some ? at : kLocalBatch];
        some &= some - 1;
      }
#pragma unroll
      for (int b = 0; b < kLocalAtOnce; ++b) {
        const unsigned long long x = both(q[b].x), y = both(q[b].y), z = both(q[b].z);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const unsigned long long ex = add2(g.x[h], x), ey = add2(g.y[h], y), ez = add2(g.z[h], z);
          const unsigned long long d = add2(add2(mul2(ex, ex), mul2(ey, ey)), mul2(ez, ez));
          hit[2 * h] += __uint_as_float(uint32_t(d)) <= a.r2;
          hit[2 * h + 1] += __uint_as_float(uint32_t(d >> 32)) <= a.r2;
        }
      }
    }
    if (r != kListEnd) r = __float_as_uint(sm.node[r].w);
  }
#pragma unroll
  for (uint32_t v = 0; v < 4; ++v)
    if (g.n[v] > a.thr && hit[v]) {
      g.n[v] -= hit[v];
      g.changed |= 1u << v;
      if (g.n[v] <= a.thr) a.off[__ldca(a.rank + g.i0 + 32u * v + lane)] = pass;
    }
}
__device__ __forceinline__ void local_group_store(const LoopArgs& a, const LocalGroup& g) {
#pragma unroll
  for (uint32_t v = 0; v < 4; ++v)
    if ((g.changed >> v) & 1u) a.cnt[g.i0 + 32u * v + (threadIdx.x & 31u)] = g.n[v];
}

__global__ __launch_bounds__(kLoopThreads, 1) void thin_local_kernel(const LoopArgs a) {
  extern __shared__ __align__(16) unsigned char local_smem[];
  LocalSmem& sm = *reinterpret_cast<LocalSmem*>(local_smem);
  __shared__ uint32_t tmp[2][32];
  __shared__ uint32_t s_next;
  if (block_error_raised(a.err)) {
    if (blockIdx.x == 0 && threadIdx.x == 0) a.ctr[kCtrPasses] = 1u;
    return;
  }
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t m = a.st2->nitems;
  const uint32_t groups = a.ctr[kCtrGroups];
  const uint64_t gwarps = uint64_t(gridDim.x) * (kLoopThreads / 32);
  const uint64_t gw = uint64_t(warp) * gridDim.x + blockIdx.x;
  const uint32_t gt = blockIdx.x * kLoopThreads + threadIdx.x, gthreads = gridDim.x * kLoopThreads;
  for (uint64_t k = gt; k < m; k += gthreads) {
    const uint32_t e = __ldg(a.list + k);
    const float4 w = __ldg(a.pos + e);
    a.lnode[k] = make_float4(-w.x, -w.y, -w.z, __uint_as_float(__ldg(a.ecell + e)));
    a.off[k] = 0u;
    a.gone[k] = 0;
    a.rank[e] = static_cast<uint32_t>(k);
  }
  if (threadIdx.x == 0)  // (NaN: within no radius, also where its square overflows)
    sm.node[kLocalBatch] = make_float4(NAN, NAN, NAN, __uint_as_float(kListEnd));
  LocalGroup mine{};  // (no entries: no count is above the threshold)
  mine.nb = kNoCell;
  if (gw < groups) local_group_load(a, gw, mine);
  uint32_t target = 0, first = 0, pass = 0, writer = 0, buf = 0;
  if (!grid_barrier(a.ctr + kCtrBar, target, a.spin_limit, a.err)) return;
  float4 ahead = make_float4(0.0f, 0.0f, 0.0f, 0.0f);  // the place of list entry first + thread
  if (threadIdx.x < m) ahead = __ldcg(a.lnode + threadIdx.x);
  while (int64_t(pass) < a.max_passes) {
    ++pass;
    const bool writes = blockIdx.x == writer;  // the block that writes this pass's deletions
    writer = writer + 1u < gridDim.x ? writer + 1u : 0u;
    // 1. the next `batch` marked entries of the list
    for (uint32_t h = threadIdx.x; h < kLocalHeads; h += kLoopThreads) sm.head[h] = kListEnd;
    uint32_t found = 0;
    auto take = [&](bool in, uint32_t r, uint32_t k, bool fresh) {
      if (!in || r >= a.batch) return;
      const float4 w = fresh ? __ldcg(a.lnode + k) : ahead;
      const uint32_t c = __float_as_uint(w.w);
      const uint32_t old = atomicExch(&sm.head[c & (kLocalHeads - 1u)], r);
      sm.cell[r] = c;
      sm.node[r] = make_float4(w.x, w.y, w.z, __uint_as_float(old));
      if (writes) a.gone[k] = 1;
      if (r + 1 == a.batch) s_next = k + 1;
    };
    for (uint32_t k0 = first;;) {
      const uint32_t ka = k0 + threadIdx.x, kb = ka + kLoopThreads;
      const uint32_t fa = ka < m ? __ldcg(a.off + ka) : ~0u, fb = kb < m ? __ldcg(a.off + kb) : ~0u;
      const bool ina = fa == 0u || fa == pass, inb = fb == 0u || fb == pass;
      const uint32_t ba = __ballot_sync(kFullMask, ina), bb = __ballot_sync(kFullMask, inb);
      if (lane == 0) tmp[buf][warp] = __popc(ba) | (__popc(bb) << 16);
      __syncthreads();
      const uint32_t v = tmp[buf][lane];
      buf ^= 1u;
      const uint32_t tot = __reduce_add_sync(kFullMask, v);
      const uint32_t pre = __reduce_add_sync(kFullMask, lane < warp ? v : 0u);
      const uint32_t lt = (1u << lane) - 1u;
      take(ina, found + (pre & 0xffffu) + __popc(ba & lt), ka, k0 != first);
      take(inb, found + (tot & 0xffffu) + (pre >> 16) + __popc(bb & lt), kb, true);
      found += (tot & 0xffffu) + (tot >> 16);
      if (found > a.batch || m - k0 <= 2u * kLoopThreads) break;
      k0 += 2u * kLoopThreads;  // (stays below m)
    }
    if (found <= a.batch) break;  // (the same in every block) the last pass
    __syncthreads();
    first = s_next;
    // 2. the counts
    local_gather(a, sm, pass, mine);
    for (uint64_t u = gw + gwarps; u < groups; u += gwarps) {
      LocalGroup more;
      local_group_load(a, u, more);
      local_gather(a, sm, pass, more);
      local_group_store(a, more);
    }
    if (first + threadIdx.x < m) ahead = __ldcg(a.lnode + first + threadIdx.x);
    if (!grid_barrier(a.ctr + kCtrBar, target, a.spin_limit, a.err)) return;
  }
  local_group_store(a, mine);
  for (uint64_t k = gt; k < m; k += gthreads)
    if (__ldcg(a.gone + k)) a.dead[__ldg(a.list + k)] = 1;
  if (blockIdx.x == 0 && threadIdx.x == 0) a.ctr[kCtrPasses] = pass;
}

// keep flag per input point (zeroed before: invalid points stay 0): not deleted by a batch
// (the flags the last pass has set are of marked points: those go anyway),
// and its count at most the threshold at the end (the last pass deletes the points still
// marked); number kept.
__global__ __launch_bounds__(256) void thin_keep_kernel(const State* st,
                                                        const float4* __restrict__ pos,
                                                        const uint32_t* __restrict__ cnt,
                                                        const uint8_t* __restrict__ dead,
                                                        uint32_t thr, uint8_t* keep,
                                                        uint32_t* kept, const int* err) {
  if (error_raised(err)) return;  // every keep flag stays 0, the count 0
  uint32_t c = 0;
  const int64_t m = st->nitems;
  for (int64_t i = blockIdx.x * int64_t(256) + threadIdx.x; i < m; i += int64_t(gridDim.x) * 256) {
    const bool k = !dead[i] && cnt[i] <= thr;
    if (k) keep[__float_as_uint(pos[i].w)] = 1;
    c += k;
  }
  __syncwarp();
  c = __reduce_add_sync(kFullMask, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(kept, c);
}

// ---- recounted --------------------------------------------------------------------------

// One pass: every remaining point counts the other remaining points within r in the 27
// cells around it (squared distance, binary32, ((dx*dx + dy*dy) + dz*dz)) and is marked
// when the count exceeds the threshold.  Counting stops once it exceeds the threshold.
__global__ __launch_bounds__(256) void thin_count_kernel(
    const State* st, const int32_t* __restrict__ p2v, const uint32_t* __restrict__ sidx,
    const uint32_t* __restrict__ cstart, const uint32_t* __restrict__ vcnt,
    const uint32_t* __restrict__ nb, const float4* __restrict__ pos, uint8_t* state, float r2,
    int64_t threshold, uint32_t* marked_count, const int* err) {
  if (error_raised(err)) return;  // nothing marked: the loop ends after one pass
  const int64_t m = st->nitems;
  uint32_t marked = 0;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < m;
       i += int64_t(gridDim.x) * blockDim.x) {
    if (!(state[i] & kAlive)) continue;
    const float4 me = pos[i];
    const uint32_t row = static_cast<uint32_t>(p2v[sidx[i]]);
    int64_t cnt = 0;
    for (int o = 0; o < kNb && cnt <= threshold; ++o) {
      const uint32_t c = nb[size_t(row) * kNb + o];
      if (c == kNoCell) continue;
      const int64_t j0 = cstart[c], j1 = j0 + vcnt[c];
      int64_t j = j0;
      for (; j + 4 <= j1 && cnt <= threshold; j += 4) {  // four at a time: their loads overlap
        float4 q[4];
        bool alive[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          alive[u] = (state[j + u] & kAlive) != 0 && j + u != i;
          q[u] = pos[j + u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) cnt += alive[u] && dist2(q[u], me.x, me.y, me.z) <= r2;
      }
      for (; j < j1 && cnt <= threshold; ++j) {
        if (j == i || !(state[j] & kAlive)) continue;
        if (dist2(pos[j], me.x, me.y, me.z) <= r2) ++cnt;
      }
    }
    if (cnt > threshold) {
      state[i] = kAlive | kMarked;
      ++marked;
    }
  }
  for (int off = 16; off; off >>= 1) marked += __shfl_xor_sync(kFullMask, marked, off);
  if ((threadIdx.x & 31) == 0 && marked) atomicAdd(marked_count, marked);
}

// The arrays of this form that the kept counts' cells, groups and flags have overwritten.
__global__ __launch_bounds__(256) void thin_refill_kernel(const State* st,
                                                          const float4* __restrict__ pos,
                                                          const uint32_t* __restrict__ prio,
                                                          uint32_t* sprio, uint32_t* sidx,
                                                          uint8_t* state, const int* err) {
  if (error_raised(err)) return;
  const int64_t m = st->nitems;
  for (int64_t i = blockIdx.x * int64_t(256) + threadIdx.x; i < m; i += int64_t(gridDim.x) * 256) {
    const uint32_t p = __float_as_uint(pos[i].w);
    sprio[i] = prio[p];
    sidx[i] = p;
    state[i] = kAlive;
  }
}

__device__ __forceinline__ uint64_t select_key(const uint32_t* sprio, const uint32_t* sidx,
                                               int64_t i) {
  return (uint64_t(sprio[i]) << 32) | sidx[i];
}

// Histogram of one 8-bit digit of the marked points' keys that match the prefix so far.
__global__ __launch_bounds__(256) void thin_hist_kernel(const State* st, const uint8_t* state,
                                                        const uint32_t* __restrict__ sprio,
                                                        const uint32_t* __restrict__ sidx,
                                                        uint64_t prefix, uint64_t mask, int shift,
                                                        uint32_t* hist, const int* err) {
  __shared__ uint32_t h[256];
  if (block_error_raised(err)) return;
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t m = st->nitems;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < m;
       i += int64_t(gridDim.x) * blockDim.x) {
    if (state[i] != (kAlive | kMarked)) continue;
    const uint64_t k = select_key(sprio, sidx, i);
    if ((k & mask) == prefix) atomicAdd(&h[(k >> shift) & 255u], 1u);
  }
  __syncthreads();
  if (h[threadIdx.x]) atomicAdd(&hist[threadIdx.x], h[threadIdx.x]);
}

// Deletes the marked points whose key, cut to the decided digits, is <= prefix (all
// marked points when mask == 0); unmarks the rest for the next pass.
__global__ __launch_bounds__(256) void thin_delete_kernel(const State* st, uint8_t* state,
                                                          const uint32_t* __restrict__ sprio,
                                                          const uint32_t* __restrict__ sidx,
                                                          uint64_t prefix, uint64_t mask,
                                                          const int* err) {
  if (error_raised(err)) return;
  const int64_t m = st->nitems;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < m;
       i += int64_t(gridDim.x) * blockDim.x) {
    if (state[i] != (kAlive | kMarked)) continue;
    const bool del = (select_key(sprio, sidx, i) & mask) <= prefix;
    state[i] = del ? 0 : kAlive;
  }
}

// keep flag per input point (the buffer was zeroed: invalid points stay 0), number kept.
__global__ __launch_bounds__(256) void thin_output_kernel(const State* st, const uint8_t* state,
                                                          const uint32_t* __restrict__ sidx,
                                                          uint8_t* keep, uint32_t* kept,
                                                          const int* err) {
  if (error_raised(err)) return;  // every keep flag stays 0, the count 0
  const int64_t m = st->nitems;
  uint32_t c = 0;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < m;
       i += int64_t(gridDim.x) * blockDim.x) {
    const bool a = state[i] & kAlive;
    keep[sidx[i]] = a ? 1 : 0;
    c += a;
  }
  for (int off = 16; off; off >>= 1) c += __shfl_xor_sync(kFullMask, c, off);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(kept, c);
}

__global__ void thin_finish_kernel(const uint32_t* kept, int64_t* out_num_kept) {
  *out_num_kept = *kept;
}

vg_status thin_status(cudaError_t e) { return e == cudaSuccess ? VG_OK : VG_ERR_CUDA; }

// Blocks of the loop's cooperative launch (one an SM), 0 where it cannot run.
int thin_loop_grid() {
  int v = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, thin_loop_kernel, kLoopThreads, 0) !=
      cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return v > 0 ? num_sms() : 0;
}

// The same of thin_local_kernel.
int thin_local_grid() {
  int v = 0;
  if (cudaFuncSetAttribute(thin_local_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(sizeof(LocalSmem))) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, thin_local_kernel, kLoopThreads,
                                                    sizeof(LocalSmem)) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return v > 0 ? num_sms() : 0;
}

// Whether the loop keeps counts, by estimated microseconds beside what both forms share.  Kept:
// 100 for its launches, every candidate pair once, a deleted point 4.5 ns and 1.5 more for each
// 1000 candidates, and 10 a pass.  Recounted: a pass takes 130 of host round trips and, a point,
// 0.3 ns, 1.2 for each 1000 candidates up to 1500 (threads of crowded cells end last) and 0.25
// beyond, and 0.5 for 1000 tested until the threshold is passed.  Passes: where the candidates of
// a point are many times the threshold, most points are deleted.  Measured both ways, kept
// against recounted: 640x480 frame (3600 candidates a point), threshold 20, batches of half the
// points 2944 and 1683 us, of an eighth 4063 and 6666; 1M points of 53 candidates, threshold
// 2, half 4102 and 1185, a sixteenth 4981 and 4623; 200,000 of 675, threshold 20, half 883 and
// 593, a quarter 993 and 1074.
bool keep_counts(int64_t n, unsigned long long pairs, int64_t batch, int64_t threshold) {
  if (n <= 0) return false;
  const double nn = double(n), pp = double(pairs), want = double(threshold) + 1.0;
  const double c = pp / nn;  // candidates of a point
  const double gone = pp > 0.0 ? std::max(0.0, 1.0 - 3.0 * want / c) * nn : 0.0;
  const double passes = std::max(1.0, gone / double(batch));
  const double kept = 100.0 + pp / 1.4e6 + (4.5e-3 + 1.5e-6 * c) * gone + 10.0 * passes;
  const double point = 3e-4 + 1.2e-6 * std::min(c, 1500.0) + 2.5e-7 * std::max(c - 1500.0, 0.0) +
                       5e-7 * std::min(c, 6.5 * want);
  return kept <= passes * (130.0 + point * nn);
}

// Whether a pass is thin_local_kernel's, by estimated cycles: 6000 and, for every round of the
// grid's warps over the groups, 2500 and 500 a deleted point that a group meets; scattered, 18,000
// and one per 90 candidates.  Both sides measured: 640x480 frame at 0.05 m, batches of 1000 (one
// round, 13 points a group, 3600 candidates): 7.0 us a pass against 23; 200K points of 84
// candidates (13 rounds): 25 against 14; 1280x720 at 0.02 m (several rounds of small cells): 18
// against 11.
bool local_lists(uint32_t groups, uint32_t batch, double pairs, double n, int grid) {
  const double rounds = std::ceil(double(groups) / (double(grid) * (kLoopThreads / 32)));
  const double met = double(batch) * pairs / n;  // candidates of a batch
  return batch <= kLocalBatch && 6000.0 + rounds * (2500.0 + 500.0 * met / n) <= 18000.0 + met / 90.0;
}

int grid_for(int64_t n) {
  const int64_t b = ceil_div(n < 1 ? 1 : n, 256);
  const int64_t cap = int64_t(num_sms()) * 8;
  return static_cast<int>(b < cap ? b : cap);
}

}  // namespace
}  // namespace vg

using namespace vg;

extern "C" {

size_t vg_thin_workspace_bytes(int64_t n_points) {
  if (n_points < 0 || n_points > kMaxPoints) return 0;
  return thin_layout(n_points).total;
}

vg_status vg_thin(const float* xyz, int64_t n, float* origin, float cell, float radius,
                  int64_t threshold, int64_t batch, const uint32_t* priority, uint8_t* out_keep,
                  int64_t* out_num_kept, int32_t* out_passes, int32_t* out_error,
                  void* workspace, size_t workspace_bytes, int flags, vg_stream_t stream_) {
  if (!(cell > 0.0f) || !std::isfinite(cell)) return VG_ERR_INVALID_ARG;
  if (!(radius > 0.0f) || !(radius <= cell)) return VG_ERR_INVALID_ARG;  // 27 cells suffice
  if (threshold < 0 || batch < 1) return VG_ERR_INVALID_ARG;
  if ((flags & ~VG_ORIGIN_FROM_MIN) != 0) return VG_ERR_INVALID_ARG;
  if (!origin || !out_keep || !out_num_kept || (n > 0 && (!xyz || !priority)))
    return VG_ERR_INVALID_ARG;
  if (n < 0 || n > kMaxPoints) return VG_ERR_INVALID_ARG;
  const ThinLayout L = thin_layout(n);
  if (!workspace || workspace_bytes < L.total) return VG_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255) != 0 ||
      (reinterpret_cast<uintptr_t>(xyz) & 3) != 0 || (reinterpret_cast<uintptr_t>(priority) & 3) != 0 ||
      (reinterpret_cast<uintptr_t>(out_num_kept) & 7) != 0 || (reinterpret_cast<uintptr_t>(origin) & 3) != 0)
    return VG_ERR_ALIGN;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  char* ws = static_cast<char*>(workspace);
  const SortLayout S = sort_layout(n, 1);
  State* st = reinterpret_cast<State*>(ws + S.state);
  int* err = out_error ? reinterpret_cast<int*>(out_error) : &st->error;
  uint64_t* vkeys = reinterpret_cast<uint64_t*>(ws + L.vkeys);
  float* vcent = reinterpret_cast<float*>(ws + L.pos);
  float4* pos = reinterpret_cast<float4*>(ws + L.pos);
  uint32_t* cnt = reinterpret_cast<uint32_t*>(ws + L.cnt);
  uint32_t* vcnt = reinterpret_cast<uint32_t*>(ws + L.vcnt);
  int64_t* vnum = reinterpret_cast<int64_t*>(ws + L.vnum);
  int32_t* p2v = reinterpret_cast<int32_t*>(ws + L.p2v);
  uint32_t* cstart = reinterpret_cast<uint32_t*>(ws + L.cstart);
  uint32_t* nb = reinterpret_cast<uint32_t*>(ws + L.nb);
  uint32_t* entry = reinterpret_cast<uint32_t*>(ws + L.vkeys);  // (once the cells' keys are read)
  uint32_t* list = entry + (n < 1 ? 1 : n);
  uint32_t* sprio = reinterpret_cast<uint32_t*>(ws + L.sprio);
  uint32_t* sidx = reinterpret_cast<uint32_t*>(ws + L.sidx);
  uint8_t* state = reinterpret_cast<uint8_t*>(ws + L.state);
  uint32_t* ctr = reinterpret_cast<uint32_t*>(ws + L.ctr);
  uint32_t* hist = reinterpret_cast<uint32_t*>(ws + L.hist);
  if (out_passes) *out_passes = 0;

  // grouping: the decimation's sort path, wide layout (point_to_voxel = each point's cell)
  const bool from_min = (flags & VG_ORIGIN_FROM_MIN) != 0;
  FramesArg fr{nullptr, 1, n, from_min ? nullptr : origin, from_min ? origin : nullptr, nullptr,
               cell, 0};
  SegOut out{vkeys, vcent, vcnt, nullptr, n, vnum, nullptr, p2v};
  vg_status s = run_frames(xyz, fr, from_min, out, out_error, workspace,
                           frames_workspace_bytes(n, 1, VG_METHOD_SORT), VG_METHOD_SORT, stream);
  if (s != VG_OK) return s;
  cudaError_t e = n > 0 ? cudaMemsetAsync(out_keep, 0, size_t(n), stream) : cudaSuccess;
  if (e == cudaSuccess) e = cudaMemsetAsync(ctr, 0, kCtrWords * sizeof(uint32_t), stream);
  if (e != cudaSuccess) return VG_ERR_CUDA;
  uint32_t* idx0 = reinterpret_cast<uint32_t*>(ws + S.idx0);
  uint32_t* idx1 = reinterpret_cast<uint32_t*>(ws + S.idx1);
  const int g = grid_for(n);
  // the entries' coordinates, an array each (16-byte boundaries), in the sort's key buffers
  float* sx = reinterpret_cast<float*>(ws + S.keys0);
  float* sy = sx + align_up(size_t(n < 1 ? 1 : n), 4);
  float* sz = sy + align_up(size_t(n < 1 ? 1 : n), 4);
  unsigned long long pairs = 0;
  uint32_t groups = 0;
  if (n > 0) {
    thin_neighbors_kernel<<<num_sms() * 8, 256, 0, stream>>>(
        vnum, vkeys, vcnt, nb, ctr, err);
    thin_setup_kernel<<<g, 256, 0, stream>>>(st, idx0, idx1, xyz, priority, p2v, cstart, pos, sx,
                                             sy, sz, sprio, sidx, entry, state, err);
    uint32_t c[4];
    static_assert(kCtrAll == kCtrPairs + 2, "read together");
    e = cudaMemcpyAsync(c, ctr + kCtrPairs, sizeof(c), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return VG_ERR_CUDA;
    pairs = c[0] | ((unsigned long long)c[1] << 32);
    groups = c[2];
  }
  const int64_t max_passes = n / batch + 2;  // every pass but the last deletes `batch` points
  const float r2 = radius * radius;
  int32_t passes = 0;
  const int loop_grid = n > 0 ? thin_loop_grid() : 0;
  if (keep_counts(n, pairs, batch, threshold) && loop_grid > 0) {
    const uint32_t thr = static_cast<uint32_t>(threshold < 0xfffffffell ? threshold : 0xfffffffell);
    State* st2 = reinterpret_cast<State*>(ws + L.st2);
    uint64_t* keys0 = reinterpret_cast<uint64_t*>(ws + S.keys0);
    uint64_t* keys1 = reinterpret_cast<uint64_t*>(ws + S.keys1);
    uint32_t* lb_a = reinterpret_cast<uint32_t*>(ws + S.lb_a);
    uint32_t* lb_b = reinterpret_cast<uint32_t*>(ws + S.lb_b);
    e = cudaMemsetAsync(st2, 0, sizeof(State), stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(state, 0, size_t(n), stream);
    if (e != cudaSuccess) return VG_ERR_CUDA;
    uint32_t* ecell = sprio;  // (the recounted form's arrays)
    uint32_t* group = sidx;
    thin_full_count_kernel<<<static_cast<int>(ceil_div(n, kFullThreads)), kFullThreads, 0,
                             stream>>>(st, p2v, cstart, vcnt, nb, pos, sx, sy, sz, cnt, ecell, group,
                                       ctr, r2, err);
    thin_prio_kernel<<<g, 256, 0, stream>>>(n, p2v, entry, cnt, priority, thr, keys0, st2, err);
    // Where a point has fewer candidates than the threshold on average, mostly none is marked:
    // one more look from the host then saves the sort, the list and the loop (400,000 points of
    // 4 candidates 645 -> 605 us a call, counted afresh every pass 590).
    uint32_t marked = 1;
    if (double(pairs) < (double(threshold) + 1.0) * double(n)) {
      e = cudaMemcpyAsync(&marked, &st2->nitems, sizeof(marked), cudaMemcpyDeviceToHost, stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
      if (e != cudaSuccess) return VG_ERR_CUDA;
    }
    if (marked) {
      e = cudaMemsetAsync(lb_a, 0, size_t(S.sort_tiles) * kRadix * sizeof(uint32_t), stream);
      if (e == cudaSuccess)
        e = launch_sort(st2, keys0, idx0, keys1, idx1, lb_a, lb_b, n, kNarrowPasses, false,
                        spin_limit(), err, stream);  // (32-bit priorities)
      if (e != cudaSuccess) return VG_ERR_CUDA;
      thin_list_kernel<<<g, 256, 0, stream>>>(st2, idx0, idx1, entry, list, err);
    }
    LoopArgs la{};
    la.st2 = st2;
    la.list = list;
    la.ecell = ecell;
    la.cstart = cstart;
    la.vcnt = vcnt;
    la.nb = nb;
    la.pos = pos;
    la.group = group;
    la.cnt = cnt;
    la.dead = state;
    la.ctr = ctr;
    la.r2 = r2;
    la.thr = thr;
    la.batch = static_cast<uint32_t>(batch < n ? batch : n);
    la.pairs_per_point = double(pairs) / double(n);
    la.max_passes = max_passes;
    la.spin_limit = spin_limit();
    la.err = err;
    void* args[] = {&la};
    // the sort's buffers again
    const int local_grid =
        local_lists(groups, la.batch, double(pairs), double(n), loop_grid) ? thin_local_grid() : 0;
    if (marked == 0) {
      // (nothing to delete: one pass)
    } else if (local_grid > 0) {
      // 16 bytes a point from keys1 to the end of idx1, 5 in keys0, 4 in the entries of points
      la.lnode = reinterpret_cast<float4*>(keys1);
      la.off = reinterpret_cast<uint32_t*>(keys0);
      la.gone = reinterpret_cast<uint8_t*>(la.off + align_up(size_t(n), 4));
      la.rank = entry;
      e = launch_cooperative(reinterpret_cast<const void*>(thin_local_kernel), local_grid,
                             kLoopThreads, args, sizeof(LocalSmem), stream);
    } else {
      // the deleted lists' heads (a cell each) and nodes (16 bytes a point of the batch, in
      // the 16 bytes a point from keys1 to the end of idx1), or `sel`
      e = cudaMemsetAsync(keys0, 0, size_t(n) * sizeof(uint64_t), stream);
      if (e != cudaSuccess) return VG_ERR_CUDA;
      la.sel = reinterpret_cast<uint32_t*>(keys0);
      la.head = reinterpret_cast<unsigned long long*>(keys0);
      la.node = reinterpret_cast<float4*>(keys1);
      e = launch_cooperative(reinterpret_cast<const void*>(thin_loop_kernel), loop_grid,
                             kLoopThreads, args, 0, stream);
    }
    if (e == cudaSuccess) {
      thin_keep_kernel<<<g, 256, 0, stream>>>(st, pos, cnt, state, thr, out_keep, ctr + kCtrKept,
                                              err);
      thin_finish_kernel<<<1, 1, 0, stream>>>(ctr + kCtrKept, out_num_kept);
      uint32_t run = 1;
      if (marked)
        e = cudaMemcpyAsync(&run, ctr + kCtrPasses, sizeof(run), cudaMemcpyDeviceToHost, stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
      if (out_passes) *out_passes = static_cast<int32_t>(run);
      return thin_status(e == cudaSuccess ? cudaGetLastError() : e);
    }
    if (e != cudaErrorCooperativeLaunchTooLarge) return VG_ERR_CUDA;
    thin_refill_kernel<<<g, 256, 0, stream>>>(st, pos, priority, sprio, sidx, state, err);
    e = cudaSuccess;  // (the launch does not fit: counted afresh every pass)
  }
  for (; n > 0 && passes < max_passes; ++passes) {
    uint32_t marked = 0;
    e = cudaMemsetAsync(ctr, 0, sizeof(uint32_t), stream);
    if (e != cudaSuccess) return VG_ERR_CUDA;
    thin_count_kernel<<<g, 256, 0, stream>>>(st, p2v, sidx, cstart, vcnt, nb, pos, state, r2,
                                             threshold, ctr, err);
    e = cudaMemcpyAsync(&marked, ctr, sizeof(uint32_t), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return VG_ERR_CUDA;
    if (int64_t(marked) <= batch) {  // the last pass: every marked point goes
      thin_delete_kernel<<<g, 256, 0, stream>>>(st, state, sprio, sidx, ~0ull, 0ull, err);
      ++passes;
      break;
    }
    // radix select of the `batch` smallest keys among the marked, 8 bits a round
    uint64_t prefix = 0, mask = 0;
    int64_t want = batch;
    for (int shift = 56; shift >= 0; shift -= 8) {
      uint32_t h[256];
      e = cudaMemsetAsync(hist, 0, sizeof(h), stream);
      if (e != cudaSuccess) return VG_ERR_CUDA;
      thin_hist_kernel<<<g, 256, 0, stream>>>(st, state, sprio, sidx, prefix, mask, shift, hist,
                                                  err);
      e = cudaMemcpyAsync(h, hist, sizeof(h), cudaMemcpyDeviceToHost, stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
      if (e != cudaSuccess) return VG_ERR_CUDA;
      int d = 0;
      while (d < 255 && want > int64_t(h[d])) want -= h[d++];
      prefix |= uint64_t(d) << shift;
      mask |= 0xffull << shift;
      if (want == int64_t(h[d])) break;  // the whole bucket goes: no finer digit needed
    }
    thin_delete_kernel<<<g, 256, 0, stream>>>(st, state, sprio, sidx, prefix, mask, err);
  }
  if (n > 0) {
    thin_output_kernel<<<g, 256, 0, stream>>>(st, state, sidx, out_keep, ctr + kCtrKept, err);
    thin_finish_kernel<<<1, 1, 0, stream>>>(ctr + kCtrKept, out_num_kept);
  } else {
    e = cudaMemsetAsync(out_num_kept, 0, sizeof(int64_t), stream);
  }
  if (out_passes) *out_passes = passes;
  return thin_status(e == cudaSuccess ? cudaGetLastError() : e);
}

}  // extern "C"
