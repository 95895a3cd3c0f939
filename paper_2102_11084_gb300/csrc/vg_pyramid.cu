// Step a6: the count-weighted octree pyramid.
//
// arXiv 2102.11084 reduces the cloud "iteratively with an ordered subdivision of space"
// (abstract, Sec. II-C) and recalls the octree, whose cells split into eight children
// (Sec. I).  Level 0 is the decimation at leaf L; level k+1 merges level k into parents
// key >> 3 (edge 2L): because Morton order is preserved by the shift, the children of a
// parent are adjacent rows of level k (at most 8), so no re-sort is needed.  n' = sum n;
// the parent's fixed-point sum is the children's sums moved to the parent corner:
//   S' = sum (S_child + n_child * round((c_child - C_parent) / u0)),
// all in units u0 = L/2^20 (the level-0 unit), and the centroid is C' + (S'/n')*u0 in
// binary32 -- the same formula as level 0 with leaf 2^k L for the corner.
//
// One kernel per level, tiles of 1024 rows (ticketed): the tile's run heads are found with
// coalesced loads (a ballot word per warp and step), ranked by a bounded chained scan that
// the whole block waits in, and compacted, so that consecutive threads take consecutive
// parents.  Bound by latency (one wait and three dependent loads a level).  A 1280x720 frame
// at 0.01 m (390K rows, three merges): 152 us a level with eight rows a thread and one
// thread walking the chained scan, 12 us now.
#include "vg_device.cuh"
#include "vg_internal.h"

namespace vg {
namespace {

static_assert(kMergeThreads == 256, "block_lookback");
constexpr int kMergeWarps = kMergeThreads / 32;

__global__ __launch_bounds__(kMergeThreads) void pyramid_merge_kernel(
    State* st, const FrameState* __restrict__ fs, int level, uint64_t* keys, float* centroids,
    uint32_t* counts, const long long* __restrict__ sums_in, long long* __restrict__ sums_out,
    int64_t* level_offsets, int64_t cap, uint32_t* lb, uint32_t spin_limit, int* err) {
  __shared__ int s_tile;
  __shared__ uint32_t s_bits[kMergeItems * kMergeWarps];  // heads among 32 consecutive rows
  __shared__ uint32_t s_before[kMergeItems * kMergeWarps];
  __shared__ uint32_t s_total;
  __shared__ uint32_t s_lb[kMergeWarps][2];
  __shared__ uint16_t s_head[kMergeTile];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // An earlier step failed: take no ticket.  Every ticket taken is processed, so no tile
  // ever waits for one that a returning block skipped.
  if (block_error_raised(err)) return;
  if (t == 0) s_tile = static_cast<int>(atomicAdd(&st->tile_ctr[kMaxPasses + level], 1u));
  __syncthreads();
  const int tile = s_tile;
  const int64_t off_prev = level_offsets[level - 1];
  const int64_t off_cur = level_offsets[level];
  const int64_t vprev = off_cur - off_prev;
  const int64_t base = int64_t(tile) * kMergeTile;
  if (base >= vprev) return;
  const int cnt = static_cast<int>(vprev - base < kMergeTile ? vprev - base : kMergeTile);

  const float o[3] = {fs[0].origin[0], fs[0].origin[1], fs[0].origin[2]};
  const float leaf0 = fs[0].leaf;
  const float inv_unit0 = quant_inv_unit(leaf0);
  const float leaf_child = __fmul_rn(leaf0, float(1u << (level - 1)));
  const float leaf_par = __fmul_rn(leaf0, float(1u << level));
  const uint64_t* ck = keys + off_prev;
  const uint32_t* cn = counts + off_prev;
  const long long* cs = sums_in;

  // run heads of the tile's rows
  uint64_t k[kMergeItems], kp[kMergeItems];
#pragma unroll
  for (int j = 0; j < kMergeItems; ++j) {
    const int li = j * kMergeThreads + t;
    const int64_t r = base + li;
    k[j] = li < cnt ? ck[r] : 0ull;
    kp[j] = li < cnt && r > 0 ? ck[r - 1] : ~0ull;
  }
#pragma unroll
  for (int j = 0; j < kMergeItems; ++j) {
    const int li = j * kMergeThreads + t;
    const uint32_t b = __ballot_sync(kFullMask, li < cnt && (k[j] >> 3) != (kp[j] >> 3));
    if (lane == 0) s_bits[j * kMergeWarps + warp] = b;
  }
  __syncthreads();
  static_assert(kMergeItems * kMergeWarps == 32, "one warp ranks the head words");
  if (warp == 0) {
    const uint32_t c = __popc(s_bits[lane]);
    uint32_t inc = c;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(kFullMask, inc, off);
      if (lane >= off) inc += y;
    }
    s_before[lane] = inc - c;
    if (lane == 31) {
      s_total = inc;
      st_relaxed(lb + tile, (tile == 0 ? kFlagPrefix : kFlagAggregate) | inc);
    }
  }
  __syncthreads();
  const uint32_t total = s_total;
#pragma unroll
  for (int j = 0; j < kMergeItems; ++j) {
    const uint32_t b = s_bits[j * kMergeWarps + warp];
    if ((b >> lane) & 1u)
      s_head[s_before[j * kMergeWarps + warp] + __popc(b & ((1u << lane) - 1u))] =
          static_cast<uint16_t>(j * kMergeThreads + t);
  }
  const uint32_t excl = block_lookback(lb, tile, spin_limit, err, s_lb);
  if (t == 0) {
    if (tile > 0) st_relaxed(lb + tile, kFlagPrefix | ((excl + total) & kValueMask));
    if (base + kMergeTile >= vprev) level_offsets[level + 1] = off_cur + excl + total;
  }
  __syncthreads();

  for (uint32_t p = t; p < total; p += kMergeThreads) {
    const int64_t r = base + s_head[p];
    uint64_t ckey[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) ckey[c] = r + c < vprev ? ck[r + c] : ~0ull;
    const uint64_t pkey = ckey[0] >> 3;
    Acc acc = acc_zero();
    uint32_t odd[3] = {0, 0, 0};  // points of the children on the upper side of each axis
    bool in = true;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      in = in && r + c < vprev && (ckey[c] >> 3) == pkey;
      if (!in) continue;
      const uint32_t n = cn[r + c];
      acc.n += n;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        acc.s[a] += cs[3 * (r + c) + a];
        odd[a] += (ckey[c] >> a) & 1u ? n : 0u;
      }
    }
    // A child on the lower side of an axis has its parent's corner there (2 i * leaf is
    // i * (2 leaf) before rounding too); one on the upper side moves its n points by the
    // one shift of that parent and axis.
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (odd[a] == 0) continue;
      const uint32_t pi = key_axis(pkey, a);
      const float C = voxel_corner(pi, o[a], leaf_par);
      const float cc = voxel_corner(2u * pi + 1u, o[a], leaf_child);
      const double shift = (double(cc) - double(C)) * double(inv_unit0);
      acc.s[a] += static_cast<long long>(odd[a]) * __double2ll_rn(shift);
    }
    const int64_t lr = int64_t(excl) + p;
    const int64_t out = off_cur + lr;
    if (out >= cap) {
      set_error(err, kErrCapacity);
      continue;
    }
    float cent[3];
    acc_centroid(pkey, acc, o, leaf_par, leaf0, cent);
    keys[out] = pkey;
    counts[out] = acc.n;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      centroids[3 * out + a] = cent[a];
      sums_out[3 * lr + a] = acc.s[a];
    }
  }
}

}  // namespace

cudaError_t launch_pyramid_merge(State* st, const FrameState* fs, int level, uint64_t* keys,
                                 float* centroids, uint32_t* counts, const long long* sums_in,
                                 long long* sums_out, int64_t* level_offsets, int64_t cap,
                                 uint32_t* lb, int64_t n_max, uint32_t spin_limit, int* err,
                                 cudaStream_t stream) {
  if (n_max == 0) return cudaSuccess;
  const int tiles = static_cast<int>(ceil_div(n_max, kMergeTile));
  pyramid_merge_kernel<<<tiles, kMergeThreads, 0, stream>>>(st, fs, level, keys, centroids, counts,
                                                            sums_in, sums_out, level_offsets, cap,
                                                            lb, spin_limit, err);
  return cudaGetLastError();
}

}  // namespace vg
