// Grouping by hashing (the alternative to sorting every point): steps a2-a5 for clouds
// with many points per voxel.
//
// arXiv 2102.11084 Sec. II-C keeps a (cell, point) table in GPU global memory from which
// the number of points of every cell is known.  Here that table is an open-addressing
// hash table in HBM keyed by the voxel's sort key: every point adds its fixed-point
// offset and a count into its voxel's slot, so only the V occupied slots -- not the N
// points -- are then radix-sorted into key order.  Same key, same accumulator and same
// centroid formula as the sort path, so both paths give identical bits.
//
//   hash_insert_kernel   key per point; runs of equal keys within 32 consecutive points (eight
//                        threads' four) merged and queued by warp; 32 queued runs at a time,
//                        in a crowded cloud merged once more, claim or find their slots and
//                        add to them
//   hash_insert_p2v_kernel  the same for calls that want point_to_voxel: points of a warp with
//                        equal keys are merged (match.any) and their leader claims/updates one
//                        slot, which every point of the group records
//   hash_compact_kernel  occupied slots -> dense (key, slot) list, digit-0 histogram
//   (radix passes over the V entries, compacted-input mode)
//   hash_finalize_kernel sorted (key, slot) -> key, count, centroid rows; slot -> row
//   hash_p2v_kernel      point -> row through its slot (only when asked for)
//
// Slot claiming: where empty slots have zero accumulators (a voxel map), EMPTY -> key by
// compare-and-swap and everyone adds with atomics.  Else EMPTY -> LOCKED, the winner writes
// the slot's accumulator and then publishes the key with a release store; others that see
// LOCKED wait (bounded) and then add with atomics after an acquire load of the key.
//
// The insert is bound by instruction issue (keys, offsets) and by L2's atomics: 64 posed
// frames (29M points) 417 us; runs within a thread's four points only, 475; merging by
// match.any lane group by lane group with four atomics a group, 954.
// In a crowded cloud without order (few cells, or one cell with a tenth of the points) the atomics
// meet on a few addresses, at 1.3 cycles a lane each: the queue's runs of one key are merged
// first (queue_merge).  50M shuffled points of 2 cells 16.9 -> 1.7 ms, of 10 cells 6.7 -> 3.6 (merging
// every point's group by match.any, as the point_to_voxel form does: 5.2 and 5.3); half of the
// points in one of 1M cells 27.5 -> 9.0.  The merge is out of line and behind a test of two ballots:
// in line it spilled, and the 64 frames took 5 % longer; tested by up to four keys of every drain, 7 %.
#include "vg_device.cuh"
#include "vg_internal.h"
#include "vg_stream.cuh"

namespace vg {
namespace {

constexpr unsigned long long kEmpty = ~0ull;
constexpr unsigned long long kLocked = ~0ull - 1ull;
constexpr uint32_t kNoSlot = 0xffffffffu;

// Adds a run (va = x | y << 32, vb = z | points << 32) to an accumulator.
__device__ __forceinline__ void acc_atomic(HashAcc* t, unsigned long long va,
                                           unsigned long long vb) {
  const unsigned long long oa = atomicAdd(&t->a, va), ob = atomicAdd(&t->b, vb);
  const unsigned long long cx = ((oa & 0xffffffffull) + (va & 0xffffffffull)) >> 32;
  const unsigned long long cy = oa + va < oa ? 1ull : 0ull;
  const unsigned long long cz = ((ob & 0xffffffffull) + (vb & 0xffffffffull)) >> 32;
  if (cx | cy | cz) atomicAdd(&t->c, cx | (cy << 21) | (cz << 42));
}

// The points and the (unbiased) sums of an accumulator.
__device__ __forceinline__ Acc acc_read(const HashAcc* t) {
  const unsigned long long a = __ldcg(&t->a), b = __ldcg(&t->b), c = __ldcg(&t->c);
  const unsigned long long cx = c & 0x1fffffull, cy = (c >> 21) & 0x1fffffull, cz = c >> 42;
  Acc r;
  r.n = static_cast<uint32_t>((b >> 32) - cz);
  const unsigned long long s[3] = {(a & 0xffffffffull) + (cx << 32), (a >> 32) + (cy << 32) - cx,
                                   (b & 0xffffffffull) + (cz << 32)};
#pragma unroll
  for (int x = 0; x < 3; ++x)
    r.s[x] = static_cast<long long>(s[x]) + static_cast<long long>(r.n) * kQMin;
  return r;
}

// Adds a run to the slot of `key`; returns the slot or kNoSlot (error recorded).
__device__ __forceinline__ uint32_t table_add(const HashTable& tab, uint64_t key,
                                              unsigned long long va, unsigned long long vb,
                                              uint32_t spin_limit, int* err) {
  uint32_t h = static_cast<uint32_t>(hash64(key)) & tab.mask;
  for (uint32_t probe = 0; probe <= tab.mask; ++probe) {
    if (tab.zeroed) {
      unsigned long long k = __ldcg(&tab.keys[h]);
      if (k == kEmpty) {
        k = atomicCAS(&tab.keys[h], kEmpty, key);
        if (k == kEmpty) k = key;
      }
      if (k == key) {
        acc_atomic(&tab.acc[h], va, vb);
        return h;
      }
      h = (h + 1) & tab.mask;
      continue;
    }
    unsigned long long k = ld_acquire64(&tab.keys[h]);
    if (k == kEmpty) {
      const unsigned long long prev = atomicCAS(&tab.keys[h], kEmpty, kLocked);
      if (prev == kEmpty) {
        tab.acc[h].a = va;
        tab.acc[h].b = vb;
        tab.acc[h].c = 0ull;
        st_release64(&tab.keys[h], key);
        return h;
      }
      k = ld_acquire64(&tab.keys[h]);
    }
    uint32_t spins = 0;
    while (k == kLocked) {
      if (++spins > spin_limit) {
        set_error(err, kErrTimeout);
        return kNoSlot;
      }
      if (spins > 16) __nanosleep(32);
      k = ld_acquire64(&tab.keys[h]);
    }
    if (k == key) {
      acc_atomic(&tab.acc[h], va, vb);
      return h;
    }
    h = (h + 1) & tab.mask;
  }
  set_error(err, kErrCapacity);
  return kNoSlot;
}

// Folds the block's valid points and largest key into the state.  Contains __syncthreads.
__device__ __forceinline__ void insert_stats(State* st, uint32_t nvalid, unsigned long long kmax,
                                             bool range_bad, int* err) {
  __shared__ unsigned long long wmax[kStreamThreads / 32];
  __shared__ uint32_t wcount[kStreamThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (__any_sync(kFullMask, range_bad) && lane == 0) set_error(err, kErrRange);
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    nvalid += __shfl_xor_sync(kFullMask, nvalid, off);
    const unsigned long long other = __shfl_xor_sync(kFullMask, kmax, off);
    kmax = other > kmax ? other : kmax;
  }
  if (lane == 0) {
    wcount[warp] = nvalid;
    wmax[warp] = kmax;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t cnt = 0;
    unsigned long long m = 0;
    for (int w = 0; w < kStreamThreads / 32; ++w) {
      cnt += wcount[w];
      m = wmax[w] > m ? wmax[w] : m;
    }
    if (cnt) {
      atomicAdd(&st->nvalid, cnt);
      atomicMax(&st->maxkey, m);
    }
  }
}

// Runs waiting for their slots, a queue a warp: at most 31 left over and 128 new ones.  (They
// are added in one place: table_add in line after each of a thread's points outgrew the
// instruction cache.)
constexpr int kQueue = 160;
struct InsertQueue {
  unsigned long long key[kQueue];
  unsigned long long xy[kQueue];  // sum x | sum y << 32
  uint32_t zn[kQueue];            // sum z | points << 26
  unsigned long long hot;         // a key that came back, or the last drain's first
};
constexpr size_t kInsertSmem = (kStreamThreads / 32) * sizeof(InsertQueue);

// A crowded cloud's drain (below): merges the warp's runs of one key where three or more meet;
// the first one's lane keeps their sums, the others nothing (kNoKey).
struct QueueRun {
  uint64_t key;
  unsigned long long a, b;  // as table_add's va, vb
};
__device__ __noinline__ QueueRun queue_merge(QueueRun r, unsigned long long* hot_key) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t mine = r.key, hot = *hot_key;
  uint32_t untried = __ballot_sync(kFullMask, mine != kNoKey);
  uint64_t k = __any_sync(kFullMask, mine == hot) ? hot : __shfl_sync(kFullMask, mine, 0);
  for (int misses = 0; untried && misses < 4;) {
    const uint32_t same = __ballot_sync(kFullMask, mine == k) & untried;
    if (__popc(same) >= 3) {
      const bool in = (same >> lane) & 1u, first = int(lane) == __ffs(same) - 1;
      uint32_t w[4] = {uint32_t(r.a), uint32_t(r.a >> 32), uint32_t(r.b), uint32_t(r.b >> 32)};
#pragma unroll
      for (int c = 0; c < 4; ++c)  // (32 runs of 26 bits: below 2^32)
        w[c] = __reduce_add_sync(kFullMask, in ? w[c] : 0u);
      if (first) {
        r.a = w[0] | ((unsigned long long)w[1] << 32);
        r.b = w[2] | ((unsigned long long)w[3] << 32);
        *hot_key = k;
      } else if (in) {
        r.key = kNoKey;
      }
    } else {
      ++misses;
    }
    untried &= ~same;
    k = __shfl_sync(kFullMask, mine, __ffs(untried) - 1);
  }
  return r;
}

template <bool kPosed>
__global__ __launch_bounds__(kStreamThreads, 3) void hash_insert_kernel(
    const float* __restrict__ xyz, FramesArg fr, int have_extent, State* st, FrameState* fs,
    HashTable tab, uint32_t spin_limit, int* err) {
  __shared__ ChunkSmem sm;
  extern __shared__ __align__(8) unsigned char hi_smem[];
  const int F = fr.nframes;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  InsertQueue& q = reinterpret_cast<InsertQueue*>(hi_smem)[warp];
  uint32_t qn = 0;  // queued runs (the same in every lane)
  if (lane == 0) q.hot = kNoKey;
  __syncwarp();
  const uint32_t T = build_chunk_map(fr, sm.off, sm.cstart, sm.tmp, err);
  const uint32_t key_shift = frame_prologue(fr, have_extent != 0, st, fs, T, sm, err);
  // a warp takes every W-th piece of 128 points: no block waits for its slowest warp, and the
  // dense parts of a cloud are shared out
  constexpr uint32_t kPieces = kStreamThreads / 32;  // of a chunk
  const uint64_t pieces = uint64_t(T) * kPieces, W = uint64_t(gridDim.x) * kPieces;
  const bool xyz_vec = (reinterpret_cast<uintptr_t>(xyz) & 15) == 0;
  uint32_t nvalid = 0;
  unsigned long long kmax = 0;
  bool range_bad = false;
  Pose P;
  int pose_f = -1;
  float vn[12];  // the next piece's points
  int fn = 0;
  auto load = [&](uint64_t pc) {
    const uint32_t c = static_cast<uint32_t>(pc / kPieces);
    fn = chunk_frame(sm.cstart, F, c);
    const int64_t start = sm.off[fn] + int64_t(c - sm.cstart[fn]) * kChunk;
    load4(xyz, start + int64_t(pc % kPieces) * 128 + lane * kStreamPoints,
          min(start + kChunk, sm.off[fn + 1]), xyz_vec && (start & 3) == 0, vn);
  };
  const uint64_t first = uint64_t(blockIdx.x) * kPieces + warp;
  if (first < pieces) load(first);
  for (uint64_t pc = first; pc < pieces; pc += W) {
    const int f = fn;
    float v[12];
#pragma unroll
    for (int x = 0; x < 12; ++x) v[x] = vn[x];
    if (pc + W < pieces) load(pc + W);
    if (kPosed) {
      if (f != pose_f) {
        load_pose(fr, f, P);
        pose_f = f;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) pose_point(P, v[3 * j], v[3 * j + 1], v[3 * j + 2]);
    }
    const float o[3] = {sm.org[f][0], sm.org[f][1], sm.org[f][2]};
    const float leaf = sm.leaf[f];
    const float rleaf = sm.rleaf[f];
    const float inv_unit = sm.inv_unit[f];
    // a thread's points and their runs (z carries the points above its 26 bits)
    uint64_t key[4];
    uint32_t w[4][3];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t ijk[3];
      float fi[3];
      key[j] = kNoKey;
      w[j][0] = w[j][1] = w[j][2] = 0;
      if (!point_index(v[3 * j], v[3 * j + 1], v[3 * j + 2], o, leaf, rleaf, ijk, fi, &range_bad))
        continue;
      key[j] = key_compose(static_cast<uint32_t>(f), morton3(ijk[0], ijk[1], ijk[2]), key_shift);
#pragma unroll
      for (int a = 0; a < 3; ++a)
        w[j][a] = quant_biased(v[3 * j + a], voxel_corner(fi[a], o[a], leaf), inv_unit);
      w[j][2] |= 1u << 26;
      ++nvalid;
      kmax = key[j] > kmax ? key[j] : kmax;
    }
    const LaneRuns r = lane_runs<4>(key);
    run_sums<4, 3>(w, r);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool end = (r.tail >> j) & 1u;
      const uint32_t m = __ballot_sync(kFullMask, end);
      if (end) {
        const uint32_t i = qn + __popc(m & ((1u << lane) - 1u));
        q.key[i] = key[j];
        q.xy[i] = w[j][0] | ((unsigned long long)w[j][1] << 32);
        q.zn[i] = w[j][2];
      }
      qn += __popc(m);
    }
    __syncwarp();
    const uint32_t left = pc + W < pieces ? 31u : 0u;  // (the warp's last piece empties the queue)
    while (qn > left) {
      const uint32_t take = min(qn, 32u);
      qn -= take;
      QueueRun r{kNoKey, 0ull, 0ull};
      if (uint32_t(lane) < take) {
        const uint32_t b = q.zn[qn + lane];
        r = QueueRun{q.key[qn + lane], q.xy[qn + lane],
                     (b & 0x3ffffffu) | ((unsigned long long)(b >> 26) << 32)};
      }
      // crowded: a quarter of the runs have lane 0's key, or two have one that the warp has
      // met before (pieces of a scan lie apart: theirs do not come back)
      const uint64_t lead = __shfl_sync(kFullMask, r.key, 0), hot = q.hot;
      const int again = __popc(__ballot_sync(kFullMask, r.key == hot && hot != kNoKey));
      if (again >= 2 || __popc(__ballot_sync(kFullMask, r.key == lead)) >= 8)
        r = queue_merge(r, &q.hot);
      else if (again == 0 && lane == 0)
        q.hot = lead;
      if (r.key != kNoKey) (void)table_add(tab, r.key, r.a, r.b, spin_limit, err);
      __syncwarp();
    }
    __syncwarp();
  }
  __syncwarp();
  insert_stats(st, nvalid, kmax, range_bad, err);
}

template <bool kPosed>
__global__ __launch_bounds__(kStreamThreads) void hash_insert_p2v_kernel(
    const float* __restrict__ xyz, FramesArg fr, int have_extent, State* st, FrameState* fs,
    HashTable tab, uint32_t* __restrict__ point_slot, uint32_t spin_limit, int* err) {
  __shared__ ChunkSmem sm;
  __shared__ int s_q[kStreamThreads / 32][32][3];
  const int F = fr.nframes;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t T = build_chunk_map(fr, sm.off, sm.cstart, sm.tmp, err);
  const uint32_t key_shift = frame_prologue(fr, have_extent != 0, st, fs, T, sm, err);
  uint32_t c0, c1;
  block_range(T, &c0, &c1);
  const bool xyz_vec = (reinterpret_cast<uintptr_t>(xyz) & 15) == 0;
  uint32_t nvalid = 0;
  unsigned long long kmax = 0;
  bool range_bad = false;
  Pose P;
  int pose_f = -1;
  for (uint32_t c = c0; c < c1; ++c) {
    const int f = chunk_frame(sm.cstart, F, c);
    const int64_t start = sm.off[f] + int64_t(c - sm.cstart[f]) * kChunk;
    const int64_t end = min(start + kChunk, sm.off[f + 1]);
    const int64_t p0 = start + int64_t(threadIdx.x) * kStreamPoints;
    float v[12];
    load4(xyz, p0, end, xyz_vec && (start & 3) == 0, v);
    if (kPosed) {
      if (f != pose_f) {
        load_pose(fr, f, P);
        pose_f = f;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) pose_point(P, v[3 * j], v[3 * j + 1], v[3 * j + 2]);
    }
    const float o[3] = {sm.org[f][0], sm.org[f][1], sm.org[f][2]};
    const float leaf = sm.leaf[f];
    const float rleaf = sm.rleaf[f];
    const float inv_unit = sm.inv_unit[f];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint64_t local = 0;
      uint32_t ijk[3];
      float fi[3];
      const bool ok = point_index(v[3 * j], v[3 * j + 1], v[3 * j + 2], o, leaf, rleaf, ijk, fi,
                                  &range_bad);
      if (ok) local = morton3(ijk[0], ijk[1], ijk[2]);
      const uint64_t key = ok ? key_compose(static_cast<uint32_t>(f), local, key_shift) : 0;
      uint32_t slot = kNoSlot;
      const uint32_t vm = __ballot_sync(kFullMask, ok);
      if (ok) {
        ++nvalid;
        kmax = key > kmax ? key : kmax;
        const Acc a = point_acc(local, v[3 * j], v[3 * j + 1], v[3 * j + 2], o, leaf, inv_unit);
        s_q[warp][lane][0] = static_cast<int>(a.s[0]);
        s_q[warp][lane][1] = static_cast<int>(a.s[1]);
        s_q[warp][lane][2] = static_cast<int>(a.s[2]);
        const uint32_t peers = __match_any_sync(vm, key);
        const int leader = __ffs(peers) - 1;
        __syncwarp(vm);
        if (lane == leader) {
          Acc g = acc_zero();
          for (uint32_t m = peers; m; m &= m - 1) {
            const int l = __ffs(m) - 1;
            g.n += 1;
            g.s[0] += s_q[warp][l][0];
            g.s[1] += s_q[warp][l][1];
            g.s[2] += s_q[warp][l][2];
          }
          // (biased sums of at most 32 points: below 2^26)
          const unsigned long long b = uint64_t(g.n) * uint64_t(-kQMin);
          slot = table_add(tab, key, (unsigned long long)(g.s[0] + b) |
                                         ((unsigned long long)(g.s[1] + b) << 32),
                           (unsigned long long)(g.s[2] + b) | ((unsigned long long)g.n << 32),
                           spin_limit, err);
        }
        slot = __shfl_sync(vm, slot, leader);
        __syncwarp(vm);
      }
      if (p0 + j < end) point_slot[p0 + j] = slot;
    }
  }
  insert_stats(st, nvalid, kmax, range_bad, err);
}

// Occupied slots -> dense (key, slot) entries for the radix sort; counts them into
// st->nitems and histograms their digit 0.  Tiles of 2048 slots, a block scan and one atomic a
// tile (an atomic on the one counter every 32 slots took 154 us for 8.4M slots, 25
// now).
constexpr int kCompactItems = 8;
__global__ __launch_bounds__(256) void hash_compact_kernel(HashTable tab, State* st,
                                                           uint64_t* __restrict__ keys,
                                                           uint32_t* __restrict__ slots,
                                                           const int* err) {
  __shared__ uint32_t hist[kRadix];
  __shared__ uint32_t tmp[8];
  __shared__ uint32_t s_base;
  if (block_error_raised(err)) return;  // an earlier step failed
  hist[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t H = tab.mask + 1;  // (a multiple of 1024)
  for (uint64_t base = uint64_t(blockIdx.x) * (256 * kCompactItems); base < H;
       base += uint64_t(gridDim.x) * (256 * kCompactItems)) {
    unsigned long long k[kCompactItems];
    uint32_t occ = 0;
#pragma unroll
    for (int q = 0; q < kCompactItems; q += 2) {
      const uint64_t h = base + 512u * (q / 2) + 2u * threadIdx.x;
      k[q] = k[q + 1] = kEmpty;
      if (h < H) {
        const ulonglong2 w = __ldcg(reinterpret_cast<const ulonglong2*>(tab.keys + h));
        k[q] = w.x;
        k[q + 1] = w.y;
      }
    }
#pragma unroll
    for (int q = 0; q < kCompactItems; ++q) occ += k[q] != kEmpty && k[q] != kLocked;
    uint32_t total;
    uint32_t pos = block_excl_scan(occ, &total, tmp);
    if (total == 0) continue;  // (the same in every thread)
    if (threadIdx.x == 0) s_base = atomicAdd(&st->nitems, total);
    __syncthreads();
    pos += s_base;
#pragma unroll
    for (int q = 0; q < kCompactItems; ++q)
      if (k[q] != kEmpty && k[q] != kLocked) {
        keys[pos] = k[q];
        slots[pos] = static_cast<uint32_t>(base + 512u * (q / 2) + 2u * threadIdx.x + (q & 1));
        atomicAdd(&hist[k[q] & (kRadix - 1)], 1u);
        ++pos;
      }
    __syncthreads();
  }
  __syncthreads();
  if (hist[threadIdx.x]) atomicAdd(&st->hist[0][threadIdx.x], hist[threadIdx.x]);
}

// Empties a zeroed table: the occupied slots' keys and accumulators.
__global__ __launch_bounds__(256) void hash_clear_kernel(HashTable tab) {
  const uint64_t H = uint64_t(tab.mask) + 1;
  for (uint64_t h = (uint64_t(blockIdx.x) * 256 + threadIdx.x) * 2; h < H;
       h += uint64_t(gridDim.x) * 512) {
    ulonglong2* kp = reinterpret_cast<ulonglong2*>(tab.keys + h);
    const ulonglong2 k = __ldcg(kp);
    if (k.x == kEmpty && k.y == kEmpty) continue;
    *kp = make_ulonglong2(kEmpty, kEmpty);
    if (k.x != kEmpty) tab.acc[h] = HashAcc{0ull, 0ull, 0ull, 0ull};
    if (k.y != kEmpty) tab.acc[h + 1] = HashAcc{0ull, 0ull, 0ull, 0ull};
  }
}

// Sorted (key, slot) entries -> output rows.
__global__ __launch_bounds__(256) void hash_finalize_kernel(
    const State* st, const FrameState* __restrict__ fs, int nframes,
    const uint64_t* __restrict__ keys0, const uint32_t* __restrict__ idx0,
    const uint64_t* __restrict__ keys1, const uint32_t* __restrict__ idx1, HashTable tab,
    uint32_t* __restrict__ slot_rank, SegOut out, int* err) {
  if (error_raised(err)) return;  // an earlier step failed
  const int64_t V = st->nitems;
  const int passes = max(1, sort_passes(st->maxkey));
  const uint64_t* K = (passes & 1) ? keys1 : keys0;
  const uint32_t* I = (passes & 1) ? idx1 : idx0;
  const uint32_t key_shift = st->key_shift;
  for (int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x; i < V; i += int64_t(gridDim.x) * 256) {
    const uint64_t key = K[i];
    const uint32_t slot = I[i];
    const uint32_t f = key_frame(key, key_shift);
    if (i >= out.cap) {
      set_error(err, kErrCapacity);
    } else {
      const Acc a = acc_read(&tab.acc[slot]);
      const uint64_t local = key_local(key, key_shift);
      const float o[3] = {fs[f].origin[0], fs[f].origin[1], fs[f].origin[2]};
      const float leaf = fs[f].leaf;
      float c[3];
      acc_centroid(local, a, o, leaf, leaf, c);
      out.keys[i] = local;
      out.counts[i] = a.n;
      out.centroids[3 * i] = c[0];
      out.centroids[3 * i + 1] = c[1];
      out.centroids[3 * i + 2] = c[2];
      if (out.sums) {
        out.sums[3 * i] = a.s[0];
        out.sums[3 * i + 1] = a.s[1];
        out.sums[3 * i + 2] = a.s[2];
      }
    }
    if (slot_rank) slot_rank[slot] = static_cast<uint32_t>(i);
    if (out.frame_offsets) {
      if (i > 0) {
        const uint32_t fp = key_frame(K[i - 1], key_shift);
        for (uint32_t g = fp + 1; g <= f; ++g) out.frame_offsets[g] = i;
      }
      if (i == V - 1)
        for (uint32_t g = f + 1; g <= uint32_t(nframes); ++g) out.frame_offsets[g] = V;
    }
    if (i == V - 1) *out.num_voxels = V;
  }
}

__global__ __launch_bounds__(256) void hash_p2v_kernel(const uint32_t* __restrict__ point_slot,
                                                       const uint32_t* __restrict__ slot_rank,
                                                       int64_t n, int32_t* __restrict__ p2v,
                                                       const int* err) {
  if (error_raised(err)) return;  // an earlier step failed
  for (int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * 256) {
    const uint32_t s = point_slot[i];
    p2v[i] = s == kNoSlot ? -1 : static_cast<int32_t>(slot_rank[s]);
  }
}

}  // namespace

cudaError_t launch_hash_insert(const float* xyz, const FramesArg& fr, bool have_extent, State* st,
                               FrameState* fs, const HashTable& tab, uint32_t* point_slot,
                               uint32_t spin_limit, int* err, cudaStream_t stream) {
  const int g = stream_grid(fr), ext = have_extent ? 1 : 0;
  const int64_t chunks = max_chunks(fr.n, fr.nframes);
  if (point_slot && posed(fr))
    hash_insert_p2v_kernel<true><<<g, kStreamThreads, 0, stream>>>(xyz, fr, ext, st, fs, tab,
                                                                   point_slot, spin_limit, err);
  else if (point_slot)
    hash_insert_p2v_kernel<false><<<g, kStreamThreads, 0, stream>>>(xyz, fr, ext, st, fs, tab,
                                                                    point_slot, spin_limit, err);
  else if (posed(fr))
    hash_insert_kernel<true><<<persistent_grid(reinterpret_cast<const void*>(
                                                   hash_insert_kernel<true>),
                                               kStreamThreads, kInsertSmem, chunks),
                               kStreamThreads, kInsertSmem, stream>>>(xyz, fr, ext, st, fs, tab,
                                                                      spin_limit, err);
  else
    hash_insert_kernel<false><<<persistent_grid(reinterpret_cast<const void*>(
                                                    hash_insert_kernel<false>),
                                                kStreamThreads, kInsertSmem, chunks),
                                kStreamThreads, kInsertSmem, stream>>>(xyz, fr, ext, st, fs, tab,
                                                                       spin_limit, err);
  return cudaGetLastError();
}

void warm_hash_config() {  // (allows the shared memory, once a device)
  for (const void* fn : {reinterpret_cast<const void*>(hash_insert_kernel<true>),
                         reinterpret_cast<const void*>(hash_insert_kernel<false>)})
    (void)persistent_grid(fn, kStreamThreads, kInsertSmem, 1);
}


cudaError_t launch_hash_clear(const HashTable& tab, cudaStream_t stream) {
  const int64_t want = ceil_div(int64_t(tab.mask) + 1, 512), cap = int64_t(num_sms()) * 8;
  hash_clear_kernel<<<static_cast<int>(want < cap ? want : cap), 256, 0, stream>>>(tab);
  return cudaGetLastError();
}

cudaError_t launch_hash_compact(const HashTable& tab, State* st, uint64_t* keys, uint32_t* slots,
                                const int* err, cudaStream_t stream) {
  const int64_t H = int64_t(tab.mask) + 1;
  const int64_t want = ceil_div(H, 256 * kCompactItems);
  const int64_t cap = int64_t(num_sms()) * 8;
  hash_compact_kernel<<<static_cast<int>(want < cap ? want : cap), 256, 0, stream>>>(tab, st, keys,
                                                                                    slots, err);
  return cudaGetLastError();
}

cudaError_t launch_hash_finalize(const State* st, const FrameState* fs, int nframes,
                                 const uint64_t* keys0, const uint32_t* idx0,
                                 const uint64_t* keys1, const uint32_t* idx1,
                                 const HashTable& tab, uint32_t* slot_rank, int64_t n_max,
                                 const SegOut& out, int* err, cudaStream_t stream) {
  if (n_max == 0) return cudaSuccess;
  // (n_max bounds the voxels; a block a possible 256 of them took 77 us for 8.4M slots)
  const int64_t want = ceil_div(n_max, 256), most = int64_t(num_sms()) * 8;
  hash_finalize_kernel<<<static_cast<int>(want < most ? want : most), 256, 0, stream>>>(
      st, fs, nframes, keys0, idx0, keys1, idx1, tab, slot_rank, out, err);
  return cudaGetLastError();
}

cudaError_t launch_hash_p2v(const uint32_t* point_slot, const uint32_t* slot_rank, int64_t n,
                            int32_t* p2v, const int* err, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  const int64_t want = ceil_div(n, 256);
  const int64_t cap = int64_t(num_sms()) * 16;
  hash_p2v_kernel<<<static_cast<int>(want < cap ? want : cap), 256, 0, stream>>>(
      point_slot, slot_rank, n, p2v, err);
  return cudaGetLastError();
}

}  // namespace vg
