// Scratch layout and launch of the occupancy-trie grouping (vg_trie.cu).
#pragma once
#include "vg_internal.h"

namespace vg {

constexpr int kTrThreads = 1024;    // threads of a block (one block an SM)
constexpr int kTrDigitBits = 7;     // a slot of the trie: 2^7 children, one bit each
constexpr uint32_t kTrDigit = (1u << kTrDigitBits) - 1u;
constexpr int kTrWords = (1 << kTrDigitBits) / 32;
constexpr size_t kTrSlotBytes = kTrWords * 4 + 8;  // bits and record
constexpr size_t kTrRowBytes = 32;                 // sums, carries and key
static_assert(kTrWords == 4, "a slot's bits are one 16-byte word, its record three prefixes");
constexpr int kTrMaxGrid = 1024;    // blocks of the launch at most
// Bits of the first level (one bit per key prefix): 2 MB up to kTrMaxPoints points, where
// clearing and ranking more costs as much as another level's three barriers; up to 32 MB
// above, where another level is another pass over the runs.
constexpr int kTrRootBits = 24;
constexpr int kTrRootBitsLarge = 28;
// Up to so many points every call takes the trie.  Above, its accesses miss L2 where the cells
// are many (a shuffled cloud of 2.5M points: 268 us at 0.02 m, the radix sort 247; 2.0M: 206
// against 224), so the cells must be few: 2 of 5 sampled pairs of consecutive points share a
// cell (camera frames at 5 mm to 0.1 m: 2 of 5 come with cells for at most a quarter of the
// points, 1 of 5 with more than half), and the cells fit a quarter of the points.
constexpr int64_t kTrMaxPoints = int64_t(1) << 21;
constexpr int64_t kTrCellShare = 4;
constexpr uint32_t kTrSame = 2, kTrSameOf = 5;

// Blocks of the launch for so many chunks of points: one a chunk, but enough of them to clear
// and rank the first level, and at most one an SM.
constexpr int64_t trie_grid(int64_t chunks, int sms) {
  const int64_t most = sms < kTrMaxGrid ? sms : kTrMaxGrid;
  const int64_t least = most > 1 ? most / 2 : 1;
  return chunks < least ? least : (chunks < most ? chunks : most);
}

// Scratch, from `base` on: the first level's bits and records, two buffers of slots (16 B of
// bits and an 8 B record each; the second one holds the rows' sums and keys once the rows are
// known), the runs of every warp (each warp's list has a place for every point it may read),
// the blocks' totals; with attributes, from `att_base` on, the runs' and the rows' sums.
struct TrieLayout {
  size_t root, rootrec, x, y, run, runhi, pslot, mask, stat, total;
  size_t runatt, rowatt, att_total;
  int64_t slots;  // slots (and rows) the buffers hold
};
constexpr TrieLayout trie_layout(int64_t n, int frames, size_t base, size_t att_base = 0) {
  TrieLayout L{};
  const int64_t nn = n < 1 ? 1 : n;
  const int root_bits = nn <= kTrMaxPoints ? kTrRootBits : kTrRootBitsLarge;
  L.slots = nn <= kTrMaxPoints ? nn : nn / kTrCellShare;
  const size_t places = size_t(max_chunks(nn, frames)) * kChunk;
  size_t off = align_up(base, 256);
  L.root = off;
  off = align_up(off + (size_t(1) << (root_bits - 3)), 256);
  L.rootrec = off;
  off = align_up(off + (size_t(1) << (root_bits - kTrDigitBits)) * 8, 256);
  L.x = off;
  off = align_up(off + size_t(L.slots) * kTrSlotBytes, 256);
  L.y = off;
  off = align_up(off + size_t(L.slots) * kTrRowBytes, 256);
  L.run = off;
  off = align_up(off + places * 16, 256);
  L.runhi = off;
  off = align_up(off + places * 4, 256);
  L.pslot = off;
  off = align_up(off + places * 4, 256);
  L.mask = off;
  off = align_up(off + places / 32 * 8, 256);
  L.stat = off;
  off = align_up(off + 8 * size_t(kTrMaxGrid) * sizeof(uint32_t), 256);
  L.total = off;
  off = align_up(att_base, 256);
  L.runatt = off;
  off = align_up(off + places * 8, 256);
  L.rowatt = off;
  off = align_up(off + size_t(L.slots) * 16, 256);
  L.att_total = off;
  return L;
}
static_assert(kTrRowBytes >= kTrSlotBytes, "the second buffer holds slots too");
static_assert((63 - kTrRootBits + kTrDigitBits - 1) / kTrDigitBits + 1 <= 8, "levels");

// Whether the grouping runs on this device, and its launch.  Up to kTrMaxPoints points it
// needs nothing before it and writes every row (two kernels).  Above, it follows the extent
// kernel (with its sample) on a cleared state, and either writes every row (kRowsWritten)
// or leaves the call to the kernels behind it.
bool trie_available(bool posed);
cudaError_t launch_trie(const float* xyz, const FramesArg& fr, State* st, FrameState* fs, char* ws,
                        const TrieLayout& L, const SegOut& out, uint32_t spin_limit, int* err,
                        cudaStream_t stream);
void warm_trie_config();

}  // namespace vg
