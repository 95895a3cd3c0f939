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
// Word of a slot's child d among the words of its level.  (The number of the child's bit, slot
// x 2^7 + d, passes 32 bits from 2^25 slots on; the word's does not.)
constexpr uint32_t trie_word(uint32_t slot, uint32_t d) { return slot * kTrWords + (d >> 5); }
constexpr int kTrMaxGrid = 1024;    // blocks of the launch at most
// Bits of the first level at most (one bit per key prefix).  Up to kTrMidPoints points 2^26,
// 2^24 of which (2 MB) every call of at most kTrMaxPoints clears while the extents are found
// and the rest, where the keys' width calls for more, with a barrier of its own: less than
// another level's three barriers and pass over the runs (1M shuffled points of 32-bit keys: 155
// us with 24 bits and two further levels, 106 with 25 and one).  Above, 32 MB where the keys
// are that wide.
constexpr int kTrRootClear = 24;
constexpr int kTrRootBits = 26;
constexpr int kTrRootBitsLarge = 28;
// Up to kTrMaxPoints points every call takes the trie.  Above, its accesses miss L2 where the
// cells are many: a shuffled map takes 238 to 255 us at 2,621,440 points (0.05 to 0.02 m), the
// radix sort 258; at 3.5M 308 to 386 against 293.  (Shuffled keys wider than 33 bits lose below
// the line too: from 1.08 times the sort's time at 1.6M points of random keys to 1.49 at 2.62M.  The
// sort path behind every call of that size, to leave them to, costs 22 us a call.)  So the
// kernel looks, on the device, and takes the calls
//   * whose cells are few: 2 of 5 sampled pairs of consecutive points share a cell (camera
//     frames at 5 mm to 0.1 m: 2 of 5 come with cells for at most a quarter of the points, 1
//     of 5 with more than half); above kTrMidPoints they must fit a quarter of the points;
//   * up to kTrMidPoints points, whose keys have at most 27 bits (one level or a nearly empty
//     second: 4M points of 26-bit keys 210 us, the radix sort 316), or more than 32 where half
//     of the sampled pairs lie within 32 leaves (a scan of 4M points in its order 428 us, the
//     radix sort's wide layout 480; shuffled, every level's accesses miss: 874 against 486).
constexpr int64_t kTrMaxPoints = int64_t(5) << 19;
constexpr int64_t kTrMidPoints = int64_t(1) << 22;
constexpr int64_t kTrCellShare = 4;
constexpr uint32_t kTrMidBits = 27;
constexpr uint32_t kTrSame = 2, kTrSameOf = 5;

// Points a prefix, on average, up to which a further level is marked unseen.
constexpr int64_t kTrSparse = 4;

// Slots of a further level, and rows, that a call's buffers hold.
constexpr int64_t trie_slots(int64_t n) { return n <= kTrMidPoints ? n : n / kTrCellShare; }
static_assert(trie_word(static_cast<uint32_t>(trie_slots(kMaxPoints)) - 1u, kTrDigit) ==
                  uint64_t(trie_slots(kMaxPoints) - 1) * kTrWords + (kTrDigit >> 5),
              "32-bit word numbers for the largest call");

constexpr int trie_root_bits(int64_t n) {
  return n <= kTrMidPoints ? kTrRootBits : kTrRootBitsLarge;
}

// Blocks of the launch for so many chunks of points: one a chunk, but enough of them to clear
// and rank the first level, and at most one an SM.
constexpr int64_t trie_grid(int64_t chunks, int sms) {
  const int64_t most = sms < kTrMaxGrid ? sms : kTrMaxGrid;
  const int64_t least = most > 1 ? most / 2 : 1;
  return chunks < least ? least : (chunks < most ? chunks : most);
}

// Scratch, from `base` on: the first level's bits and records, two buffers of slots (16 B of
// bits and an 8 B record each; the second one holds the rows' sums and keys once the rows are
// known), the runs of every block (each block's list has a place for every point it may read),
// the blocks' totals; with attributes, from `att_base` on, the runs' and the rows' sums.
struct TrieLayout {
  size_t root, rootrec, x, y, run, runhi, pslot, mask, first, stat, total;
  size_t runatt, rowatt, att_total;
  int64_t slots;  // slots (and rows) the buffers hold
};
constexpr TrieLayout trie_layout(int64_t n, int frames, size_t base, size_t att_base = 0) {
  TrieLayout L{};
  const int64_t nn = n < 1 ? 1 : n;
  const int root_bits = trie_root_bits(nn);
  L.slots = trie_slots(nn);
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
  off = align_up(off + places / 4, 256);
  L.first = off;
  off = align_up(off + places / 32 * 4, 256);
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
