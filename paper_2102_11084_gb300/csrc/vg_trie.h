// Scratch layout and launch of the occupancy-trie grouping (vg_trie.cu).
#pragma once
#include "vg_internal.h"

namespace vg {

constexpr int kTrThreads = 1024;    // threads of a block (one block an SM)
constexpr int kTrDigitBits = 8;     // a slot of the trie: 2^8 children, one bit each
constexpr int kTrWords = (1 << kTrDigitBits) / 32;
constexpr int kTrMaxGrid = 1024;    // blocks of the launch at most
// Bits of the first level (one bit per key prefix, cleared by every call): 2 MB up to
// kTrSmallPoints points, where clearing and ranking more costs as much as another level's
// three barriers; 32 MB above, where another level is another pass over the points.
constexpr int kTrRootBits = 24;
constexpr int kTrRootBitsLarge = 28;
constexpr int64_t kTrSmallPoints = int64_t(1) << 22;

constexpr int trie_root_bits(int64_t n) {
  return n <= kTrSmallPoints ? kTrRootBits : kTrRootBitsLarge;
}

// Scratch, from `base` on: the first level's bits and records, two buffers of slots (32 B of
// bits and a 16 B record each; the second one holds the rows' sums, keys and attribute sums
// once the rows are known), a word per point, the blocks' totals.
struct TrieLayout {
  size_t root, rootrec, x, y, pslot, stat, total;
  int64_t slots;  // slots (and rows) the buffers hold
};
constexpr TrieLayout trie_layout(int64_t n, size_t base) {
  TrieLayout L{};
  const int64_t nn = n < 1 ? 1 : n;
  const int rb = trie_root_bits(nn);
  L.slots = nn;
  size_t off = align_up(base, 256);
  L.root = off;
  off = align_up(off + (size_t(1) << (rb - 3)), 256);
  L.rootrec = off;
  off = align_up(off + (size_t(1) << (rb - kTrDigitBits)) * 16, 256);
  L.x = off;
  off = align_up(off + size_t(L.slots) * 48, 256);
  L.y = off;
  off = align_up(off + size_t(L.slots) * 48, 256);
  L.pslot = off;
  off = align_up(off + size_t(nn) * sizeof(uint32_t), 256);
  L.stat = off;
  off = align_up(off + 8 * size_t(kTrMaxGrid) * sizeof(uint32_t), 256);
  L.total = off;
  return L;
}

// Whether the grouping runs on this device, and its launch (two kernels).
bool trie_available(bool posed);
cudaError_t launch_trie(const float* xyz, const FramesArg& fr, State* st, FrameState* fs, char* ws,
                        const TrieLayout& L, const SegOut& out, uint32_t spin_limit, int* err,
                        cudaStream_t stream);
void warm_trie_config();

}  // namespace vg
