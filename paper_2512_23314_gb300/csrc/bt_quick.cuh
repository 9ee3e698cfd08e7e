// bt_quick.cuh -- the level pass by first occurrences (bt_quick.cu).
#pragma once

#include <functional>

#include "bt_internal.cuh"

namespace bt {

// Blocks of at least this many bytes hold a selected gram (16 + 12 - 1).
constexpr uint64_t kQuickMinB = 27;

// The selected grams of the text in order: position x[e] and distance D[e] to
// the gram's first occurrence; idx[j] = the first entry at or after position
// 32 j, idx[nw] their number; minima of D per 1 KiB and 64 KiB of positions.
struct QList {
  const uint32_t* idx;
  const uint32_t* x;
  const uint32_t* D;
  const uint32_t* seg1;
  const uint32_t* seg2;
  uint64_t nw;
};

// Device scalars of a level.
struct QuickStatus {
  unsigned long long nopen[2];  // open blocks, open pairs
  unsigned long long nitems, npairs, nmarked, nsusp;
  unsigned long long fp_tail, lo_tail, lo_tailpair;  // keys that end in the short last block
  unsigned long long cands, hits;
  unsigned long long work;    // of the search of the open keys (kWalkWork, kTestWork)
  unsigned long long probes;  // slots passed by the long walks of their registration
  unsigned int pretail, tail_F, tail_off;
  unsigned int total;  // entries of the list
  unsigned int redo;   // how far the search of the open keys is (ChaseState)
};

struct QuickBuild {
  bool ready = false;
  Scratch mem;
  Arena open;  // tables of a level's open keys
  uint32_t *idx = nullptr, *x = nullptr, *D = nullptr, *seg1 = nullptr, *seg2 = nullptr;
  QList list{};
  QuickStatus* qs = nullptr;
  QuickStatus* qs_host = nullptr;  // in the thread's pinned page
  std::function<int()> expand;  // ctx.H for the scan of every window
  explicit QuickBuild(cudaStream_t s) : mem(s) { open.s = s; }
  ~QuickBuild() { open.release(); }
};

// Returned by quick_level: this level goes by the scan of every window.
constexpr int kEveryWindow = -1;

int quick_list(BuildCtx& ctx, QuickBuild& qb);
int quick_level(BuildCtx& ctx, QuickBuild& qb, uint32_t l, uint64_t last_start);

// bt_level.cu
int alloc_level_arrays(Level& v, uint64_t words, cudaStream_t s);
int launch_children(BuildCtx& ctx, uint32_t l, uint64_t bn, uint64_t* next_st);

}  // namespace bt
