// bt_batch.cuh -- types shared by the host driver and the persistent kernel of
// the batched build (bt_batch.cu).
//
// A batch is built by one persistent kernel per size class of documents.
// Every CTA (one to an SM, narrower ones for short documents; for few long
// documents: every cluster of CTAs) takes the next
// document from a device work queue (an atomic
// counter over the documents in decreasing length) and builds that
// document's whole tree by itself, level by level (section 3's levels, the
// Karp-Rabin pass of section 3.1, then the pruning post-pass and the
// rank/select counters), with a barrier of the CTA between the steps.  No
// step of a document needs the host, so one launch builds thousands of
// documents, each with the same result as a standalone build.
#pragma once

#include "bt_internal.cuh"
#include "bt_quick.cuh"

namespace bt {

constexpr uint32_t kBMaxLevels = 40;       // documents with more levels use the standard path
constexpr uint64_t kBMaxText = 1ull << 30; // longest document of the batched path
// One document of a batch (host -> device).
struct BDoc {
  const uint8_t* T;     // device text
  uint64_t n;
  uint32_t sigma, L;
  uint32_t index;       // position in the caller's arrays
  uint32_t lv_off;      // first entry of this document in the level arrays
};

// Per level of a finished document (device -> host).
struct BLevelRes {
  uint64_t c, b, nmarked;
  uint32_t arity, cw;
  uint64_t stats[BT_ST_FIELDS];
};

// Per document (device -> host).
struct BRes {
  int status;              // BT_OK, BT_EINVAL (alphabet), BT_ENOMEM (pool), BT_EINTERNAL
  uint32_t S;
  uint64_t leaf_bytes;     // bytes of leaf text
  uint64_t out_off;        // the tree's arrays: pool + out_off
  uint64_t out_bytes;      // bytes taken from the pool (or needed, with BT_ENOMEM)
  // SM clock cycles the CTA (a cluster's leading one) spent per phase: set-up (alphabet, prefix
  // fingerprints), tables (block and pair fingerprints), window scan,
  // verification / marks / pointers / split, pruning, output and counters.
  unsigned long long cycles[6];
};

// Where the arrays of a finished tree lie in its pool region, in bytes from
// the region's start.  The same function runs on the device (to write the
// tree) and on the host (to point the bt_tree at it).
struct OutLevel {
  uint64_t mw, mr, rec, cnt, pc;
};
__host__ __device__ inline uint64_t out_align(uint64_t x) { return (x + 255) & ~255ull; }
__host__ __device__ inline uint64_t out_align16(uint64_t x) { return (x + 15) & ~15ull; }

// The level queries start at (as for a single text): the lowest one with all
// blocks whose prefix table stays within an eighth of the text, or 8 KiB; at
// most 1024 blocks, as one CTA fills the table.
__host__ __device__ inline uint32_t out_base(uint32_t L, const uint64_t* c, const uint64_t* b, uint64_t n, uint32_t S) {
  uint32_t base = 0;
  for (uint32_t l = 1; l < L; l++) {
    if (c[l] != (n + b[l] - 1) / b[l] || c[l] > 1024) break;
    const uint64_t bytes = (c[l] + 1) * S * 4;
    if (bytes <= n / 8 || bytes <= (8u << 10)) base = l;
  }
  return base;
}

// c[l]: blocks of level l after pruning; cw[l]: counter bytes; S symbols;
// leaf_alloc: leaf text bytes (rounded).  Returns the region's size.
__host__ __device__ inline uint64_t out_layout(uint32_t L, uint32_t base, const uint64_t* c, const uint32_t* cw, uint32_t S,
                                               uint64_t leaf_alloc, OutLevel* lv, uint64_t* view,
                                               uint64_t* pre, uint64_t* leaf, uint64_t* sym) {
  uint64_t o = 0;
  *view = o;
  o = out_align16(o + sizeof(TreeView));
  for (uint32_t l = 0; l < L; l++) {
    const uint64_t words = (c[l] + 31) / 32;
    lv[l].rec = o;
    o = out_align16(o + c[l] * 8 + 8);
    lv[l].mw = o;
    o = out_align16(o + words * 4 + 4);
    lv[l].mr = o;
    o = out_align16(o + (words + 1) * 4);
    lv[l].cnt = o;
    if (l >= base) o = out_align16(o + counter_stride(c[l]) * S * cw[l]);
    lv[l].pc = o;
    if (l >= base) o = out_align16(o + counter_stride(c[l]) * S * cw[l]);
  }
  *pre = o;
  o = out_align16(o + (c[base] + 1) * (uint64_t)S * 4);
  *leaf = o;
  o = out_align16(o + leaf_alloc + 16);
  *sym = o;
  o = out_align16(o + 256 * sizeof(int16_t));
  return o;
}

constexpr uint32_t kCommonBytes = 4096;  // first of all: what a cluster's CTAs share

// Scratch of one CTA (or cluster) for one document: offsets in bytes from its
// region.  Level l may hold at most cmax[l] = ceil(n / b_l) blocks.
struct ScratchLayout {
  uint64_t Hs;                                  // u64[n / 32 + 2]: prefix fingerprints H(32 j)
  uint64_t big;                                 // the list's positions and distances, u32[n] each; later, for
                                                // levels by the window scan, u64[n + 1]: H at every position
  uint64_t idx, seg1, seg2, first;              // the list's index and segment minima; the first-occurrence table
  uint64_t cells;
  uint64_t st[kBMaxLevels], lo[kBMaxLevels], off[kBMaxLevels];  // u64[cmax]
  uint64_t ptr[kBMaxLevels], mw[kBMaxLevels], mr[kBMaxLevels];  // u32
  uint64_t temp;                                // per-level work area (reused)
  uint64_t total;
};

__host__ __device__ inline uint64_t pow2_ge(uint64_t x) {
  uint64_t p = 16;
  while (p < x) p <<= 1;
  return p;
}

// Bytes of the per-level work area for a level of at most cm blocks of b bytes:
// the level pass (by first occurrences, or for short blocks the tables of the
// window scan) or the pruning pass, whichever is larger.
__host__ __device__ inline uint64_t temp_bytes(uint64_t cm, uint64_t b) {
  const uint64_t cap = pow2_ge(2 * cm);
  const uint64_t quick = out_align(cm * 4 + 4) * 4      // A, X, flags, wpop
                         + out_align(cm * 8 + 8)        // items
                         + out_align(cm + 8)            // ps
                         + out_align(cap * 32) + out_align(cap * 16)               // block and pair tables
                         + out_align(2 * cap * 16) + out_align(2 * cap * 8)        // gram table and bounds
                         + out_align(8 * cm + 1024)     // bitmap
                         + out_align(cm * 8 + 8) * 6;   // islot, igram, differ, susp (two per block), exlo
  const uint64_t scan = out_align(cm * 8 + 8) * 6       // fpB, exBL, job_of, susp, exlo, spare
                        + out_align(cm * 4 + 4) * 4     // slotB, slotP, mismatch, wpop
                        + out_align(cm + 8)             // pm
                        + out_align(cm * 32 + 32)       // jobs
                        + out_align(cap * 32) + out_align(cap * 16);
  const uint64_t level = b >= kQuickMinB && quick > scan ? quick : scan;  // (the first may end up as the second)
  const uint64_t prune = out_align(cm + 8) * 5          // hit_v, hit2, tgt_w, gone, mk2
                         + out_align(cm * 4 + 4) * 7    // state, indeg, fq x2, nidx, wpop, ptr2
                         + out_align(cm * 8 + 8) * 5;   // t1, t2, st2, off2, lo2
  return level > prune ? level : prune;
}

__host__ __device__ inline uint64_t scratch_layout(uint64_t n, uint32_t L, const uint64_t* b, ScratchLayout* s) {
  uint64_t o = kCommonBytes, temp = 0;
  s->Hs = o;
  o = out_align(o + (n / 32 + 2) * 8);
  s->big = o;
  o = out_align(o + (n + 64) * 8);
  s->idx = o;
  o = out_align(o + (n / 32 + 2) * 4);
  s->seg1 = o;
  o = out_align(o + (n / 1024 + 2) * 4);
  s->seg2 = o;
  o = out_align(o + (n / 65536 + 2) * 4);
  s->cells = 1024;
  while (s->cells < n / 8) s->cells <<= 1;
  s->first = o;
  o = out_align(o + s->cells * 4);
  for (uint32_t l = 0; l < L; l++) {
    const uint64_t cm = (n + b[l] - 1) / b[l];
    const uint64_t words = (cm + 31) / 32;
    const uint64_t tb = temp_bytes(cm, b[l]);
    if (tb > temp) temp = tb;
    s->st[l] = o;
    o = out_align(o + cm * 8 + 8);
    s->lo[l] = o;
    o = out_align(o + cm * 8 + 8);
    s->off[l] = o;
    o = out_align(o + cm * 8 + 8);
    s->ptr[l] = o;
    o = out_align(o + cm * 4 + 4);
    s->mw[l] = o;
    o = out_align(o + words * 4 + 4);
    s->mr[l] = o;
    o = out_align(o + (words + 1) * 4 + 4);
  }
  s->temp = o;
  o = out_align(o + temp);
  s->total = o;
  return o;
}

// Kernel parameters of one class launch.
struct BParams {
  const BDoc* docs;
  uint32_t ndocs;
  unsigned int* next;             // work-queue counter
  const uint64_t* sizes;          // block sizes, docs[d].lv_off + l
  BRes* res;
  BLevelRes* lres;
  char* scratch;
  uint64_t scratch_per_cta;
  char* pool;
  unsigned long long* pool_used;
  uint64_t pool_cap;
  uint64_t B;                     // Karp-Rabin base
  int prune;
  uint64_t max_rounds;
  uint32_t dyn_words;             // 32-bit words of dynamic shared memory
};

}  // namespace bt
