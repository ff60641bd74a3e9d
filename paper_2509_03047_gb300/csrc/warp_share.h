// warp_share.h -- how one sweep launch shares its warps among the (element
// type, alignment) classes of the chunks it covers.  Host code on plain
// arrays (the no-allocation fingerprint plans with it too).
//
// A warp sweeps a range of one class only.  The classes are not equally
// costly per block: a bf16 block holds twice the elements of an fp32 block,
// so the fingerprint spends almost half as much again on it, while
// pack and unpack are bound by memory in every class.  The warps are shared
// in proportion to each class's blocks times its weight (percent of an fp32
// block), so that the classes' warps finish together.  The classes of shifted
// chunks take the launch's first warps, those of aligned chunks the others,
// and within either range each class's warps are spread round-robin over the
// CTAs, so an SM runs a mix of element types (place_warps).  Within a class the
// ranges are cut by an estimated cost per segment (seg_cost, SegWalk::to_cost).
#pragma once

#include <cstdint>

#include "layout.h"

#ifndef FR_MIX_W_BF16
// Fingerprint: a bf16 block costs 1.45 fp32 blocks.  Measured, GPT-2 small
// (1.7 GB) / Llama-8B shard (14 GB) in us: 1.35 293 / 2085, 1.40 289 / 2079,
// 1.45 283 / 2092, 1.50 283 / 2103.  A compromise: the shard alone is best at
// 1.40, by 0.6%, GPT-2 small at 1.45, by 2%.
#define FR_MIX_W_BF16 145
#endif
#ifndef FR_MIX_W_BF16_PACK
#define FR_MIX_W_BF16_PACK 100  // pack and unpack: memory-bound, all blocks alike
#endif
// Fingerprint: a block of a chunk off the 16-byte boundary costs 0.25 fp32
// blocks more (0.15 / 0.25 / 0.4: 539 / 529 / 560 us for 2.5 GB of views); pack
// and unpack even it out with their units.
#ifndef FR_MIX_W_SHIFT
#define FR_MIX_W_SHIFT 25
#endif
#ifndef FR_MIX_W_BYTES
#define FR_MIX_W_BYTES 100
#endif
// Within a class, warp ranges (whole 16 KiB sum segments) are cut by an
// estimated cost per segment, in units of one 512-byte block's sweep:
// FR_SPLIT_BLK per block it holds, FR_SPLIT_SEG for its end (the sums'
// check, fold and store), and FR_SPLIT_PIECE more if it begins a chunk (the
// warp's pipeline starts over on a new address and the CRC streams are
// folded at the end of the previous piece).  Measured on GB300: by bytes
// alone short segments are underpriced (gpt2s fingerprint -3 points against
// equal segment counts); these costs beat equal counts by up to half a point
// on the fragmented and small states.
#ifndef FR_SPLIT_BLK
#define FR_SPLIT_BLK 1
#endif
#ifndef FR_SPLIT_SEG
#define FR_SPLIT_SEG 2
#endif
#ifndef FR_SPLIT_PIECE
#define FR_SPLIT_PIECE 16
#endif

// A pack or unpack launch keeps FR_DYN_PCT percent of each class's segments
// out of the warps' own runs, as units that warps claim at run time, of
// FR_UNIT_SEGS segments or a few more (unit_segs).  Measured on GB300, pack /
// unpack of GPT-2 small: no units 562 / 564 us; 8% in units of 1, 2 and 4
// segments 547 / 538, 545 / 538, 549 / 540; 4% of 1 553 / 548.
#ifndef FR_DYN_PCT
#define FR_DYN_PCT 8
#endif
// The classes of shifted chunks keep FR_DYN_PCT_MIXED percent in a launch that
// holds aligned classes too.  They have SMs of their own (place_warps), on which
// a block of unpack takes longer, and pack and unpack share one plan, so no
// weight suits both (10% more warps for them: unpack 351 -> 337 us below, but
// flat views' pack 777 -> 811).  Measured with 8 / 12 / 16 / 24 percent, 1 GB in
// eight fp32 tensors, one of them shifted: unpack 350 / 342 / 335 / 331 us, pack
// 333 either way; 2.5 GB of flat views, pack and unpack with both tables: 1,585 /
// 1,592 / 1,588 / 1,593.  Where every class is shifted 16 percent cost unpack 1%.
#ifndef FR_DYN_PCT_MIXED
#define FR_DYN_PCT_MIXED 16
#endif
#ifndef FR_UNIT_SEGS
#define FR_UNIT_SEGS 2
#endif
// A large state starts with larger units, 1 / FR_UNIT_SHARE of a warp's share of
// what is left but at most FR_UNIT_MAX segments (256 KiB): with 32 KiB ones the
// last 8% of a 32 GB state was 77,000 records, 512 for a 16 MiB chunk (its pack
// 10,179 us, 10,155 with larger ones; smaller states equal).  The two values
// matter little: pack of 32 GB with a share of 1, 2, 4, 8, 16: 10,140 / 10,148 /
// 10,152 / 10,153 / 10,160 us, with a maximum of 2, 16, 64: 10,161 / 10,152 /
// 10,154; GPT-2 small, the Llama-8B shard and the fragmented states move by 0.2%.
#ifndef FR_UNIT_SHARE
#define FR_UNIT_SHARE 4
#endif
#ifndef FR_UNIT_MAX
#define FR_UNIT_MAX 16
#endif
// A class has units only from FR_CLAIM_MIN segments per warp on.  Measured, no
// units / units, us, by segments per warp: pack of 130 MB (2.6) 50.0 / 49.6, 159
// MB (3.2) 61.5 / 59.9, 203 MB (4.1) 76.2 / 73.0, 300 MB (5.9) 107 / 102; GPT-2
// small restored in 32 batches (2.2) 1,650 / 1,665, in 24 (2.9) 1,474 / 1,485, in
// 16 (4.4) 1,470 / 1,461.  With 4 no batched restore loses and a state of 3 to 4
// segments per warp forgoes 2%.
#ifndef FR_CLAIM_MIN
#define FR_CLAIM_MIN 4
#endif

namespace frk {

enum : int { kShareFingerprint = 1, kSharePack = 2 };

// Weight of a block of element type `dt` for a launch of kind `kind`.
inline double block_weight(uint32_t dt, int kind) {
  if (dt == kDtF32) return 100.0;
  if (dt == kDtBf16) return kind == kShareFingerprint ? FR_MIX_W_BF16 : FR_MIX_W_BF16_PACK;
  return FR_MIX_W_BYTES;
}
// Of sweep class `cls`.
inline double class_weight(uint32_t cls, int kind) {
  return block_weight(cls / 2, kind) + ((cls & 1u) == 0 && kind == kShareFingerprint ? FR_MIX_W_SHIFT : 0);
}

// wc[q] = warps of class q (q < n <= W): W shared in proportion to cost[q] > 0,
// every class at least one, largest shortfall first for the remainder.
inline void share_warps(const double* cost, int n, uint64_t W, uint64_t* wc) {
  double total = 0.0;
  for (int q = 0; q < n; ++q) total += cost[q];
  uint64_t given = 0;
  for (int q = 0; q < n; ++q) {
    const uint64_t w = static_cast<uint64_t>(static_cast<double>(W) * cost[q] / total);
    wc[q] = w > 0 ? w : 1;
    given += wc[q];
  }
  while (given < W) {
    int best = 0;
    double gap = -1e300;
    for (int q = 0; q < n; ++q) {
      const double g = static_cast<double>(W) * cost[q] / total - static_cast<double>(wc[q]);
      if (g > gap) gap = g, best = q;
    }
    ++wc[best];
    ++given;
  }
  while (given > W) {  // only when many tiny classes each took one
    int best = 0;
    for (int q = 1; q < n; ++q)
      if (wc[q] > wc[best]) best = q;
    --wc[best];
    --given;
  }
}

// Estimated cost of a segment of `blocks` blocks; `first`: it begins a chunk.
inline uint64_t seg_cost(uint64_t blocks, bool first) {
  return FR_SPLIT_BLK * blocks + FR_SPLIT_SEG + (first ? FR_SPLIT_PIECE : 0);
}

// How many of the last segments of sweep class `cls`, of n in all and shared by
// Wq warps, are cut into units (none for the fingerprint, see mode_claims, nor
// while the warps have too few segments each for a tail to even out).  `mixed`:
// the launch holds classes of both alignments.
inline uint64_t claimed_segs(uint64_t n, uint64_t Wq, int kind, uint32_t cls, bool mixed) {
  const uint64_t percent = mixed && (cls & 1u) == 0 ? FR_DYN_PCT_MIXED : FR_DYN_PCT;
  return kind == kShareFingerprint || n < FR_CLAIM_MIN * Wq ? 0 : n * percent / 100;
}
// Segments of the unit cut where `left` remain: a share of what is left, so
// that a large state has few units and a chunk of it few records, down to
// FR_UNIT_SEGS and single segments at the end, so that no warp starts a long
// unit when the others run out of work.
inline uint64_t unit_segs(uint64_t left, uint64_t Wq) {
  const uint64_t least = left > Wq ? FR_UNIT_SEGS : 1, share = left / (FR_UNIT_SHARE * Wq);
  const uint64_t n = share < least ? least : share < FR_UNIT_MAX ? share : FR_UNIT_MAX;
  return n < left ? n : left;
}

// slot[q * stride + j] = launch-warp index of class q's j-th warp, for the m
// classes q in `qs`, which share the launch warps [first, first + count); warp
// w is warp w % warps_per_cta of CTA w / warps_per_cta.  The range's warps are
// taken one per CTA in turn, and each class takes a run of consecutive ones,
// so every whole CTA of the range holds the floor or the ceiling of its share
// of every class.  The sum of wc[q] is count.
inline void spread_range(const uint64_t* wc, const int* qs, int m, uint64_t first, uint64_t count, int warps_per_cta,
                         uint32_t* slot, uint64_t stride) {
  const uint64_t wpc = static_cast<uint64_t>(warps_per_cta), end = first + count;
  uint64_t cta = first / wpc, row = 0;  // the next candidate: warp `row` of `cta`
  for (int k = 0; k < m; ++k) {
    for (uint64_t j = 0; j < wc[qs[k]];) {
      const uint64_t w = cta * wpc + row;
      if (w >= first && w < end) slot[static_cast<uint64_t>(qs[k]) * stride + j++] = static_cast<uint32_t>(w);
      if (++cta * wpc >= end) cta = first / wpc, ++row;
    }
  }
}

// The warps of a launch's classes (class q is sweep class cls[q]): those of
// shifted chunks on the first CTAs, those of aligned chunks on the others (one
// CTA may hold both), each spread over its CTAs.  Element types share every
// SM on purpose; but every class is a loop of its own, and four of them
// outgrow an SM's instruction cache (2.5 GB of views, every class on every SM
// / alignments apart: fingerprint 839 / 711 us with 37% of the instruction
// fetches missing, pack 932 / 918).
inline void place_warps(const uint32_t* cls, const uint64_t* wc, int n, int warps_per_cta, uint32_t* slot,
                        uint64_t stride) {
  uint64_t first = 0;
  for (uint32_t aligned = 0; aligned < 2; ++aligned) {
    int qs[kClassCount], m = 0;
    uint64_t count = 0;
    for (int q = 0; q < n; ++q)
      if ((cls[q] & 1u) == aligned) {
        qs[m++] = q;
        count += wc[q];
      }
    spread_range(wc, qs, m, first, count, warps_per_cta, slot, stride);
    first += count;
  }
}

}  // namespace frk
