// seg_walk.h -- a walk over the sum segments of one sweep class, in chunk
// order, that cuts it into runs of pieces.  Host code on plain arrays (the
// no-allocation fingerprint plans with it too).
//
// A position is a segment boundary: segment `seg` of chunk list[k], with the
// estimated cost (seg_cost) and the number of all segments before it.  Both
// ways to move on skip whole chunks and compute the place inside the last one,
// so a cut costs O(chunks + runs), not O(segments): a prefix sum over the
// 860,000 segments of a 14 GB state took 10 ms of a plan's creation.
#pragma once

#include <algorithm>
#include <cstdint>

#include "gf2.cuh"
#include "layout.h"
#include "warp_share.h"

namespace frk {

class SegWalk {
 public:
  // `list`: the n chunks of the class that have a body, in order.
  SegWalk(ChunkDesc* chunks, const uint32_t* list, uint64_t n) : chunks_(chunks), list_(list), n_(n) {}

  uint64_t segs() const { return segs_; }  // segments before the position
  uint64_t cost() const { return before_ + cost_in(seg_); }  // and their cost

  // Moves `count` segments on (to the end at most).
  void skip(uint64_t count) {
    uint64_t to = segs_ + count;
    while (k_ < n_ && segs_ - seg_ + n_seg() <= to) next_chunk();
    if (k_ < n_ && to > segs_) {
      seg_ += to - segs_;
      segs_ = to;
    }
  }
  // Moves to the last boundary of at most `cost` and at most `segs` segments
  // before it (or stays).
  void to_cost(uint64_t cost, uint64_t segs) {
    while (k_ < n_ && before_ + cost_in(n_seg()) <= cost && segs_ - seg_ + n_seg() <= segs) next_chunk();
    if (k_ == n_ || before_ + FR_SPLIT_PIECE > cost) return;
    // inside this chunk: i segments, all whole, cost FR_SPLIT_PIECE + i * (a whole segment's)
    uint64_t i = std::min<uint64_t>((cost - before_ - FR_SPLIT_PIECE) / seg_cost(kSegBlocks, false), n_seg() - 1);
    i = std::min(i, segs - (segs_ - seg_));
    if (i > seg_) {
      segs_ += i - seg_;
      seg_ = i;
    }
  }

  // Emits the pieces from here to `end`, a later position of the same class:
  // piece(descriptor, blocks after it in its chunk's body) for each chunk
  // overlapped, `index` being the first piece's.  Sets the chunks' first_rec
  // and n_recs.  Returns the number of pieces.
  template <class Piece>
  uint32_t emit(const SegWalk& end, uint32_t index, const Piece& piece) const {
    uint64_t k = k_, off = seg_ * kSegBlocks;
    uint32_t count = 0;
    for (; k < end.k_ || (k == end.k_ && k < n_ && off < end.seg_ * kSegBlocks); ++k, off = 0) {
      ChunkDesc& d = chunks_[list_[k]];
      const uint64_t nb = d.len / kBlockBytes;
      const uint64_t to = k == end.k_ ? end.seg_ * kSegBlocks : nb;
      PieceDesc pd;
      pd.addr = d.addr + off * kBlockBytes;
      pd.payload_off = d.payload_off + off * kBlockBytes;
      pd.seg = d.seg_base + static_cast<uint32_t>(off / kSegBlocks);
      pd.nblk = static_cast<uint32_t>(to - off);
      pd.chunk = list_[k];
      pd.unused = 0;
      if (d.n_recs == 0) d.first_rec = index + count;
      d.n_recs += 1;
      piece(pd, nb - to);
      ++count;
    }
    return count;
  }

 private:
  uint64_t blocks() const { return chunks_[list_[k_]].len / kBlockBytes; }
  uint64_t n_seg() const { return (blocks() + kSegBlocks - 1) / kSegBlocks; }
  // cost of this chunk's first i segments
  uint64_t cost_in(uint64_t i) const {
    if (i == 0) return 0;
    return FR_SPLIT_PIECE + FR_SPLIT_SEG * i + FR_SPLIT_BLK * std::min<uint64_t>(i * kSegBlocks, blocks());
  }
  void next_chunk() {
    before_ += cost_in(n_seg());
    segs_ += n_seg() - seg_;
    seg_ = 0;
    ++k_;
  }

  ChunkDesc* chunks_;
  const uint32_t* list_;
  uint64_t n_;
  uint64_t k_ = 0, seg_ = 0;          // the position: segment seg_ of chunk list_[k_]
  uint64_t segs_ = 0, before_ = 0;    // segments before it; cost of the chunks before k_
};

}  // namespace frk
