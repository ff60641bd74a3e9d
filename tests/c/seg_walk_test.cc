// seg_walk_test.cc -- checks the planner's segment walk (csrc/seg_walk.h)
// against the plain rule it stands for: split_ranges over the prefix sums of
// every segment's cost (split_ranges.h).  Exits 0 and prints "seg_walk ok".
#include <cstdio>
#include <cstring>
#include <vector>

#include "seg_walk.h"
#include "split_ranges.h"

using namespace frk;

#define EXPECT(c)                                                    \
  do {                                                               \
    if (!(c)) {                                                      \
      std::fprintf(stderr, "%s:%d check failed: %s\n", __FILE__, __LINE__, #c); \
      return 1;                                                      \
    }                                                                \
  } while (0)

// One class of chunks with the given lengths, its first n_fix segments cut
// into Wq runs, the rest into units of `unit` segments.
static int check(const std::vector<uint64_t>& lens, uint64_t Wq, uint64_t dyn_percent, uint64_t unit) {
  std::vector<ChunkDesc> chunks(lens.size() + 1);  // a chunk of another class first: ids are not positions
  std::vector<uint32_t> list;
  std::vector<uint64_t> cost(1, 0), seg_chunk, seg_off;
  std::memset(chunks.data(), 0, chunks.size() * sizeof(ChunkDesc));
  uint64_t addr = 1 << 20, payload = 4096, segs = 7;
  for (size_t i = 0; i < lens.size(); ++i) {
    ChunkDesc& d = chunks[i + 1];
    d.addr = addr;
    d.len = lens[i];
    d.payload_off = payload;
    d.seg_base = static_cast<uint32_t>(segs);
    const uint64_t nb = d.len / kBlockBytes;
    if (nb) list.push_back(static_cast<uint32_t>(i + 1));
    for (uint64_t j = 0; j < nb; j += kSegBlocks) {
      cost.push_back(cost.back() + seg_cost(std::min<uint64_t>(kSegBlocks, nb - j), j == 0));
      seg_chunk.push_back(i + 1);
      seg_off.push_back(j);
    }
    segs += (nb + kSegBlocks - 1) / kSegBlocks;
    addr += d.len + 48;
    payload = align_up(payload + d.len, kPayloadAlign);
  }
  const uint64_t n = seg_chunk.size(), n_fix = n - n * dyn_percent / 100;
  std::vector<uint64_t> bnd(Wq + 1);
  split_ranges([&](uint64_t i) { return cost[i]; }, n_fix, Wq, bnd.data());

  SegWalk at(chunks.data(), list.data(), list.size()), fixed = at;
  fixed.skip(n_fix);
  EXPECT(fixed.segs() == n_fix && fixed.cost() == cost[n_fix]);
  std::vector<PieceDesc> pieces;
  std::vector<uint64_t> after;
  auto piece = [&](const PieceDesc& pd, uint64_t blocks_after) {
    pieces.push_back(pd);
    after.push_back(blocks_after);
  };
  auto run = [&](const SegWalk& to) {
    const size_t first = pieces.size();
    const uint32_t got = at.emit(to, static_cast<uint32_t>(first), piece);
    at = to;
    return got == pieces.size() - first;
  };
  for (uint64_t w = 1; w <= Wq; ++w) {
    SegWalk to = at;
    to.to_cost(static_cast<uint64_t>(static_cast<unsigned __int128>(cost[n_fix]) * w / Wq), n_fix);
    EXPECT(to.segs() == bnd[w] && to.cost() == cost[bnd[w]]);
    EXPECT(run(to));
  }
  while (at.segs() < n) {
    SegWalk to = at;
    to.skip(unit);
    EXPECT(to.segs() == std::min(n, at.segs() + unit));
    EXPECT(run(to));
  }
  // the pieces cover every segment once, in order, and never two chunks
  uint64_t s = 0;
  for (size_t r = 0; r < pieces.size(); ++r) {
    const PieceDesc& pd = pieces[r];
    ChunkDesc& d = chunks[pd.chunk];
    const uint64_t nb = d.len / kBlockBytes;
    EXPECT(s < n && seg_chunk[s] == pd.chunk && pd.nblk > 0);
    EXPECT(pd.addr == d.addr + seg_off[s] * kBlockBytes && pd.payload_off == d.payload_off + seg_off[s] * kBlockBytes);
    EXPECT(pd.seg == d.seg_base + seg_off[s] / kSegBlocks);
    EXPECT(after[r] == nb - seg_off[s] - pd.nblk);
    EXPECT(r >= d.first_rec && r < d.first_rec + d.n_recs);
    EXPECT(after[r] == 0 || pd.nblk % kSegBlocks == 0);
    s += (pd.nblk + kSegBlocks - 1) / kSegBlocks;
  }
  EXPECT(s == n);
  uint64_t recs = 0;
  for (const ChunkDesc& d : chunks) recs += d.n_recs;
  EXPECT(recs == pieces.size());
  return 0;
}

int main() {
  uint32_t x = 12345;
  auto next = [&](uint32_t m) { return (x = x * 1103515245u + 12345u, (x >> 8) % m); };
  for (int kind = 0; kind < 4; ++kind)
    for (int trial = 0; trial < 40; ++trial) {
      std::vector<uint64_t> lens;
      const uint32_t count = 1 + next(kind == 3 ? 3 : 60);
      for (uint32_t i = 0; i < count; ++i)
        lens.push_back(kind == 0   ? next(2000)
                       : kind == 1 ? 512 * (1 + next(200)) + next(512)
                       : kind == 2 ? 16384 * (1 + next(4))
                                   : (1 << 20) * (1 + next(40)) + next(700));
      for (uint64_t Wq : {1ull, 2ull, 7ull, 152ull, 2432ull})
        for (uint64_t dyn : {0ull, 8ull, 50ull})
          if (check(lens, Wq, dyn, 1 + next(4))) return 1;
    }
  // units: all of the claimed segments, never growing, single ones at the end
  for (uint64_t n : {1ull, 5ull, 152ull, 3041ull, 20000ull, 155000ull, 2000000ull})
    for (uint64_t Wq : {1ull, 40ull, 1520ull, 3040ull}) {
      uint64_t left = n, before = FR_UNIT_MAX;
      while (left > 0) {
        const uint64_t u = unit_segs(left, Wq);
        EXPECT(u >= 1 && u <= left && u <= before && (left > Wq || u == 1));
        before = u;
        left -= u;
      }
    }
  if (check({}, 5, 0, 1) || check({100, 511, 0}, 5, 8, 2)) return 1;
  std::printf("seg_walk ok\n");
  return 0;
}
