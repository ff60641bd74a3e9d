// plan_units.cc -- prints the claimable units of a plan's pack and unpack
// launches.  Input: "SMs chunk_bytes batches tensors", then per tensor "address
// bytes dtype".  Output: a line "batch class units" for every sweep class with a
// chunk body in the batch; batch -1 is the whole-state launch.
#include <cinttypes>
#include <cstdio>

#include "fake_cuda.h"

#include "api.cu"

static void print(fr_plan p, const Decomp& D, size_t b, int label) {
  const BatchInfo& bi = D.batches[b];
  uint32_t units[kClassCount] = {};
  bool any[kClassCount] = {};
  for (uint64_t c = bi.c_begin; c < bi.c_end; ++c)
    if (p->chunks[c].len >= kBlockBytes) any[p->chunks[c].sweep_class] = true;
  for (uint32_t u = 0; u < bi.n_units; ++u) ++units[D.d_units[bi.unit_off + u].cls];
  for (uint32_t q = 0; q < kClassCount; ++q)
    if (any[q]) std::printf("%d %u %u\n", label, q, units[q]);
}

int main() {
  uint64_t chunk = 0, n = 0;
  uint32_t batches = 0;
  if (std::scanf("%d %" SCNu64 " %u %" SCNu64, &fake::sm_count, &chunk, &batches, &n) != 4) return 1;
  std::vector<fr_tensor> t(n);
  for (fr_tensor& x : t) {
    uint64_t addr = 0, bytes = 0;
    uint32_t dtype = 0;
    if (std::scanf("%" SCNu64 " %" SCNu64 " %u", &addr, &bytes, &dtype) != 3) return 1;
    x = fr_tensor{reinterpret_cast<void*>(addr), bytes, dtype, 0};
  }
  fr_plan p = nullptr;
  if (fr_plan_create_batched(t.data(), n, chunk, batches, &p) != FR_OK) return 1;
  print(p, whole_for(p, kModePack), 0, -1);
  if (p->n_batches > 1)
    for (uint32_t b = 0; b < p->n_batches; ++b) print(p, batch_for(p, kModePack), b, static_cast<int>(b));
  return 0;
}
