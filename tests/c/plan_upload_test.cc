// plan_upload_test.cc -- when fr_plan_create returns, the plan's tables are in
// device memory: no part of their copy may still be on its way, since a call on
// a non-blocking stream is not ordered after the legacy stream that copies them.
// Exits 0 and prints "plan_upload ok".
#include <cstdio>

#include "fake_cuda.h"

#include "api.cu"

#define EXPECT(c)                                                    \
  do {                                                               \
    if (!(c)) {                                                      \
      std::fprintf(stderr, "%s:%d check failed: %s\n", __FILE__, __LINE__, #c); \
      return 1;                                                      \
    }                                                                \
  } while (0)

// Every piece of decomposition D lies in the one tensor [addr, addr + bytes), the claim counters are zero.
static int check_decomp(const Decomp& D, uint64_t addr, uint64_t bytes) {
  EXPECT(D.n_recs > 0);
  uint64_t blocks = 0;
  for (uint64_t i = 0; i < D.n_recs; ++i) {
    const PieceDesc& d = D.d_pieces[i];
    EXPECT(d.addr >= addr && d.addr + uint64_t(d.nblk) * kBlockBytes <= addr + bytes);
    blocks += d.nblk;
  }
  EXPECT(blocks == bytes / kBlockBytes);
  if (D.d_queue != nullptr)
    for (size_t b = 0; b < D.batches.size(); ++b) EXPECT(D.d_queue[kQueueWords * b] == 0);
  return 0;
}

int main() {
  const uint64_t addr = 1ull << 40, bytes = 300ull << 20;
  const fr_tensor t = {reinterpret_cast<void*>(addr), bytes, FR_DT_F32, 0};
  for (uint32_t batches : {1u, 5u}) {
    fr_plan p = nullptr;
    EXPECT(fr_plan_create_batched(&t, 1, 1 << 20, batches, &p) == FR_OK);
    EXPECT(fake::pending.empty());
    bool units = false;
    for (const Decomp& D : p->whole) {
      if (check_decomp(D, addr, bytes)) return 1;
      units |= D.d_queue != nullptr;
    }
    EXPECT(units);
    if (batches > 1)
      if (check_decomp(p->batched[p->geo[kModePack]], addr, bytes)) return 1;
    EXPECT(*p->d_status == 0);
    EXPECT(p->d_crc_xor[0] == host_crc_xor_term(1 << 20));
    fr_plan_destroy(p);
  }
  std::printf("plan_upload ok\n");
  return 0;
}
