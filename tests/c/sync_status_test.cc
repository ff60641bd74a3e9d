// sync_status_test.cc -- fr_sync_status returns a recorded condition once, and
// has cleared it in device memory when it returns: a call on a non-blocking
// stream, which may record the next condition at once, is not ordered after the
// legacy stream.  Exits 0 and prints "sync_status ok".
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

int main() {
  const fr_tensor t = {reinterpret_cast<void*>(1ull << 40), 1 << 20, FR_DT_F32, 0};
  fr_plan p = nullptr;
  EXPECT(fr_plan_create(&t, 1, 1 << 16, &p) == FR_OK);
  for (void* stream : {static_cast<void*>(nullptr), reinterpret_cast<void*>(0x1234)}) {
    EXPECT(fr_sync_status(p, stream) == FR_OK);
    *p->d_status = kStatusCapacity;
    EXPECT(fr_sync_status(p, stream) == FR_ERR_CAPACITY);
    EXPECT(*p->d_status == 0);
    *p->d_status = kStatusCapacity;  // the next call's
    fake::finish_all();
    EXPECT(fr_sync_status(p, stream) == FR_ERR_CAPACITY);
    EXPECT(fr_sync_status(p, stream) == FR_OK);
  }
  fr_plan_destroy(p);
  std::printf("sync_status ok\n");
  return 0;
}
