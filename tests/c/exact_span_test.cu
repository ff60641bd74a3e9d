// exact_span_test.cu -- the two ways to redo a lane's share of a sum segment
// exactly (csrc/sweep_impl.cuh), lane by lane (slow_span) and by the whole warp
// (slow_span_by_warp), return the same bits for every length of a segment, and
// both agree with sums in 64 bits.  Built with FR_SEG_BLOCKS as given, 32 blocks
// a segment or more.  Exits 0 and prints "exact_span ok".
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "sweep_impl.cuh"

using namespace frk;

#define EXPECT(c)                                                    \
  do {                                                               \
    if (!(c)) {                                                      \
      std::fprintf(stderr, "%s:%d check failed: %s\n", __FILE__, __LINE__, #c); \
      return 1;                                                      \
    }                                                                \
  } while (0)
#define CUDA(c) EXPECT((c) == cudaSuccess)

// One warp: lane l's share of the n blocks at p, both ways.
template <int DT, bool SHIFT>
__global__ void both(const uint8_t* p, uint32_t n, Exact* by_lane, Exact* by_warp) {
  const uint32_t lane = threadIdx.x;
  const uint8_t* sp = p + lane * 16;
  by_lane[lane] = slow_span<DT, SHIFT>(sp, n);
  __syncwarp();
  for (uint32_t l = 0; l < 32; ++l) {
    const Exact x = slow_span_by_warp<DT, SHIFT>(sp, n, l, lane);
    if (lane == l) by_warp[lane] = x;
  }
}

static uint32_t g_seed = 1;
static uint32_t next() { return (g_seed = g_seed * 1664525u + 1013904223u) >> 8; }

// A value of kind 0 (ordinary), 1 (mostly tiny or huge squares, zeros and non-finite values among them) or 2 (tiny only).
static float value(int kind) {
  const float x = static_cast<float>(static_cast<int>(next() % 20001) - 10000) * 1e-3f;
  if (kind == 0) return next() % 97 == 0 ? NAN : x;
  if (kind == 2) return x * 1e-25f;
  switch (next() % 8) {
    case 0: return x * 1e-25f;
    case 1: return x * 1e-40f;  // subnormal
    case 2: return x * 1e17f;
    case 3: return x * 1e25f;
    case 4: return 0.0f;
    case 5: return next() % 3 ? -INFINITY : NAN;
    default: return x;
  }
}

template <int DT, bool SHIFT>
static int check(int kind, uint32_t n) {
  constexpr int kBytes = DT == kDtF32 ? 4 : 2;
  const size_t shift = SHIFT ? 4 : 0, bytes = n * size_t(kBlockBytes), per_lane = 16 / kBytes;
  std::vector<uint8_t> host(bytes);
  std::vector<double> sum(32, 0.0);
  std::vector<uint32_t> count(32, 0);
  for (size_t e = 0; e < bytes / kBytes; ++e) {
    float f = value(kind);
    uint32_t w;
    std::memcpy(&w, &f, 4);
    if (DT != kDtF32) w &= 0xFFFF0000u;
    std::memcpy(&f, &w, 4);
    const uint32_t bits = DT == kDtF32 ? w : w >> 16;
    std::memcpy(&host[e * kBytes], &bits, kBytes);
    const size_t lane = e / per_lane % 32;
    if (std::isfinite(f)) sum[lane] += static_cast<double>(f) * f;
    else ++count[lane];
  }
  uint8_t* dev = nullptr;
  Exact* out = nullptr;
  CUDA(cudaMalloc(&dev, bytes + 16));
  CUDA(cudaMalloc(&out, 64 * sizeof(Exact)));
  CUDA(cudaMemset(dev, 0, bytes + 16));
  CUDA(cudaMemcpy(dev + shift, host.data(), bytes, cudaMemcpyHostToDevice));
  both<DT, SHIFT><<<1, 32>>>(dev + shift, n, out, out + 32);
  CUDA(cudaGetLastError());
  Exact got[64];
  CUDA(cudaMemcpy(got, out, sizeof got, cudaMemcpyDeviceToHost));
  CUDA(cudaFree(dev));
  CUDA(cudaFree(out));
  // a lane's m elements are added within m^2 u^2 of their sum, u = 2^-24
  const double m = double(n) * per_lane, bound = m * m * 0x1p-48;
  for (int l = 0; l < 32; ++l) {
    EXPECT(std::memcmp(&got[l].d, &got[32 + l].d, 8) == 0);
    EXPECT(got[l].nonfinite == got[32 + l].nonfinite && got[l].nonfinite == count[l]);
    EXPECT(std::fabs(got[l].d - sum[l]) <= bound * sum[l]);
  }
  return 0;
}

int main() {
  for (int kind = 0; kind < 3; ++kind)
    for (uint32_t n : {1u, 2u, 31u, 32u, 33u, 63u, 64u})
      if (n <= kSpan) {
        if (check<kDtF32, false>(kind, n) || check<kDtF32, true>(kind, n) || check<kDtBf16, false>(kind, n) ||
            check<kDtBf16, true>(kind, n)) {
          std::fprintf(stderr, "kind %d, %u blocks of %u\n", kind, n, kSpan);
          return 1;
        }
      }
  std::printf("exact_span ok\n");
  return 0;
}
