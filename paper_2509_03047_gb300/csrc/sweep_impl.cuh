// sweep_impl.cuh -- the bandwidth-bound body sweep of fingerprint / pack / unpack.
//
// Restoration of a rank's state from a data-parallel replica (FlashRecovery,
// arXiv 2509.03047, Sec. III-E) is, on one GPU, a sweep over every byte of
// the param / master / Adam-m / Adam-v tensors: checksum it, and for the
// transfer copy it into (pack) or out of (unpack) a flat buffer.  This kernel
// does the whole-512-byte-block part of every chunk in one HBM pass:
//
//  * copy engine: each lane moves 16 bytes per block with a coalesced 128-bit
//    load and (pack/unpack) a coalesced 128-bit store, whatever the tensor's
//    alignment (take16);
//  * CRC-32C: the 128 words of a block are 128 interleaved CRC streams
//    (lane l owns streams 4l..4l+3, four independent dependency chains), each
//    advanced by s <- (s ^ w) * x^4096 with four byte lookups in tables kept in
//    shared memory.  Every lane has a private copy of each table entry in its
//    own bank, so the 32 lookups of a warp never conflict.  At the end of a
//    piece each lane's streams are multiplied to their place and XORed into the
//    raw CRC of the piece;
//  * non-finite count and sum of squares, fused on the same registers: each
//    square is added to a packed f32x2 running sum by one FMA, and the
//    addition's error -- including the square's own rounding for fp32 -- is
//    recovered to second order by a TwoSum whose low term is a second FMA
//    (two_sum_sq), then flushed into fp64.  A 16 KiB segment whose running
//    sum is not finite (NaN/Inf input, or overflow) or is tiny with non-zero
//    input is redone element by element, exactly, from a reload of its
//    16-byte units (slow_span), so the fast path never needs a per-element
//    test.
//
// No tensor cores: nothing here is a contraction.  One CTA per SM, with a warp
// count per mode (the 128 KiB of lane-replicated tables fill most of shared
// memory).  The plan sorts chunks into classes by element type and by whether
// they start on a 16-byte boundary; each class has its own block stream, cut
// into per-warp runs of pieces, and its own code specialization, so each warp
// runs a single loop variant.  A call launches once for all its classes
// (sweep_kernel); its warps then claim the last few percent of the work as
// small units.  sweep_{fp,pack,unpack,unpack_fp}.cu each instantiate one mode.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "gf2.cuh"
#include "kernels.h"
#include "layout.h"

namespace frk {

namespace {

// Warps and threads of one mode's CTA.
template <int MODE>
struct Cta {
  static constexpr int kWarps = sweep_warps(MODE);
  static constexpr int kThreads = kWarps * 32;
};
constexpr int kTableBytes = 4 * 256 * 32 * 4;  // 4 tables x 256 entries x 32 lanes x 4 B
// Pipeline geometry (compile-time), tuned on GB300 by timing the 31.8 GB
// Llama-70B shard.  The read-only fingerprint gains from bulk L2 prefetch
// exactly one span ahead (none: -9 points; two spans: -25) and from 8-block
// register stages; pack and unpack lose by the prefetch (their write stream
// evicts the prefetched lines before use, and DRAM reads grow by ~20%), so
// they rely on 4-block register stages and more warps (kernels.h).
#ifndef FR_STAGE_FP
#define FR_STAGE_FP 8
#endif
// The fingerprint of shifted chunks takes the shorter stage: its loop holds
// the realignment too, and with 8-block stages the loops of two element types
// outgrow the instruction cache (2.5 GB of views: 567 us, 560 with 4).
#ifndef FR_STAGE_FP_SHIFT
#define FR_STAGE_FP_SHIFT 4
#endif
// Up to this many lanes of a segment that need the exact fallback take it in
// turn by the whole warp (slow_span_by_warp), more take it side by side
// (slow_span).  In turn, each lane costs 3.5 us more; side by side they cost the
// same together however many.  Measured, fingerprint of 15 MB of fp32 as a
// graph, us, in turn / side by side, NaN lanes in one segment: 1 lane 17 / 25, 2
// lanes 20 / 25, 3 lanes 24 / 25, 4 lanes 27 / 25; in every segment: 22 / 27, 30 /
// 27, 37 / 27, 44 / 27.  Among lanes whose squares are tiny (span_end_slow) only
// one is taken so: their squares are added one by one in fp64 (256 MB of
// exp(N(ln 1e-12, 3^2)): fingerprint, up to 1 / 2 lanes in turn, 409 / 426).
#ifndef FR_SLOW_WARP_LANES
#define FR_SLOW_WARP_LANES 2
#endif
#ifndef FR_STAGE_PACK
#define FR_STAGE_PACK 4
#endif
#ifndef FR_STAGE_UNPACK
#define FR_STAGE_UNPACK 4
#endif
#ifndef FR_LOADFIRST_FP
#define FR_LOADFIRST_FP 0
#endif
#ifndef FR_LOADFIRST_PACK
#define FR_LOADFIRST_PACK 0
#endif
#ifndef FR_LOADFIRST_UNPACK
#define FR_LOADFIRST_UNPACK 1
#endif
// Blocks per validity span: one sum segment (a power of two, a multiple of
// every stage).
constexpr uint32_t kSpan = static_cast<uint32_t>(kSegBlocks);

constexpr int kSlowWarpLanes = FR_SLOW_WARP_LANES;

typedef unsigned long long u64;

__device__ const ByteTables4 g_braid = make_mul_tables(kBraidMul);

extern __shared__ __align__(16) uint8_t g_smem[];

// ------------------------------------------------------------------ tables

// Table k, entry i, lane l lives at byte
//   (k >> 1) * 65536 + i * 256 + (k & 1) * 128 + l * 4,
// i.e. bank l.  The address of (table k, byte k of x, this lane) is one
// byte-permute: byte 0 = l*4, byte 1 = byte k of x.
// Every thread of a kThreads-thread CTA stores its share of 16-byte units;
// the loop is unrolled so a thread's table loads all issue before the first
// store waits on one (a rolled loop made the fill a chain of ~16 L2 round
// trips, about 3 us per launch).
template <int kThreads>
__device__ __forceinline__ void fill_tables() {
  constexpr int kUnits = kTableBytes / 16;
  constexpr int kIters = (kUnits + kThreads - 1) / kThreads;
  uint32_t v[kIters];
#pragma unroll
  for (int it = 0; it < kIters; ++it) {
    const int q = static_cast<int>(threadIdx.x) + it * kThreads;
    const int k = q >> 11, i = (q & 2047) >> 3;
    v[it] = q < kUnits ? g_braid.t[k][i] : 0u;
  }
#pragma unroll
  for (int it = 0; it < kIters; ++it) {
    const int q = static_cast<int>(threadIdx.x) + it * kThreads;
    if (q < kUnits) {
      const int k = q >> 11, rem = q & 2047, i = rem >> 3, g = rem & 7;
      const uint32_t off = (k >> 1) * 65536 + i * 256 + (k & 1) * 128 + g * 16;
      *reinterpret_cast<uint4*>(g_smem + off) = make_uint4(v[it], v[it], v[it], v[it]);
    }
  }
}

__device__ __forceinline__ uint32_t tab(uint32_t off) {
  return *reinterpret_cast<const uint32_t*>(g_smem + off);
}

// (s ^ w) * x^4096 for this lane's stream, given x = s ^ w.
__device__ __forceinline__ uint32_t braid_step(uint32_t x, uint32_t lb) {
  const uint32_t t0 = tab(__byte_perm(x, lb, 0x5504));
  const uint32_t t1 = tab(__byte_perm(x, lb, 0x5514) + 128);
  const uint32_t t2 = tab(__byte_perm(x, lb, 0x5524) + 65536);
  const uint32_t t3 = tab(__byte_perm(x, lb, 0x5534) + 65536 + 128);
  return (t0 ^ t1) ^ (t2 ^ t3);
}

// The piece-end fold.  A lane joins its four streams by Horner with x^32, then
// multiplies by x^(128 (31 - l)), its place among the lanes, and by the
// unbraid factor at once, and the lanes are XORed.  x^32 comes from byte
// tables (read-only, in L1).  The product (n << 4k) * M_l, for nibble position
// k, nibble value n and lane l's multiplier M_l, sits at word
// (16k + n) * 32 + l of a 16 KiB table behind the braid tables in shared
// memory: the 32 lanes' lookups of a nibble position fall in 32 banks.  A warp
// pays the fold once per piece; as a tree of five shuffles and multiplications
// by byte tables, 24 lookups of up to 8 lines each, it was as much load/store
// work as 10 blocks (40,000 chunks of 1.5 KB on average: step 253 -> 243 us).
__device__ const ByteTables4 g_x32 = make_mul_tables(gf_xpow(32));

constexpr int kLaneFoldWords = 8 * 16 * 32;
struct alignas(16) LaneFoldTable {
  uint32_t t[kLaneFoldWords];
};
__host__ __device__ constexpr LaneFoldTable make_lane_fold_table() {
  LaneFoldTable out{};
  for (int l = 0; l < 32; ++l) {
    const uint32_t m = gf_mulmod(gf_xpow(128ull * static_cast<uint64_t>(31 - l)), kUnbraid);
    for (int k = 0; k < 8; ++k) {
      uint32_t bit[4] = {};
      for (int j = 0; j < 4; ++j) bit[j] = gf_mulmod(1u << (4 * k + j), m);
      for (int n = 0; n < 16; ++n) {
        uint32_t v = 0;
        for (int j = 0; j < 4; ++j)
          if (n & (1 << j)) v ^= bit[j];
        out.t[(16 * k + n) * 32 + l] = v;
      }
    }
  }
  return out;
}
__device__ const LaneFoldTable g_lane_fold = make_lane_fold_table();
constexpr int kSweepSmem = kTableBytes + kLaneFoldWords * 4;

// Starts this thread's share of the lane table on its way to shared memory;
// finish_lane_fold waits for it.
template <int kThreads>
__device__ __forceinline__ void start_lane_fold() {
  const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(g_smem + kTableBytes));
  for (int q = static_cast<int>(threadIdx.x); q < kLaneFoldWords / 4; q += kThreads)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(base + 16u * q), "l"(g_lane_fold.t + 4 * q) : "memory");
}
__device__ __forceinline__ void finish_lane_fold() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// a * x^32 mod P.
__device__ __forceinline__ uint32_t mul_x32(uint32_t a) {
  return (__ldg(&g_x32.t[0][a & 255u]) ^ __ldg(&g_x32.t[1][(a >> 8) & 255u])) ^
         (__ldg(&g_x32.t[2][(a >> 16) & 255u]) ^ __ldg(&g_x32.t[3][a >> 24]));
}
// a * M_l mod P for the calling lane l (lb = 4l).
__device__ __forceinline__ uint32_t mul_lane(uint32_t a, uint32_t lb) {
  const uint8_t* T = g_smem + kTableBytes + lb;
  uint32_t r[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) r[k] = *reinterpret_cast<const uint32_t*>(T + (16 * k + ((a >> (4 * k)) & 15u)) * 128);
  return (r[0] ^ r[1] ^ r[2]) ^ (r[3] ^ r[4] ^ r[5]) ^ (r[6] ^ r[7]);
}

// ------------------------------------------------------------------ memory

// 16 bytes at p, a multiple of 16.  (Non-coherent: see wait_for_kernel_before.)
__device__ __forceinline__ uint4 ld_unit(const uint8_t* p) {
  uint4 v;
  asm("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0,%1,%2,%3}, [%4];"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p));
  return v;
}

// The same, kept in L1 for the neighbour lane.
__device__ __forceinline__ uint4 ld_unit_l1(const uint8_t* p) {
  uint4 v;
  asm("ld.global.nc.L2::256B.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

__device__ __forceinline__ void st_unit(uint8_t* p, const uint4& v) {
  asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z),
               "r"(v.w)
               : "memory");
}

// Chunks that do not start on a 16-byte boundary move in 16-byte granules all
// the same.  Reading, a lane's unit lies across two granules of the tensor:
// lane l loads the one it ends in, as part of the block's pipeline, and the one
// it starts in -- lane l - 1's, or lane 31's of the block before -- again from
// L1 when it needs it; take16 cuts the unit out.  Writing, lane l stores the
// granule its unit starts in, whose first bytes are the end of the unit before
// it, taken from the packed buffer in the same way.  So every lane holds the
// same 16 bytes of the chunk as for an aligned chunk, and neither the CRC
// streams nor the order of the sums change with the alignment.  A granule of
// the tensor is only read if it holds a byte of the piece, so no read reaches
// a page that the tensor does not; its other bytes are dropped, and never
// written.
//
// Before, such chunks moved by 4-byte or single-byte accesses 16 bytes apart
// from lane to lane: 4 or 16 times the load and store instructions, each
// touching every line of the block.  With the neighbour's granule passed by
// shuffle instead of L1 (four shuffles, a carry and a select each) the loops
// were 12 instructions a block longer.  GB300, 2.5 GB of views at any element
// offset, us, by narrow accesses / shuffles / L1: fingerprint 1095 / 597 / 529,
// pack 1025 / 931 / 783, pack and unpack with both tables 2063 / 1917 / 1610.

// 16 bytes from byte t on (0 <= t < 16, the same in every lane) of a then b.
__device__ __forceinline__ uint4 take16(const uint4& a, const uint4& b, uint32_t t) {
  uint32_t w0 = a.x, w1 = a.y, w2 = a.z, w3 = a.w, w4 = b.x, w5 = b.y;
  if (t & 8u) {
    w0 = a.z;
    w1 = a.w;
    w2 = b.x;
    w3 = b.y;
    w4 = b.z;
    w5 = b.w;
  }
  if (t & 4u) {
    w0 = w1;
    w1 = w2;
    w2 = w3;
    w3 = w4;
    w4 = w5;
  }
  const uint32_t sh = 8u * (t & 3u);
  return make_uint4(__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh), __funnelshift_r(w2, w3, sh),
                    __funnelshift_r(w3, w4, sh));
}

// The unit at p by itself; SHIFT: p need not be a multiple of 16.
template <bool SHIFT>
__device__ __forceinline__ uint4 ld_unit_at(const uint8_t* p) {
  if (!SHIFT) return ld_unit(p);
  const uint32_t t = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(p)) & 15u;
  const uint4 a = ld_unit(p - t);
  return t ? take16(a, ld_unit(p - t + 16), t) : a;
}

// The bytes k of v with k < t (HEAD) or k >= t, as single stores from p on:
// the first and the last granule of a piece whose destination is shifted
// belong to it in part only.
template <bool HEAD>
__device__ __forceinline__ void st_part(uint8_t* p, const uint4& v, uint32_t t) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (uint32_t k = 0; k < 16; ++k)
    if (HEAD ? k < t : k >= t) p[HEAD ? k : k - t] = static_cast<uint8_t>(w[k >> 2] >> (8 * (k & 3)));
}

// ------------------------------------------------------------------ f32x2

__device__ __forceinline__ u64 pk(uint32_t lo, uint32_t hi) {
  u64 r;
  asm("mov.b64 %0, {%1,%2};" : "=l"(r) : "r"(lo), "r"(hi));
  return r;
}
__device__ __forceinline__ float lo_f(u64 v) { return __uint_as_float(static_cast<uint32_t>(v)); }
__device__ __forceinline__ float hi_f(u64 v) { return __uint_as_float(static_cast<uint32_t>(v >> 32)); }
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 sub2(u64 a, u64 b) {
  u64 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// S + C += x*x, for each half of a packed pair (S, x >= 0 in effect: squares
// and sums of squares).  t = fl(S + x*x) by one FMA; then zn = fl(S - t),
// y = t + zn, a = S - y, b = fl(x*x + zn) by a second FMA, and C takes a + b.
//  * t <= 2S: S - t is exact (Sterbenz), so zn = S - t, y = S, a = 0 and b is
//    the addition's exact error S + x*x - t rounded once.
//  * t > 2S: zn lies in [-t, -t/2], so y = t + zn is exact and equals S + d,
//    d the rounding error of S - t; a = -d exactly, and b = (error + d)
//    rounded once, with |error + d| <= ulp(t).
// Either way a + b is the error of t to within about 3u^2 t (u = 2^-24): the
// square need not be exact in fp32, so fp32 inputs need no separate residual
// term, and for bf16 inputs (exact squares) this is Knuth's TwoSum exactly.
__device__ __forceinline__ void two_sum_sq(u64& S, u64& C, u64 x) {
  const u64 t = fma2(x, x, S);
  const u64 zn = sub2(S, t);
  const u64 y = add2(t, zn);
  const u64 a = sub2(S, y);
  const u64 b = fma2(x, x, zn);
  C = add2(C, add2(a, b));
  S = t;
}

// S + C += p, error-free (Knuth's TwoSum): S takes the rounded sum, C the
// rounding error.
__device__ __forceinline__ void two_sum_acc(u64& S, u64& C, u64 p) {
  const u64 t = add2(S, p);
  const u64 z = sub2(t, S);
  const u64 y = sub2(t, z);
  const u64 a = sub2(S, y);
  const u64 b = sub2(p, z);
  C = add2(C, add2(a, b));
  S = t;
}

struct FpAcc {
  u64 A, CA, B, CB;  // two f32x2 accumulators with their error terms
};

template <int DT>
__device__ __forceinline__ void fp_unit(const uint4& v, FpAcc& f) {
  if (DT == kDtF32) {
    two_sum_sq(f.A, f.CA, pk(v.x, v.y));
    two_sum_sq(f.B, f.CB, pk(v.z, v.w));
  } else {
    // bf16 pairs: the low element is the low half-word
    const u64 y0 = pk(v.x << 16, v.x & 0xFFFF0000u), y1 = pk(v.y << 16, v.y & 0xFFFF0000u);
    const u64 y2 = pk(v.z << 16, v.z & 0xFFFF0000u), y3 = pk(v.w << 16, v.w & 0xFFFF0000u);
    two_sum_sq(f.A, f.CA, y0);
    two_sum_sq(f.B, f.CB, y2);
    two_sum_sq(f.A, f.CA, y1);
    two_sum_sq(f.B, f.CB, y3);
  }
}

struct Exact {
  double d;
  uint32_t nonfinite;
};


// (hi, lo) += x * x exactly, for pair_square(|x|) or x = 0: the fp32 product and
// its FMA residual, by TwoSum.
__device__ __forceinline__ void add_pair_square(float& hi, float& lo, float x) {
  const float p = x * x;
  const float e = __fmaf_rn(x, x, -p);
  const float t = hi + p;
  const float z = t - hi;
  lo += ((hi - (t - z)) + (p - z)) + e;
  hi = t;
}

// Exact sum of squares of elements added one by one, in order, given as fp32
// bit patterns (a bf16 element in the high half).  A non-finite element is
// counted; a square that pair_square takes is added to the float pair (hi, lo);
// any other sets `odd`, and the caller adds it (odd_elem).  No branch and no fp64
// instruction: predicated off, those still take turns on the narrow pipe, and
// with them in the loop a NaN cost the launch 13 us, without 2.
struct ExactSum {
  float hi = 0.0f, lo = 0.0f;
  uint32_t nonfinite = 0;
  bool odd = false;
  __device__ __forceinline__ void add(uint32_t f) {
    const bool inf_nan = (f & 0x7F800000u) == 0x7F800000u;
    const float ax = fabsf(__uint_as_float(f));
    const bool fast = ax == 0.0f || pair_square(ax);  // false for NaN and Inf
    nonfinite += inf_nan ? 1u : 0u;
    odd |= !fast && !inf_nan;
    add_pair_square(hi, lo, fast ? __uint_as_float(f) : 0.0f);  // (a zero square changes nothing)
  }
  template <int DT>
  __device__ __forceinline__ void add_word(uint32_t w) {
    add(DT == kDtF32 ? w : w << 16);
    if (DT != kDtF32) add(w & 0xFFFF0000u);
  }
};

// Whether an element, given as fp32 bits, has a square that ExactSum leaves out
// (tiny or huge, rare), and the sum of those of a word, in fp64, where the
// square of an fp32 value is exact.
__device__ __forceinline__ bool odd_elem(uint32_t f) {
  const float ax = fabsf(__uint_as_float(f));
  return (f & 0x7F800000u) != 0x7F800000u && ax != 0.0f && !pair_square(ax);
}
template <int DT>
__device__ __forceinline__ bool odd_word(uint32_t w) {
  return DT == kDtF32 ? odd_elem(w) : odd_elem(w << 16) || odd_elem(w & 0xFFFF0000u);
}
template <int DT>
__device__ __forceinline__ void add_odd(double& d, uint32_t w) {
#pragma unroll
  for (int h = 0; h < (DT == kDtF32 ? 1 : 2); ++h) {
    const uint32_t f = DT == kDtF32 ? w : h == 0 ? w << 16 : w & 0xFFFF0000u;
    if (!odd_elem(f)) continue;
    const double xd = static_cast<double>(__uint_as_float(f));
    d = __dadd_rn(d, __dmul_rn(xd, xd));
  }
}

// Exact per-element fallback for this lane's units of `n` blocks, the first at sp:
// non-finite elements are counted; each finite square is added exactly --
// for |x| in [2^-40, 2^56] as its fp32 product and FMA residual into an
// unevaluated float pair by TwoSum, else (tiny or huge values, rare) in fp64,
// where the square of an fp32 value is exact.  Its error, under n^2 u^2 of
// the sum for the n elements of a lane, is far inside the sums' bound.  The
// segment was just swept (its lines are mostly in L2); the lane first
// prefetches all its units into L1, so the reloads do not wait for L2 one by
// one, and the float pair keeps the arithmetic off GB300's narrow fp64 pipe.
// (Loading the units in register batches instead makes the compiler spill in
// the hot loop that calls this.)
template <int DT, bool SHIFT>
__device__ __noinline__ Exact slow_span(const uint8_t* sp, uint32_t n) {
  for (uint32_t b = 0; b < n; ++b) asm volatile("prefetch.global.L1 [%0];" ::"l"(sp + b * kBlockBytes));
  float hi = 0.0f, lo = 0.0f;
  double d = 0.0;
  uint32_t nonfinite = 0;
  for (uint32_t b = 0; b < n; ++b) {
    const uint4 v = ld_unit_at<SHIFT>(sp + b * kBlockBytes);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int h = 0; h < (DT == kDtF32 ? 1 : 2); ++h) {
        const uint32_t f = DT == kDtF32 ? w[j] : (h == 0 ? w[j] << 16 : w[j] & 0xFFFF0000u);
        if ((f & 0x7F800000u) == 0x7F800000u) {
          ++nonfinite;
          continue;
        }
        const float x = __uint_as_float(f);
        const float ax = fabsf(x);
        if (pair_square(ax)) {
          add_pair_square(hi, lo, x);
        } else if (ax != 0.0f) {
          const double xd = static_cast<double>(x);
          d = __dadd_rn(d, __dmul_rn(xd, xd));
        }
      }
    }
  }
  return Exact{(static_cast<double>(hi) + static_cast<double>(lo)) + d, nonfinite};
}

// The same for lane l's units, in every lane: lane k loads the unit of block
// k (of 32 at a time), and all lanes add the words in the order slow_span does,
// taking them from lane k by shuffle.  One lane that needs the fallback (one
// NaN) is the common case, and its warp may be all that a launch still waits
// for: this way it waits for one load, not for 32 in turn.  GB300, a 15 MB state with 3 NaNs
// (L2-resident, as a graph), us: fingerprint 24.5 -> 17.3, pack 24.7 -> 16.9;
// without NaN 15.2.
template <int DT, bool SHIFT>
__device__ __noinline__ Exact slow_span_by_warp(const uint8_t* sp, uint32_t n, uint32_t l, uint32_t lane) {
  const uint8_t* first = sp + (static_cast<int32_t>(l) - static_cast<int32_t>(lane)) * 16;  // lane l's first unit
  ExactSum x;
  double d = 0.0;  // the squares that x leaves out, in the same order
#pragma unroll 1
  for (uint32_t g = 0; g < kSpan; g += 32) {  // (one pass unless a segment is built larger)
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (g + lane < n) v = ld_unit_at<SHIFT>(first + (g + lane) * kBlockBytes);
#pragma unroll 1
    for (uint32_t k = g; k < n && (kSpan <= 32 || k < g + 32); ++k) {
      x.add_word<DT>(__shfl_sync(0xFFFFFFFFu, v.x, k - g));
      x.add_word<DT>(__shfl_sync(0xFFFFFFFFu, v.y, k - g));
      x.add_word<DT>(__shfl_sync(0xFFFFFFFFu, v.z, k - g));
      x.add_word<DT>(__shfl_sync(0xFFFFFFFFu, v.w, k - g));
    }
    if (x.odd) {
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
      uint32_t odd = 0;  // the words of this lane's unit that hold one
#pragma unroll
      for (int j = 0; j < 4; ++j) odd |= (odd_word<DT>(w[j]) ? 1u : 0u) << j;
#pragma unroll 1
      for (uint32_t m = __ballot_sync(0xFFFFFFFFu, odd != 0); m != 0; m &= m - 1) {
        const int k = __ffs(static_cast<int>(m)) - 1;
        const uint32_t o = __shfl_sync(0xFFFFFFFFu, odd, k);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t wj = __shfl_sync(0xFFFFFFFFu, w[j], k);
          if (o >> j & 1u) add_odd<DT>(d, wj);
        }
      }
    }
  }
  return Exact{(static_cast<double>(x.hi) + static_cast<double>(x.lo)) + d, x.nonfinite};
}

// Whether this lane's units of `n` blocks hold only (signed) zeros.
template <int DT, bool SHIFT>
__device__ __noinline__ bool span_is_zero(const uint8_t* sp, uint32_t n) {
  constexpr uint32_t kMask = (DT == kDtF32) ? 0x7FFFFFFFu : 0x7FFF7FFFu;
  uint32_t acc = 0;
  for (uint32_t b = 0; b < n; ++b) {
    const uint4 v = ld_unit_at<SHIFT>(sp + b * kBlockBytes);
    acc |= (v.x | v.y | v.z | v.w) & kMask;
  }
  return acc == 0;
}

// The span's sum as an unevaluated float pair (hi, lo): the four fp32 partial
// sums are merged error-free in fp32 (TwoSum); the error terms (about 2^-24
// of the sum) are merged with plain fp32 adds, which costs about 2^-48
// relative.  No fp64 work: GB300's fp64 pipe is narrow.
__device__ __forceinline__ void fold_to_pair(const FpAcc& f, float& hi, float& lo) {
  u64 s = f.A, c = add2(f.CA, f.CB);
  two_sum_acc(s, c, f.B);
  const float a = lo_f(s), b = hi_f(s);
  const float t = a + b;
  const float z = t - a;
  const float err = (a - (t - z)) + (b - z);
  hi = t;
  lo = (lo_f(c) + hi_f(c)) + err;
}

// ------------------------------------------------------------------ piece

// Bulk prefetch of [p, p + bytes) into L2 (TMA unit; no registers held).
__device__ __forceinline__ void prefetch_l2(const uint8_t* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// The same, issued by lane 0 only, as a predicated instruction (no branch).
__device__ __forceinline__ void prefetch_l2_lane0(const uint8_t* p, uint32_t bytes, uint32_t lane) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.eq.u32 q, %2, 0;\n\t@q cp.async.bulk.prefetch.L2.global [%0], %1;\n\t}" ::"l"(p),
      "r"(bytes), "r"(lane)
      : "memory");
}

// Per-mode pipeline geometry: blocks per lane held in registers one stage
// ahead, and whether the next span (kSpan blocks) is prefetched into L2.
// Unpack with fingerprint values does pack's work per byte (copy, CRC, sums),
// so it takes pack's geometry.
template <int MODE, bool SHIFT>
struct Geo {
  static constexpr bool kPackLike = MODE == kModePack || MODE == kModeUnpackFp;
  static constexpr int kStage = MODE == kModeFingerprint ? (SHIFT ? FR_STAGE_FP_SHIFT : FR_STAGE_FP)
                                                         : (kPackLike ? FR_STAGE_PACK : FR_STAGE_UNPACK);
  static constexpr bool kPrefetch = MODE == kModeFingerprint;
  // Issue a unit's reload before consuming it (more load lead, one register
  // copy) or after (no copy): latency-bound modes want the former.
  static constexpr bool kLoadFirst = MODE == kModeFingerprint ? FR_LOADFIRST_FP
                                     : (kPackLike ? FR_LOADFIRST_PACK : FR_LOADFIRST_UNPACK);
  static_assert(kSpan % kStage == 0, "a span holds whole stages");
};

// State of one lane while it sweeps a piece.
template <int MODE, int DT>
struct Lane {
  uint32_t s[4];  // CRC streams 4l..4l+3
  FpAcc f;        // fp32 sums of the current span
  uint32_t nonfinite;
  // shifted pieces only
  uint32_t t;  // take16's t
  bool first;  // destination, lane 0: no block stored yet
};

// One unit `v`, which goes to wp; `up`: where it was loaded.
template <int MODE, int DT, bool SHIFT>
__device__ __forceinline__ void do_unit(Lane<MODE, DT>& L, const uint4& v, const uint8_t* up, uint8_t* wp, uint32_t lb) {
  constexpr bool kFp = mode_sums(MODE) && (DT != kDtBytes);
  if (MODE != kModeFingerprint) {
    if (SHIFT && mode_unpacks(MODE)) {
      // (16 bytes before a payload are still in the packed buffer)
      const uint4 g = take16(ld_unit_l1(up - 16), v, L.t);
      if (!L.first)
        st_unit(wp, g);
      else
        st_part<true>(wp + 16 - L.t, v, L.t);
      L.first = false;
    } else {
      st_unit(wp, v);
    }
  }
  L.s[0] = braid_step(L.s[0] ^ v.x, lb);
  L.s[1] = braid_step(L.s[1] ^ v.y, lb);
  L.s[2] = braid_step(L.s[2] ^ v.z, lb);
  L.s[3] = braid_step(L.s[3] ^ v.w, lb);
  if (kFp) fp_unit<DT>(v, L.f);
}

// The lanes' float pairs added in a fixed tree by TwoSum; lane 0 stores the
// segment's sum in pair form (seg_value).
__device__ __forceinline__ void store_pair_sum(float hi, float lo, double* seg, uint32_t lane) {
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) {
    const float oh = __shfl_down_sync(0xFFFFFFFFu, hi, m);
    const float ol = __shfl_down_sync(0xFFFFFFFFu, lo, m);
    const float t = hi + oh;
    const float z = t - hi;
    const float err = (hi - (t - z)) + (oh - z);
    lo = (lo + ol) + err;
    hi = t;
  }
  if (lane == 0) *reinterpret_cast<float2*>(seg) = make_float2(lo, hi);
}

// End of a segment some lane of which has a running sum `tot` outside
// [2^-60, 2^120): the lane's fast sums stand if finite and not small (fp32
// underflow is then below 2^-77 relative), or if its elements are all zero;
// else the lane's share is summed exactly from a reload.  Lanes that all took
// the fast path with sums far from fp32 overflow are added in pair form, else
// in fp64.  Returns the lane's non-finite elements.
template <int DT, bool SHIFT>
__device__ __noinline__ uint32_t span_end_slow(FpAcc f, float tot, const uint8_t* sp, uint32_t n, double* seg,
                                               uint32_t lane) {
  bool ok = tot < __int_as_float(0x7F800000);
  if (ok && !(tot >= 0x1p-60f)) ok = span_is_zero<DT, SHIFT>(sp, n);
  float hi = 0.0f, lo = 0.0f;
  double d = 0.0;
  uint32_t nonfinite = 0;
  if (ok) fold_to_pair(f, hi, lo);
  if (__all_sync(0xFFFFFFFFu, ok && tot < 0x1p120f)) {
    store_pair_sum(hi, lo, seg, lane);
    return 0;
  }
  if (ok) d = static_cast<double>(hi) + static_cast<double>(lo);
  uint32_t bad = __ballot_sync(0xFFFFFFFFu, !ok);
  const bool tiny = __any_sync(0xFFFFFFFFu, !ok && tot < 1.0f);  // (else NaN, Inf or overflow)
  if (__popc(bad) > (tiny ? 1 : kSlowWarpLanes)) {
    bad = 0;
    if (!ok) {
      const Exact x = slow_span<DT, SHIFT>(sp, n);
      d = x.d;
      nonfinite = x.nonfinite;
    }
  }
  for (; bad != 0; bad &= bad - 1) {
    const uint32_t l = static_cast<uint32_t>(__ffs(static_cast<int>(bad))) - 1u;
    const Exact x = slow_span_by_warp<DT, SHIFT>(sp, n, l, lane);
    if (lane == l) {
      d = x.d;
      nonfinite = x.nonfinite;
    }
  }
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) d += __shfl_down_sync(0xFFFFFFFFu, d, m);
  if (lane == 0) *seg = -d;
  return nonfinite;
}

// End of a span (one segment) of `n` blocks, the lane's first unit at sp.  The
// common case in line, all else behind one vote and one call: the loops of two
// element types only just fit an SM's instruction cache (fingerprint of 4.2 GB
// in 50,000 tensors 694 -> 679 us, of the Llama-8B shard 2132 -> 2078).
template <int MODE, int DT, bool SHIFT>
__device__ __forceinline__ void span_end(Lane<MODE, DT>& L, const uint8_t* sp, uint32_t n, double* seg,
                                         uint32_t lane) {
  const u64 ab = add2(L.f.A, L.f.B);
  const float tot = lo_f(ab) + hi_f(ab);
  if (__all_sync(0xFFFFFFFFu, tot >= 0x1p-60f && tot < 0x1p120f)) {
    float hi, lo;
    fold_to_pair(L.f, hi, lo);
    store_pair_sum(hi, lo, seg, lane);
  } else {
    L.nonfinite += span_end_slow<DT, SHIFT>(L.f, tot, sp, n, seg, lane);
  }
  L.f.A = L.f.CA = L.f.B = L.f.CB = 0ull;
}

// A run of `n` consecutive pieces of one class, a warp's own or a unit it
// claimed: piece i (from r on) is get(i, whether more
// follow), its record recs[i].  SHIFT: the
// tensor side (source, or destination for unpack) of the class's chunks does
// not start on a 16-byte boundary; the packed side always does.
//
// Pipeline: for the fingerprint, lane 0 prefetches whole spans into L2 one span
// ahead with the bulk-copy unit; each lane keeps kStage 16-byte units of the
// next stage in flight in registers, which therefore mostly wait for L2.  Each
// span is one sum segment: its fp32 sums start at zero, are checked at its end,
// and are replaced by an exact sum from a reload when they fail.  (Loading a
// piece's first stage before the piece before it is folded gained pack 0.3%
// and cost the fingerprint of the Llama-8B shard 3%.)
template <int MODE, int DT, bool SHIFT, class Get>
__device__ __forceinline__ void sweep_run(uint8_t* packed, double* segs, Record* recs, const Get& get, uint32_t r,
                                          uint32_t n, uint32_t lane) {
  constexpr bool kFp = mode_sums(MODE) && (DT != kDtBytes);
  constexpr uint32_t kStage = Geo<MODE, SHIFT>::kStage;
  constexpr bool kPrefetch = Geo<MODE, SHIFT>::kPrefetch;
  constexpr bool kShiftSrc = SHIFT && !mode_unpacks(MODE), kShiftDst = SHIFT && mode_unpacks(MODE);
  constexpr uint32_t kStageBytes = kStage * kBlockBytes;
  constexpr uint32_t kSpanBytes = kSpan * kBlockBytes;
  constexpr bool kSpans = MODE == kModeFingerprint;  // whole spans in a loop of their own
  const uint32_t lb = lane << 2;

  Lane<MODE, DT> L;
  const uint8_t* lp;  // the next stage's loads
  uint8_t* wp;
  uint32_t left;  // blocks not swept yet
  double* seg;
  uint4 cur[kStage];
  auto load = [&](const uint8_t* q) { return SHIFT ? ld_unit_l1(q) : ld_unit(q); };
  // Starts piece r.  (Every unit is given a value: a register that is only set
  // under a condition is live, to the compiler, around every loop that
  // encloses this one, through the code of every class -- 1,000 bytes of
  // spills.)
  auto begin = [&]() {
    const PieceDesc d = get(r, n > 1);
    uint8_t* tensor = reinterpret_cast<uint8_t*>(d.addr);
    uint8_t* pk = packed + d.payload_off;
    lp = mode_unpacks(MODE) ? pk : tensor;
    wp = mode_unpacks(MODE) ? tensor : pk;
    left = d.nblk;
    seg = segs + d.seg;
    if (kShiftSrc) {
      L.t = static_cast<uint32_t>(d.addr) & 15u;
      lp += 16u - L.t;
    }
    if (kShiftDst) {
      const uint32_t before = static_cast<uint32_t>(d.addr) & 15u;
      L.t = 16u - before;
      wp -= before;
      L.first = lane == 0;
    }
    // the first span goes to L2 now; each later one about a span before use
    if (kPrefetch) prefetch_l2_lane0(lp, (left < kSpan ? left : kSpan) * kBlockBytes, lane);
    lp += lane * 16;
    wp += lane * 16;
#pragma unroll
    for (uint32_t u = 0; u < kStage; ++u)
      cur[u] = u < left ? load(lp + u * kBlockBytes) : make_uint4(0u, 0u, 0u, 0u);
    lp += kStageBytes;
  };
  // Where the block in cur[u] was loaded, and this lane's unit of it.
  auto place = [&](uint32_t u) { return lp + u * kBlockBytes - kStageBytes; };
  auto unit = [&](uint32_t u) { return kShiftSrc ? take16(ld_unit_l1(place(u) - 16), cur[u], L.t) : cur[u]; };
  // One stage whose following stage is whole.
  auto stage = [&]() {
#pragma unroll
    for (uint32_t u = 0; u < kStage; ++u) {
      if (Geo<MODE, SHIFT>::kLoadFirst) {
        const uint4 v = unit(u);
        cur[u] = load(lp + u * kBlockBytes);
        do_unit<MODE, DT, SHIFT>(L, v, place(u), wp + u * kBlockBytes, lb);
      } else {
        do_unit<MODE, DT, SHIFT>(L, unit(u), place(u), wp + u * kBlockBytes, lb);
        cur[u] = load(lp + u * kBlockBytes);
      }
    }
    lp += kStageBytes;
    wp += kStageBytes;
  };

  if (n == 0) return;
  begin();
  for (;;) {
    L.s[0] = L.s[1] = L.s[2] = L.s[3] = 0;
    L.f = FpAcc{0ull, 0ull, 0ull, 0ull};
    L.nonfinite = 0;
    // A piece goes stage by stage while the stage after it is whole (a stage
    // loads the next one), then the last blocks, under two stages of them, one
    // at a time, the registers moving up.  A short piece runs through all of
    // this code once, and fetching it is what it waits for; so the last blocks
    // take the code of one block, not of a stage, and pack and unpack have one
    // loop of stages and one place for the end of a span after it.  The
    // fingerprint, bound by issue, has whole spans in a loop without a branch
    // before the stages that are left, and the piece's end apart.  (40,000
    // chunks of 1.5 KB on average, step: two predicated stages at the end and
    // separate loops 221 us, one block at a time 198, one loop 189; with one
    // loop the fingerprint of the Llama-8B shard loses 3%.)
    uint32_t done = 0;  // blocks of the current span swept
    if constexpr (kSpans) {
      while (left >= kSpan + kStage) {
        if (kPrefetch && lane == 0) {
          const uint32_t m = left - kSpan < kSpan ? left - kSpan : kSpan;
          prefetch_l2(lp - kStageBytes + kSpanBytes, m * kBlockBytes);
        }
#pragma unroll 1
        for (uint32_t st = 0; st < kSpan / kStage; ++st) stage();
        if (kFp)
          span_end<MODE, DT, kShiftSrc>(L, lp - kSpanBytes - kStageBytes - (kShiftSrc ? 16 - L.t : 0), kSpan, seg, lane);
        ++seg;
        left -= kSpan;
      }
      if (kPrefetch && left > kSpan)
        prefetch_l2_lane0(lp - kStageBytes + kSpanBytes, (left - kSpan) * kBlockBytes, lane);
#pragma unroll 1
      for (; left >= 2 * kStage; left -= kStage, done += kStage) stage();
    } else {
#pragma unroll 1
      while (left >= 2 * kStage) {
        stage();
        left -= kStage;
        done += kStage;
        if (done == kSpan) {
          if (kFp)
            span_end<MODE, DT, kShiftSrc>(L, lp - kSpanBytes - kStageBytes - (kShiftSrc ? 16 - L.t : 0), kSpan, seg, lane);
          ++seg;
          done = 0;
        }
      }
    }
    for (;;) {
      do_unit<MODE, DT, SHIFT>(L, unit(0), place(0), wp, lb);
#pragma unroll
      for (uint32_t u = 0; u + 1 < kStage; ++u) cur[u] = cur[u + 1];
      if (left > kStage) cur[kStage - 1] = load(lp);
      lp += kBlockBytes;
      wp += kBlockBytes;
      ++done;
      --left;
      if (kSpans && left == 0) break;
      if (done == kSpan || left == 0) {
        if (kFp)
          span_end<MODE, DT, kShiftSrc>(L, lp - (done + kStage) * kBlockBytes - (kShiftSrc ? 16 - L.t : 0), done, seg,
                                        lane);
        if (left == 0) break;
        ++seg;
        done = 0;
      }
    }
    // the open span (the piece's last): its first unit, blocks and slot
    const uint8_t* sp = lp - (done + kStage) * kBlockBytes - (kShiftSrc ? 16 - L.t : 0);
    double* last_seg = seg;
    Record* rec = recs + r;
    // a shifted destination ends in the first granule after the blocks, with the
    // end of the last unit
    if (kShiftDst && lane == 0) st_part<false>(wp, ld_unit_l1(lp - kStageBytes - 16), L.t);
    ++r;
    const bool more = --n > 0;
    if (kSpans && kFp) span_end<MODE, DT, kShiftSrc>(L, sp, done, last_seg, lane);

    // ---- fold the 128 streams into the raw CRC of the piece
    uint32_t v = mul_x32(L.s[0]) ^ L.s[1];
    v = mul_x32(v) ^ L.s[2];
    v = mul_x32(v) ^ L.s[3];
    v = __reduce_xor_sync(0xFFFFFFFFu, mul_lane(v, lb));
    const uint32_t nonfinite = kFp ? __reduce_add_sync(0xFFFFFFFFu, L.nonfinite) : 0u;
    if (lane == 0) *rec = Record{v, nonfinite, 0.0};
    if (!more) return;
    begin();
  }
}

// One run by its class's code.  (Plain unpack only copies and checksums, so
// it runs every element type as bytes.)
template <int MODE>
__device__ __forceinline__ void sweep_class(const SweepParams& p, const RunDesc& rd, uint32_t lane) {
  // a piece's descriptor says all its sweep needs: one dependent load, and the
  // next one's is on its way to L1
  auto get = [&](uint32_t r, bool more) {
    if (more && lane == 0) asm volatile("prefetch.global.L1 [%0];" ::"l"(p.pieces + r + 1));
    return p.pieces[r];
  };
  if constexpr (!mode_sums(MODE)) {
    if (rd.cls & 1u)
      sweep_run<MODE, kDtBytes, false>(p.packed, p.segs, p.recs, get, rd.first, rd.n, lane);
    else
      sweep_run<MODE, kDtBytes, true>(p.packed, p.segs, p.recs, get, rd.first, rd.n, lane);
  } else {
    switch (rd.cls) {
      case kDtF32 * 2 + 1: sweep_run<MODE, kDtF32, false>(p.packed, p.segs, p.recs, get, rd.first, rd.n, lane); break;
      case kDtBf16 * 2 + 1: sweep_run<MODE, kDtBf16, false>(p.packed, p.segs, p.recs, get, rd.first, rd.n, lane); break;
      case kDtBytes * 2 + 1: sweep_run<MODE, kDtBytes, false>(p.packed, p.segs, p.recs, get, rd.first, rd.n, lane); break;
      case kDtF32 * 2: sweep_run<MODE, kDtF32, true>(p.packed, p.segs, p.recs, get, rd.first, rd.n, lane); break;
      case kDtBf16 * 2: sweep_run<MODE, kDtBf16, true>(p.packed, p.segs, p.recs, get, rd.first, rd.n, lane); break;
      default: sweep_run<MODE, kDtBytes, true>(p.packed, p.segs, p.recs, get, rd.first, rd.n, lane); break;
    }
  }
}

// Whether a mode's warps claim units: pack and unpack, which are bound by
// memory latency and whose warps' rates differ from SM to SM by a few percent.
// The fingerprint keeps a static split: it is bound by instruction issue, and
// the start of each unit (claim, descriptors, first loads: about 4 us against
// 10 us for its 32 KiB) costs its launch more than the tail (GPT-2 small: its
// SMs end between 270 and 282 us without units, all at 295 with 8% in units).
__host__ __device__ constexpr bool mode_claims(int m) { return m != kModeFingerprint; }

// The CTA's shared memory: braid tables, lane table.
template <int MODE>
__device__ __forceinline__ void fill_smem() {
  start_lane_fold<Cta<MODE>::kThreads>();
  fill_tables<Cta<MODE>::kThreads>();
  finish_lane_fold();
  __syncthreads();
}

// Every class of a batch in one launch: each warp sweeps a run of its own
// class, and the plan spreads each class's warps over all CTAs, so warps that
// wait on memory and warps that are bound by instruction issue share every
// SM.  For pack and unpack the runs cover most of each class's blocks; the
// rest is cut into units that warps claim one at a time once their own run is
// done, so the launch ends when the work does, not when its slowest warp
// does.  Which warp sweeps a unit changes nothing in the results: a piece's
// record and segment sums have fixed slots.
//
// The claim counter needs no reset: every warp claims until it is refused
// once, so a launch makes exactly n_units + (its warps) claims, and atomicInc
// wraps to zero on the last of them.  (A claim made before the sweep it
// follows, to hide its round trip, holds a unit back from idle warps: GPT-2
// small's unpack lost 4%.)
template <int MODE>
__global__ void __launch_bounds__(Cta<MODE>::kThreads, 1) sweep_kernel(SweepParams p) {
  fill_smem<MODE>();
  wait_for_kernel_before();
  const uint32_t lane = threadIdx.x & 31u;
  RunDesc rd = p.warps[blockIdx.x * Cta<MODE>::kWarps + (threadIdx.x >> 5)];
  for (;;) {
    sweep_class<MODE>(p, rd, lane);
    if (!mode_claims(MODE) || p.n_units == 0) return;
    uint32_t u = 0;
    if (lane == 0) u = atomicInc(p.queue, p.n_units + gridDim.x * Cta<MODE>::kWarps - 1);
    u = __shfl_sync(0xFFFFFFFFu, u, 0);
    if (u >= p.n_units) return;
    rd = p.units[u];
  }
}

// List mode (re-sending failed chunks): warp w sweeps the whole body of chunk
// ids[w] into recs[w].  Every variant is a separate function, so this cold
// kernel's dispatch does not burden the registers of the hot ones.
template <int MODE, int DT, bool ALIGNED>
__device__ __noinline__ void list_piece(const ListParams& p, uint64_t w, uint32_t lane) {
  auto get = [&](uint32_t, bool) {
    const ChunkDesc cd = p.chunks[p.ids[w]];
    PieceDesc d;
    d.addr = cd.addr;
    d.payload_off = cd.payload_off;
    d.seg = cd.seg_base;
    d.nblk = static_cast<uint32_t>(cd.len / kBlockBytes);
    return d;
  };
  sweep_run<MODE, DT, !ALIGNED>(p.packed, p.segs, p.recs + w, get, 0, 1, lane);
}

template <int MODE>
__global__ void __launch_bounds__(Cta<MODE>::kThreads, 1) list_kernel(const __grid_constant__ ListParams p) {
  fill_smem<MODE>();
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t w = static_cast<uint64_t>(blockIdx.x) * Cta<MODE>::kWarps + (threadIdx.x >> 5);
  if (w >= p.n) return;
  const ChunkDesc cd = p.chunks[p.ids[w]];
  if (cd.len < static_cast<uint64_t>(kBlockBytes)) return;
  const bool aligned = (cd.sweep_class & 1u) != 0;
  const uint32_t dt = mode_sums(MODE) ? cd.dtype : kDtBytes;
  if (dt == kDtF32) {
    if (aligned) list_piece<MODE, kDtF32, true>(p, w, lane);
    else list_piece<MODE, kDtF32, false>(p, w, lane);
  } else if (dt == kDtBf16) {
    if (aligned) list_piece<MODE, kDtBf16, true>(p, w, lane);
    else list_piece<MODE, kDtBf16, false>(p, w, lane);
  } else {
    if (aligned) list_piece<MODE, kDtBytes, true>(p, w, lane);
    else list_piece<MODE, kDtBytes, false>(p, w, lane);
  }
}

template <int MODE>
cudaError_t launch_list(const ListParams& p, cudaStream_t s) {
  if (p.n == 0) return cudaSuccess;
  const uint64_t ctas = (p.n + Cta<MODE>::kWarps - 1) / Cta<MODE>::kWarps;
  list_kernel<MODE><<<static_cast<unsigned>(ctas), Cta<MODE>::kThreads, kSweepSmem, s>>>(p);
  return cudaGetLastError();
}

}  // namespace

// Opt the kernels of one mode in to their shared-memory size; launch them.
template <int MODE>
cudaError_t configure_mode() {
  cudaError_t e = cudaFuncSetAttribute(sweep_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmem);
  if constexpr (MODE != kModeFingerprint) {  // no call fingerprints a list
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(list_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmem);
  }
  return e;
}

template <int MODE>
cudaError_t launch_mode(const SweepParams& p, int n_ctas, cudaStream_t s) {
  return launch_chained(sweep_kernel<MODE>, n_ctas, Cta<MODE>::kThreads, kSweepSmem, s, p);
}

}  // namespace frk
