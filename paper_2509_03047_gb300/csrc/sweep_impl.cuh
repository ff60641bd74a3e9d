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
//    piece the streams are folded with GF(2) multiplications by constants and
//    warp shuffles into the raw CRC of the piece;
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
// outgrow the instruction cache (2.5 GB of views: 686 us, 597 with 4).
#ifndef FR_STAGE_FP_SHIFT
#define FR_STAGE_FP_SHIFT 4
#endif
// Up to this many lanes of a segment that need the exact fallback take it in
// turn by the whole warp (slow_span_by_warp), more take it side by side
// (slow_span).
#ifndef FR_SLOW_WARP_LANES
#define FR_SLOW_WARP_LANES 4
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

// The piece-end fold multiplies by seven constants: x^32 (Horner inside the
// lane), x^128 ... x^2048 (the shuffle tree) and the unbraid factor.  Each
// multiply is four byte lookups in that constant's tables (read-only, cached
// in L1) instead of a 32-step bit loop: a warp pays the fold once per piece,
// which matters for states of many small tensors.
struct FoldTables {
  ByteTables4 m[7];
};
__host__ __device__ constexpr FoldTables make_fold_tables() {
  FoldTables f{};
  f.m[0] = make_mul_tables(gf_xpow(32));
  f.m[1] = make_mul_tables(gf_xpow(128));
  f.m[2] = make_mul_tables(gf_xpow(256));
  f.m[3] = make_mul_tables(gf_xpow(512));
  f.m[4] = make_mul_tables(gf_xpow(1024));
  f.m[5] = make_mul_tables(gf_xpow(2048));
  f.m[6] = make_mul_tables(kUnbraid);
  return f;
}
__device__ const FoldTables g_fold = make_fold_tables();

// a * (constant i) mod P.
__device__ __forceinline__ uint32_t mul_fold(int i, uint32_t a) {
  const ByteTables4& T = g_fold.m[i];
  return (__ldg(&T.t[0][a & 255u]) ^ __ldg(&T.t[1][(a >> 8) & 255u])) ^
         (__ldg(&T.t[2][(a >> 16) & 255u]) ^ __ldg(&T.t[3][a >> 24]));
}

// ------------------------------------------------------------------ memory

// 16 bytes at p, a multiple of 16.
__device__ __forceinline__ uint4 ld_unit(const uint8_t* p) {
  uint4 v;
  asm("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0,%1,%2,%3}, [%4];"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p));
  return v;
}

__device__ __forceinline__ void st_unit(uint8_t* p, const uint4& v) {
  asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z),
               "r"(v.w)
               : "memory");
}

// Chunks that do not start on a 16-byte boundary move in 16-byte granules all
// the same.  A lane's unit lies across two granules.  Reading, lane l loads
// the one its unit ends in and gets the one it starts in from lane l - 1 by
// shuffle (lane 0: from lane 31's of the block before); take16 cuts the unit
// out.  Writing, lane l stores the granule its unit starts in, whose first
// bytes are the end of lane l - 1's unit.  So every lane holds the same 16
// bytes of the chunk as for an aligned chunk, and neither the CRC streams nor
// the order of the sums change with the alignment.  A granule is only read if
// it holds a byte of the piece, so no read reaches a page that the tensor does
// not; its other bytes are dropped, and never written.
//
// Before, such chunks moved by 4-byte or single-byte accesses 16 bytes apart
// from lane to lane: 4 or 16 times the load and store instructions, each
// touching every line of the block.  GB300, 2.5 GB of views at any element
// offset, us: fingerprint 1095 -> 597, pack 1025 -> 931, unpack 1495 -> 791.

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

// Lane `from`'s v.
__device__ __forceinline__ uint4 shfl4(const uint4& v, uint32_t from) {
  return make_uint4(__shfl_sync(0xFFFFFFFFu, v.x, from), __shfl_sync(0xFFFFFFFFu, v.y, from),
                    __shfl_sync(0xFFFFFFFFu, v.z, from), __shfl_sync(0xFFFFFFFFu, v.w, from));
}
__device__ __forceinline__ uint4 select4(bool c, const uint4& a, const uint4& b) {
  return make_uint4(c ? a.x : b.x, c ? a.y : b.y, c ? a.z : b.z, c ? a.w : b.w);
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


// Exact sum of squares of elements added one by one, in order, given as fp32
// bit patterns (a bf16 element in the high half).  A non-finite element is
// counted; the square of one with |x| = 0 or in [2^-40, 2^56] is added exactly
// -- the fp32 product and its FMA residual -- to the float pair (hi, lo) by
// TwoSum; any other sets `odd`, and odd_squares adds it.  No branch and no fp64
// instruction: predicated off, those still take turns on the narrow pipe, and
// with them in the loop a NaN cost the launch 13 us, without 2.
struct ExactSum {
  float hi = 0.0f, lo = 0.0f;
  uint32_t nonfinite = 0;
  bool odd = false;
  __device__ __forceinline__ void add(uint32_t f) {
    const bool inf_nan = (f & 0x7F800000u) == 0x7F800000u;
    const float ax = fabsf(__uint_as_float(f));
    const bool fast = ax == 0.0f || (ax >= 0x1p-40f && ax <= 0x1p56f);  // false for NaN and Inf
    nonfinite += inf_nan ? 1u : 0u;
    odd |= !fast && !inf_nan;
    const float x = fast ? __uint_as_float(f) : 0.0f;  // (a zero square changes nothing)
    const float p = x * x;
    const float e = __fmaf_rn(x, x, -p);
    const float t = hi + p;
    const float z = t - hi;
    lo += ((hi - (t - z)) + (p - z)) + e;
    hi = t;
  }
  template <int DT>
  __device__ __forceinline__ void add_word(uint32_t w) {
    add(DT == kDtF32 ? w : w << 16);
    if (DT != kDtF32) add(w & 0xFFFF0000u);
  }
};

// The squares that ExactSum leaves out (tiny or huge values, rare), of the
// calling lane's units of `n` blocks, the first at sp, in order: in fp64, where
// the square of an fp32 value is exact.
template <int DT, bool SHIFT>
__device__ __noinline__ double odd_squares(const uint8_t* sp, uint32_t n) {
  double d = 0.0;
#pragma unroll 1
  for (uint32_t b = 0; b < n; ++b) {
    const uint4 v = ld_unit_at<SHIFT>(sp + b * kBlockBytes);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < (DT == kDtF32 ? 4 : 8); ++j) {
      const uint32_t f = DT == kDtF32 ? w[j & 3] : ((j & 1) ? w[j / 2] & 0xFFFF0000u : w[j / 2] << 16);
      const float ax = fabsf(__uint_as_float(f));
      if ((f & 0x7F800000u) == 0x7F800000u || ax == 0.0f || (ax >= 0x1p-40f && ax <= 0x1p56f)) continue;
      const double xd = static_cast<double>(__uint_as_float(f));
      d = __dadd_rn(d, __dmul_rn(xd, xd));
    }
  }
  return d;
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
        if (ax >= 0x1p-40f && ax <= 0x1p56f) {
          const float p2 = x * x;
          const float e = __fmaf_rn(x, x, -p2);
          const float t = hi + p2;
          const float z = t - hi;
          lo += ((hi - (t - z)) + (p2 - z)) + e;
          hi = t;
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
// k, and all lanes add the words in the order slow_span does, taking them from
// lane k by shuffle.  One lane that needs the fallback (one NaN) is the common
// case, and its warp may be all that a launch still waits for: this way it
// waits for one load, not for 32 in turn.  GB300, a 15 MB state with 3 NaNs
// (L2-resident, as a graph), us: fingerprint 24.5 -> 17.3, pack 24.7 -> 16.9;
// without NaN 15.2.
template <int DT, bool SHIFT>
__device__ __noinline__ Exact slow_span_by_warp(const uint8_t* sp, uint32_t n, uint32_t l, uint32_t lane) {
  const uint8_t* first = sp + (static_cast<int32_t>(l) - static_cast<int32_t>(lane)) * 16;  // lane l's first unit
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (lane < n) v = ld_unit_at<SHIFT>(first + lane * kBlockBytes);
  ExactSum x;
#pragma unroll 1
  for (uint32_t k = 0; k < n; ++k) {
    x.add_word<DT>(__shfl_sync(0xFFFFFFFFu, v.x, k));
    x.add_word<DT>(__shfl_sync(0xFFFFFFFFu, v.y, k));
    x.add_word<DT>(__shfl_sync(0xFFFFFFFFu, v.z, k));
    x.add_word<DT>(__shfl_sync(0xFFFFFFFFu, v.w, k));
  }
  const double d = x.odd ? odd_squares<DT, SHIFT>(first, n) : 0.0;
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
  uint32_t t;     // take16's t
  uint4 carry;    // lane 0: lane 31's granule (source) or unit (destination) of the previous block
  bool first;     // destination, lane 0: no block stored yet
};

template <int MODE, int DT, bool SHIFT>
__device__ __forceinline__ void do_unit(Lane<MODE, DT>& L, const uint4& v, uint8_t* wp, uint32_t lb) {
  constexpr bool kFp = mode_sums(MODE) && (DT != kDtBytes);
  if (MODE != kModeFingerprint) {
    if (SHIFT && mode_unpacks(MODE)) {
      const uint4 y = shfl4(v, (lb / 4 + 31) & 31u);
      const uint4 g = take16(select4(lb == 0, L.carry, y), v, L.t);
      L.carry = y;
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

// End of a span (one segment) of `n` blocks, the lane's first unit at sp: the fast sums are kept if finite and
// either large enough that fp32 underflow is negligible (below 2^-77 relative)
// or made of zeros only; otherwise the segment is summed exactly from a
// reload.  The lanes' sums are then added in a fixed tree and lane 0 stores
// the segment's sum (a float pair, see seg_value) at its index.
template <int MODE, int DT, bool SHIFT>
__device__ __forceinline__ void span_end(Lane<MODE, DT>& L, const uint8_t* sp, uint32_t n, double* seg,
                                         uint32_t lane) {
  const u64 ab = add2(L.f.A, L.f.B);
  const float tot = lo_f(ab) + hi_f(ab);
  bool ok = tot < __int_as_float(0x7F800000);
  if (ok && !(tot >= 0x1p-60f)) ok = span_is_zero<DT, SHIFT>(sp, n);
  float hi = 0.0f, lo = 0.0f;
  double d = 0.0;
  if (ok) fold_to_pair(L.f, hi, lo);
  uint32_t bad = __ballot_sync(0xFFFFFFFFu, !ok);
  if (__popc(bad) > kSlowWarpLanes) {
    bad = 0;
    if (!ok) {
      const Exact x = slow_span<DT, SHIFT>(sp, n);
      d = x.d;
      L.nonfinite += x.nonfinite;
    }
  }
  for (; bad != 0; bad &= bad - 1) {
    const uint32_t l = static_cast<uint32_t>(__ffs(static_cast<int>(bad))) - 1u;
    const Exact x = slow_span_by_warp<DT, SHIFT>(sp, n, l, lane);
    if (lane == l) {
      d = x.d;
      L.nonfinite += x.nonfinite;
    }
  }
  L.f.A = L.f.CA = L.f.B = L.f.CB = 0ull;
  // The lanes' sums are added in a fixed tree: as float pairs by TwoSum when
  // every lane took the fast path with a sum far from fp32 overflow (no fp64
  // work), else in fp64 (rare).  Lane 0 stores the form seg_value() reads.
  if (__all_sync(0xFFFFFFFFu, ok && tot < 0x1p120f)) {
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
  } else {
    if (ok) d = static_cast<double>(hi) + static_cast<double>(lo);
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) d += __shfl_down_sync(0xFFFFFFFFu, d, m);
    if (lane == 0) *seg = -d;
  }
}

// One piece: `nblk` 512-byte blocks from `src` (to `dst` for pack/unpack).
// SHIFT: the tensor side (source, or destination for unpack) does not start
// on a 16-byte boundary; the packed side always does.
//
// Pipeline: for the fingerprint, lane 0 prefetches whole spans into L2 one span
// ahead with the bulk-copy unit; each lane keeps kStage 16-byte units of the next stage in
// flight in registers, which therefore mostly wait for L2.  Each span is one
// sum segment: its fp32 sums start at zero, are checked at its end, and are
// replaced by an exact sum from a reload when they fail.
template <int MODE, int DT, bool SHIFT>
__device__ __forceinline__ void sweep_piece(const uint8_t* __restrict__ src, uint8_t* __restrict__ dst,
                                            uint32_t nblk, uint32_t lane, Record* rec, double* seg) {
  constexpr bool kFp = mode_sums(MODE) && (DT != kDtBytes);
  constexpr uint32_t kStage = Geo<MODE, SHIFT>::kStage;
  constexpr bool kPrefetch = Geo<MODE, SHIFT>::kPrefetch;
  constexpr bool kShiftSrc = SHIFT && !mode_unpacks(MODE), kShiftDst = SHIFT && mode_unpacks(MODE);
  constexpr uint32_t kStageBytes = kStage * kBlockBytes;
  constexpr uint32_t kSpanBytes = kSpan * kBlockBytes;
  const uint32_t lb = lane << 2;

  Lane<MODE, DT> L;
  L.s[0] = L.s[1] = L.s[2] = L.s[3] = 0;
  L.f = FpAcc{0ull, 0ull, 0ull, 0ull};
  L.nonfinite = 0;
  const uint8_t* lp = src;
  uint8_t* wp = dst;
  if (kShiftSrc) {
    L.t = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(src)) & 15u;
    lp += 16u - L.t;
    L.carry = lane == 0 ? ld_unit(lp - 16) : make_uint4(0u, 0u, 0u, 0u);
  }
  if (kShiftDst) {
    const uint32_t before = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(dst)) & 15u;
    L.t = 16u - before;
    wp -= before;
    L.carry = make_uint4(0u, 0u, 0u, 0u);
    L.first = lane == 0;
  }

  // The first span goes to L2 now; each later one about a span before use.
  if (kPrefetch) prefetch_l2_lane0(lp, (nblk < kSpan ? nblk : kSpan) * kBlockBytes, lane);

  // (Every unit is given a value here: a register that is only set under a
  // condition is live, to the compiler, around every loop that encloses this
  // one, through the code of every class -- 1,000 bytes of spills.)
  uint4 cur[kStage];
  lp += lane * 16;
  wp += lane * 16;
#pragma unroll
  for (uint32_t u = 0; u < kStage; ++u)
    cur[u] = u < nblk ? ld_unit(lp + u * kBlockBytes) : make_uint4(0u, 0u, 0u, 0u);
  lp += kStageBytes;  // the next stage's loads

  // This lane's unit of the next block, which is in cur[u].
  auto unit = [&](uint32_t u) {
    if (!kShiftSrc) return cur[u];
    const uint4 y = shfl4(cur[u], (lane + 31) & 31u);
    const uint4 before = select4(lane == 0, L.carry, y);
    L.carry = y;
    return take16(before, cur[u], L.t);
  };
  // One stage whose following stage is whole.
  auto stage = [&]() {
#pragma unroll
    for (uint32_t u = 0; u < kStage; ++u) {
      if (Geo<MODE, SHIFT>::kLoadFirst) {
        const uint4 v = unit(u);
        cur[u] = ld_unit(lp + u * kBlockBytes);
        do_unit<MODE, DT, SHIFT>(L, v, wp + u * kBlockBytes, lb);
      } else {
        do_unit<MODE, DT, SHIFT>(L, unit(u), wp + u * kBlockBytes, lb);
        cur[u] = ld_unit(lp + u * kBlockBytes);
      }
    }
    lp += kStageBytes;
    wp += kStageBytes;
  };

  // Three loops cover a piece: (1) whole spans whose following stage is
  // whole too, each span (one sum segment) a call-free loop of kSpan/kStage
  // stages with no branch, preceded by the L2 prefetch of the next span and
  // followed by its validity check -- the bulk of a long piece; (2) the
  // stages left whose following stage is still whole, fewer than a span; (3)
  // the last one or two stages, predicated.  Loop (2) keeps the predicated
  // drain, which runs at about half the rate, to under 2 * kStage blocks.
  uint32_t left = nblk;  // blocks not swept yet
  while (left >= kSpan + kStage) {
    if (kPrefetch && lane == 0) {
      const uint32_t n = left - kSpan < kSpan ? left - kSpan : kSpan;
      prefetch_l2(lp - kStageBytes + kSpanBytes, n * kBlockBytes);
    }
#pragma unroll 1
    for (uint32_t st = 0; st < kSpan / kStage; ++st) stage();
    if (kFp) span_end<MODE, DT, kShiftSrc>(L, lp - kSpanBytes - kStageBytes - (kShiftSrc ? 16 - L.t : 0), kSpan, seg, lane);
    ++seg;
    left -= kSpan;
  }
  if (kPrefetch && left > kSpan)
    prefetch_l2_lane0(lp - kStageBytes + kSpanBytes, (left - kSpan) * kBlockBytes, lane);
  uint32_t done = 0;  // blocks of the current span swept, whole stages
#pragma unroll 1
  for (; left >= 2 * kStage; left -= kStage, done += kStage) stage();
  while (left > 0) {
#pragma unroll
    for (uint32_t u = 0; u < kStage; ++u) {
      if (u < left) {
        do_unit<MODE, DT, SHIFT>(L, unit(u), wp + u * kBlockBytes, lb);
        if (kStage + u < left) cur[u] = ld_unit(lp + u * kBlockBytes);
      }
    }
    lp += kStageBytes;
    wp += kStageBytes;
    const uint32_t n = left < kStage ? left : kStage;
    left -= n;
    if (kFp && (left == 0 || done + n == kSpan)) {
      span_end<MODE, DT, kShiftSrc>(L, lp - (done + 2 * kStage) * kBlockBytes - (kShiftSrc ? 16 - L.t : 0), done + n, seg,
                                    lane);
      ++seg;
      done = 0;
    } else {
      done += n;
    }
  }

  // A shifted destination ends in the first granule after the blocks.
  if (kShiftDst && lane == 0) st_part<false>(dst - (16u - L.t) + static_cast<uint64_t>(nblk) * kBlockBytes, L.carry, L.t);

  // ---- fold the 128 streams into the raw CRC of the piece
  uint32_t v = mul_fold(0, L.s[0]) ^ L.s[1];
  v = mul_fold(0, v) ^ L.s[2];
  v = mul_fold(0, v) ^ L.s[3];
  {
    uint32_t o;
    o = __shfl_down_sync(0xFFFFFFFFu, v, 1);
    v = mul_fold(1, v) ^ o;
    o = __shfl_down_sync(0xFFFFFFFFu, v, 2);
    v = mul_fold(2, v) ^ o;
    o = __shfl_down_sync(0xFFFFFFFFu, v, 4);
    v = mul_fold(3, v) ^ o;
    o = __shfl_down_sync(0xFFFFFFFFu, v, 8);
    v = mul_fold(4, v) ^ o;
    o = __shfl_down_sync(0xFFFFFFFFu, v, 16);
    v = mul_fold(5, v) ^ o;
  }

  uint32_t nonfinite = L.nonfinite;
  if (kFp) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) nonfinite += __shfl_down_sync(0xFFFFFFFFu, nonfinite, m);
  }
  if (lane == 0) {
    Record r;
    r.crc = mul_fold(6, v);
    r.nonfinite = nonfinite;
    r.unused = 0.0;
    *rec = r;
  }
}

// A run of consecutive pieces of one class: a warp's own range, or a unit it
// claimed.  A piece's descriptor says all its sweep needs, so a piece costs
// one dependent load before its data, and the next one's is already in L1.
// ALIGNED: every chunk of the class starts on a 16-byte boundary of its
// tensor's memory; else none does.
template <int MODE, int DT, bool ALIGNED>
__device__ __forceinline__ void sweep_run(const SweepParams& p, uint32_t r, uint32_t n, uint32_t lane) {
  for (; n > 0; --n, ++r) {
    const PieceDesc d = p.pieces[r];
    if (n > 1 && lane == 0) asm volatile("prefetch.global.L1 [%0];" ::"l"(p.pieces + r + 1));
    uint8_t* tensor = reinterpret_cast<uint8_t*>(d.addr);
    uint8_t* packed = (MODE == kModeFingerprint) ? nullptr : p.packed + d.payload_off;
    sweep_piece<MODE, DT, !ALIGNED>(mode_unpacks(MODE) ? packed : tensor, mode_unpacks(MODE) ? tensor : packed, d.nblk,
                                    lane, p.recs + r, p.segs + d.seg);
  }
}

// One run by its class's code.  (Plain unpack only copies and checksums, so
// it runs every element type as bytes.)
template <int MODE>
__device__ __forceinline__ void sweep_class(const SweepParams& p, const RunDesc& rd, uint32_t lane) {
  if constexpr (!mode_sums(MODE)) {
    if (rd.cls & 1u)
      sweep_run<MODE, kDtBytes, true>(p, rd.first, rd.n, lane);
    else
      sweep_run<MODE, kDtBytes, false>(p, rd.first, rd.n, lane);
  } else {
    switch (rd.cls) {
      case kDtF32 * 2 + 1: sweep_run<MODE, kDtF32, true>(p, rd.first, rd.n, lane); break;
      case kDtBf16 * 2 + 1: sweep_run<MODE, kDtBf16, true>(p, rd.first, rd.n, lane); break;
      case kDtBytes * 2 + 1: sweep_run<MODE, kDtBytes, true>(p, rd.first, rd.n, lane); break;
      case kDtF32 * 2: sweep_run<MODE, kDtF32, false>(p, rd.first, rd.n, lane); break;
      case kDtBf16 * 2: sweep_run<MODE, kDtBf16, false>(p, rd.first, rd.n, lane); break;
      default: sweep_run<MODE, kDtBytes, false>(p, rd.first, rd.n, lane); break;
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
  fill_tables<Cta<MODE>::kThreads>();
  __syncthreads();
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
__device__ __noinline__ void list_piece(uint8_t* tensor, uint8_t* packed, uint32_t n, uint32_t lane, Record* rec,
                                        double* segs) {
  sweep_piece<MODE, DT, !ALIGNED>(mode_unpacks(MODE) ? packed : tensor, mode_unpacks(MODE) ? tensor : packed, n, lane,
                                  rec, segs);
}

template <int MODE>
__global__ void __launch_bounds__(Cta<MODE>::kThreads, 1) list_kernel(ListParams p) {
  fill_tables<Cta<MODE>::kThreads>();
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t w = static_cast<uint64_t>(blockIdx.x) * Cta<MODE>::kWarps + (threadIdx.x >> 5);
  if (w >= p.n) return;
  const ChunkDesc cd = p.chunks[p.ids[w]];
  const uint32_t nb = static_cast<uint32_t>(cd.len / kBlockBytes);
  if (nb == 0) return;
  uint8_t* tensor = reinterpret_cast<uint8_t*>(cd.addr);
  uint8_t* packed = p.packed + cd.payload_off;
  const bool aligned = (cd.sweep_class & 1u) != 0;
  const uint32_t dt = mode_sums(MODE) ? cd.dtype : kDtBytes;
  double* segs = p.segs + cd.seg_base;
  Record* rec = p.recs + w;
  if (dt == kDtF32) {
    if (aligned) list_piece<MODE, kDtF32, true>(tensor, packed, nb, lane, rec, segs);
    else list_piece<MODE, kDtF32, false>(tensor, packed, nb, lane, rec, segs);
  } else if (dt == kDtBf16) {
    if (aligned) list_piece<MODE, kDtBf16, true>(tensor, packed, nb, lane, rec, segs);
    else list_piece<MODE, kDtBf16, false>(tensor, packed, nb, lane, rec, segs);
  } else {
    if (aligned) list_piece<MODE, kDtBytes, true>(tensor, packed, nb, lane, rec, segs);
    else list_piece<MODE, kDtBytes, false>(tensor, packed, nb, lane, rec, segs);
  }
}

template <int MODE>
cudaError_t launch_list(const ListParams& p, cudaStream_t s) {
  if (p.n == 0) return cudaSuccess;
  const uint64_t ctas = (p.n + Cta<MODE>::kWarps - 1) / Cta<MODE>::kWarps;
  list_kernel<MODE><<<static_cast<unsigned>(ctas), Cta<MODE>::kThreads, kTableBytes, s>>>(p);
  return cudaGetLastError();
}

}  // namespace

// Opt the kernels of one mode in to their shared-memory size; launch them.
template <int MODE>
cudaError_t configure_mode() {
  cudaError_t e = cudaFuncSetAttribute(sweep_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTableBytes);
  if constexpr (MODE != kModeFingerprint) {  // no call fingerprints a list
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(list_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTableBytes);
  }
  return e;
}

template <int MODE>
cudaError_t launch_mode(const SweepParams& p, int n_ctas, cudaStream_t s) {
  sweep_kernel<MODE><<<n_ctas, Cta<MODE>::kThreads, kTableBytes, s>>>(p);
  return cudaGetLastError();
}

}  // namespace frk
