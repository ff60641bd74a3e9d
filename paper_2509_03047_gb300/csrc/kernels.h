// kernels.h -- launchers of the device kernels (internal to libflashrec).
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

#include "layout.h"
#include "../../include/flashrec.h"

namespace frk {

// Sweep modes.  kModeUnpackFp is unpack + verify that also computes the
// fingerprint values (non-finite count, sum of squares) of the restored bytes
// on the same pass, so a restore needs no separate fingerprint sweep.
enum : int { kModeFingerprint = 0, kModePack = 1, kModeUnpack = 2, kModeUnpackFp = 3 };
// Direction: the packed buffer is the source.
__host__ __device__ constexpr bool mode_unpacks(int m) { return m == kModeUnpack || m == kModeUnpackFp; }
// Whether the mode computes non-finite counts and sums of squares.
__host__ __device__ constexpr bool mode_sums(int m) { return m != kModeUnpack; }

struct SweepParams {
  const PieceDesc* pieces;
  const RunDesc* warps;   // one run per warp of the launch, of any class
  Record* recs;           // one per piece
  double* segs;           // segment sums of squares (all modes but kModeUnpack)
  uint8_t* packed;        // pack: destination; unpack: source; fingerprint: unused
  // Work units of any class, claimed one at a time by warps that have
  // finished their own run.  *queue counts the claims: zero when a launch
  // starts and again when it ends.  n_units = 0: no units, queue unused.
  const RunDesc* units;
  uint32_t* queue;
  uint32_t n_units;
};

struct FinalizeParams {
  const ChunkDesc* chunks;
  const Record* recs;
  const double* segs;
  const PieceDesc* pieces;  // per record: its piece (read only without rec_mul)
  const uint32_t* rec_mul;  // per record: x^(8 * bytes after it in its chunk's body); null: computed here
  const uint32_t* crc_xor;  // per chunk: CRC preset/final-XOR term for its length; null: computed here
  uint64_t n_chunks;        // chunks of the whole plan
  uint64_t c_begin, c_end;  // chunks to finalize: [c_begin, c_end), or list positions if ids != null
  const uint32_t* ids;      // list mode: chunk ids; the record of list position i is recs[i]
  uint8_t* packed;  // pack: destination; unpack: source
  FpEntry* out_fp;  // fingerprint: output table; pack, unpack-fp: optional table (null: none)
  uint8_t* flags;   // unpack: per-chunk verdict
};

// Geometry of the sweep kernels: one CTA per SM, with a warp count per mode
// (measured on GB300 with the 31.8 GB shard: the issue-bound fingerprint
// wants 16 warps with deep per-warp stages -- 20 warps cost it 7 points; the
// latency-bound pack and unpack want 20 warps in flight -- 2 points more).
#ifndef FR_WARPS_FP
#define FR_WARPS_FP 16
#endif
#ifndef FR_WARPS_PACK
#define FR_WARPS_PACK 20
#endif
#ifndef FR_WARPS_UNPACK
#define FR_WARPS_UNPACK 20
#endif
#ifndef FR_WARPS_UNPACK_FP
#define FR_WARPS_UNPACK_FP 20
#endif
__host__ __device__ constexpr int sweep_warps(int mode) {
  return mode == kModeFingerprint ? FR_WARPS_FP
         : mode == kModePack      ? FR_WARPS_PACK
         : mode == kModeUnpack    ? FR_WARPS_UNPACK
                                  : FR_WARPS_UNPACK_FP;
}

// A call is a chain of two to three kernels that each need the one before whole.
// Every kernel of the chain is launched so that its blocks may start while that
// one ends (programmatic stream serialization): launching them, and filling
// their tables in shared memory, overlaps with it, and every thread then waits
// for it, and with it for all before it, before it touches memory that any
// kernel writes.  A kernel of someone else's in between is waited for whole.
// GB300, us, launched one after the other -> so: GPT-2 small fingerprint 280 ->
// 276, pack 539 -> 534, unpack 538 -> 532; 4.2 GB in 50,000 tensors, fingerprint
// 677 -> 672; GPT-2 small restored in 16 batches 1540 -> 1465; a 15 MB state's
// restore step 39.3 -> 37.4.  No kernel lets the next start before its own blocks
// end (griddepcontrol.launch_dependents): finalize's blocks on the SMs that finish
// first slow the sweep's last ones.  With the trigger / without, us: fingerprint
// of 64 MB 22.7 / 20.1, 256 MB 57.9 / 57.1, 1 GB 178 / 175, 1.7 to 14 GB equal,
// 32 GB in 16 MiB chunks 4,935 / 4,945 (a mix of bf16 and fp32 of 320 to 400 MB 1
// us less with it); pack and unpack of GPT-2 small in 16 batches 1547 / 1461.
template <class... P>
cudaError_t launch_chained(void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t s, const P&... args) {
  cudaLaunchAttribute overlap = {};
  overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  overlap.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(static_cast<unsigned>(grid));
  c.blockDim = dim3(static_cast<unsigned>(block));
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &overlap;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, args...);
  return cudaGetLastError();
}
#ifdef __CUDACC__
// In every thread of such a kernel, before its first access to global memory
// other than the constant tables: the kernel before has ended, its writes are
// visible.  That also makes the non-coherent loads (ld.global.nc, __ldg) of the
// state and the packed buffer valid, which ask for memory that nobody writes
// while the kernel reads it, although a block may have started while the kernel
// before still wrote it: none comes before this wait, since every address comes
// from a table that is read after it, and from the wait on nothing writes what
// a call reads until the call's end.  (A shifted unpack's first load reaches 16
// bytes before the payload, which another stream's pack may be writing: they
// are dropped.)  Plain loads instead, which keep their order with the stores
// before them: 2.5 GB of views, pack 781 -> 944 us, unpack 788 -> 1,003; aligned
// states equal but for the Llama-8B step, 8,377 -> 8,399.
__device__ __forceinline__ void wait_for_kernel_before() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The one rule, in the sweeps' exact fallback and in finalize's tails, by which
// the square of a finite element is added exactly to a float pair: |x| = ax in
// [2^-40, 2^56], where the fp32 product and its FMA residual are the square (the
// residual is not subnormal) and a lane's squares stay far from overflow.  A
// zero adds nothing; any other square is added in fp64.
__device__ __forceinline__ bool pair_square(float ax) { return ax >= 0x1p-40f && ax <= 0x1p56f; }
#endif

// Per device, before the first launch: opt the sweep kernels in to their
// shared-memory size.
cudaError_t configure_sweep_fp();
cudaError_t configure_sweep_pack();
cudaError_t configure_sweep_unpack();
cudaError_t configure_sweep_unpack_fp();

// List mode: one warp per listed chunk sweeps its whole body into recs[i].
struct ListParams {
  const ChunkDesc* chunks;
  const uint32_t* ids;
  uint64_t n;
  Record* recs;
  double* segs;
  uint8_t* packed;
};

// Every class of a batch in one launch (per-run class in RunDesc).
cudaError_t launch_sweep_fp(const SweepParams& p, int n_ctas, cudaStream_t s);
cudaError_t launch_sweep_pack(const SweepParams& p, int n_ctas, cudaStream_t s);
cudaError_t launch_sweep_unpack(const SweepParams& p, int n_ctas, cudaStream_t s);
cudaError_t launch_sweep_unpack_fp(const SweepParams& p, int n_ctas, cudaStream_t s);
inline cudaError_t launch_sweep(int mode, const SweepParams& p, int n_ctas, cudaStream_t s) {
  return mode == kModeFingerprint ? launch_sweep_fp(p, n_ctas, s)
         : mode == kModePack      ? launch_sweep_pack(p, n_ctas, s)
         : mode == kModeUnpackFp  ? launch_sweep_unpack_fp(p, n_ctas, s)
                                  : launch_sweep_unpack(p, n_ctas, s);
}
cudaError_t launch_list_pack(const ListParams& p, cudaStream_t s);
cudaError_t launch_list_unpack(const ListParams& p, cudaStream_t s);
cudaError_t launch_list_unpack_fp(const ListParams& p, cudaStream_t s);
inline cudaError_t launch_list_sweep(int mode, const ListParams& p, cudaStream_t s) {
  return mode == kModePack ? launch_list_pack(p, s)
                           : (mode == kModeUnpackFp ? launch_list_unpack_fp(p, s) : launch_list_unpack(p, s));
}

cudaError_t launch_finalize(int mode, const FinalizeParams& p, cudaStream_t s);
// Ascending ids of the set flags, first `cap` of them, and the true count.
cudaError_t launch_compact_flags(const uint8_t* flags, uint64_t n, uint32_t* out, uint64_t cap,
                                 uint64_t* count, uint32_t* status, cudaStream_t s);
// Ascending ids of the differing 16-byte entries, first `cap`, true count.
cudaError_t launch_diff(const FpEntry* a, const FpEntry* b, uint64_t n, uint32_t* out, uint64_t cap,
                        uint64_t* count, cudaStream_t s);

// Set the calling thread's fr_last_error message and return the status
// (FR_ERR_INVALID_ARG with `what`, FR_ERR_CUDA with the CUDA error's text).
fr_status report_invalid(const char* where, const char* what);
fr_status report_cuda(const char* where, cudaError_t e);

}  // namespace frk
