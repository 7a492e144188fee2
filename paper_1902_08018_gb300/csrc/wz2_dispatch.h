// wz2_dispatch.h -- host-side entry points of the WZ2 kernels, one translation
// unit per rate (wz2_r<rate>.cu) so that the instantiations build in parallel.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "wz2_batch.h"

namespace whff {

// Polls of a bounded device-side wait (tensor-core kernels) before it gives up
// and records WHFF_ETIMEOUT: about a second of try_wait.
constexpr uint32_t kWaitPolls = 1u << 22;

// Raise the dynamic shared-memory limit of a kernel.  The limit belongs to the kernel on
// one device, and a process may use several; it is set on a device's first launch (the
// two calls cost 1 to 2 us, which a small pass would see).  device: the current one, -1 asks.
// carveout: ask for all of the SM's memory as shared memory, too.
template <auto Kern>
int raise_smem(int bytes, bool carveout, int device = -1) {
  static std::atomic<uint64_t> done{0};  // a bit per device; devices from 64 on always set it
  if (device < 0 && cudaGetDevice(&device) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  const uint64_t bit = device < 64 ? 1ull << device : 0;
  if (done.load(std::memory_order_acquire) & bit) return 0;
  if (cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess ||
      (carveout && cudaFuncSetAttribute(Kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                        cudaSharedmemCarveoutMaxShared) != cudaSuccess)) {
    cudaGetLastError();
    return -1;
  }
  done.fetch_or(bit, std::memory_order_release);
  return 0;
}

// Blocks up to which a one-column pass of the lift transforms x in its kernel: that
// saves a launch and costs seven additions per block.  Transform launched / fused, us:
//   4096^2 (2^20 blocks), rate 16: 20.9 / 17.7
//   16384^2 (2^24), rates 8 12 16 20 24: 83.3 86.8 97.4 114.7 129.1 / 82.6 84.3 94.0 111.5 124.9
//   20480^2: 121.0 127.0 144.2 170.2 194.2 / 122.0 123.5 139.9 168.2 189.4
//   32768^2 (2^26): 277.1 290.4 334.5 410.5 467.6 / 286.7 292.7 332.1 410.0 463.2
// Rate 8, bound by decode instructions, loses from 20480^2 on; rate 12 at 32768^2;
// the others gain up to there, the longest measured.
// An x that the kernel cannot take 16 bytes at a time (N not a multiple of 4, or an
// unaligned x; the transform's own output always is) is read word by word for every
// block, which pays only up to 2^22 blocks:
//   4095^2, rates 8 12 16: 25.7 25.7 25.7 / 18.2 18.5 18.6;  8191^2: 37.5 38.2 40.5 / 35.0 36.7 39.0
//   12289^2: 59.5 59.6 65.1 / 64.3 65.8 71.5;  16383^2: 89.1 90.8 101.8 / 105.9 107.3 116.5
// Lane groups (groups8), whose rows are short, have less to hide such loads behind: up to
// 2^19 blocks.  Rate 16: 16000 x 378 (380000) 17.4 / 15.5, 32000 x 378 16.2 / 18.7,
// 64000 x 378 20.3 / 24.0, 20000 x 999 30.4 / 37.6.
constexpr int64_t wz2_fuse_blocks(int rate, bool x_fast, bool groups8) {
  return (int64_t)1 << (!x_fast ? (groups8 ? 19 : 22) : rate == 8 ? 24 : rate == 12 ? 25 : 26);
}

// Blocks up to which the one-column kernels with four or eight blocks in flight add the
// segments of shared bands themselves.  The fence and the atomics of that make the loop
// before them slower, a launch of its own costs 2 us.  In the kernel / launched, us:
//   378 x 32768, rate 16, four in flight: 20.6 / 22.6; eight: 18.5 / 20.6
//   8192^2 (2^22 blocks): 35.9 / 36.0; 40.1 / 38.3
//   16384^2, rates 8 12 16, four: 82.1 86.2 95.8 / 78.0 81.6 94.0
//   32768^2: 285.2 293.0 334.7 / 258.9 275.8 329.2; rate 8, eight: 278.4 / 253.8
// With two in flight the loop gains nothing (16384^2: 84.2 84.3 94.1 / 86.2 87.7 96.0;
// 32768^2: 282.3 282.1 332.4 / 280.1 287.7 330.2), so they always add their own.
constexpr int64_t wz2_finish_blocks(int unroll) { return unroll == 2 ? INT64_MAX : (int64_t)1 << 21; }

struct Wz2Step {
  const uint8_t* stream;
  int64_t M, N, BM, BN;
  const float* x;
  int64_t ldx;
  bool x_vec_ok;
  int64_t L;       // blocks per warp range
  int maxseg;      // most ranges sharing one band
  double* ws;
  double* y;
  int64_t ldy;
  double* state;
  double decay;
  int64_t ctas;    // grid size (persistent)
  int unroll;      // blocks in flight per lane: 2, 4 or 8 (R = 1), 2 otherwise
  bool lift;
  int R;           // 1, 2, 4 or 8
  bool red32;      // fold lanes with the FP32 pair butterfly (short bands)
  bool groups8;    // four 8-lane groups per warp, one band each (short bands)
  float* xt;       // lift: scratch for (2G)^T x, 4 BN floats per right-hand side (8 columns)
  bool staged;     // R = 1: stream each warp's range through shared memory by bulk copies
  int* status;     // device status word (bounded waits of the staged kernel)
  unsigned* seen;  // per band: counts the segments of the pass (see finish_shared_band)
  int device;      // the current one, where the handle lives
};

// Bytes a handle's device stream allocation carries past the stream, so that
// 16-byte-rounded bulk copies of the last blocks stay inside it.
constexpr int kStreamPad = 256;


struct Wz2Batch {
  const dev::BatchEntry* entries;  // device table
  const int64_t* row_begin;        // device prefix of rows
  int nentries;
  int64_t total_blocks, total_rows, L;
  int64_t ctas;
  bool any_shared;                 // some band is split between warp ranges
  bool lift;
  int R;
};

// A batch of one scaled format (BF16, FP16, FP8, FP32): same tables, units
// are 16-byte column chunks (BN of them per band), stream = the payload.
int scaled_batched_launch(int fmt, const Wz2Batch& b, cudaStream_t st);

// state step of a batch (rate independent; defined in the rate-16 unit)
int wz2_batched_state_launch(const dev::BatchState* table, const int64_t* row_begin, int n, int64_t total_rows,
                             cudaStream_t st);

struct ScaledStep {
  int fmt;  // 2 BF16, 3 FP16, 4 FP8 E4M3
  const uint8_t* payload;
  const float* scales;
  int64_t M, N, ld, TN;
  const float* x;
  int64_t ldx;
  bool x_vec_ok;
  int64_t L;
  int maxseg;
  double* ws;
  double* y;
  int64_t ldy;
  double* state;
  double decay;
  int64_t ctas;
  int R;
  bool red32;
  bool groups8;  // four 8-lane groups per warp, one band each (short bands)
  unsigned* seen;  // per band: counts the segments of the pass
};
int scaled_launch(const ScaledStep& a, cudaStream_t st);  // scaled.cu

// Tensor-core pass of up to 32 right-hand sides over a WZ2 matrix (mma.cu).
struct MmaStep {
  int rate;
  bool lift;
  const uint8_t* stream;
  int64_t M, N, BM, BN;
  const float* x;
  int64_t ldx;
  int R;           // 1..32 (padded to 16 or 32 inside)
  int64_t L;       // (tile, stage) items per CTA: tile = 32 bands, stage = 16 blocks
  int ctas;        // persistent grid, ceil(items / L)
  int maxseg;      // most CTAs sharing one tile
  double* ws;      // tiles x maxseg x R x 128 FP64 partials
  uint8_t* btiles; // B operand pieces of every 16-block stage (built per pass)
  double* y;
  int64_t ldy;
  double* state;
  double decay;
  int* status;
  uint32_t spin;   // polls of an in-loop mbarrier wait before it gives up (kWaitPolls)
  const void* map; // CUtensorMap in device memory of the whole stored matrix, or null
  int paired;      // two maps, 128 bytes apart: the even and the odd bands
  int64_t band0;   // first band of this pass in it (row views)
  int device;      // the current one, where the handle lives
  int sms;         // its SMs
};
int mma_launch(const MmaStep& a, cudaStream_t st);

// The tensor-core passes of a batch that share one width class (NR 16 or 32),
// in one persistent launch (mma.cu).  members / passes: device tables.
struct MmaBatchStep {
  int rate;
  bool lift;
  int nr;
  const dev::MmaMember* members;
  const dev::MmaPass* passes;
  int nmem;
  int64_t total, L;  // items of all members, items per CTA
  int ctas;
  int64_t bt_threads, fin_threads;
  int* status;
  uint32_t spin;
  int sms;           // SMs of the device
};
int mma_batch_launch(const MmaBatchStep& a, cudaStream_t st);
int mma_max_members();  // most members of one batched launch
// item ranges per SM of the tensor-core kernel at this rate for R <= nr (0 on error)
int mma_occupancy(int rate, bool lift, int nr);
int scaled_occupancy(int fmt, bool groups8);  // resident CTAs per SM of the R = 1 kernel

// Tensor-core pass of up to 32 right-hand sides over a BF16 / FP16 / FP8
// matrix (scaled_mma.cu): items (tile of 128 rows, stage of 64 columns).
struct ScaledMmaStep {
  int fmt;
  const uint8_t* payload;
  const float* scales;
  int64_t M, N, ld, TN;
  const float* x;
  int64_t ldx;
  int R;           // 1..32 (padded to 16 or 32 inside)
  int64_t L;       // items per CTA
  int ctas;
  int maxseg;      // most CTAs sharing one tile
  double* ws;      // tiles x maxseg x R x 128 FP64 partials
  uint8_t* btiles; // B operand pieces of every stage (built per pass)
  double* y;
  int64_t ldy;
  double* state;
  double decay;
  int* status;
  uint32_t spin;
  const void* tmap;  // CUtensorMap of the whole stored matrix (A tiles by TMA), or null
  int64_t row0;      // first row of this pass within that matrix (row views)
  int* colexp;       // FP16 with tmap: 32 ints of scratch for the per-column exponents of x
  int device;        // the current one, where the handle lives
  int sms;         // its SMs
};
int scaled_mma_launch(const ScaledMmaStep& a, cudaStream_t st);
// Host: encode the TMA map of a WZ2 stream (BM bands of BN blocks, box one stage:
// 32 bands x 16 blocks), or, where its rows are 8 bytes off 16, the maps of the
// even and of the odd bands (box 16 bands, 16 bytes more per row; the odd rows
// start 8 bytes in).  out: 256 bytes.  Returns the number of maps, 0 if none.
int wz2_tma_map(void* out, const void* stream, int64_t BM, int64_t BN, int rate);
// Host: encode the TMA map of a BF16, FP16 (fmt 3) or FP8 (fmt 4) payload (M x ld
// elements, row-major, box 64 x 128, 128-byte swizzle, FP8 64) into out (a
// CUtensorMap, 128 bytes, 64-byte aligned); 0 on success.
int scaled_tma_map(void* out, const void* payload, int64_t M, int64_t ld, int fmt);
// resident CTAs per SM for R <= 32 (0 on error); tma: the TMA-fed BF16 kernel
int scaled_mma_occupancy(int fmt, bool tma);

// Fixed-accuracy (WZ3) pass: (2G)^T x, then persistent ranges (R = 1: a warp's,
// of L runs of the pass's bands in band-major order; R = 8: a CTA's, of L
// (group of 8 bands, run) units); the last range of a shared band adds its
// segments.  band0 is the first band of a
// row view within the matrix (its index is the matrix's).
struct Wz3Step {
  const uint64_t* index;  // the matrix's run index (BM_total x RB)
  const uint8_t* area;    // the block area
  int64_t band0;
  int64_t M, N, BM, BN, RB;
  const float* x;
  int64_t ldx;
  float* xt;  // scratch: (2G)^T x, 4 BN floats per right-hand side
  int R;      // 1 or 8
  int64_t L;      // R = 1: runs per warp range; R = 8: (group of 8 bands, run) units per CTA
  int maxseg;     // most ranges sharing one band
  int64_t ctas;   // grid size
  double* ws;     // BM x maxseg x R x 4 segment partials when maxseg > 1
  double* y;
  int64_t ldy;
  double* state;
  double decay;
  unsigned* seen;  // per band: counts the segments of the pass
};
int wz3_launch(const Wz3Step& a, cudaStream_t st);
int wz3_occupancy();  // resident CTAs per SM of the R = 1 kernel (0 on error)
int wz3_decompress(const uint64_t* index, const uint8_t* area, int64_t M, int64_t N, double* out, int64_t ldo,
                   cudaStream_t st);

template <int RATE>
int wz2_launch(const Wz2Step& a, cudaStream_t st);
template <int RATE>
int wz2_batched_launch(const Wz2Batch& b, cudaStream_t st);
template <int RATE>
int wz2_decompress(const uint8_t* stream, int64_t M, int64_t N, int64_t BN, int64_t nblocks, double* out,
                   int64_t ldo, bool lift, cudaStream_t st);
// resident CTAs per SM of the R = 1 kernel for the given unroll (0 on error)
template <int RATE>
int wz2_occupancy(bool lift, int unroll);
// resident CTAs per SM of the staged R = 1 kernel (0 on error)
template <int RATE>
int wz2_stream_occupancy(bool lift);

}  // namespace whff
