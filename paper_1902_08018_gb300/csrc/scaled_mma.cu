// Tensor-core (tcgen05) passes for the scaled formats: instantiation unit.
#include <algorithm>

#include <cudaTypedefs.h>

#include "scaled_mma.cuh"
#include "scaled_mma_fp8.cuh"
#include "scaled_mma_tma.cuh"
#include "wz2_dispatch.h"

namespace whff {

template <int FMT, int NR>
static int scaled_mma_one(const ScaledMmaStep& a, cudaStream_t st) {
  using S = dev::ScaledMmaSmem<FMT, NR>;
  auto kern = dev::scaled_mma_kernel<FMT, NR>;
  constexpr bool kF16 = FMT == 3;
  const bool tma = (FMT == 2 || FMT == 3) && a.tmap != nullptr;
  const bool fp8 = FMT == 4 && a.tmap != nullptr;
  if (fp8   ? raise_smem<dev::fp8_mma_kernel<NR>>(dev::Fp8Smem<NR>::kBytes, false, a.device)
      : tma ? raise_smem<dev::scaled_mma_tma_kernel<NR, kF16>>(dev::TmaSmem<NR>::kBytes, true, a.device)
            : raise_smem<dev::scaled_mma_kernel<FMT, NR>>(S::kBytes, true, a.device))
    return -1;
  const int nstages = (int)((a.N + 63) / 64);
  const int tiles = (int)((a.M + 127) / 128);
  const dev::MmaPass pass{a.x, a.y, a.btiles, a.ws, a.ldx, a.ldy, a.N, a.M, 0, 0, 0, nstages, tiles, a.R, a.maxseg};
  const int64_t bthreads = (int64_t)nstages * dev::kMmaStageBlocks * NR;
  const bool f16_pieces = tma && kF16;  // FP16 A by TMA: FP16 B pieces of x scaled per column
  if (f16_pieces) {
    dev::f16_colexp_kernel<<<(unsigned)NR, 256, 0, st>>>(a.x, a.ldx, a.N, a.R, a.colexp);
    dev::f16_mma_btiles<NR><<<(unsigned)((bthreads + 255) / 256), 256, 0, st>>>(pass, a.colexp, bthreads);
  } else {
    dev::wz2_mma_btiles<false, NR><<<(unsigned)((bthreads + 255) / 256), 256, 0, st>>>(pass, nullptr, 1, bthreads);
  }
  if (fp8) {
    const int per = dev::mma_ranges_per_cta(a.ctas, a.sms, dev::kFp8Ranges);
    dev::fp8_mma_kernel<NR><<<(unsigned)((a.ctas + per - 1) / per), dev::kMmaDecodeThreads, dev::Fp8Smem<NR>::kBytes, st>>>(
        *static_cast<const CUtensorMap*>(a.tmap), a.row0, a.scales, a.TN, a.btiles, a.ws, nstages, a.R, a.maxseg,
        (int64_t)tiles * nstages, a.L, per, a.status, a.spin);
  } else if (tma) {
    dev::scaled_mma_tma_kernel<NR, kF16><<<(unsigned)a.ctas, dev::kTmaThreads, dev::TmaSmem<NR>::kBytes, st>>>(
        *static_cast<const CUtensorMap*>(a.tmap), a.row0, a.scales, a.TN, a.btiles, a.ws, nstages, a.R, a.maxseg,
        (int64_t)tiles * nstages, a.L, a.status, a.spin);
  } else {
    kern<<<(unsigned)a.ctas, dev::kMmaThreads, S::kBytes, st>>>(a.payload, a.scales, a.M, a.ld, a.TN, a.btiles,
                                                                a.ws, nstages, a.R, a.maxseg,
                                                                (int64_t)tiles * nstages, a.L, a.status, a.spin);
  }
  const int64_t fin = (int64_t)tiles * a.R * 128;
  dev::scaled_mma_finish<<<(unsigned)((fin + 255) / 256), 256, 0, st>>>(a.ws, a.M, nstages, a.R, a.maxseg, tiles, a.L,
                                                                       a.y, a.ldy, f16_pieces ? a.colexp : nullptr);
  if (a.state)
    dev::wz2_mma_state<<<(unsigned)((a.M + 255) / 256), 256, 0, st>>>(a.y, a.ldy, a.R, a.M, a.state, a.decay);
  return 0;
}

template <int FMT>
static int scaled_mma_fmt(const ScaledMmaStep& a, cudaStream_t st) {
  return a.R <= 16 ? scaled_mma_one<FMT, 16>(a, st) : scaled_mma_one<FMT, 32>(a, st);
}

int scaled_mma_launch(const ScaledMmaStep& a, cudaStream_t st) {
  if (a.R < 1 || a.R > 32 || a.ctas < 1 || a.L < 1) return -1;
  switch (a.fmt) {
    case 2: return scaled_mma_fmt<2>(a, st);
    case 3: return scaled_mma_fmt<3>(a, st);
    case 4: return scaled_mma_fmt<4>(a, st);
    default: return -1;
  }
}

// Resident CTAs per SM from the kernel's registers, shared memory and TMEM
// columns (as for the fixed-allocation tensor-core kernel).
template <int FMT, int NR>
static int scaled_mma_occ_one() {
  using S = dev::ScaledMmaSmem<FMT, NR>;
  auto kern = dev::scaled_mma_kernel<FMT, NR>;
  cudaFuncAttributes fa;
  int dev = 0, smem_sm = 0, regs_sm = 0, reserved = 0;
  if (raise_smem<dev::scaled_mma_kernel<FMT, NR>>(S::kBytes, true) ||
      cudaFuncGetAttributes(&fa, kern) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const int warps = dev::kMmaThreads / 32;
  const int regs_warp = (fa.numRegs * 32 + 255) / 256 * 256;
  const int by_regs = regs_sm / (regs_warp * warps);
  const int by_smem = smem_sm / (S::kBytes + (int)fa.sharedSizeBytes + reserved);
  const int by_tmem = 512 / (int)dev::mma_tmem_cols<NR>();
  return std::min(std::min(by_regs, by_smem), by_tmem);
}

// Resident CTAs per SM of the TMA-fed kernel, from its registers, shared
// memory and TMEM columns (the occupancy API reported one CTA where two fit).
template <int NR, bool F16>
static int scaled_tma_occ_one() {
  auto kern = dev::scaled_mma_tma_kernel<NR, F16>;
  cudaFuncAttributes fa;
  int dev = 0, smem_sm = 0, regs_sm = 0, reserved = 0;
  if (raise_smem<dev::scaled_mma_tma_kernel<NR, F16>>(dev::TmaSmem<NR>::kBytes, true) ||
      cudaFuncGetAttributes(&fa, kern) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const int warps = dev::kTmaThreads / 32;
  const int regs_warp = (fa.numRegs * 32 + 255) / 256 * 256;
  const int by_regs = regs_sm / (regs_warp * warps);
  const int by_smem = smem_sm / (dev::TmaSmem<NR>::kBytes + (int)fa.sharedSizeBytes + reserved);
  const int by_tmem = 512 / (int)dev::mma_tmem_cols<NR>();
  return std::min(std::min(by_regs, by_smem), by_tmem);
}

int scaled_mma_occupancy(int fmt, bool tma) {
  switch (fmt) {
    case 2:
      return tma ? std::min(scaled_tma_occ_one<16, false>(), scaled_tma_occ_one<32, false>())
                 : std::min(scaled_mma_occ_one<2, 16>(), scaled_mma_occ_one<2, 32>());
    case 3:
      return tma ? std::min(scaled_tma_occ_one<16, true>(), scaled_tma_occ_one<32, true>())
                 : std::min(scaled_mma_occ_one<3, 16>(), scaled_mma_occ_one<3, 32>());
    case 4: return std::min(scaled_mma_occ_one<4, 16>(), scaled_mma_occ_one<4, 32>());
    default: return 0;
  }
}

}  // namespace whff

namespace whff {

static PFN_cuTensorMapEncodeTiled_v12000 tma_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
      cudaGetLastError();
      return nullptr;
    }
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  return encode;
}

int wz2_tma_map(void* out, const void* stream, int64_t BM, int64_t BN, int rate) {
  const auto encode = tma_encoder();
  const cuuint64_t words = (cuuint64_t)rate / 2, inner = (cuuint64_t)BN * words;
  if (!encode || inner >= (1ull << 31) - 2 || BM >= (1ll << 31)) return 0;
  const int maps = inner % 4 ? 2 : 1;
  for (int k = 0; k < maps; ++k) {
    const cuuint64_t rows = maps == 1 ? (cuuint64_t)BM : (cuuint64_t)(BM + 1 - k) / 2;
    const cuuint64_t dims[2] = {inner + 2 * k, rows ? rows : 1};
    const cuuint64_t strides[1] = {inner * 4 * maps};
    const cuuint32_t box[2] = {(cuuint32_t)(16 * words + (maps == 2 ? 4 : 0)), (cuuint32_t)(32 / maps)};
    const cuuint32_t estr[2] = {1, 1};
    // no odd band: an empty map is not encodable, and its one row is never wanted below BM
    const uint8_t* base = static_cast<const uint8_t*>(stream) + (k && rows ? inner * 4 - 8 : 0);
    if (encode(reinterpret_cast<CUtensorMap*>(static_cast<uint8_t*>(out) + 128 * k), CU_TENSOR_MAP_DATA_TYPE_UINT32, 2,
               const_cast<uint8_t*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return 0;
  }
  return maps;
}

int scaled_tma_map(void* out, const void* payload, int64_t M, int64_t ld, int fmt) {
  const auto encode = tma_encoder();
  if (!encode) return -1;
  const bool fp8 = fmt == 4;
  const cuuint64_t dims[2] = {(cuuint64_t)ld, (cuuint64_t)M};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * (fp8 ? 1 : 2)};  // bytes between rows (ld % 16 == 0)
  const cuuint32_t box[2] = {64, 128};                             // one stage: 64 columns x 128 rows
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode(static_cast<CUtensorMap*>(out),
                            fp8        ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                            : fmt == 3 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                       : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                            2, const_cast<void*>(payload), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            fp8 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : -1;
}

}  // namespace whff
