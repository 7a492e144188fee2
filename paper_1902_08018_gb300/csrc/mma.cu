// Tensor-core (tcgen05) launches for many right-hand sides: instantiation unit.
#include <algorithm>

#include "mma_kernels.cuh"
#include "wz2_dispatch.h"

namespace whff {

constexpr int kMaxMembers = 64;  // members of one batched tensor-core launch (their table sits in smem)

// Shared memory of a batch's kernel, which grows with its table: set for every launch.
// (Raised once for the largest table, the calls saved had a batch of ten matrices of 1024
// to 8192 take 200 us a pass among others instead of 192: the pace of the submissions
// matters there, a pause of the host in their place gave 192 as well.)
template <int RATE, bool LIFT, int NR>
static int mma_set_batch_smem(int bytes) {
  auto kern = dev::wz2_mma_kernel<RATE, LIFT, NR, true>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess ||
      cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) !=
          cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  return 0;
}

template <int RATE, bool LIFT, int NR>
static int mma_one(const MmaStep& a, cudaStream_t st) {
  using S = dev::MmaSmem<RATE, NR>;
  const int smem = S::kBytes;
  if (raise_smem<dev::wz2_mma_kernel<RATE, LIFT, NR, false>>(smem, true, a.device)) return -1;
  const int nstages = (int)((a.BN + dev::kMmaStageBlocks - 1) / dev::kMmaStageBlocks);
  const int tiles = (int)((a.BM + dev::kMmaBands - 1) / dev::kMmaBands);
  const dev::MmaMember mem{a.stream, a.btiles, a.ws, a.BM, a.BN, 0, nstages, tiles, a.R, a.maxseg, a.map, a.paired, a.band0};
  const dev::MmaPass pass{a.x, a.y, a.btiles, a.ws, a.ldx, a.ldy, a.N, a.M, 0, 0, 0, nstages, tiles, a.R, a.maxseg};
  const int64_t bthreads = (int64_t)nstages * dev::kMmaStageBlocks * NR;
  dev::wz2_mma_btiles<LIFT, NR><<<(unsigned)((bthreads + 255) / 256), 256, 0, st>>>(pass, nullptr, 1, bthreads);
  const int per = dev::mma_ranges_per_cta(a.ctas, a.sms, dev::kMmaRanges<RATE>);
  dev::wz2_mma_kernel<RATE, LIFT, NR, false><<<(unsigned)((a.ctas + per - 1) / per), dev::kMmaDecodeThreads, smem, st>>>(
      mem, nullptr, 1, (int64_t)tiles * nstages, a.L, per, a.status, a.spin);
  const int64_t fin_threads = (int64_t)tiles * a.R * 32;
  dev::wz2_mma_finish<LIFT><<<(unsigned)((fin_threads + 255) / 256), 256, 0, st>>>(pass, nullptr, 1, fin_threads,
                                                                                  a.L);
  if (a.state)
    dev::wz2_mma_state<<<(unsigned)((a.M + 255) / 256), 256, 0, st>>>(a.y, a.ldy, a.R, a.M, a.state, a.decay);
  return 0;
}

template <int RATE>
static int mma_rate(const MmaStep& a, cudaStream_t st) {
  const int nr = a.R <= 16 ? 16 : 32;
  if (a.lift) return nr == 16 ? mma_one<RATE, true, 16>(a, st) : mma_one<RATE, true, 32>(a, st);
  return nr == 16 ? mma_one<RATE, false, 16>(a, st) : mma_one<RATE, false, 32>(a, st);
}

// A batch's passes of one width class in one persistent launch: B tiles of
// every pass, the tensor-core kernel over the concatenated item sequence,
// every pass's finish (the states are the caller's).
template <int RATE, bool LIFT, int NR>
static int mma_batch_one(const MmaBatchStep& a, cudaStream_t st) {
  using S = dev::MmaSmem<RATE, NR>;
  const int smem = S::kBytes + a.nmem * (int)sizeof(dev::MmaMember);
  if (mma_set_batch_smem<RATE, LIFT, NR>(smem)) return -1;
  const dev::MmaMember m0{};
  const dev::MmaPass p0{};
  dev::wz2_mma_btiles<LIFT, NR><<<(unsigned)((a.bt_threads + 255) / 256), 256, 0, st>>>(p0, a.passes, a.nmem,
                                                                                       a.bt_threads);
  const int per = dev::mma_ranges_per_cta(a.ctas, a.sms, dev::kMmaRanges<RATE>);
  dev::wz2_mma_kernel<RATE, LIFT, NR, true><<<(unsigned)((a.ctas + per - 1) / per), dev::kMmaDecodeThreads, smem, st>>>(
      m0, a.members, a.nmem, a.total, a.L, per, a.status, a.spin);
  dev::wz2_mma_finish<LIFT><<<(unsigned)((a.fin_threads + 255) / 256), 256, 0, st>>>(p0, a.passes, a.nmem,
                                                                                    a.fin_threads, a.L);
  return 0;
}

template <int RATE>
static int mma_batch_rate(const MmaBatchStep& a, cudaStream_t st) {
  if (a.lift) return a.nr == 16 ? mma_batch_one<RATE, true, 16>(a, st) : mma_batch_one<RATE, true, 32>(a, st);
  return a.nr == 16 ? mma_batch_one<RATE, false, 16>(a, st) : mma_batch_one<RATE, false, 32>(a, st);
}

int mma_batch_launch(const MmaBatchStep& a, cudaStream_t st) {
  if ((a.nr != 16 && a.nr != 32) || a.nmem < 1 || a.nmem > kMaxMembers || a.ctas < 1 || a.L < 1) return -1;
  switch (a.rate) {
    case 8: return mma_batch_rate<8>(a, st);
    case 12: return mma_batch_rate<12>(a, st);
    case 16: return mma_batch_rate<16>(a, st);
    case 20: return mma_batch_rate<20>(a, st);
    case 24: return mma_batch_rate<24>(a, st);
    default: return -1;
  }
}

int mma_max_members() { return kMaxMembers; }

int mma_launch(const MmaStep& a, cudaStream_t st) {
  if (a.R < 1 || a.R > 32 || a.ctas < 1 || a.L < 1) return -1;
  switch (a.rate) {
    case 8: return mma_rate<8>(a, st);
    case 12: return mma_rate<12>(a, st);
    case 16: return mma_rate<16>(a, st);
    case 20: return mma_rate<20>(a, st);
    case 24: return mma_rate<24>(a, st);
    default: return -1;
  }
}

// Item ranges per SM of a pass (0 if the kernel cannot run here): one resident
// CTA takes them one after another.
template <int RATE, bool LIFT, int NR>
static int mma_occ_one() {
  cudaFuncAttributes fa;
  if (mma_set_batch_smem<RATE, LIFT, NR>(dev::MmaSmem<RATE, NR>::kBytes + kMaxMembers * (int)sizeof(dev::MmaMember)) ||
      cudaFuncGetAttributes(&fa, dev::wz2_mma_kernel<RATE, LIFT, NR, true>) != cudaSuccess ||
      fa.maxThreadsPerBlock < dev::kMmaDecodeThreads) {
    cudaGetLastError();
    return 0;
  }
  return dev::kMmaRanges<RATE>;
}

template <int RATE>
static int mma_occ_rate(bool lift, int nr) {
  if (lift) return nr <= 16 ? mma_occ_one<RATE, true, 16>() : mma_occ_one<RATE, true, 32>();
  return nr <= 16 ? mma_occ_one<RATE, false, 16>() : mma_occ_one<RATE, false, 32>();
}

int mma_occupancy(int rate, bool lift, int nr) {
  switch (rate) {
    case 8: return mma_occ_rate<8>(lift, nr);
    case 12: return mma_occ_rate<12>(lift, nr);
    case 16: return mma_occ_rate<16>(lift, nr);
    case 20: return mma_occ_rate<20>(lift, nr);
    case 24: return mma_occ_rate<24>(lift, nr);
    default: return 0;
  }
}

}  // namespace whff
