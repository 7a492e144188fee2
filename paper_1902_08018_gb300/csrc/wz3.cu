// Fixed-accuracy (WZ3) launches: instantiation unit.
#include "wz2_dispatch.h"
#include "wz3_kernels.cuh"

namespace whff {

int wz3_launch(const Wz3Step& a, cudaStream_t st) {
  if (a.R != 1 && a.R != 8) return -1;
  // (2G)^T x once per pass, 4 BN floats per right-hand side
  const uint64_t* index = a.index + a.band0 * a.RB;  // the view's first band
  const unsigned threads = dev::kWarpsPerCta * 32;
  if (a.R == 8) {
    dev::wz3_xt8_kernel<<<(unsigned)a.RB, 256, 0, st>>>(a.x, a.ldx, a.N, a.RB, a.xt);
    dev::wz3_gemv8_kernel<<<(unsigned)a.ctas, threads, 0, st>>>(index, a.area, a.M, a.BM, (int)a.BN, (int)a.RB, a.xt,
                                                                a.L, a.maxseg, a.ws, a.y, a.ldy, a.state, a.decay, a.seen);
    return 0;
  }
  dev::wz2_xt_kernel<<<(unsigned)((a.BN + 255) / 256), 256, 0, st>>>(a.x, a.ldx, a.N, 1, a.BN, a.xt, 4 * a.BN);
  dev::wz3_gemv_kernel<<<(unsigned)a.ctas, threads, 0, st>>>(index, a.area, a.M, a.BM, (int)a.BN, (int)a.RB, a.xt,
                                                                a.L, a.maxseg, a.ws, a.y, a.ldy, a.state, a.decay, a.seen);
  return 0;
}

int wz3_occupancy() {
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, dev::wz3_gemv_kernel, dev::kWarpsPerCta * 32, 0) !=
      cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return occ;
}

int wz3_decompress(const uint64_t* index, const uint8_t* area, int64_t M, int64_t N, double* out, int64_t ldo,
                   cudaStream_t st) {
  const int64_t BM = (M + 3) / 4, BN = (N + 3) / 4, RB = (BN + 31) / 32, nb = BM * BN;
  auto kern = dev::out_vec_ok(out, ldo) ? &dev::wz3_decompress_kernel<true> : &dev::wz3_decompress_kernel<false>;
  kern<<<(unsigned)((nb + 255) / 256), 256, 0, st>>>(index, area, M, N, BN, RB, nb, out, ldo);
  return 0;
}

}  // namespace whff
