// gemv_kernels.cuh -- the fused decode + GEMV kernels of the control step and
// their FP64 epilogue (Sec. 4.4: FP32 products, FP64 reduction; Sec. 2.1:
// carried state), plus the decode-only kernels (Sec. 5.2).
//
// Work split (WZ1): one warp owns one 4-row band of A (one block row) over a
// column range; lanes take consecutive 4x4 blocks, so a warp streams one
// contiguous run of the compressed stream per iteration.  (The fixed-
// allocation and scaled formats use the persistent range schedule of
// wz2_kernels.cuh / scaled_kernels.cuh.)  Each lane keeps compensated FP32 sums
// (TwoSum: hi + lo) per row and right-hand side; the warp folds them with
// shuffles (fold.cuh) and widens the totals.  With one column range per band the warp finishes y and the
// state itself; with several (split-K, for wide matrices whose few rows
// cannot fill the GPU -- the cuBLAS failure mode of Sec. 5.1) the FP64
// partials go to a workspace and a second kernel sums them in split order.
#pragma once
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <cstdint>

#include "decode_out.cuh"
#include "fold.cuh"
#include "wz1_decode.cuh"

namespace whff {
namespace dev {

constexpr int kWarpsPerCta = 8;

__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float p) {
  const float s = hi + p;
  const float bp = s - hi;
  const float err = (hi - (s - bp)) + (p - bp);
  hi = s;
  lo += err;
}

// The band of values z (value k of the fold: column k / 4, row k % 4) that a lane
// holds, written to y, the state (column by column) or the partials.
// MIX 1: the lift's 2G mixing of a column's four rows and 2^-3; MIX 2: 2^3 (no
// transform); MIX 0: as they are.  All 32 lanes call it; `lane` is the lane in
// its group of GL.
//   part != nullptr: value k goes to part[k] (mixed): a segment of a shared band;
//   else row i of the band is row row0 + i of y (and of the state), below M.
//   active = false: a group without a piece writes nothing.
template <int MIX, int R, int GL>
__device__ __forceinline__ void band_write(double (&z)[4 * R >= GL ? 4 * R / GL : 1], int lane, int64_t row0, int64_t M,
                                           double* __restrict__ part, double* __restrict__ y, int64_t ldy,
                                           double* __restrict__ state, double decay, bool active) {
  constexpr unsigned kAll = 0xFFFFFFFFu;
  constexpr int N = 4 * R;
  constexpr int C = N >= GL ? N / GL : 1;  // values per lane
  constexpr int S = N >= GL ? 1 : GL / N;  // lanes per value
  const int first = fold_index<N, GL>(lane), base = (threadIdx.x & 31) - lane;
  // the value k of the group: lane k / C * S holds it
  auto from = [&](int k, int own) { return __shfl_sync(kAll, z[own], base + k / C * S); };
  if (MIX == 1) {  // y = (2G) z * 2^-3, 2G rows (2,-1,-1,0), (2,-1,1,0), (2,1,-1,-1), (2,1,1,1)
    double t[C];
    const int q = first & ~3;
    if constexpr (C >= 4) {  // whole columns in the lane
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const int i = c & 3, b = c & ~3;
        double v = times_pow2(z[b], 1);
        v = i < 2 ? v - z[b + 1] : v + z[b + 1];
        v = i & 1 ? v + z[b + 2] : v - z[b + 2];
        if (i >= 2) v = i == 2 ? v - z[b + 3] : v + z[b + 3];
        t[c] = times_pow2(v, -3);
      }
    } else {
      const double z0 = from(q, 0), z1 = from(q + 1, C == 2 ? 1 : 0), z2 = from(q + 2, 0),
                   z3 = from(q + 3, C == 2 ? 1 : 0);
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const int i = (first + c) & 3;
        double v = times_pow2(z0, 1) + negate_if(z1, i < 2);
        v += negate_if(z2, !(i & 1));
        v += i < 2 ? 0.0 : negate_if(z3, i == 2);
        t[c] = times_pow2(v, -3);
      }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) z[c] = t[c];
  } else if (MIX == 2) {
#pragma unroll
    for (int c = 0; c < C; ++c) z[c] = times_pow2(z[c], 3);
  }
  const bool writer = active && lane % S == 0;
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const int k = first + c;
    const int64_t row = row0 + (k & 3);
    if (!writer) continue;
    if (part) part[k] = z[c];
    else if (row < M) y[(int64_t)(k >> 2) * ldy + row] = z[c];
  }
  if (state != nullptr) {
    if constexpr (R == 1) {
      const int64_t row = row0 + (first & 3);
      if (writer && !part && row < M) state[row] = decay * state[row] + z[0];
    } else {  // lane i of the group gathers row i's columns in order
      const int i = lane & 3;
      const int64_t row = row0 + i;
      const bool mine = active && !part && lane < 4 && row < M;
      double s = mine ? state[row] : 0.0;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        double v;
        if constexpr (C == 1) v = from(4 * r + i, 0);
        else if constexpr (C == 2) {
          const double a = from(4 * r + i, 0), b = from(4 * r + i, 1);
          v = i & 1 ? b : a;
        } else {
          v = 0.0;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const double a = from(4 * r + c, c);
            if (i == c) v = a;
          }
        }
        s = decay * s + v;
      }
      if (mine) state[row] = s;
    }
  }
}

// Fold a lane's (hi, lo) sums for 4 rows x R columns over its group of GL lanes
// (fold.cuh) and write them.  red32: the FP32 pair fold, else the triple one.
template <int MIX, int R, int GL = 32>
__device__ __forceinline__ void band_finish(const float (&hi)[4][R], const float (&lo)[4][R], int lane, int64_t row0,
                                            int64_t M, double* __restrict__ part, double* __restrict__ y, int64_t ldy,
                                            double* __restrict__ state, double decay, bool red32, bool active = true) {
  constexpr int N = 4 * R;
  if constexpr (R > 1) asm volatile("" : "+r"(lane));  // the fold's lane constants stay out of the caller's loops
  float h[N], l[N];
#pragma unroll
  for (int k = 0; k < N; ++k) h[k] = hi[k & 3][k >> 2], l[k] = lo[k & 3][k >> 2];
  double z[N >= GL ? N / GL : 1];
  if (red32) fold_lanes<N, GL, false>(h, l, lane, z);
  else fold_lanes<N, GL, true>(h, l, lane, z);
  band_write<MIX, R, GL>(z, lane, row0, M, part, y, ldy, state, decay, active);
}

// a / b for non-negative operands, in 32 bits where they fit.
__device__ __forceinline__ int64_t div64(int64_t a, int64_t b) {
  return ((uint64_t)a | (uint64_t)b) >> 32 ? a / b : (int64_t)((uint32_t)a / (uint32_t)b);
}

// x[4J .. 4J+3] of column r, zero beyond N.
__device__ __forceinline__ float4 load_x4(const float* __restrict__ x, int64_t ldx, int r, int64_t c0, int64_t N,
                                          bool vec_ok) {
  const float* p = x + (int64_t)r * ldx + c0;
  if (vec_ok && c0 + 3 < N) return __ldg(reinterpret_cast<const float4*>(p));
  float4 v;
  v.x = c0 < N ? __ldg(p) : 0.f;
  v.y = c0 + 1 < N ? __ldg(p + 1) : 0.f;
  v.z = c0 + 2 < N ? __ldg(p + 2) : 0.f;
  v.w = c0 + 3 < N ? __ldg(p + 3) : 0.f;
  return v;
}

// --------------------------------------------------------------- WZ1 GEMV
// Four warps to a block of the embedded coder's kernels: the SMs' shares of a
// grid differ by less than with eight (10000^2 in three splits: 12.4 blocks per
// SM, not 6.2), 36 warps fit an SM, and rate 64 fits 48 KB of shared memory.
// wz1_gemv_kernel, rate 16, 10000^2 (0.2 GB), one column: 451 us with a group
// test per iteration; 268 us with table lookups; 241 us with whole planes two at
// a time and four-warp blocks.  1026 warp instructions per 32 blocks, bound by
// the integer pipe (74 % busy): the parse about half of them, the bit transpose,
// lift and products the rest.
constexpr int kWz1Threads = 128;
template <int NW32, int R>
__global__ void __launch_bounds__(kWz1Threads)
    wz1_gemv_kernel(const uint8_t* __restrict__ stream, int64_t M, int64_t N, int64_t BM, int64_t BN,
                    const float* __restrict__ x, int64_t ldx, bool x_vec_ok, int ksplit, int64_t jchunk,
                    double* __restrict__ ws, double* __restrict__ y, int64_t ldy, double* __restrict__ state,
                    double decay) {
  __shared__ Wz1Smem<NW32, kWz1Threads> sm;
  wz1_smem_init(sm);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t I = (int64_t)blockIdx.x * (kWz1Threads / 32) + warp;
  if (I >= BM) return;  // whole warp
  const int split = blockIdx.y;
  const int64_t J0 = (int64_t)split * jchunk;
  const int64_t J1 = min(BN, J0 + jchunk);

  float hi[4][R], lo[4][R];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int r = 0; r < R; ++r) hi[i][r] = lo[i][r] = 0.f;

  const int64_t rowblk = I * BN;
  uint32_t next[NW32];
  if (J0 + lane < J1) load_block<NW32>(stream, rowblk + J0 + lane, next);
  for (int64_t J = J0 + lane; J < J1; J += 32) {
    uint32_t w[NW32];
#pragma unroll
    for (int i = 0; i < NW32; ++i) w[i] = next[i];
    if (J + 32 < J1) load_block<NW32>(stream, rowblk + J + 32, next);  // on its way while this one is decoded
    int32_t q[16];
    int emax;
    const bool nz = decode_block(w, sm, q, emax);
    if (!nz) continue;
    const float scale = __int_as_float((emax - 26 + 127) << 23);  // 2^(emax-26), a normal float
    float a[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = __int2float_rn(q[i]);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float4 xv = load_x4(x, ldx, r, 4 * J, N, x_vec_ok);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float p = a[4 * i] * xv.x;
        p = fmaf(a[4 * i + 1], xv.y, p);
        p = fmaf(a[4 * i + 2], xv.z, p);
        p = fmaf(a[4 * i + 3], xv.w, p);
        two_sum_acc(hi[i][r], lo[i][r], p * scale);
      }
    }
  }
  // several splits: the partial of column r, row i goes to ws[(split R + r) Mpad + i]; a column's
  // rows are then consecutive, as in y
  const bool part = ksplit > 1;
  band_finish<0, R>(hi, lo, lane, 4 * I, part ? 4 * BM : M, nullptr, part ? ws + (int64_t)split * R * 4 * BM : y,
                    part ? 4 * BM : ldy, part ? nullptr : state, decay, false);
}

// ------------------------------------------------------- scaled-format GEMV
// Element decode: FMT 2 = BF16, 3 = FP16, 4 = FP8 E4M3.  A lane reads 16
// bytes: V = 8 (16-bit) or 16 (8-bit) consecutive elements of one row.
template <int FMT>
struct ScaledTraits;
template <>
struct ScaledTraits<2> {
  static constexpr int V = 8;
  __device__ static __forceinline__ void decode(uint4 raw, float (&f)[8]) {
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
  }
};
template <>
struct ScaledTraits<3> {
  static constexpr int V = 8;
  __device__ static __forceinline__ void decode(uint4 raw, float (&f)[8]) {
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      __half2_raw hr;
      hr.x = (unsigned short)(w[i] & 0xFFFF);
      hr.y = (unsigned short)(w[i] >> 16);
      const float2 v = __half22float2(__half2(hr));
      f[2 * i] = v.x;
      f[2 * i + 1] = v.y;
    }
  }
};
template <>
struct ScaledTraits<4> {
  static constexpr int V = 16;
  __device__ static __forceinline__ void decode(uint4 raw, float (&f)[16]) {
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __half2_raw lo = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(w[i] & 0xFFFF), __NV_E4M3);
      const __half2_raw hi = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(w[i] >> 16), __NV_E4M3);
      const float2 a = __half22float2(__half2(lo));
      const float2 b = __half22float2(__half2(hi));
      f[4 * i] = a.x;
      f[4 * i + 1] = a.y;
      f[4 * i + 2] = b.x;
      f[4 * i + 3] = b.y;
    }
  }
};

// FP32 storage (the uncompressed comparison): four values per 16 bytes.
template <>
struct ScaledTraits<7> {
  static constexpr int V = 4;
  __device__ static __forceinline__ void decode(uint4 raw, float (&f)[4]) {
    f[0] = __uint_as_float(raw.x);
    f[1] = __uint_as_float(raw.y);
    f[2] = __uint_as_float(raw.z);
    f[3] = __uint_as_float(raw.w);
  }
};

// bytes per element of a scaled format
template <int FMT>
__host__ __device__ constexpr int scaled_elem_bytes() {
  return FMT == 4 ? 1 : FMT == 7 ? 4 : 2;
}

// --------------------------------------------------- split-K epilogue (FP64)
static __global__ void splitk_epilogue_kernel(const double* __restrict__ ws, int ksplit, int R, int64_t Mpad, int64_t M,
                                       double* __restrict__ y, int64_t ldy, double* __restrict__ state,
                                       double decay) {
  const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= M) return;
  double s = state ? state[row] : 0.0;
  for (int r = 0; r < R; ++r) {
    double t = 0.0;
    for (int k = 0; k < ksplit; ++k) t += ws[((int64_t)k * R + r) * Mpad + row];
    y[(int64_t)r * ldy + row] = t;
    s = decay * s + t;
  }
  if (state) state[row] = s;
}

// ------------------------------------------------------------- decode only
// Thread per block (WZ1) or per 16-byte chunk (scaled); results as decode_out.cuh says.
template <int NW32, bool VEC>
__global__ void __launch_bounds__(kWz1Threads)
    wz1_decompress_kernel(const uint8_t* __restrict__ stream, int64_t M, int64_t N, int64_t BN, int64_t nblocks,
                          double* __restrict__ out, int64_t ldo) {
  using Smem = Wz1Smem<NW32, kWz1Threads>;
  __shared__ __align__(16) Smem sm;
  static_assert(sizeof(Smem) >= (kWz1Threads / 32) * 512 * 8, "turns the rows round: 4 x 128 doubles a warp");
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = b < nblocks;
  int64_t I = 0, J = 0;
  unit_of(live ? b : nblocks - 1, BN, I, J);
  uint32_t w[NW32];
  load_block<NW32>(stream, live ? b : nblocks - 1, w);
  wz1_smem_init(sm);  // while the words are on their way
  int32_t q[16];
  int emax;
  const bool nz = decode_block(w, sm, q, emax);
  uint2 d[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) d[k] = nz ? f64_from_f32(__int2float_rn(q[k]), emax - 26) : make_uint2(0u, 0u);
  if constexpr (!VEC) __syncthreads();  // the decoder's words have been read
  store_units<VEC, 4, 4>(d, live, I, J, BN, M, N, out, ldo, reinterpret_cast<double*>(&sm) + (threadIdx.x >> 5) * 512);
}

template <int FMT, bool VEC>
__global__ void __launch_bounds__(256)
    scaled_decompress_kernel(const uint8_t* __restrict__ payload, const float* __restrict__ scales, int64_t M,
                             int64_t N, int64_t ld, int64_t TN, double* __restrict__ out, int64_t ldo) {
  using T = ScaledTraits<FMT>;
  constexpr int V = T::V;
  constexpr int EB = scaled_elem_bytes<FMT>();
  __shared__ double turn[VEC ? 1 : 8 * 32 * V];
  const int64_t chunks_per_row = ld / V;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = t < M * chunks_per_row;
  int64_t row = 0, j = 0;
  unit_of(live ? t : M * chunks_per_row - 1, chunks_per_row, row, j);
  const int64_t c = j * V;
  const uint4 raw = __ldcs(reinterpret_cast<const uint4*>(payload + ((uint64_t)row * ld + c) * EB));
  float f[V];
  T::decode(raw, f);
  const float s = __ldg(scales + (row / 128) * TN + c / 128);
  uint2 d[V];
#pragma unroll
  for (int v = 0; v < V; ++v) d[v] = f64_product(f[v], s);
  store_units<VEC, 1, V>(d, live, row, j, chunks_per_row, M, N, out, ldo,
                         turn + (VEC ? 0 : (threadIdx.x >> 5) * 32 * V));
}

}  // namespace dev
}  // namespace whff
