// decode_out.cuh -- FP64 results of the decode-only kernels, built and written
// without the FP64 pipe.
//
// GB300 retires about two FP64 operations per SM and clock, so a conversion and
// a multiply per entry (the obvious (double)t * scale) alone took 230 us on an
// 8192^2 matrix, more than twice its HBM time.  Every decoded entry is exact in
// FP64, so its bits are put together with integer instructions instead.
// A block's row is 32 bytes of the output: one 256-bit store per lane covers
// whole sectors, a warp's store 1 KB in a row; four 8-byte stores 32 bytes apart
// sent every sector to L2 four times.
// wz2_decompress_kernel at rate 16, 8192^2 (0.13 GB in, 0.54 GB out): 283 us with
// FP64 conversions and 8-byte stores, 110 us (6.1 TB/s) this way.
#pragma once
#include <cstdint>

namespace whff {
namespace dev {

// f * 2^e as FP64 bits (lo, hi): f a normal FP32 value or a zero, the result normal.
__device__ __forceinline__ uint2 f64_from_f32(float f, int e) {
  const uint32_t u = __float_as_uint(f), m = u & 0x7FFFFFFFu;
  const uint32_t hi = (u & 0x80000000u) | ((m >> 3) + ((uint32_t)(896 + e) << 20));
  return m ? make_uint2(u << 29, hi) : make_uint2(0u, u);
}

// t * 2^e as FP64 bits: |t| < 2^53, the result normal or zero.
__device__ __forceinline__ uint2 f64_from_int(int64_t t, int e) {
  const uint64_t a = (uint64_t)(t < 0 ? -t : t);
  if (!a) return make_uint2(0u, 0u);
  const int lz = __clzll((long long)a);
  const uint64_t m = a << lz;  // leading one at bit 63; (m >> 43) carries it into the exponent
  const uint32_t hi = ((uint32_t)(m >> 43) + ((uint32_t)(1085 - lz + e) << 20)) | (t < 0 ? 0x80000000u : 0u);
  return make_uint2((uint32_t)(m >> 11), hi);
}

// f * s as FP64 bits, exact (24 x 24 significant bits).  Values outside the
// normal FP32 range (and infinities, NaN) take the FP64 multiply.
__device__ __forceinline__ uint2 f64_product(float f, float s) {
  const uint32_t uf = __float_as_uint(f), us = __float_as_uint(s);
  const uint32_t ef = (uf >> 23) & 255u, es = (us >> 23) & 255u;
  const uint32_t sign = (uf ^ us) & 0x80000000u;
  if (es - 1u >= 254u || (ef - 1u >= 254u && (uf & 0x7FFFFFFFu))) {
    const double d = (double)s * (double)f;
    return make_uint2((uint32_t)__double2loint(d), (uint32_t)__double2hiint(d));
  }
  const uint64_t p = (uint64_t)((uf & 0x7FFFFFu) | 0x800000u) * ((us & 0x7FFFFFu) | 0x800000u);
  const uint32_t top = (uint32_t)(p >> 47);  // 1: the product of the significands is at least 2
  const uint64_t m = p << (6 - top);         // leading one at bit 52
  const uint32_t hi = sign | ((uint32_t)(m >> 32) + ((ef + es + 768u + top) << 20));
  return (uf & 0x7FFFFFFFu) ? make_uint2((uint32_t)m, hi) : make_uint2(0u, sign);
}

__device__ __forceinline__ double f64_of(uint2 v) { return __hiloint2double((int)v.y, (int)v.x); }

// Four values to a 32-byte aligned address, one 256-bit store.
__device__ __forceinline__ void store_f64x4(double* p, uint2 a, uint2 b, uint2 c, uint2 d) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};\n" ::"l"(p), "d"(f64_of(a)), "d"(f64_of(b)), "d"(f64_of(c)),
               "d"(f64_of(d))
               : "memory");
}

// Each lane holds ROWS x W consecutive values, d[r * W + c], of unit j of
// line i (units of W columns, U to a line; consecutive lanes hold consecutive
// units, the next line's after the last one).  VEC: the output takes 32-byte
// stores (aligned, leading dimension a multiple of 4).  Otherwise the warp
// turns its values round in `sm` (ROWS x W x 32 doubles of its own) and writes
// each row's run of values with the lanes side by side, whatever its alignment.
// All 32 lanes call it; live = the lane holds a unit (the first lanes do).
template <bool VEC, int ROWS, int W>
__device__ __forceinline__ void store_units(const uint2 (&d)[ROWS * W], bool live, int64_t i, int64_t j, int64_t U,
                                            int64_t M, int64_t N, double* __restrict__ out, int64_t ldo, double* sm) {
  static_assert(W % 4 == 0, "whole 32-byte stores");
  if constexpr (VEC) {
    if (!live) return;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const int64_t row = (int64_t)ROWS * i + r;
      if (row >= M) break;
      double* p = out + row * ldo + W * j;
#pragma unroll
      for (int c = 0; c < W; c += 4) {
        if (W * j + c + 3 < N) {
          store_f64x4(p + c, d[r * W + c], d[r * W + c + 1], d[r * W + c + 2], d[r * W + c + 3]);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (W * j + c + q < N) p[c + q] = f64_of(d[r * W + c + q]);
        }
      }
    }
  } else {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
      for (int c = 0; c < W; ++c) sm[(r * 32 + lane) * W + c] = f64_of(d[r * W + c]);
    const int64_t i0 = __shfl_sync(0xFFFFFFFFu, i, 0), j0 = __shfl_sync(0xFFFFFFFFu, j, 0);
    const int n = __popc(__ballot_sync(0xFFFFFFFFu, live));
    __syncwarp();
#pragma unroll 1
    for (int k = 0; k < W; ++k) {
      const int q = 32 * k + lane, owner = q / W;
      if (owner >= n) continue;
      int64_t ii = i0, jj = j0 + owner;
      while (jj >= U) jj -= U, ++ii;
      const int64_t col = W * jj + q % W;
      if (col >= N) continue;
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        const int64_t row = (int64_t)ROWS * ii + r;
        if (row < M) out[row * ldo + col] = sm[r * 32 * W + q];
      }
    }
  }
}

// Whether an FP64 output takes 32-byte stores.
inline bool out_vec_ok(const double* out, int64_t ldo) {
  return reinterpret_cast<uintptr_t>(out) % 32 == 0 && ldo % 4 == 0;
}

// Line and unit of linear unit b, U units to a line.
__device__ __forceinline__ void unit_of(int64_t b, int64_t U, int64_t& i, int64_t& j) {
  if ((b | U) >> 32) {
    i = b / U;
  } else {
    i = (uint32_t)b / (uint32_t)U;
  }
  j = b - i * U;
}

}  // namespace dev
}  // namespace whff
