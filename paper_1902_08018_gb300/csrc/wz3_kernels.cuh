// wz3_kernels.cuh -- zfp's fixed-accuracy mode read GPU-first ("WZ3"):
// decode and fused decode + GEMV kernels.
//
// A WZ3 matrix keeps WZ2's blocks (block exponent, shift K, lifted
// coefficients in sequency order, offset-binary fields) but chooses K per
// block for an absolute tolerance and one field width W per run of up to 32
// blocks of a band.  A run is exactly what one warp takes in one iteration:
// lane l decodes block 32 run + l, and since W is the same for the whole run
// the warp switches once, uniformly, onto a field extractor compiled for that
// width (no per-lane prefix sums, no dynamic register indexing).  The run's
// first byte comes from one index entry (offset | W << 56) that every lane
// reads, and its words are interleaved across its blocks (word k of block b
// at word k nb + b), so each of the warp's loads is one coalesced sweep.
// As for WZ2 with the lift, the product works in the transform domain:
// y_band = (2G) sum_J s_J V_J ((2G)^T x_J) 2^-3 with s_J = 2^(E+K-154), the
// (2G) mixing once per band in FP64 (band_finish with the lift's mix).
#pragma once
#include <cstdint>

#include "wz2_kernels.cuh"

namespace whff {
namespace dev {

__host__ __device__ constexpr int wz3_block_bytes(int W) { return 8 * ((13 + 16 * W + 63) / 64); }

template <int W>
struct Wz3Layout {
  static constexpr int kWords = wz3_block_bytes(W) / 4;  // 32-bit words of a block
  static constexpr uint32_t kMask = (1u << W) - 1u;
  static_assert(W >= 1 && W <= 31, "WZ3 field widths are 1..31");
};

template <int W, int K, int NW>
__device__ __forceinline__ uint32_t wz3_field(const uint32_t (&w)[NW]) {
  constexpr int off = 13 + W * K;
  constexpr int wi = off / 32, sh = off % 32;
  if constexpr (sh + W <= 32) {
    return (w[wi] >> sh) & Wz3Layout<W>::kMask;
  } else {
    return __funnelshift_r(w[wi], w[wi + 1], sh) & Wz3Layout<W>::kMask;
  }
}

// The 16 fields of a width-W block, placed in block order (t[4 i + j] for
// coefficient (i, j)): up to 23 bits already OR'd into the mantissa of 2^23
// (so that one packed subtraction of 2^23 + 2^(W-1) gives the exact value),
// wider ones raw.  Only this part depends on W at compile time, so the code a
// run's width selects stays small.
template <int W, int... Ks>
__device__ __forceinline__ void wz3_fields_to(const uint32_t (&w)[16], uint32_t (&t)[16],
                                              std::integer_sequence<int, Ks...>) {
  constexpr uint32_t kOr = W <= 23 ? 0x4B000000u : 0u;
  ((t[seq_index(Ks)] = wz3_field<W, Ks>(w) | kOr), ...);
}

// Fields for the run's width W (1..31), a switch that is uniform over the warp.
__device__ __forceinline__ void wz3_fields_w(int W, const uint32_t (&w)[16], uint32_t (&t)[16]) {
  switch (W) {
#define WZ3_F(WW) \
  case WW:        \
    wz3_fields_to<WW>(w, t, std::make_integer_sequence<int, 16>{}); \
    break;
    WZ3_F(1) WZ3_F(2) WZ3_F(3) WZ3_F(4) WZ3_F(5) WZ3_F(6) WZ3_F(7) WZ3_F(8) WZ3_F(9) WZ3_F(10) WZ3_F(11) WZ3_F(12)
    WZ3_F(13) WZ3_F(14) WZ3_F(15) WZ3_F(16) WZ3_F(17) WZ3_F(18) WZ3_F(19) WZ3_F(20) WZ3_F(21) WZ3_F(22) WZ3_F(23)
    WZ3_F(24) WZ3_F(25) WZ3_F(26) WZ3_F(27) WZ3_F(28) WZ3_F(29) WZ3_F(30)
    default:  // 31 (wider runs are refused when the matrix is made resident)
      wz3_fields_to<31>(w, t, std::make_integer_sequence<int, 16>{});
#undef WZ3_F
  }
}

// The lane's block of a run of nb blocks (word-interleaved: word k of block
// b at word k nb + b of the run), so that each load instruction of the warp
// reads 8 nb consecutive bytes.  An idle lane (past the band's end) and every
// lane of a zero run load nothing.
__device__ __forceinline__ void wz3_load_run(const uint8_t* __restrict__ area, uint64_t e, int lane, int nb,
                                             bool active, uint32_t (&w)[16]) {
  const int W = (int)(e >> 56);
  const int nw = wz3_block_bytes(W) / 8;  // 64-bit words of a block (uniform over the warp)
  const uint2* p = reinterpret_cast<const uint2*>(area + (e & 0x00FFFFFFFFFFFFFFull)) + lane;
  if (nb == 32) {  // a whole run: constant offsets
    if (W != 0) {
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k < nw) {
          const uint2 v = __ldcs(p + k * 32);
          w[2 * k] = v.x;
          w[2 * k + 1] = v.y;
        }
    }
  } else if (active && W != 0) {
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < nw) {
        const uint2 v = __ldcs(p + k * nb);
        w[2 * k] = v.x;
        w[2 * k + 1] = v.y;
      }
  }
}

// A block's products added into the lane's sums (one column): p_i = s * sum_b
// V[i][b] xt[b] (xt the transformed x of the block's column chunk J), then
// hi/lo[i][0] += p_i by TwoSum.  Rows
// (0, 1) and (2, 3) go in packed FP32 pairs; each half rounds as the scalar
// chain (product, three FMAs in b order, the scale, TwoSum) would.
// wz3_values gives V[h][b] = (value (2h, b), value (2h + 1, b)) and s.
__device__ __forceinline__ void wz3_values(const uint32_t (&w)[16], int W, float2 (&V)[2][4], float& s) {
  uint32_t t[16];
  wz3_fields_w(W, w, t);
  // exact: (2^23 + field) - (2^23 + 2^(W-1))
  float bias = 8388608.0f + (float)(1u << (W - 1));
  if (W > 23) {  // the integer conversion, round to nearest
    const uint32_t half = 1u << (W - 1);
    bias = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) t[k] = __float_as_uint(__int2float_rn((int32_t)(t[k] - half)));
  }
  const float2 b2 = make_float2(bias, bias);
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int b = 0; b < 4; ++b)
      V[h][b] = sub_f2(make_float2(__uint_as_float(t[8 * h + b]), __uint_as_float(t[8 * h + 4 + b])), b2);
  const uint32_t E = w[0] & 0xFFu, K = (w[0] >> 8) & 31u;
  s = E ? __uint_as_float((E + K - 27u) << 23) : 0.f;  // 2^(E+K-154); E >= 28 for a nonzero block
}

__device__ __forceinline__ void wz3_accumulate(const float2 (&V)[2][4], float s, const float* __restrict__ xt, int J,
                                               float (&hi)[4][1], float (&lo)[4][1]) {
  const float2 s2 = make_float2(s, s);
  const float4 x = __ldg(reinterpret_cast<const float4*>(xt + 4 * J));
  const float2 x0 = make_float2(x.x, x.x), x1 = make_float2(x.y, x.y), x2 = make_float2(x.z, x.z),
               x3 = make_float2(x.w, x.w);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float2 q = mul_f2(V[h][0], x0);
    q = fma_f2(V[h][1], x1, q);
    q = fma_f2(V[h][2], x2, q);
    q = fma_f2(V[h][3], x3, q);
    float2 H = make_float2(hi[2 * h][0], hi[2 * h + 1][0]), Lo = make_float2(lo[2 * h][0], lo[2 * h + 1][0]);
    two_sum_acc2(H, Lo, mul_f2(q, s2));
    hi[2 * h][0] = H.x, hi[2 * h + 1][0] = H.y, lo[2 * h][0] = Lo.x, lo[2 * h + 1][0] = Lo.y;
  }
}

// Persistent warp ranges over the runs in band-major order (units = runs):
// warp g takes runs [g L, (g + 1) L) of the pass's bands, band I of the pass
// being band0 + I of the matrix (index points at band0's first entry).  A
// band whose runs all lie in the range is finished here (y, state); a band
// shared by several ranges leaves one FP64 partial per range in
// ws[I maxseg + seg][4], which its last warp adds up.  The index entry of
// the next run is read while the lanes decode the current one.  One column.
static __global__ void __launch_bounds__(kWarpsPerCta * 32, 4)
    wz3_gemv_kernel(const uint64_t* __restrict__ index, const uint8_t* __restrict__ area, int64_t M, int64_t BM,
                    int BN, int RB, const float* __restrict__ xt, int64_t L, int maxseg,
                    double* __restrict__ ws, double* __restrict__ y, int64_t ldy, double* __restrict__ state,
                    double decay, unsigned* __restrict__ seen) {
  const int lane = threadIdx.x & 31;
  const int64_t g = (int64_t)blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5);
  const int64_t total = BM * RB;
  const int64_t u0 = g * L, u1 = min(total, u0 + L);
  if (u0 >= u1) return;  // warp-uniform; nothing below synchronises across warps
  int64_t I = u0 / RB;  // band of the current piece
  float hi[4][1], lo[4][1];
#pragma unroll
  for (int i = 0; i < 4; ++i) hi[i][0] = lo[i][0] = 0.f;
  uint64_t e_nxt = __ldg(index + u0);  // the same word for every lane
  for (int64_t ub = u0; ub < u1;) {  // the range's piece of band I: runs [ub, ue)
    const int64_t ue = min(u1, (I + 1) * RB);
#pragma unroll 1
    for (int64_t u = ub; u < ue; ++u) {
      const uint64_t e = e_nxt;
      if (u + 1 < u1) e_nxt = __ldg(index + u + 1);
      const int q = (int)(u - I * RB);  // run within the band
      const int nb = min(32, BN - 32 * q);
      const int W = (int)(e >> 56);
      uint32_t w[16];
      wz3_load_run(area, e, lane, nb, lane < nb, w);
      if (W != 0 && lane < nb) {  // a zero run adds 0
        float2 V[2][4];
        float s;
        wz3_values(w, W, V, s);
        wz3_accumulate(V, s, xt, 32 * q + lane, hi, lo);
      }
    }
    const int64_t g_lo = div64(I * RB, L), g_hi = div64((I + 1) * RB - 1, L);
    const bool shared = g_lo != g_hi;
    band_finish<1, 1>(hi, lo, lane, 4 * I, M, shared ? ws + (I * maxseg + (g - g_lo)) * 4 : nullptr, y, ldy, state,
                      decay, false);
    if (shared)
      finish_shared_band(seen, ws, I, M, (int)(g - g_lo), (int)(g_hi - g_lo + 1), maxseg, 1, y, ldy, state, decay);
#pragma unroll
    for (int i = 0; i < 4; ++i) hi[i][0] = lo[i][0] = 0.f;
    ++I;
    ub = ue;
  }
}

// Eight right-hand sides: the x of a block is 128 bytes, three times its stored
// bits, so what x costs decides.  The eight warps of a CTA take the same runs of
// eight neighbouring bands side by side and share the x chunks through L1; with
// a range of one band after another to each warp every x chunk came from L2
// (8.6 GB a pass at 32768^2).  CTA c takes units [c L, c L + L) of the sequence
// (group of 8 bands, run), group-major; warp w the group's band w.
// The chain of a row takes scalar FMAs (their operands need no doubling into
// pairs; a packed instruction takes two issue cycles of the FMA pipe anyway), the
// TwoSum packed ones on rows 2h and 2h + 1.
// The 32 sums of a band (r, i) are folded over the lanes as triples
// (fold.cuh), lane 4 r + i ending with that of row i and column r: FP64 butterflies cost
// 2600 cycles of GB300's FP64 pipe per band piece.  Pairs would take 3 us less of a
// pass, and give up digits that FP64 kept.
// 8192^2 at 1e-7 (0.18 GB, one pass of 8 columns): 269 us and 12 us of segment
// epilogue with warp ranges and FP64 folds, 117 us with all launches this way, at 56 % of
// the issue slots; the FMA pipe (128 FMAs and 96 packed ones per 32 blocks, and
// the moves between them) is what bounds it now, at 57 us of pipe time.

// (2G)^T x of 8 columns as the kernel reads it: for run q and column r the run's
// 32 blocks, 16 bytes each, xt[((q 8 + r) 32 + block) 4 + b], so that every load
// of a warp is 512 bytes in a row at a constant offset.  Thread per (q, r,
// block); blocks past the last one get zeros.  The same FP32 operations as
// wz2_xt_kernel.
static __global__ void wz3_xt8_kernel(const float* __restrict__ x, int64_t ldx, int64_t N, int64_t RB,
                                      float* __restrict__ xt) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= RB * 256) return;
  const int blk = (int)t & 31, r = (int)(t >> 5) & 7;
  const int64_t q = t >> 8, col = 4 * (32 * q + blk);
  const float* xr = x + r * ldx + col;
  float xv[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) xv[c] = col + c < N ? xr[c] : 0.f;
  const float a = xv[0] + xv[1], b = xv[2] + xv[3], c = xv[0] + xv[2], d = xv[1] + xv[3];
  reinterpret_cast<float4*>(xt)[t] = make_float4(2.f * (a + b), b - a, d - c, xv[3] - xv[2]);
}

// A block's products into the sums of 8 columns, hi/lo[h][r] the rows (2h, 2h + 1):
// the chain of wz3_accumulate.  xq: the lane's block in the run's part of the x
// that wz3_xt8_kernel lays out.
__device__ __forceinline__ void wz3_accumulate8(const float2 (&V)[2][4], float s, const float* __restrict__ xq,
                                                f32p (&hi)[2][8], f32p (&lo)[2][8]) {
  const f32p s2 = pair_of(s, s);
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const float4 x = __ldg(reinterpret_cast<const float4*>(xq + 128 * r));
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float a = V[h][0].x * x.x, b = V[h][0].y * x.x;
      a = fmaf(V[h][1].x, x.y, a), b = fmaf(V[h][1].y, x.y, b);
      a = fmaf(V[h][2].x, x.z, a), b = fmaf(V[h][2].y, x.z, b);
      a = fmaf(V[h][3].x, x.w, a), b = fmaf(V[h][3].y, x.w, b);
      two_sum_scaled_p(hi[h][r], lo[h][r], pair_of(a, b), s2);
    }
  }
}

// Bring the run of index entry e to L2: a lane per 128-byte line.
__device__ __forceinline__ void wz3_prefetch_run(const uint8_t* __restrict__ area, uint64_t e, int lane, int nb) {
  const uint32_t bytes = (uint32_t)(nb * wz3_block_bytes((int)(e >> 56)));
  const uint8_t* p = area + (e & 0x00FFFFFFFFFFFFFFull);
  if (128 * (uint32_t)lane < bytes) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 128 * lane));
}

__device__ __forceinline__ int64_t wz3_groups(int64_t BM) { return (BM + 7) / 8; }

static __global__ void __launch_bounds__(kWarpsPerCta * 32, 2)
    wz3_gemv8_kernel(const uint64_t* __restrict__ index, const uint8_t* __restrict__ area, int64_t M, int64_t BM,
                     int BN, int RB, const float* __restrict__ xt, int64_t L, int maxseg, double* __restrict__ ws,
                     double* __restrict__ y, int64_t ldy, double* __restrict__ state, double decay, unsigned* __restrict__ seen) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t u0 = (int64_t)blockIdx.x * L, u1 = min(wz3_groups(BM) * RB, u0 + L);
  for (int64_t ub = u0; ub < u1;) {  // the range's piece of group G: runs [q0, q1) of each of its bands
    const int64_t G = ub / RB, ue = min(u1, (G + 1) * RB);
    const int q0 = (int)(ub - G * RB), q1 = (int)(ue - G * RB);
    ub = ue;
    const int64_t I = 8 * G + warp;
    if (I >= BM) continue;  // whole warp
    f32p hi[2][8], lo[2][8];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int r = 0; r < 8; ++r) hi[h][r] = lo[h][r] = 0;
    const uint64_t* idx = index + I * RB;
    uint64_t e0 = __ldg(idx + q0), e1 = __ldg(idx + min(q0 + 1, q1 - 1)), e2 = __ldg(idx + min(q0 + 2, q1 - 1));
#pragma unroll 1
    for (int q = q0; q < q1; ++q) {
      const uint64_t e = e0;
      e0 = e1, e1 = e2;
      wz3_prefetch_run(area, e1, lane, min(32, BN - 32 * min(q + 2, q1 - 1)));
      e2 = __ldg(idx + min(q + 3, q1 - 1));
      const int W = (int)(e >> 56), left = BN - 32 * q;
      if (W == 0 || lane >= left) continue;  // a zero run adds 0
      uint32_t w[16];
      wz3_load_run(area, e, lane, min(32, left), true, w);
      float2 V[2][4];
      float s;
      wz3_values(w, W, V, s);
      wz3_accumulate8(V, s, xt + 1024 * (int64_t)q + 4 * lane, hi, lo);
    }
    __syncwarp();
    float h[32], l[32];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float2 a = halves_of(hi[k][r]), b = halves_of(lo[k][r]);
        h[4 * r + 2 * k] = a.x, h[4 * r + 2 * k + 1] = a.y;
        l[4 * r + 2 * k] = b.x, l[4 * r + 2 * k + 1] = b.y;
      }
    double z[1];
    fold_lanes<32, 32, true>(h, l, lane, z);
    const int64_t c_lo = div64(G * RB, L), c_hi = div64((G + 1) * RB - 1, L);
    const bool shared = c_lo != c_hi;
    band_write<1, 8, 32>(z, lane, 4 * I, M, shared ? ws + (I * maxseg + (blockIdx.x - c_lo)) * 32 : nullptr, y, ldy,
                         state, decay, true);
    if (shared)
      finish_shared_band(seen, ws, I, M, (int)(blockIdx.x - c_lo), (int)(c_hi - c_lo + 1), maxseg, 8, y, ldy, state, decay);
  }
}

// Decode: thread per block, the exact definition -- T = (2G) V (2G)^T in
// integers, times 2^(K+emax-30), exact in FP64 -- written row-major (ldo) as
// decode_out.cuh says, rows and columns past M, N dropped.
template <bool VEC>
static __global__ void __launch_bounds__(256)
    wz3_decompress_kernel(const uint64_t* __restrict__ index, const uint8_t* __restrict__ area, int64_t M, int64_t N,
                          int64_t BN, int64_t RB, int64_t nblocks, double* __restrict__ out, int64_t ldo) {
  __shared__ double turn[VEC ? 1 : 8 * 512];
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = b < nblocks;
  int64_t I = 0, J = 0;
  unit_of(live ? b : nblocks - 1, BN, I, J);
  const int64_t run = J / 32;
  const uint64_t e = index[I * RB + run];
  const int W = (int)(e >> 56);
  int64_t T[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) T[k] = 0;
  int scale_exp = 0;
  bool zero = W == 0;
  if (!zero) {
    const int nw = wz3_block_bytes(W) / 8;
    const int64_t nb = min((int64_t)32, BN - 32 * run);
    // word-interleaved run: word k of block b at word k nb + b
    const uint64_t* wp = reinterpret_cast<const uint64_t*>(area + (e & 0x00FFFFFFFFFFFFFFull)) + (J - 32 * run);
    uint64_t w[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) w[k] = k < nw ? wp[k * nb] : 0ull;
    const int E = (int)(w[0] & 0xFF), K = (int)((w[0] >> 8) & 31);
    zero = E == 0;
    scale_exp = K + (E - 127) - 30;
    const uint64_t mask = (1ull << W) - 1ull;
    int64_t V[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int o = 13 + W * k, wi = o >> 6, sh = o & 63;
      uint64_t u = w[wi] >> sh;
      if (sh + W > 64) u |= w[wi + 1] << (64 - sh);
      V[seq_index(k)] = (int64_t)(u & mask) - ((int64_t)1 << (W - 1));
    }
    // (2G) applied to the columns, then to the rows
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t s2 = 2 * V[j], x = V[4 + j], yv = V[8 + j], z = V[12 + j];
      V[j] = s2 - x - yv, V[4 + j] = s2 - x + yv, V[8 + j] = s2 + x - yv - z, V[12 + j] = s2 + x + yv + z;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int64_t s2 = 2 * V[4 * r], x = V[4 * r + 1], yv = V[4 * r + 2], z = V[4 * r + 3];
      T[4 * r] = s2 - x - yv, T[4 * r + 1] = s2 - x + yv, T[4 * r + 2] = s2 + x - yv - z,
            T[4 * r + 3] = s2 + x + yv + z;
    }
  }
  uint2 d[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) d[k] = zero ? make_uint2(0u, 0u) : f64_from_int(T[k], scale_exp);
  store_units<VEC, 4, 4>(d, live, I, J, BN, M, N, out, ldo, turn + (VEC ? 0 : (threadIdx.x >> 5) * 512));
}

}  // namespace dev
}  // namespace whff
