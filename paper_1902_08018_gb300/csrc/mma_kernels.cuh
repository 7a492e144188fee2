// mma_kernels.cuh -- many right-hand sides on the 5th-generation tensor cores.
//
// With R right-hand sides the step Y = A X is a dense contraction (Sec. 4.4's
// GEMV becomes a GEMM), so for R >= 4 (the default crossover) the WZ2 kernels run
// it on tcgen05.  In the transform domain the contraction is
//     Z_band = sum_J (s_J V_J) ((2G)^T X_J),   Y_band = (2G) Z_band * 2^-3,
// a GEMM whose A operand is the stored integer coefficients times a
// power-of-two block scale, and whose B operand is the transformed x.
//
// Precision (the 1e-6 bar): a coefficient of a W-bit field has at most W-1
// significant bits, so A splits EXACTLY into PA = ceil((W-1)/8) BF16 pieces
// (1 at rate 8, 2 at rates 12 and 16, 3 at 20 and 24); B (FP32) into three
// BF16 pieces (8+8+8 bits, exact).  The products A_p B_q with p+q <= 2 are
// issued (kind::f16, BF16 in, FP32 accumulate in TMEM); the dropped ones are
// below 2^-24 of |a||x|.  The tensor cores' FP32 accumulate is not a
// round-to-nearest sum, so the products go to three accumulators by size:
// A_0 B_0; the 2^-8 terms A_0 B_1 + A_1 B_0; the 2^-16 terms A_0 B_2 + A_1 B_1
// + A_2 B_0.  With the B pieces side by side along N, one instruction
// A_p [B_0 .. B_{2-p}] (N = (3-p) NR) writes accumulators p..2, so a K step
// takes PA instructions.  The accumulators cover at most kMmaDrainStages
// stages of one tile (16 blocks = 64 columns of K each) and are then added
// and drained into TwoSum FP32 registers, so FP32 rounding never sees long
// sums.
//
// Tiles are 32 bands = 128 coefficient rows, stages 16 blocks of K.  The sequence
// of (tile, stage) items is split into equal contiguous ranges; one CTA per SM is
// resident and takes its ranges' stages through three rings with a role each:
//  * copies: the stage's B tile (bulk copy) and its compressed words (tiled copy)
//    into shared memory, five or six stages ahead;
//  * decode: twelve warps in quartets, a quartet a stage; a thread turns a block
//    into its BF16 pieces and stores them straight to TMEM, where A is read from:
//    the 16x256b store gives lane l the row l / 4 and four values of K, so a
//    block's four rows land at TMEM lanes 8a + band % 8 of its bands' quarter;
//  * issue: one elected lane starts the stage's MMAs (A from TMEM, B from shared
//    memory) and commits them to the stage's and the group's barriers;
//  * drain: eight warps add a finished group's three accumulators into TwoSum
//    registers; a range's sums go to the workspace as one FP64 segment partial.
// wz2_mma_finish adds a band's segments in order and mixes with 2G, wz2_mma_state
// applies the state.
// A in shared memory cost 32 KB of stores and as many of operand reads per stage,
// and the register-fed words a barrier of the whole CTA per stage; measured per
// stage's MMAs (N = 96 and 64), A from TMEM takes 324 clocks, from shared memory
// 426 (N = 48 and 32: 175 and 349).  WZ2-lift 16, 12288^2, 32 columns: 131 us
// before, 79 us now (pass 156 -> 102 us); rate 12 batches of 1024..8192 at 16 and
// 32 columns: 67 + 54 -> 44 + 40 us.  The same MMAs in the same groups: the results
// are the same bits.  What bounds it now is the issuing warp's turn-around per
// stage (about 1200 clocks of waits, issue and commits), not the tensor pipe (27 %
// busy) nor HBM.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>

#include <cstdint>
#include <utility>

#include "whff.h"
#include "bulk.cuh"
#include "wz2_kernels.cuh"

namespace whff {
namespace dev {

constexpr int kMmaThreads = 256;       // 8 warps; warps w and w+4 share TMEM lanes 32(w%4)..
constexpr int kMmaBands = 32;         // 128 coefficient rows per tile
constexpr int kMmaStageBlocks = 16;   // K = 64 per stage
constexpr int kMmaKSteps = 4;         // K = 16 per instruction
constexpr int kMmaDrainStages = 2;    // stages of one tile accumulated in TMEM between drains


// 64-bit shared-memory matrix descriptor: start >> 4 (bits 0-13), leading
// byte offset >> 4 (16-29), stride byte offset >> 4 (32-45), descriptor
// version 1 (bit 46), no swizzle (bits 61-63 = 0).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
         (1ull << 46);
}

// Instruction descriptor, kind::f16: F32 accumulator (bits 4-5 = 1), A and B
// BF16 (bits 7-9 = 1, 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at 24.
__device__ __forceinline__ constexpr uint32_t mma_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// The same with A and B FP16 (bits 7-9 and 10-12 = 0).
__device__ __forceinline__ constexpr uint32_t mma_idesc_f16(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// Byte offset of element (row, k) in a 16-wide K-step tile (no swizzle,
// K-major): core matrix (row/8, k/8) of 8 rows x 16 bytes, 2 along K.
__device__ __forceinline__ uint32_t tile_off(int row, int k) {
  return (uint32_t)(((row >> 3) * 2 + (k >> 3)) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// Exact split of a float with at most 24 significant bits into three BF16.
__device__ __forceinline__ void split3(float v, __nv_bfloat16& a, __nv_bfloat16& b, __nv_bfloat16& c) {
  a = __float2bfloat16_rn(v);
  const float r1 = v - __bfloat162float(a);
  b = __float2bfloat16_rn(r1);
  c = __float2bfloat16_rn(r1 - __bfloat162float(b));
}

__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 lo, __nv_bfloat16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

// BF16 pieces of one A coefficient: its field has at most W-1 significant bits.
template <int RATE>
struct MmaPieces {
  static constexpr int kBits = Wz2Layout<RATE>::kW - 1;
  static constexpr int kA = kBits <= 8 ? 1 : kBits <= 16 ? 2 : 3;
};

// B operand of one stage: per K step, the 3 pieces one after another along N
// (a 3 NR x 16 BF16 tile).
template <int NR>
struct MmaBTile {
  static constexpr int kBTile = NR * 16 * 2;  // one piece, one K step
  static constexpr int kB = 3 * kMmaKSteps * kBTile;
};

// TMEM columns: two accumulator groups of three NR-column accumulators,
// rounded up to the power of two that tcgen05.alloc takes.
template <int NR>
__host__ __device__ constexpr uint32_t mma_tmem_cols() {
  return 6 * NR <= 32 ? 32u : 6 * NR <= 64 ? 64u : 6 * NR <= 128 ? 128u : 256u;
}

// Shared memory of wz2_mma_kernel: a ring of kNB B tiles and of as many stages'
// compressed words, the barriers, the TMEM
// slot and the abort flag; the member table follows kBytes.
template <int RATE, int NR>
struct MmaSmem {
  static constexpr int kNA = MmaPieces<RATE>::kA == 3 ? 3 : 4;  // A buffers in TMEM
  static constexpr int kB = MmaBTile<NR>::kB;
  static constexpr int kNB = RATE >= 20 ? 5 : 6;
  static constexpr int kBB = 2 * RATE;  // bytes of a block
  static constexpr int kRowBytes = kMmaStageBlocks * kBB;  // a band's words, rows back to back as the tiled copy writes them
  static constexpr int kWords = kMmaBands * (kRowBytes + 16);  // 16 bytes more per row, see the copies
  static constexpr int kBars = kNB * (kB + kWords);
  static constexpr int kBytes = kBars + 256;
};

// Ranges that a CTA of wz2_mma_kernel takes one after another, at most.  The ranges,
// and the accumulator groups that end with them, are those of a grid of two CTAs per
// SM (one where A takes three pieces).
template <int RATE>
constexpr int kMmaRanges = MmaPieces<RATE>::kA == 3 ? 1 : 2;

// Ranges per CTA of a pass of `ranges`: one while there is an SM for each (512^2 in
// FP8, 32 columns, replayed: 16.4 us with two, 14.4 with one).
inline int mma_ranges_per_cta(int ranges, int sms, int most) { return ranges <= sms ? 1 : most; }

// Eight columns of the three accumulators at ta, ta + stride, ta + 2 stride,
// summed big + (small + smaller): one wait for the three loads, tied to their
// registers so no use can move above it.
__device__ __forceinline__ void tmem_load_sum8(uint32_t ta, uint32_t stride, float (&v)[8]) {
  uint32_t a[8], b[8], c[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
               : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7])
               : "r"(ta));
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
               : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7])
               : "r"(ta + stride));
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
               : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3]), "=r"(c[4]), "=r"(c[5]), "=r"(c[6]), "=r"(c[7])
               : "r"(ta + 2 * stride));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                 "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7]),
                 "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(c[4]), "+r"(c[5]), "+r"(c[6]), "+r"(c[7])
               :
               : "memory");
#pragma unroll
  for (int i = 0; i < 8; i += 2) {  // packed pairs: each half rounds as a + (b + c) would
    const float2 bc = add_f2(make_float2(__uint_as_float(b[i]), __uint_as_float(b[i + 1])),
                             make_float2(__uint_as_float(c[i]), __uint_as_float(c[i + 1])));
    const float2 t = add_f2(make_float2(__uint_as_float(a[i]), __uint_as_float(a[i + 1])), bc);
    v[i] = t.x;
    v[i + 1] = t.y;
  }
}


// The B operand of every stage, built once per step: for column block J and
// right-hand side r, (2G)^T x_J (or x_J without the lift) in three BF16
// pieces, already in the shared-memory tile layout of its 16-block stage:
// out[stage][piece][kstep] = NR x 16 BF16 tile.  Thread per (stage, J, r).
// The pass of thread q in a launch-wide grid: `single` when table is null,
// else the entry with the largest begin <= q (begin = bt_begin or fin_begin).
template <bool FIN>
__device__ __forceinline__ MmaPass pass_of(const MmaPass& single, const MmaPass* __restrict__ table, int n,
                                           int64_t q) {
  if (!table) return single;
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if ((FIN ? table[mid].fin_begin : table[mid].bt_begin) <= q) lo = mid;
    else hi = mid - 1;
  }
  return table[lo];
}

// B tiles of every pass: for stage st, column block J and right-hand side r,
// (2G)^T x_J (or x_J without the lift) in three BF16 pieces, already in the
// shared-memory tile layout of the stage: out[st][kstep][piece] = NR x 16 BF16.
// Thread per (pass, stage, J in the stage, r); total threads given.
template <bool LIFT, int NR>
__global__ void wz2_mma_btiles(MmaPass single, const MmaPass* __restrict__ table, int n, int64_t threads) {
  using S = MmaBTile<NR>;
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= threads) return;
  const MmaPass ps = pass_of<false>(single, table, n, q);
  const int64_t ql = q - ps.bt_begin;
  if (ql >= (int64_t)ps.S * kMmaStageBlocks * NR) return;
  const int r = (int)(ql % NR);
  const int jl = (int)((ql / NR) % kMmaStageBlocks);
  const int64_t stage = ql / ((int64_t)NR * kMmaStageBlocks);
  const int64_t J = stage * kMmaStageBlocks + jl;
  float xt[4] = {0.f, 0.f, 0.f, 0.f};
  if (r < ps.R) {
    float xv[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) xv[c] = 4 * J + c < ps.N ? __ldg(ps.x + (int64_t)r * ps.ldx + 4 * J + c) : 0.f;
    if (LIFT) {
      const float aa = xv[0] + xv[1], bb = xv[2] + xv[3], cc = xv[0] + xv[2], dd = xv[1] + xv[3];
      xt[0] = 2.f * (aa + bb);
      xt[1] = bb - aa;
      xt[2] = dd - cc;
      xt[3] = xv[3] - xv[2];
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) xt[c] = xv[c];
    }
  }
  __nv_bfloat16 p[3][4];
#pragma unroll
  for (int b = 0; b < 4; ++b) split3(xt[b], p[0][b], p[1][b], p[2][b]);
  const int kstep = jl >> 2, kk = (jl & 3) * 4;
  uint8_t* base = ps.btiles + stage * (int64_t)S::kB;
#pragma unroll
  for (int pc = 0; pc < 3; ++pc)
    *reinterpret_cast<uint2*>(base + (kstep * 3 + pc) * S::kBTile + tile_off(r, kk)) =
        make_uint2(pack2(p[pc][0], p[pc][1]), pack2(p[pc][2], p[pc][3]));
}


// cvt.rn.bf16x2.f32: the packed pair (lo in bits 0-15, hi in bits 16-31).
__device__ __forceinline__ uint32_t bf16x2_rn(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;\n" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// The 16 coefficients of a block times its scale 2^(E+K-154), as packed pairs
// in tile-row order: P[a][h] = (V[a][2h], V[a][2h+1]).  The field is OR-ed into
// the mantissa of 2^(e+23) and one packed subtraction per pair gives the scaled
// value exactly (wz2_fields_times_scale's values, two per instruction); blocks
// beyond the trick's exponent range (|a| >= 2^103) decode unscaled and take s
// by an exact packed multiply.  A zero block decodes to zeros.
template <int RATE, bool LIFT>
__device__ __forceinline__ void mma_block_pairs(const uint32_t (&w)[Wz2Layout<RATE>::kWords], float2 (&P)[4][2]) {
  using Lay = Wz2Layout<RATE>;
  const uint32_t E = w[0] & 0xFFu, K = (w[0] >> 8) & 31u;
  const bool trick = E + K <= 258u;
  const uint32_t creg = trick ? (E ? (E + K - 4u) << 23 : 0u) : 0x4B000000u;
  const uint32_t mreg = E ? Lay::kMask : 0u;
  const float bias = E ? __uint_as_float(creg | (1u << (Lay::kW - 1))) : 0.f;
  uint32_t u[16];
  wz2_field_bits_impl<RATE>(w, mreg, creg, u, std::make_integer_sequence<int, 16>{});
  const float2 b2 = make_float2(bias, bias);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int m0 = 4 * a + 2 * h, m1 = m0 + 1;
      const int k0 = LIFT ? seq_field(m0) : m0, k1 = LIFT ? seq_field(m1) : m1;
      P[a][h] = sub_f2(make_float2(__uint_as_float(u[k0]), __uint_as_float(u[k1])), b2);
    }
  if (!trick) {
    const float s = __uint_as_float((E + K - 27u) << 23);
    const float2 s2 = make_float2(s, s);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int h = 0; h < 2; ++h) P[a][h] = mul_f2(P[a][h], s2);
  }
}

// Exact split of a pair of values (at most 8 PA significant bits each) into PA
// BF16 pairs, d[p] = piece p of (v.x, v.y): round to BF16, subtract, repeat --
// the two subtractions of each step in one packed instruction.
template <int PA>
__device__ __forceinline__ void split_pair(float2 v, uint32_t (&d)[PA]) {
#pragma unroll
  for (int p = 0; p < PA; ++p) {
    d[p] = bf16x2_rn(v.x, v.y);
    if (p + 1 < PA) v = sub_f2(v, make_float2(bf16_lo(d[p]), bf16_hi(d[p])));
  }
}

// Warps of the kernel: one issues the MMAs, three bring the compressed words and
// the B tiles in, kMmaQuartets x 4 decode, 8 drain.
constexpr int kMmaIssueWarp = 0, kMmaCopyWarp = 1, kMmaDecodeWarp = 4;
constexpr int kMmaCopyThreads = 32 * (kMmaDecodeWarp - kMmaCopyWarp);
constexpr int kMmaQuartets = 3;
constexpr int kMmaDrainWarp = kMmaDecodeWarp + 4 * kMmaQuartets;
constexpr int kMmaDecodeThreads = 32 * (kMmaDrainWarp + 8);

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(p));
  return p != 0;
}

// `bytes` (0 to 16) bytes global -> shared without a register, zeros for the rest
// of 16; both addresses 16-byte aligned.  Through L1, which fetches the sector that two
// pieces share once: past it each piece crossed the host link by itself (8192^2 at rate
// 16 in host memory, 32 columns: 1124 us; 662 us so, the link's time).
__device__ __forceinline__ void cp_async_zfill(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// Four 32-bit columns to TMEM by the warp's lanes, 16 lanes of the warp's
// quarter from taddr on: r0, r1 go to row lane / 4, columns 2 (lane % 4) and + 1;
// r2, r3 to row 8 + lane / 4.
__device__ __forceinline__ void tmem_store_16x256(uint32_t taddr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("tcgen05.st.sync.aligned.16x256b.x1.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(taddr), "r"(r0), "r"(r1), "r"(r2),
               "r"(r3)
               : "memory");
}

// Persistent grid over the item sequence of one or more passes (members):
// member k owns items [item_begin, item_begin + tiles S), item = item_begin +
// tile S + stage; range v is items [v L, v L + L), and CTA g takes the
// per_cta ranges from per_cta g on.  ws[((tile * maxseg + seg) * R + r) *
// 128 + m] of a member receives the FP64 partial of coefficient row a of band b
// of the tile, m = 32a + b, for the range's segment seg = v - (item_begin + tile
// S) / L.  Accumulator groups end with a range, so a result does not depend on
// how the ranges are dealt to the CTAs.
// `single` is the only member when table is null (one matrix); otherwise the
// nmem members of the table (a batch) are copied to shared memory.
template <int RATE, bool LIFT, int NR, bool TABLE>
__global__ void __launch_bounds__(kMmaDecodeThreads, 1)
    wz2_mma_kernel(MmaMember single, const MmaMember* __restrict__ table, int nmem, int64_t total, int64_t L,
                   int per_cta, int* __restrict__ status, uint32_t spin) {
  using SM = MmaSmem<RATE, NR>;
  constexpr int PA = MmaPieces<RATE>::kA, NB = SM::kNB, NA = SM::kNA, NQ = kMmaQuartets;
  constexpr int NW = Wz2Layout<RATE>::kWords;
  constexpr int HALF = NR / 2;  // columns drained by each of the two warps on a lane quarter
  constexpr uint32_t kACols = 8 * kMmaKSteps * PA;  // TMEM columns of a stage's A pieces
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t s_base = smem_addr(smem);
  const uint32_t b_full = s_base + SM::kBars;  // NB: the B tile in the slot has landed, and the words of a tiled copy
  const uint32_t w_full = b_full + 8 * NB;     // NB: so have the words copied in pieces (every copying thread's)
  const uint32_t done = w_full + 8 * NB;       // NB: the MMAs of the stage in the slot are done
  const uint32_t a_full = done + 8 * NB;       // NA: the stage's A pieces are in the buffer (4 arrivals)
  const uint32_t gfull = a_full + 8 * NA;      // 2: the accumulator group is complete
  const uint32_t gfree = gfull + 16;           // 2: the accumulator group has been drained (8 arrivals)
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + SM::kBars + 8 * (3 * NB + NA + 4));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  MmaMember* tab = reinterpret_cast<MmaMember*>(smem + SM::kBytes);  // the members

  // broadcast, so that the compiler knows the roles to be warp-uniform
  const int t = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, t >> 5, 0), lane = t & 31;
  const int64_t it0 = (int64_t)blockIdx.x * per_cta * L;
  const int n = (int)max((int64_t)0, min(total, it0 + per_cta * L) - it0);  // stages of this CTA
  const int len = (int)L;
  if constexpr (TABLE)
    for (int i = t; i < nmem; i += kMmaDecodeThreads) tab[i] = table[i];
  // member m (TABLE: of the batch's table; else the one matrix)
  auto mb = [&](int m) -> const MmaMember& {
    if constexpr (TABLE) return tab[m];
    return single;
  };
  if (t == 0) {
    for (int i = 0; i < NB; ++i)
      mbar_init(b_full + 8 * i, 1), mbar_init(w_full + 8 * i, kMmaCopyThreads), mbar_init(done + 8 * i, 1);
    for (int i = 0; i < NA; ++i) mbar_init(a_full + 8 * i, 4);
    for (int i = 0; i < 2; ++i) mbar_init(gfull + 8 * i, 1), mbar_init(gfree + 8 * i, 8);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    *abort_flag = 0;
  }
  if (warp == kMmaIssueWarp) {  // all of TMEM: two groups of three accumulators, then the A buffers
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(tslot)),
                 "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, *tslot, 0);
  static_assert(6 * NR + NA * (int)kACols <= 512, "accumulators and A buffers fit TMEM");
  auto a_cols = [&](uint32_t k) { return tmem + (uint32_t)(6 * NR) + k % NA * kACols; };  // of stage k
  auto fail = [&]() {  // a wait ran out: every other wait gives up
    atomicExch(status, WHFF_ETIMEOUT);
    *abort_flag = 1;
  };
  // a whole warp waits; false if the wait ran out (reported) or the CTA gave up
  auto warp_wait = [&](uint32_t bar, uint32_t parity) {
    const int r = mbar_wait_or_abort(bar, parity, spin, abort_flag);
    const bool ran_out = __any_sync(0xFFFFFFFFu, r == 0), ok = __all_sync(0xFFFFFFFFu, r > 0);
    if (ran_out && lane == 0) fail();
    return ok;
  };

  // Cursor (member, tile, stage): advances in item order, so the loops have no divisions.
  int c_m = 0;
  if constexpr (TABLE)
    while (c_m + 1 < nmem && tab[c_m + 1].item_begin <= it0) ++c_m;
  int c_tile = 0, c_st = 0;
  if (n > 0) {
    const MmaMember& me = mb(c_m);
    c_tile = (int)((it0 - me.item_begin) / me.S);
    c_st = (int)(it0 - me.item_begin - (int64_t)c_tile * me.S);
  }
  auto advance = [&]() {
    if (++c_st == mb(c_m).S) {
      c_st = 0, ++c_tile;
      if constexpr (TABLE)
        if (c_tile == tab[c_m].tiles) c_tile = 0, ++c_m;
    }
  };
  // Whether the item at the cursor, with range_left items of its range to go
  // and stage k of this CTA, closes its accumulator group at position gpos.
  auto closes = [&](int gpos, int range_left, int k) {
    return gpos + 1 == kMmaDrainStages || c_st == mb(c_m).S - 1 || range_left == 1 || k == n - 1;
  };

  // every role's end: nothing more goes to TMEM or is read from it
  auto leave = [&]() {
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
  };
  if (warp >= kMmaDecodeWarp && warp < kMmaDrainWarp) {
    // ---- decode: quartet q takes stages q, q + NQ, ...; warp w of it bands 8w .. 8w + 7
    // of the tile, lane l band l / 4 of those and the blocks l % 4 of the four K steps.
    const int q = (warp - kMmaDecodeWarp) >> 2, quarter = warp & 3, cb = lane & 3;
    const int band_l = 8 * quarter + (lane >> 2);
    for (int i = 0; i < q && i < n; ++i) advance();
    for (int k = q; k < n; k += NQ) {
      const MmaMember& me = mb(c_m);
      const bool tiled = me.map != nullptr;
      // the lane's first block in the slot (see the copies)
      const uint8_t* staged = smem + NB * SM::kB + (uint32_t)k % NB * SM::kWords + cb * SM::kBB;
      if (me.paired) {
        const int odd = ((int)me.band0 + band_l) & 1;
        staged += (odd * (kMmaBands / 2) + (band_l >> 1)) * (SM::kRowBytes + 16) + 8 * odd;
      } else if (tiled) {
        staged += band_l * SM::kRowBytes;
      } else {
        const uint32_t blk = (32 * (uint32_t)c_tile + band_l) * (uint32_t)me.BN + 16 * (uint32_t)c_st;
        staged += band_l * (SM::kRowBytes + 16) +
                  (((uint32_t)reinterpret_cast<uintptr_t>(me.stream) + blk * SM::kBB) & 8u);
      }
      if (k + NQ < n) {
#pragma unroll
        for (int i = 0; i < NQ; ++i) advance();
      }
      // the words are here
      if (!warp_wait((tiled ? b_full : w_full) + 8 * ((uint32_t)k % NB), (uint32_t)k / NB & 1u)) break;
      if (k >= NA) {  // the A buffer is free once the MMAs of the stage NA before are done
        const uint32_t p = (uint32_t)(k - NA);
        if (!warp_wait(done + 8 * (p % NB), p / NB & 1u)) break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const uint32_t a_row = a_cols((uint32_t)k) + ((uint32_t)(32 * quarter) << 16);
#pragma unroll
      for (int u = 0; u < kMmaKSteps; ++u) {
        uint32_t w[NW];
        wz2_lds<RATE>(staged + 4 * u * SM::kBB, w);  // zeros past the matrix: a zero block
        float2 P[4][2];
        mma_block_pairs<RATE, LIFT>(w, P);
        uint32_t d[4][2][PA];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int h = 0; h < 2; ++h) split_pair<PA>(P[a][h], d[a][h]);
        __syncwarp();
#pragma unroll
        for (int p = 0; p < PA; ++p) {
          const uint32_t col = a_row + (uint32_t)(8 * (p * kMmaKSteps + u));
          tmem_store_16x256(col, d[0][0][p], d[0][1][p], d[1][0][p], d[1][1][p]);
          tmem_store_16x256(col + (16u << 16), d[2][0][p], d[2][1][p], d[3][0][p], d[3][1][p]);
        }
      }
      asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(a_full + 8 * ((uint32_t)k % NA));
    }
    asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
    leave();
  } else if (warp >= kMmaDrainWarp) {
    // ---- drain: TMEM lane 32 quarter + lane holds coefficient row a = lane / 8 of band
    // 8 quarter + lane % 8.  A group's three accumulators are added and enter TwoSum sums.
    const int quarter = warp & 3, m_row = 32 * (lane >> 3) + 8 * quarter + (lane & 7);
    const int c0 = HALF * ((warp - kMmaDrainWarp) >> 2);
    const uint32_t rows = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)c0;
    float hi[HALF], lo[HALF];
#pragma unroll
    for (int r = 0; r < HALF; ++r) hi[r] = lo[r] = 0.f;
    int cur_m = c_m, cur_tile = c_tile;  // member and tile of the sums
    int v = (int)blockIdx.x * per_cta, left = len;  // the range, and its items from here on
    auto flush = [&](int range) {
      const MmaMember& me = mb(cur_m);
      const int64_t seg = range - (me.item_begin + (int64_t)cur_tile * me.S) / L;
      double* dst = me.ws + (((int64_t)cur_tile * me.maxseg + seg) * me.R) * 128 + m_row;
#pragma unroll
      for (int r = 0; r < HALF; ++r) {
        if (c0 + r < me.R) dst[(int64_t)(c0 + r) * 128] = widen(hi[r]) + widen(lo[r]);
        hi[r] = lo[r] = 0.f;
      }
    };
    int gpos = 0, acc = 0;
    uint32_t parity = 0;
    bool open = false, alive = true;
    for (int k = 0; k < n; ++k) {
      const int m = c_m, tile = c_tile;
      const bool ends = closes(gpos, left, k);
      gpos = ends ? 0 : gpos + 1;
      advance();
      if (ends) {
        if (!warp_wait(gfull + 8 * acc, parity)) {
          alive = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (open && (m != cur_m || tile != cur_tile)) flush(v);
        cur_m = m, cur_tile = tile, open = true;
        const uint32_t ta = rows + (uint32_t)(3 * acc * NR);
#pragma unroll
        for (int h = 0; h < HALF; h += 8) {
          float x[8];
          tmem_load_sum8(ta + h, NR, x);
#pragma unroll
          for (int r = 0; r < 8; r += 2) {  // TwoSum on packed pairs of columns (the same bits per half)
            float2 H = make_float2(hi[h + r], hi[h + r + 1]), Lo = make_float2(lo[h + r], lo[h + r + 1]);
            two_sum_acc2(H, Lo, make_float2(x[r], x[r + 1]));
            hi[h + r] = H.x, hi[h + r + 1] = H.y, lo[h + r] = Lo.x, lo[h + r + 1] = Lo.y;
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(gfree + 8 * acc);
        parity ^= (uint32_t)acc;
        acc ^= 1;
      }
      if (--left == 0) {
        flush(v);
        open = false, left = len, ++v;
      }
    }
    if (alive && open) flush(v);
    leave();
  } else {
    if (warp == kMmaIssueWarp) {
      // ---- issue.  The whole warp walks the stages, so that everything the MMAs take is
      // warp-uniform; lanes 0-2 wait for a stage's three barriers side by side (a wait costs
      // about 250 clocks even when its phase is over), one elected lane issues.
      int last_commit = -1, groups = 0, gpos = 0, acc = 0, buf = 0, slot = 0, left = len;
      uint32_t phase = 0, a_phase = 0, g_phase = 1;  // g_phase: the groups are free at first
      const uint64_t b_desc0 = smem_desc(s_base, 128, 256);
#pragma unroll 1
      for (int k = 0; k < n; ++k) {
        const bool init = gpos == 0, ends = closes(gpos, left, k);
        const uint32_t bar = lane == 0 ? b_full + 8 * slot : lane == 1 ? a_full + 8 * buf : gfree + 8 * acc;
        const uint32_t par = lane == 0 ? phase : lane == 1 ? a_phase : g_phase;
        int r = 1;
        if (lane < (init ? 3 : 2)) r = mbar_wait_or_abort(bar, par, spin, abort_flag);
        if (__any_sync(0xFFFFFFFFu, r <= 0)) {
          if (r == 0) fail();
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (elect_one()) {
          // A_p [B_0 .. B_{2-p}] into accumulators p..2; A_0 of the first K step of
          // a group starts all three
          const uint64_t bd0 = b_desc0 + (uint64_t)((slot * SM::kB) >> 4);
          const uint32_t d0 = tmem + (uint32_t)(3 * acc * NR), a0 = a_cols((uint32_t)buf);
#pragma unroll
          for (int ks = 0; ks < kMmaKSteps; ++ks) {
#pragma unroll
            for (int pa = 0; pa < PA; ++pa) {
              const uint32_t ad = a0 + (uint32_t)(8 * (pa * kMmaKSteps + ks));
              const uint64_t bd = bd0 + (uint64_t)((3 * ks * MmaBTile<NR>::kBTile) >> 4);
              const uint32_t accumulate = (init && ks == 0 && pa == 0) ? 0u : 1u;
              asm volatile(
                  "{\n\t.reg .pred p;\n\t"
                  "setp.ne.b32 p, %4, 0;\n\t"
                  "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d0 + (uint32_t)(pa * NR)),
                  "r"(ad), "l"(bd), "r"(mma_idesc((3 - pa) * NR)), "r"(accumulate));
            }
          }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(done +
                                                                                                          8 * slot)
                       : "memory");
          if (ends)
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                             gfull + 8 * acc)
                         : "memory");
        }
        __syncwarp();
        last_commit = k;
        if (ends) {
          g_phase ^= (uint32_t)acc;
          acc ^= 1;
          ++groups;
        }
        gpos = ends ? 0 : gpos + 1;
        advance();
        if (--left == 0) left = len;
        if (++buf == NA) buf = 0, a_phase ^= 1;
        if (++slot == NB) slot = 0, phase ^= 1;
      }
      __syncwarp();
      leave();
      if (lane == 0 && *abort_flag) {  // MMAs and their commits in flight: a second bounded chance
        if (last_commit >= 0) (void)mbar_wait(done + 8 * (last_commit % NB), (uint32_t)((last_commit / NB) & 1));
        if (groups) (void)mbar_wait(gfull + 8 * ((groups - 1) & 1), (uint32_t)(((groups - 1) >> 1) & 1));
      }
      __syncwarp();
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512u));
    } else {
      // ---- copies, NB stages ahead: the B tile, and the compressed words of the stage's 32
      // bands with zeros where the matrix ends.  One tiled copy; at rates 12 and 20 with an odd
      // number of blocks per band (rows 8 bytes off 16) two, of the even and the odd bands, the
      // odd rows starting 8 bytes into theirs; from host memory aligned 16-byte pieces (a row
      // may start 8 bytes into the first one).  A slot is refilled once its MMAs are done.
      // What the copy engine brings completes on b_full alone, which one arrival closes: this
      // warp can then wait for all of it at the end, whoever has given up before.
      constexpr bool kShift = SM::kBB % 16 != 0;
      constexpr int kRow = (kMmaStageBlocks * SM::kBB + (kShift ? 8 : 0) + 15) / 16;  // pieces of a band
      // a warp takes one row (two of 16 pieces) at a time, every third
      constexpr int kLanes = kRow <= 16 ? 16 : 32, kStep = (32 / kLanes) * (kMmaCopyThreads / 32);
      const int r0 = (warp - kMmaCopyWarp) * (32 / kLanes) + lane / kLanes, c0 = lane % kLanes;
      int issued = 0, slot = 0;
      uint32_t phase = 1;  // the slots are free at first
      const void* acquired = nullptr;  // the map that this CTA may use
      for (; issued < n; ++issued) {
        if (!warp_wait(done + 8 * slot, phase)) break;
        const MmaMember& me = mb(c_m);
        if (me.map && me.map != acquired && warp == kMmaCopyWarp) {
          acquired = me.map;
          tensormap_acquire(me.map);
          if (me.paired) tensormap_acquire(static_cast<const uint8_t*>(me.map) + 128);
        }
        const uint32_t words = s_base + NB * SM::kB + slot * SM::kWords;
        const uint32_t b_bar = b_full + 8 * slot, w_bar = w_full + 8 * slot;
        const bool tiled = me.map != nullptr;
        if (warp == kMmaCopyWarp && elect_one()) {
          constexpr uint32_t kHalf = kMmaBands / 2 * (SM::kRowBytes + 16);  // paired: odd and even bands, a map each
          if (tiled) mbar_expect_tx_only(b_bar, me.paired ? 2 * kHalf : (uint32_t)(kMmaBands * SM::kRowBytes));
          bulk_copy_g2s(s_base + slot * SM::kB, me.btiles + (int64_t)c_st * SM::kB, (uint32_t)SM::kB, b_bar);
          if (tiled) {
            const int x = c_st * kMmaStageBlocks * NW, g = (int)(me.band0 + kMmaBands * (int64_t)c_tile);
            if (me.paired) {
              tma_load_2d(words + (g & 1) * kHalf, static_cast<const uint8_t*>(me.map) + (g & 1) * 128, x, g >> 1, b_bar);
              tma_load_2d(words + (~g & 1) * kHalf, static_cast<const uint8_t*>(me.map) + (~g & 1) * 128, x, (g + 1) >> 1,
                          b_bar);
            } else {
              tma_load_2d(words, me.map, x, g, b_bar);
            }
          }
        }
        __syncwarp();
        if (tiled) {  // nothing to copy in pieces: the phase turns all the same
          mbar_arrive(w_bar);
          advance();
          if (++slot == NB) slot = 0, phase ^= 1;
          continue;
        }
        const int bands = (int)min((int64_t)kMmaBands, me.BM - kMmaBands * (int64_t)c_tile);
        const int row_bytes = (int)min((int64_t)kMmaStageBlocks, me.BN - kMmaStageBlocks * (int64_t)c_st) * SM::kBB;
        const uint8_t* src =
            me.stream + (kMmaBands * (int64_t)c_tile * me.BN + kMmaStageBlocks * (int64_t)c_st) * SM::kBB;
        const int64_t band_bytes = me.BN * SM::kBB;
        const uint8_t* row = src + r0 * band_bytes + c0 * 16;
        uint32_t dst = words + r0 * (SM::kRowBytes + 16) + c0 * 16;
#pragma unroll
        for (int i = 0; i < (kMmaBands + kStep - 1) / kStep; ++i) {
          const int r = r0 + i * kStep;
          const int shift = kShift ? (int)(reinterpret_cast<uintptr_t>(row) & 8u) : 0;
#pragma unroll
          for (int c = 0; c < kRow; c += kLanes) {
            const int bytes = r < bands ? max(0, min(16, row_bytes + shift - 16 * (c0 + c))) : 0;
            if (r < kMmaBands && c0 + c < kRow)
              cp_async_zfill(dst + 16 * c, bytes ? row - shift + 16 * c : me.btiles, bytes);
          }
          row += kStep * band_bytes;
          dst += kStep * (SM::kRowBytes + 16);
        }
        asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(w_bar) : "memory");
        advance();
        if (++slot == NB) slot = 0, phase ^= 1;
      }
      __syncwarp();
      asm volatile("cp.async.wait_all;\n" ::: "memory");
      leave();
      if (warp == kMmaCopyWarp && lane == 0 && *abort_flag)  // the engine's copies in flight land before the CTA goes
        for (int k = issued > NB ? issued - NB : 0; k < issued; ++k)
          (void)mbar_wait(b_full + 8 * (k % NB), (uint32_t)((k / NB) & 1));
    }
  }
}

// Sum each band's segment partials in order and map its 4 coefficient rows to
// y (2G mix and 2^-3 with the lift, 2^3 without).  Thread per (pass, tile,
// column, band of the tile), the band fastest, so a warp reads 32 consecutive
// partials of one row and writes 32 consecutive 4-row groups of y.
// Its few FP64 additions are 16 clocks a warp each; powers of two go through the
// exponent instead.
template <bool LIFT>
__global__ void wz2_mma_finish(MmaPass single, const MmaPass* __restrict__ table, int n, int64_t threads, int64_t L) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= threads) return;
  const MmaPass ps = pass_of<true>(single, table, n, q);
  const int64_t ql = q - ps.fin_begin;
  const int bl = (int)(ql & 31);
  const int64_t tr = ql >> 5;  // tile * R + r
  const int r = (int)(tr % ps.R);
  const int64_t tile = tr / ps.R;
  const int64_t I = 32 * tile + bl;
  if (tile >= ps.tiles || 4 * I >= ps.M) return;
  const int64_t first = ps.item_begin + tile * ps.S;
  const int nseg = (int)((first + ps.S - 1) / L - first / L + 1);
  double z[4];
  for (int a = 0; a < 4; ++a)
    z[a] = seq_sum_strided(ps.ws + ((tile * ps.maxseg) * ps.R + r) * 128 + 32 * a + bl, nseg, (int64_t)ps.R * 128);
  double yy[4];
  if (LIFT) {
    const double a = times_pow2(z[0], 1), m = a - z[1], p = a + z[1];
    yy[0] = times_pow2(m - z[2], -3);
    yy[1] = times_pow2(m + z[2], -3);
    yy[2] = times_pow2(p - z[2] - z[3], -3);
    yy[3] = times_pow2(p + z[2] + z[3], -3);
  } else {
    for (int i = 0; i < 4; ++i) yy[i] = times_pow2(z[i], 3);
  }
  for (int i = 0; i < 4; ++i)
    if (4 * I + i < ps.M) ps.y[(int64_t)r * ps.ldy + 4 * I + i] = yy[i];
}

// state <- decay * state + y[:, r] for r = 0..R-1 in order.  Thread per row.
static __global__ void wz2_mma_state(const double* __restrict__ y, int64_t ldy, int R, int64_t M,
                                     double* __restrict__ state, double decay) {
  const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= M) return;
  double s = state[row];
  for (int r = 0; r < R; ++r) s = decay * s + y[(int64_t)r * ldy + row];
  state[row] = s;
}

}  // namespace dev
}  // namespace whff
