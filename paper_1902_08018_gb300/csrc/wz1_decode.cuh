// wz1_decode.cuh -- per-thread decoder of one WZ1 block (zfp-style fixed rate,
// Sec. 4.3).
//
// Steps: header (nonzero flag, biased exponent) -> embedded plane decode up
// to the 16*rate-9 bit budget (verbatim prefix bits + group tests, last
// coefficient implied) -> 32x16 bit-matrix transpose of the plane words into
// one word per coefficient -> negabinary to two's complement -> inverse lift
// (columns, then rows; mod 2^32, arithmetic shifts) -> 16 int32 values q.
//
// The parse is a chain of data-dependent steps that the 32 lanes of a warp take
// at different places, so what counts is warp iterations: one table lookup
// takes ten stream bits of a plane's group tests at once (nearly every plane is
// one lookup, whatever the lane's bits are), and once every lane's coefficients
// are all significant the rest is 16-bit planes, two to a 32-bit window.  The
// stream words and the plane words sit in shared memory, a column per thread (a
// lane's own index never conflicts).  One group test per iteration, 19 of 32
// lanes active, took 1881 warp instructions per 32 blocks at rate 16 (10000^2: 451 us,
// now 241; see wz1_gemv_kernel).
// The decoded matrix entry is (float)q * 2^(emax-26) (round to nearest even).
//
// Sec. 5.2 observes that zfp decoding is sequential within a stream and that
// the only parallelism is to give chunks to threads; in fixed-rate mode every
// 4x4 block is such a chunk, so one thread owns one block.
#pragma once
#include <cstdint>

namespace whff {
namespace dev {

// Row-major index 4*i + j of the k-th coefficient in sequency order.
__device__ __forceinline__ constexpr int seq_index(int k) {
  constexpr int t[16] = {0, 1, 4, 5, 2, 3, 8, 12, 6, 7, 9, 13, 10, 11, 14, 15};
  return t[k];
}

__device__ __forceinline__ uint32_t asr1(uint32_t v) { return (uint32_t)((int32_t)v >> 1); }

// Inverse lift of one 4-vector (s, d, d0, e) -> (x0, x1, x2, x3), mod 2^32.
__device__ __forceinline__ void inv_lift(uint32_t& a, uint32_t& b, uint32_t& c, uint32_t& d) {
  uint32_t s = a, dd = b, d0 = c, e = d;
  uint32_t d1 = e + d0;
  uint32_t s0 = s - asr1(dd);
  uint32_t s1 = dd + s0;
  a = s0 - asr1(d0);
  b = d0 + a;
  c = s1 - asr1(d1);
  d = d1 + c;
}

// Swap of bit groups between two words of a bit matrix (s = 1, 2, 4; m the low
// group of each pair): a keeps its low groups and takes b's low ones above them.
__device__ __forceinline__ void dswap(uint32_t& a, uint32_t& b, int s, uint32_t m) {
  const uint32_t hi = a >> s;
  a = (a & m) | ((b << s) & ~m);
  b = (hi & m) | (b & ~m);
}

// Group tests of a plane, kTestBits stream bits at a time.  A plane's tests read
// T S..S T S..S T ...: a test bit T (0 ends the plane), then one bit S per
// position up to and including the first one.  The entry of (state, bits), the
// state being before a T (0) or inside an S run (1): bits 0-11 the S bits in
// order, 12 stopped inside an S run, 13 a zero T was met, byte 2 the stream bits
// taken, byte 3 the number of S bits.
constexpr int kTestBits = 10;
constexpr int kTestEntries = 2 << kTestBits;
constexpr uint32_t kInScan = 1u << 12, kPlaneDone = 1u << 13;
struct TestTable {
  uint32_t e[kTestEntries];
};
constexpr TestTable make_test_table() {
  TestTable t{};
  for (int i = 0; i < kTestEntries; ++i) {
    bool scan = i >> kTestBits, end = false;
    uint32_t out = 0, cnt = 0, pos = 0;
    while (pos < (uint32_t)kTestBits && !end) {
      const bool bit = (i >> pos) & 1;
      ++pos;
      if (!scan) {
        scan = bit;
        end = !bit;
      } else {
        if (bit) out |= 1u << cnt;
        ++cnt;
        scan = !bit;
      }
    }
    t.e[i] = out | (scan && !end ? kInScan : 0u) | (end ? kPlaneDone : 0u) | pos << 16 | cnt << 24;
  }
  return t;
}
alignas(16) static __device__ const TestTable kTestTable = make_test_table();

// Shared memory of a block of TH threads decoding NW32-word blocks: per thread a
// column of stream words (two zero words follow) and one of 16 plane pairs
// (plane k in half k % 2 of word k / 2), and the table.
template <int NW32, int TH>
struct Wz1Smem {
  uint32_t words[(NW32 + 2) * TH];
  uint32_t planes[16 * TH];
  alignas(16) uint32_t table[kTestEntries];
};

// Once per block, before the first decode; ends with a barrier.  16 bytes at a
// time, and a caller with one block a thread asks for its words first: a small
// matrix is bound by these latencies.
template <int NW32, int TH>
__device__ __forceinline__ void wz1_smem_init(Wz1Smem<NW32, TH>& sm) {
  static_assert(kTestEntries % 4 == 0, "whole 16-byte pieces");
  for (int i = threadIdx.x; i < kTestEntries / 4; i += TH)
    reinterpret_cast<uint4*>(sm.table)[i] = reinterpret_cast<const uint4*>(kTestTable.e)[i];
  sm.words[NW32 * TH + threadIdx.x] = sm.words[(NW32 + 1) * TH + threadIdx.x] = 0u;
  __syncthreads();
}

// 32 stream bits from bit pos on (pos < 32 (NW32 + 1)); zeros past the block.
template <int TH>
__device__ __forceinline__ uint32_t wz1_window(const uint32_t* __restrict__ words, int pos) {
  const uint32_t* p = words + (pos >> 5) * TH;
  return __funnelshift_r(p[0], p[TH], pos);
}

// Decode the plane stream (after the 9 header bits) of the block whose words
// are w: the 16 negabinary words u[k] in sequency order.  Bits past the budget
// read as zeros, which end a plane as the budget does; only the implied last
// coefficient has to look at the budget itself.
template <int NW32, int TH>
__device__ __forceinline__ void decode_planes(const uint32_t (&w)[NW32], Wz1Smem<NW32, TH>& sm, uint32_t (&u)[16]) {
  constexpr int kEnd = 32 * NW32;  // 16*rate bits, rate = 2*NW32
  uint32_t* words = sm.words + threadIdx.x;
  uint32_t* planes = sm.planes + threadIdx.x;
#pragma unroll
  for (int i = 0; i < NW32; ++i) words[i * TH] = w[i];
#pragma unroll
  for (int i = 0; i < 16; ++i) planes[i * TH] = 0u;
  auto put = [&](int k, uint32_t p) {  // plane k
    reinterpret_cast<uint16_t*>(planes + (k >> 1) * TH)[k & 1] = (uint16_t)p;
  };

  // leading empty planes: a zero test each, while nothing is significant yet
  const uint32_t lead = wz1_window<TH>(words, 9);
  const int z0 = lead ? __ffs(lead) - 1 : 32;
  int pos = 9 + z0, k = 31 - z0, n = 0;
#pragma unroll 1
  for (; n < 16 && k >= 0 && pos < kEnd; --k) {  // n: coefficients significant so far
    const uint32_t win = wz1_window<TH>(words, pos);
    uint32_t p = win & ((1u << n) - 1u), src = win >> n;
    pos += n;
    int scan = 0;
#pragma unroll 1
    for (;;) {
      const uint32_t e = sm.table[(scan << kTestBits) | (src & ((1u << kTestBits) - 1u))];
      const int cnt = (int)(e >> 24), run = 15 - n;  // positions n..14 have bits of their own
      uint32_t out = e & 0xFFFu;
      if (cnt > run || (cnt == run && (e & kInScan))) {  // the scan went past position 14: 15 is implied
        out &= (1u << run) - 1u;
        pos += run + __popc(out) + (1 - scan);
        p |= out << n;
        if (pos <= kEnd) p |= 1u << 15;
        n = 16;
        break;
      }
      p |= out << n;
      n += cnt;
      pos += (int)((e >> 16) & 255u);
      if (e & kPlaneDone) break;
      scan = e & kInScan ? 1 : 0;
      src = wz1_window<TH>(words, pos);
    }
    put(k, p);
  }
  if (!(k & 1) && k >= 0 && pos < kEnd) {  // whole planes: an even one alone ...
    put(k, wz1_window<TH>(words, pos));
    --k, pos += 16;
  }
  if (k >= 0 && pos < kEnd) {  // ... then (k, k - 1), one word of the stream and one of the planes at a time
    const uint32_t* src = words + (pos >> 5) * TH;
    uint32_t* dst = planes + (k >> 1) * TH;
    const uint32_t* last = src + (min(k >> 1, (kEnd - 1 - pos) >> 5)) * TH;
    uint32_t lo = *src;
#pragma unroll 1
    for (;;) {
      const uint32_t hi = src[TH];
      *dst = __byte_perm(__funnelshift_r(lo, hi, pos), 0u, 0x1032);
      if (src == last) break;
      lo = hi, src += TH, dst -= TH;
    }
  }

  // Transpose the 32 (plane) x 16 (coefficient) bit matrix: bit k of u[i] = bit
  // i of plane k.  The index bits of word (w3 w2 w1 w0) and bit (b4 .. b0), at
  // first plane (k4 k3 k2 k1) and (k0, c3 c2 c1 c0), are exchanged w3-b4, w3-b0,
  // w2-b3, w1-b2, w0-b1; coefficient (c3 c2 c1 c0) ends in word (c0 c3 c2 c1).
  uint32_t A[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) A[i] = planes[i * TH];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t a = A[i], b = A[i + 8];
    A[i] = __byte_perm(a, b, 0x5410);
    A[i + 8] = __byte_perm(a, b, 0x7632);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) dswap(A[i], A[i + 8], 1, 0x55555555u);
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (!(i & 4)) {
      const uint32_t a = A[i], b = A[i + 4];
      A[i] = __byte_perm(a, b, 0x6240);
      A[i + 4] = __byte_perm(a, b, 0x7351);
    }
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (!(i & 2)) dswap(A[i], A[i + 2], 4, 0x0F0F0F0Fu);
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (!(i & 1)) dswap(A[i], A[i + 1], 2, 0x33333333u);
#pragma unroll
  for (int i = 0; i < 16; ++i) u[i] = A[((i & 1) << 3) | (i >> 1)];
}

// Decode one block: q (row-major) after the inverse transform, and emax; false
// for a zero block, whose q mean nothing.
template <int NW32, int TH>
__device__ __forceinline__ bool decode_block(const uint32_t (&w)[NW32], Wz1Smem<NW32, TH>& sm, int32_t (&q)[16],
                                             int& emax) {
  const bool nz = w[0] & 1u;
  emax = (int)((w[0] >> 1) & 0xFFu) - 127;
  uint32_t u[16];
  decode_planes<NW32, TH>(w, sm, u);
  uint32_t c[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) c[seq_index(k)] = (u[k] ^ 0xAAAAAAAAu) - 0xAAAAAAAAu;
#pragma unroll
  for (int j = 0; j < 4; ++j) inv_lift(c[j], c[4 + j], c[8 + j], c[12 + j]);
#pragma unroll
  for (int r = 0; r < 4; ++r) inv_lift(c[4 * r], c[4 * r + 1], c[4 * r + 2], c[4 * r + 3]);
#pragma unroll
  for (int i = 0; i < 16; ++i) q[i] = (int32_t)c[i];
  return nz;
}

// Load one block's words (2*rate bytes at a 2*rate-byte-aligned address).
template <int NW32>
__device__ __forceinline__ void load_block(const uint8_t* __restrict__ base, int64_t blk, uint32_t (&w)[NW32]) {
  const uint8_t* p = base + (uint64_t)blk * (uint64_t)(4 * NW32);
  if constexpr (NW32 % 4 == 0) {
#pragma unroll
    for (int i = 0; i < NW32 / 4; ++i) {
      uint4 v = __ldcs(reinterpret_cast<const uint4*>(p) + i);
      w[4 * i] = v.x;
      w[4 * i + 1] = v.y;
      w[4 * i + 2] = v.z;
      w[4 * i + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < NW32 / 2; ++i) {
      uint2 v = __ldcs(reinterpret_cast<const uint2*>(p) + i);
      w[2 * i] = v.x;
      w[2 * i + 1] = v.y;
    }
  }
}

}  // namespace dev
}  // namespace whff
