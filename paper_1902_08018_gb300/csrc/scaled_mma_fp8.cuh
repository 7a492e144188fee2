// scaled_mma_fp8.cuh -- the tensor-core pass for FP8 E4M3 storage with A in TMEM.
//
// The roles of wz2_mma_kernel on the items of the scaled formats: a tiled copy
// brings a stage's 128 rows x 64 bytes, twelve warps widen E4M3 to BF16 (exactly)
// and store it to TMEM, one elected lane issues the MMAs, eight warps drain, scale
// and sum.  Same MMAs, same groups (the two stages of a scale tile), same ranges as
// scaled_mma_kernel<FP8>, which host-resident matrices keep: the same bits.
//
// Bound: the issuing warp's turn-around per stage, as in wz2_mma_kernel (HBM would
// take 23 us).  The register-fed kernel gave every stage a barrier of the whole CTA.
// 32 columns at 12288^2: 114.7 us a pass with it, 77.8 with this one.
#pragma once
#include <cuda.h>

#include "scaled_mma.cuh"

namespace whff {
namespace dev {

// Item ranges of a CTA at most: those of a grid of two CTAs per SM (see kMmaRanges).
constexpr int kFp8Ranges = 2;

template <int NR>
struct Fp8Smem {
  static constexpr int kNA = 6;  // A buffers in TMEM
  static constexpr int kB = MmaBTile<NR>::kB;
  static constexpr int kNB = 8;
  static constexpr int kWords = 128 * 64;  // the stage's box
  static constexpr int kBars = kNB * (kB + kWords);
  static constexpr int kBytes = kBars + 512;
};

// Eight 32-bit columns of each lane's own row to TMEM.
__device__ __forceinline__ void tmem_store_32x32_8(uint32_t taddr, const uint32_t (&a)[4], const uint32_t (&b)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"r"(taddr), "r"(a[0]),
               "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3])
               : "memory");
}

template <int NR>
__global__ void __launch_bounds__(kMmaDecodeThreads, 1)
    fp8_mma_kernel(const __grid_constant__ CUtensorMap tmap, int64_t row0, const float* __restrict__ scales, int64_t TN,
                   const uint8_t* __restrict__ btiles, double* __restrict__ ws, int S, int R, int maxseg, int64_t total,
                   int64_t L, int per_cta, int* __restrict__ status, uint32_t spin) {
  using SM = Fp8Smem<NR>;
  constexpr int NB = SM::kNB, NA = SM::kNA, NQ = kMmaQuartets;
  constexpr int HALF = NR / 2;  // columns drained by each of the two warps on a lane quarter
  constexpr uint32_t kACols = 8 * kMmaKSteps;  // TMEM columns of a stage's A
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t s_base = smem_addr(smem);
  const uint32_t b_full = s_base + SM::kBars;  // NB: the B tile in the slot has landed
  const uint32_t w_full = b_full + 8 * NB;     // NB: so have its stored values
  const uint32_t done = w_full + 8 * NB;       // NB: the MMAs of the stage in the slot are done
  const uint32_t a_full = done + 8 * NB;       // NA: the stage's A pieces are in the buffer (4 arrivals)
  const uint32_t gfull = a_full + 8 * NA;      // 2: the accumulator group is complete
  const uint32_t gfree = gfull + 16;           // 2: the accumulator group has been drained (8 arrivals)
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + SM::kBars + 8 * (3 * NB + NA + 4));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);

  // broadcast, so that the compiler knows the roles to be warp-uniform
  const int t = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, t >> 5, 0), lane = t & 31;
  const int64_t it0 = (int64_t)blockIdx.x * per_cta * L;
  const int n = (int)max((int64_t)0, min(total, it0 + per_cta * L) - it0);  // stages of this CTA
  const int len = (int)L;
  if (t == 0) {
    for (int i = 0; i < NB; ++i)
      mbar_init(b_full + 8 * i, 1), mbar_init(w_full + 8 * i, 1), mbar_init(done + 8 * i, 1);
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

  // Cursor (tile, stage): advances in item order, so the loops have no divisions.
  int c_tile = n > 0 ? (int)(it0 / S) : 0, c_st = n > 0 ? (int)(it0 - (int64_t)c_tile * S) : 0;
  auto advance = [&]() {
    if (++c_st == S) c_st = 0, ++c_tile;
  };
  // Whether the item at the cursor, with range_left items of its range to go and
  // stage k of this CTA, closes its accumulator group: the two stages of a scale tile.
  auto closes = [&](int gpos, int range_left, int k) {
    return gpos + 1 == kMmaDrainStages || (c_st & 1) || c_st == S - 1 || range_left == 1 || k == n - 1;
  };

  // every role's end: nothing more goes to TMEM or is read from it
  auto leave = [&]() {
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
  };
  if (warp >= kMmaDecodeWarp && warp < kMmaDrainWarp) {
    // ---- decode: quartet q takes stages q, q + NQ, ...; a thread a row of the tile: its 64
    // bytes (16-byte pieces swizzled by the tiled copy: piece c of row r is at c ^ (r / 2 % 4))
    // become 32 pairs of BF16, exactly.
    const int q = (warp - kMmaDecodeWarp) >> 2, quarter = warp & 3;
    const int row = 32 * quarter + lane, sw = (row >> 1) & 3;
    for (int k = q; k < n; k += NQ) {
      if (!warp_wait(w_full + 8 * ((uint32_t)k % NB), (uint32_t)k / NB & 1u)) break;  // the values are here
      if (k >= NA) {  // the A buffer is free once the MMAs of the stage NA before are done
        const uint32_t p = (uint32_t)(k - NA);
        if (!warp_wait(done + 8 * (p % NB), p / NB & 1u)) break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const uint32_t a_row = a_cols((uint32_t)k) + ((uint32_t)(32 * quarter) << 16);
      const uint4* vals = reinterpret_cast<const uint4*>(smem + NB * SM::kB + (uint32_t)k % NB * SM::kWords) + 4 * row;
#pragma unroll
      for (int c = 0; c < 4; ++c) {  // 16 values: one K step
        uint32_t d[2][1][4];
        scaled_mma_pieces<4>(vals[c ^ sw], d);
        __syncwarp();
        tmem_store_32x32_8(a_row + 8 * c, d[0][0], d[1][0]);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(a_full + 8 * ((uint32_t)k % NA));
    }
    asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
    leave();
  } else if (warp >= kMmaDrainWarp) {
    // ---- drain: TMEM lane 32 quarter + lane holds that row of the tile.  A group's three
    // accumulators are added, scaled and enter TwoSum sums as in scaled_mma_kernel.
    const int quarter = warp & 3, c0 = HALF * ((warp - kMmaDrainWarp) >> 2);
    const uint32_t rows = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)c0;
    float hi[HALF], lo[HALF];
#pragma unroll
    for (int r = 0; r < HALF; ++r) hi[r] = lo[r] = 0.f;
    int cur_tile = c_tile;  // tile of the sums
    int v = (int)blockIdx.x * per_cta, left = len;  // the range, and its items from here on
    auto flush = [&](int range) {
      const int64_t seg = range - ((int64_t)cur_tile * S) / L;
      double* dst = ws + (((int64_t)cur_tile * maxseg + seg) * R) * 128 + 32 * quarter + lane;
#pragma unroll
      for (int r = 0; r < HALF; ++r) {
        if (c0 + r < R) dst[(int64_t)(c0 + r) * 128] = widen(hi[r]) + widen(lo[r]);
        hi[r] = lo[r] = 0.f;
      }
    };
    int gpos = 0, acc = 0;
    uint32_t parity = 0;
    bool open = false, alive = true;
    for (int k = 0; k < n; ++k) {
      const int tile = c_tile, tc = c_st >> 1;
      const bool ends = closes(gpos, left, k);
      gpos = ends ? 0 : gpos + 1;
      advance();
      if (ends) {
        const float s = __ldg(scales + (int64_t)tile * TN + tc);
        if (!warp_wait(gfull + 8 * acc, parity)) {
          alive = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (open && tile != cur_tile) flush(v);
        cur_tile = tile, open = true;
        const uint32_t ta = rows + (uint32_t)(3 * acc * NR);
#pragma unroll
        for (int h = 0; h < HALF; h += 8) {
          float x[8];
          tmem_load_sum8(ta + h, NR, x);
#pragma unroll
          for (int r = 0; r < 8; r += 2) {  // packed pairs of columns: each half rounds as the scalar steps
            const float2 ps = make_float2(__fmul_rn(x[r], s), __fmul_rn(x[r + 1], s));
            float2 H = make_float2(hi[h + r], hi[h + r + 1]), Lo = make_float2(lo[h + r], lo[h + r + 1]);
            two_sum_acc2(H, Lo, ps);
            Lo = add_f2(Lo, fma_f2(make_float2(x[r], x[r + 1]), make_float2(s, s), make_float2(-ps.x, -ps.y)));
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
          // A [B_0 B_1 B_2] into the three accumulators, the group's first K step starting them
          const uint64_t bd0 = b_desc0 + (uint64_t)((slot * SM::kB) >> 4);
          const uint32_t d0 = tmem + (uint32_t)(3 * acc * NR), a0 = a_cols((uint32_t)buf);
#pragma unroll
          for (int ks = 0; ks < kMmaKSteps; ++ks) {
            const uint32_t ad = a0 + (uint32_t)(8 * ks);
            const uint64_t bd = bd0 + (uint64_t)((3 * ks * MmaBTile<NR>::kBTile) >> 4);
            const uint32_t accumulate = (init && ks == 0) ? 0u : 1u;
            asm volatile(
                "{\n\t.reg .pred p;\n\t"
                "setp.ne.b32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d0),
                "r"(ad), "l"(bd), "r"(mma_idesc(3 * NR)), "r"(accumulate));
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
    } else if (warp == kMmaCopyWarp) {
      // ---- copies, NB stages ahead: the stage's 64 columns of 128 rows (zeros past the matrix)
      // and its B tile.  A slot is refilled once the MMAs of its stage are done.
      int issued = 0, slot = 0;
      uint32_t phase = 1;  // the slots are free at first
      for (; issued < n; ++issued) {
        if (!warp_wait(done + 8 * slot, phase)) break;
        if (elect_one()) {
          bulk_copy_g2s(s_base + slot * SM::kB, btiles + (int64_t)c_st * SM::kB, (uint32_t)SM::kB, b_full + 8 * slot);
          mbar_expect_tx(w_full + 8 * slot, (uint32_t)SM::kWords);
          tma_load_2d(s_base + NB * SM::kB + slot * SM::kWords, &tmap, 64 * c_st, (int)(row0 + 128 * (int64_t)c_tile),
                      w_full + 8 * slot);
        }
        __syncwarp();
        advance();
        if (++slot == NB) slot = 0, phase ^= 1;
      }
      __syncwarp();
      leave();
      if (lane == 0 && *abort_flag)  // the copies in flight land before the CTA goes
        for (int k = issued > NB ? issued - NB : 0; k < issued; ++k) {
          (void)mbar_wait(b_full + 8 * (k % NB), (uint32_t)((k / NB) & 1));
          (void)mbar_wait(w_full + 8 * (k % NB), (uint32_t)((k / NB) & 1));
        }
    } else {
      leave();
    }
  }
}

}  // namespace dev
}  // namespace whff
