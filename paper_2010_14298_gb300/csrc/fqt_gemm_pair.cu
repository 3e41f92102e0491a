// fqt_gemm_pair.cu -- the instances of k_gemm that run on CTA pairs
// (cta_group::2, 256 x 256 super tiles), and k_gemm_wide, split-K partials of
// few rows; fqt_gemm.cu chooses between them and the single-CTA instances.
#include "fqt_gemm_core.cuh"

namespace fqt {

GemmKernel gemm_pair_kernel(int mode, int nb, int form) {
  if (mode == MODE_PARTIAL) return k_gemm<MODE_PARTIAL, 1, 0, true>;
#define FQT_GXP(NBV)                                                         \
  case NBV:                                                                  \
    return form == 2   ? k_gemm<MODE_GRADX, NBV, 2, true>                    \
           : form == 1 ? k_gemm<MODE_GRADX, NBV, 1, true>                    \
                       : k_gemm<MODE_GRADX, NBV, 0, true>;
  switch (nb) {
    FQT_GXP(1)
    FQT_GXP(4)
    FQT_GXP(8)
    FQT_GXP(16)
    FQT_GXP(32)
    FQT_GXP(64)
  }
#undef FQT_GXP
  return nullptr;
}

// ---------------------------------------------------------------------------
// grad_W partials where C fills at most one tile of 128 rows: a CTA takes g.wn
// = 128, 192 or 256 columns of X~ against all of C, so that Q_b1 is read for
// fewer column tiles and the MMA is up to 256 columns wide (with C = 64 half
// of its lanes are idle: a second atom of A past C is not even loaded).  Two
// accumulators of 256 columns alternate by exact chunk, the running sums in
// registers, as for pairs.
// With an implicit im2col operand (g.taps) the column atoms of a tile are the
// taps of one kernel row, for 64 channels: one copy of the pixels of the K
// block and of the kw - 1 beside them serves all of them, since the operand
// of tap x starts x pixels (128-byte rows) into it; the leading byte offset
// between the atoms is one row, and the swizzle follows the address.
// What bounds it: the operand copies through L2 without g.taps, then the MMAs
// (0.30 us per K block of 128 x 192, with C = 64 as with 128).
// 64 x 576 over the 802816 pixels of 256 x 56 x 56: 195 us in tiles of 128
// (all nine taps' columns, 925 MB, pass through L2), 122 with 192 columns, 98
// with one copy per kernel row.
// ---------------------------------------------------------------------------
using WideLayout = GemmLayout<MODE_PARTIAL, 0, 1, true>;

// B's bytes in a stage are a multiple of 1024 (swizzle atoms)
size_t gemm_wide_smem(uint32_t b_bytes, int stages) {
  return kFixedBytes + (size_t)stages * ((size_t)kTileBytes + b_bytes) +
         (size_t)kPartialEpiWarps * kBoxBytes + 1024;
}

__global__ void __launch_bounds__(WideLayout::threads, 1)
    k_gemm_wide(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const __grid_constant__ CUtensorMap tmOut, const GemmArgs g) {
  extern __shared__ __align__(1024) uint8_t wide_raw[];
  uint8_t *smem = wide_raw + ((1024u - (smem_u32(wide_raw) & 1023u)) & 1023u);
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kOffBar);
  uint8_t *ops = smem + kFixedBytes;
  // pixels from one image row of a stage to the next (g.taps)
  const uint32_t pitch = (uint32_t)(g.cpw + g.taps - 1);
  const uint32_t b_tx = g.taps ? (uint32_t)g.crpb * pitch * 128u : (uint32_t)g.wn * 128u;
  const uint32_t stage = (uint32_t)kTileBytes + ((b_tx + 1023u) & ~1023u);
  uint8_t *ring = ops + (size_t)g.stages * stage;
  uint64_t *full = bars, *empty = bars + kMaxStages;
  uint64_t *accf = bars + 2 * kMaxStages, *acce = accf + 4, *drain = acce + 4;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + kNumBars);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < g.stages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(&accf[i], 1);
      mbar_init(&acce[i], 4);  // the four warps of the half
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == kWarpMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  if (warp >= kGemmWarpEpi0) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(WideLayout::regs_epi));
    partial_epilogue_pair<true>(g, smem, ring, accf, acce, tmem, &tmOut, abort_flag, warp, lane);
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(WideLayout::regs_ctl));
    if (warp == kWarpTma && lane == 0) {
      // ---------------------------------------------------------- producer
      int s = 0;
      uint32_t ph = 0;
      const int nbox = g.wn / 64;
      Item t;
      bool ok = true;
      for (int64_t local = 0; ok && wide_item(g, local, t) && !*abort_flag; local += 2) {
        const bool two = g.M - t.m0 > 64;
        const uint32_t bytes = (uint32_t)(kTileBytes / 2) * (two ? 2u : 1u) + b_tx;
        // implicit im2col (see k_gemm's producer)
        int cimg = 0, cyb = 0, ccg[4] = {0, 0, 0, 0}, cx[4] = {0, 0, 0, 0}, cy[4] = {0, 0, 0, 0};
        if (g.conv) {
          cimg = (int)(t.kb0 / g.cybi);
          cyb = (int)(t.kb0 - (int64_t)cimg * g.cybi);
          if (g.taps) {
            const int tile = (int)t.n0 / g.wn, gpr = g.cin / 64;
            cy[0] = tile / gpr - g.cpad;
            ccg[0] = (tile % gpr) * 64;
            cx[0] = -g.cpad;
          }
          for (int h = 0; h < 4 && !g.taps; ++h) {
            const int d = (int)t.n0 + 64 * h, tap = d / g.cin, ky = tap / g.ckw;
            ccg[h] = d - tap * g.cin;
            cx[h] = tap - ky * g.ckw - g.cpad;
            // past the last tap: a box outside the tensor (zeros)
            cy[h] = d < g.N ? ky - g.cpad : g.cih + g.coh + 8;
          }
        }
        for (int64_t kb = t.kb0; kb < t.kb1; ++kb) {
          ok = mbar_wait(&empty[s], ph ^ 1u, g.status);
          if (!ok) break;
          mbar_expect_tx(&full[s], bytes);
          uint8_t *sa = ops + (size_t)s * stage, *sb = sa + kTileBytes;
          const int32_t kc = (int32_t)(kb * BK);
          if (g.conv) {
            const int oy0 = cyb * g.crpb;
            tma_load_4d(sa, &tmA, (int32_t)t.m0, 0, oy0, cimg, &full[s]);
            if (two)
              tma_load_4d(sa + kTileBytes / 2, &tmA, (int32_t)t.m0 + 64, 0, oy0, cimg, &full[s]);
#pragma unroll
            for (int h = 0; h < 4; ++h)
              if (h < (g.taps ? 1 : nbox))
                tma_load_4d(sb + h * (kTileBytes / 2), &tmB, ccg[h], cx[h], oy0 + cy[h], cimg,
                            &full[s]);
            if (++cyb == g.cybi) { cyb = 0; ++cimg; }
          } else {
            tma_load_2d(sa, &tmA, (int32_t)t.m0, kc, &full[s]);
            if (two) tma_load_2d(sa + kTileBytes / 2, &tmA, (int32_t)t.m0 + 64, kc, &full[s]);
            for (int h = 0; h < nbox; ++h)
              tma_load_2d(sb + h * (kTileBytes / 2), &tmB, (int32_t)t.n0 + 64 * h, kc, &full[s]);
          }
          if (++s == g.stages) { s = 0; ph ^= 1u; }
        }
      }
      if (!ok) *abort_flag = 1;
      if (*abort_flag) {
        sleep_ns(200000);  // copies in flight land before the CTA exits
      } else {
        for (int i = 0; i < g.stages; ++i) {
          if (!mbar_wait(&empty[s], ph ^ 1u, g.status)) break;
          if (++s == g.stages) { s = 0; ph ^= 1u; }
        }
      }
    } else if (warp == kWarpMma && lane == 0) {
      // -------------------------------------------------------- MMA issuer
      int s = 0, b = 0;
      uint32_t ph = 0, aph = 0u;
      const uint32_t idesc = make_idesc(true, true, BM, g.wn);
      // B of the K steps of 16 rows: offset of each (in 16 bytes), and the
      // strides between its column atoms and its groups of eight rows
      uint32_t b_lbo = g.mn_lbo, b_sbo = g.mn_sbo, boff[BK / 16];
      for (int k = 0; k < BK / 16; ++k) boff[k] = (2048u >> 4) * k;
      if (g.taps) {
        b_lbo = 128u;
        if (g.cpw < 16) b_sbo = pitch * 128u;
        for (int k = 0; k < BK / 16; ++k)
          boff[k] = (uint32_t)(16 * k / g.cpw * (int)pitch + 16 * k % g.cpw) * 8u;
      }
      Item t;
      bool ok = true;
      for (int64_t local = 0; ok && wide_item(g, local, t) && !*abort_flag; local += 2) {
        for (int64_t c0 = t.kb0; ok && c0 < t.kb1; c0 += g.kc_blocks) {
          const int64_t c1 = min(t.kb1, c0 + g.kc_blocks);
          const uint32_t par = ((aph >> b) & 1u) ^ 1u;
          ok = mbar_wait(&acce[2 * b], par, g.status) &&
               mbar_wait(&acce[2 * b + 1], par, g.status);
          if (!ok) break;
          tc_fence_after();
          const uint32_t dt = tmem + (uint32_t)(b * 2 * BN);
          for (int64_t kb = c0; kb < c1; ++kb) {
            ok = mbar_wait(&full[s], ph, g.status);
            if (!ok) break;
            tc_fence_after();
            const uint32_t a_addr = smem_u32(ops + (size_t)s * stage);
            const uint64_t da = sw128_desc_mn(a_addr, g.mn_lbo, g.mn_sbo);
            const uint64_t db = sw128_desc_mn(a_addr + (uint32_t)kTileBytes, b_lbo, b_sbo);
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
              umma_f16(dt, da + (2048u >> 4) * k, db + boff[k], idesc,
                       (kb > c0 || k > 0) ? 1u : 0u);
            umma_commit(&empty[s]);
            if (++s == g.stages) { s = 0; ph ^= 1u; }
          }
          umma_commit(&accf[2 * b]);
          umma_commit(&accf[2 * b + 1]);
          aph ^= 1u << b;
          b ^= 1;
        }
      }
      if (!ok) *abort_flag = 1;
      umma_commit(drain);  // every MMA has completed before TMEM is released
      mbar_wait(drain, 0, g.status);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kTmemCols)
                 : "memory");
  }
}

}  // namespace fqt
