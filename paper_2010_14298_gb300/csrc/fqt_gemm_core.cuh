// fqt_gemm_core.cuh -- the tensor-core contraction kernel k_gemm and its
// epilogues, shared by the translation units that instantiate it.  The head
// of fqt_gemm.cu describes the kernel.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "fqt_common.cuh"
#include "fqt_internal.h"

namespace fqt {

constexpr int BM = 128, BN = 128, BK = 64;
constexpr int kMaxStages = 8;  // operand stages (A and B fp16 tiles), chosen per launch
constexpr int kWarpTma = 0, kWarpMma = 1, kWarpEpi0 = 2;  // k_gradw's roles
constexpr int kPartialEpiWarps = 8;
// k_gemm: warpgroup 0 holds the TMA producer, the MMA issuer and grad_X's
// per-tile parameter loader (warp 3 idles); the epilogue warps follow in
// sets of four (one per TMEM lane quadrant) that take the tiles in turn.
// The epilogue's arithmetic comes in three forms (FORM):
//   0  int32 integer parts (several exact chunks, or the fp32 form's offset
//      bound below 0);
//   1  the fp32 form for tiles whose row offsets allow it, int32 for the
//      others, in the same epilogue (the fp32 form's offset bound is small);
//   2  the fp32 form only.
// In every form the rare tiles outside it (a row offset m beyond the int32
// form's, or the fp32 form's in FORM 2) are stored raw and finished by the
// CTA after its last tile (gradx_raw_fix).
// FORM 2 has four sets: without the int32 path, warpgroup 0 can hand
// registers to the epilogue warpgroups (setmaxnreg) and 104 per thread
// suffice (96 for blocks of up to 16 rows, whose parameter loader keeps 80); tiles with a long reduction use three of the sets (g.sets), so
// that the tensor cores fill a fourth accumulator while three are drained.
// Otherwise three sets at 128 registers; split-K partials use the first
// eight epilogue warps.
constexpr int kGemmWarpPar = 2, kGemmWarpEpi0 = 4;
// A pair's partials (PAIR, MODE 1) keep their int32 running sums in the
// registers of two sets (128 columns each, 128 sums per thread).
template <int MODE, int FORM, int NB = 16, bool PAIR = false>
struct GemmLayout {
  static constexpr int sets = (MODE == 0 && FORM == 2) ? 4 : (MODE == 1 && PAIR) ? 2 : 3;
  static constexpr int threads = 32 * (kGemmWarpEpi0 + 4 * sets);
  // registers per thread of the launch, and the split (0: no setmaxnreg)
  static constexpr int launch_regs = ((65536 / threads) / 8) * 8;
  static constexpr int regs_ctl = sets == 4 ? (NB <= 16 ? 80 : 64) : sets == 2 ? 80 : 0;
  static constexpr int regs_epi = sets == 4 ? (NB <= 16 ? 96 : 104) : sets == 2 ? 208 : 0;
  static_assert(regs_ctl == 0 || 128 * regs_ctl + 32 * 4 * sets * regs_epi <= threads * launch_regs,
                "register split above the launch's registers");
};
// two 128-column fp32 accumulators and 256 columns of int32 running sums
constexpr uint32_t kTmemCols = 512;

constexpr size_t kTileBytes = 16384;  // one 128 x 64 fp16 operand tile
constexpr size_t kBoxBytes = 4096;   // one 32 x 32 fp32 / int32 output box
// Shared memory, from a 1024-byte-aligned base:
//   [0, kFixedBytes)           per-warp epilogue tables and barriers
//   [kFixedBytes, +S * 32 KiB) S operand stages (A, B)
//   [..., + 8 * R * 4 KiB)     R output boxes per epilogue warp (TMA store ring)
// grad_X parameter stages (one per tile in flight), each:
//   RowPar kp      per row k: inv_sw inv_s_k, .. hz_k, .. y hr_k, m_k
//   int leads[BN]  lead row of each block;  int msum[BN]  sum of m per block
//   int cs[BM]     W~ column sums of the tile's columns;  int flag
constexpr int kParStages = 4;
constexpr size_t kParBytes = 4096;
constexpr size_t kParLeads = 2048, kParMsum = 2560, kParCs = 3072, kParFlag = 3584;
constexpr size_t kOffPar = 0;
constexpr size_t kOffBar = kOffPar + kParStages * kParBytes;
// operand full / empty, accumulator full / empty (4 each), parameter full /
// empty (4 each)
// ... + the MMA drain barrier + the byte-operand rings' barriers (carrier
// stage widened, carrier stage consumed)
constexpr size_t kNumBars = 4 * kMaxStages + 17;
// grad_X in the fp32 form with fixed blocks: one bit per tile of this CTA
// (in its order) for the tiles left raw, finished by the CTA at the end
constexpr size_t kOffRaw = (kOffBar + kNumBars * 8 + 16 + 15) & ~(size_t)15;
constexpr size_t kRawMaskBytes = 4096;
constexpr int64_t kMaxLocalTiles = (int64_t)kRawMaskBytes * 8;
constexpr size_t kFixedBytes = (kOffRaw + kRawMaskBytes + 1023) & ~(size_t)1023;

// Operand stages: `stages` of the A and B fp16 tiles (32 KB), and with byte
// operands (split-K partials) `ustages` of their 8 KB byte tiles as TMA wrote
// them (16 KB), a deeper ring of their own in front of the carrier ring.
__host__ __device__ constexpr size_t gemm_smem_bytes(int stages, int ring, int ustages = 0) {
  return kFixedBytes + (size_t)stages * 2 * kTileBytes + (size_t)ustages * kTileBytes +
         (size_t)kPartialEpiWarps * ring * kBoxBytes + 1024;  // + alignment slack
}

// MODE_GRADX: grad_X^T = W~^T Q_b2(dH)^T, i.e. M = D (output columns of
// grad_X, TMEM lanes), N = rows of dH (TMEM columns), K = C, with the
// dequantizing epilogue.  MODE_PARTIAL: raw int32 split-K partials.
enum { MODE_GRADX = 0, MODE_PARTIAL = 1 };

// Dequantization of grad_W's integer products (k_reduce, and the epilogue of
// a pair's partials when one split covers the reduction).
struct ReduceArgs {
  const int32_t *part;
  int splits;
  int64_t M, N;
  int64_t *out_i64;  // raw sums (debug)
  float *out_f32;    // grad_W
  // grad_W = inv_s1 inv_sx sum_n (a_nc + z'_1)(x_nd + z'_x)
  int64_t Kn;        // rows N of dH / X
  int oa, ob;
  // an implicit im2col X~: its padding entered the product as code 2^(bx-1);
  // P += (code(0) - ob) pad_a[tap(d)][c], pad_a = the A carriers summed over
  // the rows whose tap reads padding (taps x C), tap(d) = d / cin
  const int32_t *pad_a, *code_zero;
  int taps, cin;
  const int32_t *cs_a, *cs_b;  // column sums of Q_b1 codes (M) and X~ codes (N)
  const float *inv_a, *zero_a, *inv_b, *zero_b;
  int vec;  // four outputs per thread (N % 4 == 0, 16-byte aligned buffers)
};

struct GemmArgs {
  int64_t M, N, K;            // out is M x N, reduction over K
  int a_kmajor, b_kmajor;     // operand storage (see fqt_debug_int_gemm)
  uint32_t mn_lbo, mn_sbo;    // MN-major descriptor strides (bytes)
  int kc_blocks;              // K-blocks per exact chunk
  int m_tiles, n_tiles, splits;
  int64_t ks_blocks, kb_total;
  int64_t n_items;
  int stages, ring;           // operand stages, output boxes per epilogue warp
  int nacc;                   // TMEM accumulators in rotation (2 or 4)
  int m_fast;                 // item order: M tiles fastest (grad_X: the D
                              // tiles of the same output rows together)
  // grad_X epilogue (MODE_GRADX); rows of Q_b2 are the N dimension
  int kind;
  int og, ow;                  // centring offsets 2^(b-1) of Q_b2 and W~ codes
  const float *inv_s, *zero;   // Q_b2 metadata (1 or N entries)
  const int32_t *row_sum, *lead;
  const float *hz, *hr;        // BHQ offsets (block > 1)
  const int32_t *perm, *gsize; // adaptive BHQ groups (NB = 0): output row and
                               // group size of every stored row of Q_b2
  float raw_mmax;              // NB = 0: largest |m| of a row finished here
  float flt_mmax;              // largest |m| of a tile for the fp32 form
  float i32_mmax;              // largest |m| of a tile for the int32 form
  const int32_t *col_sum_w;    // W~ column sums over C
  const float *inv_sw, *zero_w;
  float *out;                  // grad_X (N x M row-major) for MODE_GRADX
  int sets;                    // grad_X epilogue sets in use (3 or 4)
  int bw, b2;                  // code bits of W~ and of Q_b2
  int small_p;                 // every |P| < 2^22 (block sums off the fp32 bits)
  int u8;                      // MODE_PARTIAL: byte operands, widened on chip
  int ustages;                 // ... through a ring of this many byte stages
  // MODE_PARTIAL with an implicit im2col X~ (stride 1): K blocks of 64
  // output-pixel slots = rpb output rows of pw slots (pw >= ow, the slots
  // past ow zero); A (Q_b1) and B (the NHWC codes at each tap's offset) are
  // read as 4-D boxes of (64 channels, pw, rpb, 1)
  int conv, cpw, crpb, cybi, coh, cih, cin, ckw, cpad, cow, ciw;
  int64_t cnimg;
  // a pair's (a wide tile's) partials with one split: grad_W itself (red)
  int fuse;
  int wn;                      // columns of a wide tile (k_gemm_wide)
  int taps;                    // its column atoms are the taps of a kernel row (0: consecutive)
  ReduceArgs red;
  int *status;
};

// ---------------------------------------------------------------------------
// PTX wrappers specific to the tensor-core path
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map,
                                            int32_t c0, int32_t c1,
                                            uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, int32_t c0,
                                            int32_t c1, int32_t c2, int32_t c3,
                                            uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
      "r"(smem_u32(bar))
      : "memory");
}

// The same loads issued by either CTA of a pair (cta_group::2): dst is this
// CTA's shared memory, bar the cluster address of the barrier that counts
// the bytes (the leader's).
__device__ __forceinline__ void tma_load_2d_pair(void *dst, const CUtensorMap *map, int32_t c0,
                                                 int32_t c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tma_load_4d_pair(void *dst, const CUtensorMap *map, int32_t c0,
                                                 int32_t c1, int32_t c2, int32_t c3,
                                                 uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}

// Cluster address of a shared-memory object of the pair's leader (rank 0).
__device__ __forceinline__ uint32_t leader_addr(const void *p) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
  return r;
}

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar)
               : "memory");
}

// Barrier of both CTAs of a pair (every thread of both reaches it).
__device__ __forceinline__ void cluster_sync() {
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n\t"
      "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, int32_t c0,
                                             int32_t c1, const void *src) {
  asm volatile(
      "cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
      ::"l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_u32(src))
      : "memory");
}

__device__ __forceinline__ void tma_store_3d(const CUtensorMap *map, int32_t c0,
                                             int32_t c1, int32_t c2,
                                             const void *src) {
  asm volatile(
      "cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
      ::"l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2),
      "r"(smem_u32(src))
      : "memory");
}

__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// Waits until at most n of this thread's bulk store groups still read
// shared memory (n = ring depth - 1 frees the oldest slot).
__device__ __forceinline__ void bulk_wait_read(int n) {
  switch (n) {
    case 0: asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.bulk.wait_group.read 2;" ::: "memory"); break;
    default: asm volatile("cp.async.bulk.wait_group.read 3;" ::: "memory"); break;
  }
}

__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

// UMMA shared-memory descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (stride byte offset), version 1 (bit 46).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;              // leading byte offset (unused, 16 B)
  d |= (uint64_t)(1024 >> 4) << 32;    // stride byte offset
  d |= (uint64_t)1 << 46;              // descriptor version
  d |= (uint64_t)2 << 61;              // SWIZZLE_128B
  return d;
}

// UMMA shared-memory descriptor of an MN-major operand with 128-byte
// swizzle: 64-element (128-byte) MN atoms of 8 K rows (1024 bytes); atoms
// `lbo` bytes apart along MN and `sbo` bytes apart along K.
__device__ __forceinline__ uint64_t sw128_desc_mn(uint32_t saddr, uint32_t lbo,
                                                  uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Instruction descriptor of kind::f16: A, B fp16, D fp32, M x N (128 x 128);
// bit 15 / 16 select MN-major A / B.
__host__ __device__ constexpr uint32_t make_idesc(bool a_mn, bool b_mn, int m = BM,
                                                  int n = BN) {
  return (1u << 4) | (0u << 7) | (0u << 10) | ((a_mn ? 1u : 0u) << 15) |
         ((b_mn ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t a_desc,
                                         uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// M = 256 over the two CTAs of a pair (each CTA's shared memory holds its
// 128 rows of A and its half of B's columns, at the same offsets).
__device__ __forceinline__ void umma_f16_pair(uint32_t tmem_d, uint64_t a_desc, uint64_t b_desc,
                                              uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrives on the barrier at this offset in both CTAs of the pair.
__device__ __forceinline__ void umma_commit_pair(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}

__device__ __forceinline__ void umma_commit(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
        "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
        "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]),
        "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]),
      "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]),
      "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]),
      "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}

__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// 32 columns of this warp's 32 lanes, without waiting (see tmem_wait_ld).
__device__ __forceinline__ void tmem_ld32_nw(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
        "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
        "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]),
        "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld16_nw(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
        "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
        "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld8_nw(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
        "=r"(r[6]), "=r"(r[7])
      : "r"(taddr));
}

// W consecutive columns (W = 8, 16 or 32) of this warp's 32 lanes.
template <int W>
__device__ __forceinline__ void tmem_ldw_nw(uint32_t taddr, uint32_t (&r)[W]) {
  if constexpr (W == 32) tmem_ld32_nw(taddr, r);
  else if constexpr (W == 16) tmem_ld16_nw(taddr, r);
  else tmem_ld8_nw(taddr, r);
}

// One column of this warp's 32 lanes, without waiting.
__device__ __forceinline__ uint32_t tmem_ld1_nw(uint32_t taddr) {
  uint32_t v;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(v) : "r"(taddr));
  return v;
}

// Waits for every tcgen05.ld this thread has issued.  The registers of the
// loads are passed through so that no use is scheduled before the wait.
template <int NR>
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[NR]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < NR; ++i) asm volatile("" : "+r"(r[i]));
}

// Byte offset of the 16-byte chunk `chunk` of row `row` in a 128-byte-swizzled
// K-major tile (rows of 128 bytes, 1024-byte atoms of 8 rows).
__device__ __forceinline__ uint32_t sw128_off(int row, int chunk) {
  return (uint32_t)(row * 128 + ((chunk ^ (row & 7)) << 4));
}

// The 32 rows r0 .. r0 + 31 of this thread's column j of grad_X.  The 32
// lanes of a warp hold 32 consecutive columns, so every store of a row is one
// coalesced 128-byte write; no staging is needed.
struct BoxOut {
  float *p;       // &grad_X[row r0][j]
  int64_t ld;     // row stride (D)
  int rows;       // rows of the box inside the matrix (0 .. 32)
  bool jv;        // column j inside the matrix
  __device__ __forceinline__ void st(int row, float v) const {
    if (jv && row < rows) __stcs(p + row * ld, v);
  }
  __device__ __forceinline__ void st2(int row, f32x2 v) const {
    float a, b;
    unpack2(v, a, b);
    st(row, a);
    st(row + 1, b);
  }
  // all 32 values of the box (then the lead-row overwrites, same thread)
  __device__ __forceinline__ void st32(const float (&o)[32]) const {
    if (!jv) return;
    if (rows == 32) {
#pragma unroll
      for (int i = 0; i < 32; ++i) __stcs(p + i * ld, o[i]);
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (i < rows) __stcs(p + i * ld, o[i]);
    }
  }
};


struct Item {
  int64_t m0, n0;
  int split;
  int64_t kb0, kb1;
};

__device__ __forceinline__ Item decode_item(const GemmArgs &g, int64_t it) {
  Item r;
  const int64_t tiles = (int64_t)g.m_tiles * g.n_tiles;
  r.split = (int)(it / tiles);
  const int64_t t = it - (int64_t)r.split * tiles;
  if (g.m_fast) {  // the M tiles of the same N rows side by side
    r.m0 = (t % g.m_tiles) * BM;
    r.n0 = (t / g.m_tiles) * BN;
  } else {
    r.m0 = (t / g.n_tiles) * BM;
    r.n0 = (t % g.n_tiles) * BN;
  }
  r.kb0 = (int64_t)r.split * g.ks_blocks;
  r.kb1 = min(g.kb_total, r.kb0 + g.ks_blocks);
  return r;
}

// The tiles of a CTA in its order.  A CTA on its own takes items blockIdx.x +
// local gridDim.x.  The CTAs of a pair (PAIR) take super tiles of 256 x 256,
// every (gridDim.x / 2)-th one: each CTA the 128 output rows M of its rank,
// as two tiles of 128 columns N (local = 2 super + half).  Returns false
// past the last.
template <bool PAIR>
__device__ __forceinline__ bool cta_item(const GemmArgs &g, int64_t local, Item &t) {
  if constexpr (PAIR) {
    const int64_t it = (int64_t)(blockIdx.x >> 1) + (local >> 1) * (int64_t)(gridDim.x >> 1);
    if (it >= g.n_items) return false;
    t = decode_item(g, it);
    t.m0 = 2 * t.m0 + (int64_t)(blockIdx.x & 1) * BM;
    t.n0 = 2 * t.n0 + (local & 1) * BN;
    return true;
  } else {
    const int64_t it = (int64_t)blockIdx.x + local * (int64_t)gridDim.x;
    if (it >= g.n_items) return false;
    t = decode_item(g, it);
    return true;
  }
}

// The tiles of a CTA of k_gemm_wide: items of 128 x g.wn, as two column halves
// (local = 2 item + half, the second from column 128 on).
__device__ __forceinline__ bool wide_item(const GemmArgs &g, int64_t local, Item &t) {
  const int64_t it = (int64_t)blockIdx.x + (local >> 1) * (int64_t)gridDim.x;
  if (it >= g.n_items) return false;
  t = decode_item(g, it);
  t.n0 = t.n0 / BN * g.wn + (local & 1) * BN;
  return true;
}

// The accumulator's consumer is done with it: the pair's MMA issuer (the
// leader) counts the arrivals of both CTAs.
template <bool PAIR>
__device__ __forceinline__ void acc_release(uint64_t *bar) {
  if constexpr (PAIR) mbar_arrive_cluster(leader_addr(bar));
  else mbar_arrive(bar);
}

// The items of one step of a CTA's schedule: item it, and with pairs the
// CTA's next item it + gridDim.x when it exists.  Returns their count.
__device__ __forceinline__ int group_items(const GemmArgs &g, int64_t it, bool pairs,
                                           Item (&tt)[2]) {
  tt[0] = decode_item(g, it);
  tt[1] = tt[0];
  if (pairs && it + (int64_t)gridDim.x < g.n_items) {
    tt[1] = decode_item(g, it + (int64_t)gridDim.x);
    return 2;
  }
  return 1;
}

__device__ __forceinline__ BoxOut box_out(const GemmArgs &g, const Item &t, int q, int lane,
                                          int r0) {
  BoxOut w;
  const int64_t j = t.m0 + q * 32 + lane, row0 = t.n0 + r0;
  w.jv = j < g.M;
  const int64_t left = g.N - row0;
  w.rows = left >= 32 ? 32 : (int)(left > 0 ? left : 0);
  w.ld = g.M;
  w.p = g.out + (w.rows > 0 && w.jv ? row0 * g.M + j : 0);
  return w;
}

// ---------------------------------------------------------------------------
// grad_X epilogue.  The accumulator holds P^T: TMEM lane = output column j of
// grad_X, TMEM column = row k of dH, so each thread owns one column j and the
// rows of a BHQ block are consecutive registers of one thread.
//
// Dequantization (Eq. 9).  With a the centred codes of Q_b2 (code - 2^(b-1)),
// w those of W~, the row offset 2^(b-1) + z'_k = m_k + d_k (m_k an integer,
// |d_k| <= 1/2) and y = 2^(bw-1) + z_w,
//   V_kj = sum_c (a_kc + m_k + d_k)(w_cj + y) = I_kj + y R_k + d_k U_j,
//   I_kj = P_kj + m_k CWc_j (an exact integer), CWc_j = sum_c w_cj,
//   R_k = sum_c (a_kc + m_k), U_j = CWc_j + C y = col_sum_w_j + C z_w,
// and grad_X = inv_sw diag(inv_s) Q_blk V.  The reflection is linear in the
// rows: Q V = Q I + y (Q R) 1^T + (Q d) U^T, with Q R and Q d per row (hr,
// hz; the identity for PTQ / PSQ).  Per block of nb rows with lead p,
//   (Q I)_k = I_k - beta (k != p),  (Q I)_p = rho S,
//   S = sum_k I_k, beta = kappa (rho S - I_p), rho = 1/sqrt(nb),
//   kappa = rho / (1 - rho).
// S and I_p are exact integers, beta is formed in float-float and split into
// an integer and a remainder, so I_k - beta loses nothing to the cancellation
// of the reflection: every term left in fp32 is small or row-constant.
//
// Two forms of the integer part, chosen per tile from the largest row offset
// |m_k| of its rows:
//   fp32   every |I| (2 + sqrt(nb)) below 2^24 (|I| below 2^24 without
//          reflection): one exact chunk and |m_k| <= flt_mmax;
//   int32  every |I| (2 + sqrt(nb)) below 2^31: |m_k| <= i32_mmax.  Every sum
//          then fits in int32 (wrapping partial sums are harmless) and each
//          result is one rounding of the exact integer.
// A tile outside both keeps its exact products P (as int32 bit patterns
// after several chunks) and the CTA finishes it after its last tile in int64
// and float-float (gradx_raw_fix).  Conversions to and from 64-bit integers
// run on the FP64 pipe, which is narrow on this GPU: the per-element path
// uses none.
// ---------------------------------------------------------------------------
// fp32 integers of magnitude below 2^22 to int32 with one FADD: x + 1.5 2^23
// holds x in its low mantissa bits.
constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
constexpr uint32_t kMagicBits = 0x4B400000u;

__device__ __forceinline__ uint32_t magic_bits(float x) {
  return __float_as_uint(__fadd_rn(x, kMagic));
}

__device__ __forceinline__ int magic_int(float x) { return (int)(magic_bits(x) - kMagicBits); }

// beta = kappa (rho S - I_p) split as bi + bf (bi an integer, |bi| < 2^31 in
// the int32 form) and the lead value rho S, for a block of nact >= 2 rows.
struct BlockFix {
  float bf, lead;
  int bi;
};

__device__ __forceinline__ BlockFix block_fix(const HhConst &c, long long S, int Ip) {
  const ff rS = ff_mul(c.rho, ff_from_int(S));
  const ff w = ff_add(rS, ff_neg(ff_from_i32s(Ip)));
  const ff beta = ff_mul(c.kap, w);
  BlockFix f;
  const float bi = rintf(beta.h);
  f.bi = __float2int_rn(bi);
  f.bf = __fadd_rn(__fsub_rn(beta.h, bi), beta.l);
  f.lead = ff_round(rS);
  return f;
}

// out = sc (t + hz U) + sc y hr, with kq = (sc, sc hz, sc y hr, m)
__device__ __forceinline__ float dequant(const float4 &kq, float t, float U) {
  return __fmaf_rn(kq.x, t, __fmaf_rn(kq.y, U, kq.z));
}

// The per-row terms (sc, A = sc hz, B = sc y hr, m) of a tile in shared
// memory, two rows interleaved ({sc, sc', A, A'}, {B, B', m, m'}) so that the
// epilogue dequantizes rows in packed pairs.
struct RowPair {
  f32x2 sc, A, B, m;
};

struct RowPar {
  float *p;
  __device__ __forceinline__ RowPair pair(int k) const {  // rows k, k + 1 (k even)
    const float4 x = *reinterpret_cast<const float4 *>(p + 4 * k);
    const float4 y = *reinterpret_cast<const float4 *>(p + 4 * k + 4);
    return {pack2(x.x, x.y), pack2(x.z, x.w), pack2(y.x, y.y), pack2(y.z, y.w)};
  }
  __device__ __forceinline__ float4 row(int k) const {
    const float *q = p + 8 * (k >> 1) + (k & 1);
    return make_float4(q[0], q[2], q[4], q[6]);
  }
  __device__ __forceinline__ float m(int k) const { return p[8 * (k >> 1) + (k & 1) + 6]; }
  __device__ __forceinline__ void set(int k, float sc, float A, float B, float m) const {
    float *q = p + 8 * (k >> 1) + (k & 1);
    q[0] = sc;
    q[2] = A;
    q[4] = B;
    q[6] = m;
  }
};

// dequant() of two rows
__device__ __forceinline__ f32x2 dequant2(const RowPair &q, f32x2 t, f32x2 U) {
  return fma2(q.sc, t, fma2(q.A, U, q.B));
}

// Row i of a column whose row 0 is at p (ld = the row stride in entries; one
// widening multiply-add per address).
__device__ __forceinline__ float *row_ptr(float *p, uint32_t ld, int i) {
  return reinterpret_cast<float *>(reinterpret_cast<char *>(p) + (uint64_t)ld * (uint32_t)(4 * i));
}

// The integer parts I = P + m CWc of 32 rows (one box) of this thread's
// column in the int32 form.
struct Ints {
  int v[32];
  __device__ __forceinline__ float f(int i) const { return __int2float_rn(v[i]); }
  __device__ __forceinline__ f32x2 f2(int i) const { return pack2(f(i), f(i + 1)); }
  __device__ __forceinline__ f32x2 minus2(int i, const BlockFix &b) const {
    return add2(pack2(__int2float_rn((int)((uint32_t)v[i] - (uint32_t)b.bi)),
                      __int2float_rn((int)((uint32_t)v[i + 1] - (uint32_t)b.bi))),
                pack2(-b.bf, -b.bf));
  }
};

// The exact products P of one TMEM column group: the chunk's fp32 value plus
// the int32 running sum of the earlier chunks.
__device__ __forceinline__ void load_products(uint32_t acc, uint32_t ints, bool multi, int c0,
                                              int (&P)[32]) {
  uint32_t r[32], s[32];
  tmem_ld32_nw(acc + (uint32_t)c0, r);
  if (multi) tmem_ld32_nw(ints + (uint32_t)c0, s);
  tmem_wait_ld(r);
  if (multi) tmem_wait_ld(s);
#pragma unroll
  for (int i = 0; i < 32; ++i)
    P[i] = (int)((uint32_t)__float2int_rn(__uint_as_float(r[i])) + (multi ? s[i] : 0u));
}

// Loads the products of the 32 rows at TMEM column c0 and forms I
// (|m| <= i32_mmax and |CWc| <= C 2^(bw-1) are below 2^22).
__device__ __forceinline__ void load_ints(uint32_t acc, uint32_t ints, bool multi, int c0,
                                          const RowPar &kp, float cwc, Ints &I) {
  load_products(acc, ints, multi, c0, I.v);
  const uint32_t cw = (uint32_t)magic_int(cwc);
#pragma unroll
  for (int i = 0; i < 32; ++i)
    I.v[i] = (int)((uint32_t)I.v[i] + (uint32_t)magic_int(kp.m(c0 + i)) * cw);
}

// I of one row (TMEM column col) of this thread's column.
__device__ __forceinline__ int load_int1(uint32_t acc, uint32_t ints, bool multi, int col,
                                         float m, float cwc) {
  uint32_t v[2];
  v[0] = tmem_ld1_nw(acc + (uint32_t)col);
  v[1] = multi ? tmem_ld1_nw(ints + (uint32_t)col) : 0u;
  tmem_wait_ld(v);
  const uint32_t P = (uint32_t)__float2int_rn(__uint_as_float(v[0])) + v[1];
  return (int)(P + (uint32_t)magic_int(m) * (uint32_t)magic_int(cwc));
}

// One box (32 rows r0 .. r0 + 31 of the tile) of blocks of NB <= 32 rows:
// reflection, dequantization, store into the swizzled box.
// lead products loaded per box: one per block of NB <= 32 rows
__host__ __device__ constexpr int leads_per_box(int nb) { return nb > 1 && nb <= 32 ? 32 / nb : 1; }

template <int NB>
__device__ __forceinline__ void box_small(const Ints &I, const int (&Ip)[leads_per_box(NB)],
                                          const HhConst &hc, const RowPar &kp,
                                          const int *leads, int r0, int64_t row0,
                                          int64_t N, float U, const BoxOut &w) {
  const f32x2 U2 = pack2(U, U);
  if (NB == 1) {
#pragma unroll
    for (int i = 0; i < 32; i += 2) w.st2(i, dequant2(kp.pair(r0 + i), I.f2(i), U2));
    return;
  }
  constexpr int NBB = NB > 1 ? NB : 2;
#pragma unroll
  for (int b = 0; b < 32 / NBB; ++b) {
    const int kb0 = r0 + b * NBB;
    const int64_t left = N - (row0 + b * NBB);
    const int nact = left >= NBB ? NBB : (int)(left > 0 ? left : 0);
    if (nact < 2) {  // a one-row block is not transformed
#pragma unroll
      for (int l = 0; l < NBB; l += 2)
        w.st2(b * NBB + l, dequant2(kp.pair(kb0 + l), I.f2(b * NBB + l), U2));
      continue;
    }
    long long S = 0;
#pragma unroll
    for (int l = 0; l < NBB; ++l) S += I.v[b * NBB + l];
    const BlockFix f = block_fix(nact == NBB ? hc : hh_const(nact), S, Ip[b]);
#pragma unroll
    for (int l = 0; l < NBB; l += 2)
      w.st2(b * NBB + l, dequant2(kp.pair(kb0 + l), I.minus2(b * NBB + l, f), U2));
    const int p = leads[kb0 / NBB];  // the lead row: a later store of the same thread
    w.st(b * NBB + p, dequant(kp.row(kb0 + p), f.lead, U));
  }
}

// The final chunk of one tile for this warp in the int32 form: groups of GW
// rows (a box, or one block of NB > 32 rows spanning several boxes).  raw: a
// tile outside both forms, whose row terms are units (m = 0, so I = P): its
// exact products P are stored as int32 bit patterns for gradx_raw_fix.
template <int NB, bool PAIR>
__device__ __forceinline__ void gradx_tile(const GemmArgs &g, const Item &t, uint32_t acc,
                                           uint32_t ints, bool multi, const RowPar &kp,
                                           const int *leads, const HhConst &hc, float cwc,
                                           float U, uint64_t *acce_set, int q, int lane,
                                           bool raw) {
  constexpr int GW = NB > 32 ? NB : 32;
  constexpr int NPP = leads_per_box(NB);
#pragma unroll 1
  for (int g0 = 0; g0 < BN; g0 += GW) {
    // blocks of more than 32 rows: their sums over all boxes first
    long long S_big = 0;
    int Ip_big = 0, p_big = 0;
    if (NB > 32) {
#pragma unroll 1
      for (int bx = 0; bx < GW / 32; ++bx) {
        Ints I;
        load_ints(acc, ints, multi, g0 + bx * 32, kp, cwc, I);
#pragma unroll
        for (int i = 0; i < 32; ++i) S_big += I.v[i];
      }
      p_big = leads[g0 / (NB > 32 ? NB : 1)];
      Ip_big = load_int1(acc, ints, multi, g0 + p_big, kp.m(g0 + p_big), cwc);
    }
#pragma unroll 1
    for (int bx = 0; bx < GW / 32; ++bx) {
      const int r0 = g0 + bx * 32;
      const BoxOut w = box_out(g, t, q, lane, r0);
      Ints I;
      load_ints(acc, ints, multi, r0, kp, cwc, I);
      int Ip[NPP];
#pragma unroll
      for (int b = 0; b < NPP; ++b) {
        Ip[b] = 0;
        if (NB > 1 && NB <= 32) {
          const int col = r0 + b * (32 / NPP) + leads[(r0 + b * (32 / NPP)) / (32 / NPP)];
          Ip[b] = load_int1(acc, ints, multi, col, kp.m(col), cwc);
        }
      }
      if (r0 + 32 == BN) {  // the accumulator has been read in full
        tc_fence_before();
        __syncwarp();
        if (lane == 0) acc_release<PAIR>(acce_set);
      }
      if (raw) {
        w.st32(reinterpret_cast<const float (&)[32]>(I.v));
        continue;
      }
      if constexpr (NB <= 32) {
        box_small<NB>(I, Ip, hc, kp, leads, r0, t.n0 + r0, g.N, U, w);
      } else {
        const int64_t left = g.N - (t.n0 + g0);
        const int nact = left >= NB ? NB : (int)(left > 0 ? left : 0);
        if (nact < 2) {
#pragma unroll
          for (int i = 0; i < 32; i += 2)
            w.st2(i, dequant2(kp.pair(r0 + i), I.f2(i), pack2(U, U)));
        } else {
          const BlockFix f = block_fix(nact == NB ? hc : hh_const(nact), S_big, Ip_big);
#pragma unroll
          for (int i = 0; i < 32; i += 2)
            w.st2(i, dequant2(kp.pair(r0 + i), I.minus2(i, f), pack2(U, U)));
          if (p_big >= bx * 32 && p_big < bx * 32 + 32)
            w.st(p_big - bx * 32, dequant(kp.row(g0 + p_big), f.lead, U));
        }
      }
    }
  }
}

struct BlockFixF {
  float bi, bf, lead;
};

__device__ __forceinline__ BlockFixF block_fix_f(const HhConst &c, int S, int Ip) {
  const ff rS = ff_mul(c.rho, ff_from_i32s(S));
  const ff w = ff_add(rS, ff_neg(ff_from_i32s(Ip)));
  const ff beta = ff_mul(c.kap, w);
  BlockFixF f;
  f.bi = rintf(beta.h);
  f.bf = __fadd_rn(__fsub_rn(beta.h, f.bi), beta.l);
  f.lead = ff_round(rS);
  return f;
}

// Two non-lead rows of Q I in the fp32 form: (P - bi) + m CWc is exact (every
// magnitude below 2^24), then the remainder bf.
__device__ __forceinline__ f32x2 reflect2(f32x2 P, const RowPair &q, f32x2 cwc,
                                          const BlockFixF &f) {
  return add2(fma2(q.m, cwc, add2(P, pack2(-f.bi, -f.bi))), pack2(-f.bf, -f.bf));
}

// The sum of the integers that fp32 values below 2^22 in magnitude hold, off
// the bits of v + 1.5 2^23 (n such words carry n kMagicBits).
__device__ __forceinline__ uint32_t magic_sum2(f32x2 v) {
  float a, b;
  unpack2(add2(v, pack2(kMagic, kMagic)), a, b);
  return __float_as_uint(a) + __float_as_uint(b);
}

__device__ __forceinline__ f32x2 pair_of(const uint32_t *r) {
  return pack2(__uint_as_float(r[0]), __uint_as_float(r[1]));
}
__device__ __forceinline__ void set_pair(uint32_t *r, f32x2 v) {
  float a, b;
  unpack2(v, a, b);
  r[0] = __float_as_uint(a);
  r[1] = __float_as_uint(b);
}

// (Q I)_k of a non-lead row, one at a time (the passes over raw rows).
__device__ __forceinline__ float reflect_f(float P, const float4 &kq, float cwc,
                                           const BlockFixF &f) {
  return __fsub_rn(__fmaf_rn(kq.w, cwc, __fsub_rn(P, f.bi)), f.bf);
}

// The final chunk of one tile in the fp32 form (one exact chunk, |P| < 2^22,
// |m| <= mmax).  Block sums S = sum P + CWc sum m, I_p = P_p + m_p CWc.
// raw: a tile outside the fp32 form, whose row terms are units (1, 0, 0, 0):
// no block is transformed, so the stores are its exact products P.
template <int NB, bool PAIR>
__device__ __forceinline__ void gradx_tile_f(const GemmArgs &g, const Item &t, uint32_t acc,
                                             const RowPar &kp, const int *leads,
                                             const int *msum, const HhConst &hc, float cwc,
                                             float U, uint64_t *acce_set, int q, int lane,
                                             bool raw) {
  constexpr int NBD = NB > 1 ? NB : 1;
  const int cwi = (int)cwc;
  const f32x2 cw2 = pack2(cwc, cwc), U2 = pack2(U, U);
  const int64_t j = t.m0 + q * 32 + lane;
  const bool jv = j < g.M;
  const uint32_t ld = (uint32_t)g.M;
  if constexpr (NB <= 32) {
    // one block (NB >= 8) or 16 rows (no reflection) per step, loaded from
    // TMEM on its own, so few values are live at a time
    constexpr int CH = NB >= 8 ? NB : (NB <= 1 ? 16 : 8);
    constexpr int BPC = NB > 1 ? CH / NB : 0;  // blocks per chunk
#pragma unroll 1
    for (int r0 = 0; r0 < BN; r0 += CH) {
      uint32_t r[CH];
      tmem_ldw_nw<CH>(acc + (uint32_t)r0, r);
      uint32_t pp[BPC > 0 ? BPC : 1];
#pragma unroll
      for (int b = 0; b < BPC; ++b)
        pp[b] = tmem_ld1_nw(acc + (uint32_t)(r0 + b * NBD + leads[(r0 + b * NBD) / NBD]));
      tmem_wait_ld(r);
      if (BPC > 0) tmem_wait_ld(pp);
      if (r0 + CH == BN) {  // the accumulator has been read in full
        tc_fence_before();
        __syncwarp();
        if (lane == 0) acc_release<PAIR>(acce_set);
      }
      const int64_t row0 = t.n0 + r0;
      const int64_t left = g.N - row0;
      const int rows = left >= CH ? CH : (int)(left > 0 ? left : 0);
      float *po = g.out + (jv && rows > 0 ? row0 * g.M + j : 0);
      if constexpr (NB <= 1) {
#pragma unroll
        for (int i = 0; i < CH; i += 2) {
          const RowPair kq = kp.pair(r0 + i);
          set_pair(r + i, dequant2(kq, fma2(kq.m, cw2, pair_of(r + i)), U2));
        }
      }
      int lrow[BPC > 0 ? BPC : 1];
      float lval[BPC > 0 ? BPC : 1];
#pragma unroll
      for (int b = 0; b < (BPC > 0 ? BPC : 1); ++b) {
        lrow[b] = -1;
        lval[b] = 0.0f;
      }
      if constexpr (NB > 1) {
#pragma unroll
        for (int b = 0; b < BPC; ++b) {
          const int kb0 = r0 + b * NBD;
          const int64_t lb = g.N - (t.n0 + kb0);
          const int nact = lb >= NBD ? NBD : (int)(lb > 0 ? lb : 0);
          if (nact < 2 || raw) {  // a one-row block is not transformed
#pragma unroll
            for (int l = 0; l < NBD; l += 2) {
              const RowPair kq = kp.pair(kb0 + l);
              uint32_t *v = r + b * NBD + l;
              set_pair(v, dequant2(kq, fma2(kq.m, cw2, pair_of(v)), U2));
            }
            continue;
          }
          uint32_t sb = 0u;
#pragma unroll
          for (int l = 0; l < NBD; l += 2) sb += magic_sum2(pair_of(r + b * NBD + l));
          const int S = (int)(sb - (uint32_t)NBD * kMagicBits) + cwi * msum[kb0 / NBD];
          const int p = leads[kb0 / NBD];
          const float4 kl = kp.row(kb0 + p);
          const int Ip = magic_int(__uint_as_float(pp[b])) + (int)kl.w * cwi;
          const BlockFixF f = block_fix_f(nact == NBD ? hc : hh_const(nact), S, Ip);
#pragma unroll
          for (int l = 0; l < NBD; l += 2) {
            const RowPair kq = kp.pair(kb0 + l);
            uint32_t *v = r + b * NBD + l;
            set_pair(v, dequant2(kq, reflect2(pair_of(v), kq, cw2, f), U2));
          }
          lrow[b] = b * NBD + p;
          lval[b] = dequant(kl, f.lead, U);
        }
      }
      if constexpr (NB == 0) {
        // adaptive groups: row r0 + i of the tile is row leads[r0 + i] of grad_X
        if (jv) {
#pragma unroll
          for (int i = 0; i < CH; ++i)
            if (i < rows) __stcs(g.out + (int64_t)leads[r0 + i] * g.M + j, __uint_as_float(r[i]));
        }
      } else if (jv) {
        if (rows == CH) {
#pragma unroll
          for (int i = 0; i < CH; ++i) __stcs(row_ptr(po, ld, i), __uint_as_float(r[i]));
        } else {
#pragma unroll
          for (int i = 0; i < CH; ++i)
            if (i < rows) __stcs(row_ptr(po, ld, i), __uint_as_float(r[i]));
        }
        // the lead rows: later stores of the same thread to the same address
#pragma unroll
        for (int b = 0; b < BPC; ++b)
          if (lrow[b] >= 0 && lrow[b] < rows) __stcs(po + (int64_t)lrow[b] * g.M, lval[b]);
      }
    }
  } else {
    // blocks of more than 32 rows: their sums over all boxes of 32 first
#pragma unroll 1
    for (int g0 = 0; g0 < BN; g0 += NBD) {
      uint32_t sb = 0u;
#pragma unroll 1
      for (int bx = 0; bx < NBD / 32; ++bx) {
        uint32_t r[32];
        tmem_ld32_nw(acc + (uint32_t)(g0 + bx * 32), r);
        tmem_wait_ld(r);
#pragma unroll
        for (int i = 0; i < 32; i += 2) sb += magic_sum2(pair_of(r + i));
      }
      const int S = (int)(sb - (uint32_t)NB * kMagicBits) + cwi * msum[g0 / NBD];
      const int p = leads[g0 / NBD];
      uint32_t pv[1];
      pv[0] = tmem_ld1_nw(acc + (uint32_t)(g0 + p));
      tmem_wait_ld(pv);
      const float4 kl = kp.row(g0 + p);
      const int Ip = magic_int(__uint_as_float(pv[0])) + (int)kl.w * cwi;
      const int64_t left = g.N - (t.n0 + g0);
      const int nact = left >= NB ? NB : (int)(left > 0 ? left : 0);
      const bool refl = nact >= 2 && !raw;
      const BlockFixF f = block_fix_f(nact == NB || !refl ? hc : hh_const(nact), S, Ip);
#pragma unroll 1
      for (int bx = 0; bx < NBD / 32; ++bx) {
        const int r0 = g0 + bx * 32;
        const BoxOut w = box_out(g, t, q, lane, r0);
        uint32_t r[32];
        tmem_ld32_nw(acc + (uint32_t)r0, r);
        tmem_wait_ld(r);
        if (r0 + 32 == BN) {  // the accumulator has been read in full
          tc_fence_before();
          __syncwarp();
          if (lane == 0) acc_release<PAIR>(acce_set);
        }
        if (refl) {
#pragma unroll
          for (int i = 0; i < 32; i += 2) {
            const RowPair kq = kp.pair(r0 + i);
            set_pair(r + i, dequant2(kq, reflect2(pair_of(r + i), kq, cw2, f), U2));
          }
        } else {
#pragma unroll
          for (int i = 0; i < 32; i += 2) {
            const RowPair kq = kp.pair(r0 + i);
            set_pair(r + i, dequant2(kq, fma2(kq.m, cw2, pair_of(r + i)), U2));
          }
        }
        w.st32(reinterpret_cast<const float (&)[32]>(r));
        // the lead row: a later store of the same thread
        if (refl && p >= bx * 32 && p < bx * 32 + 32)
          w.st(p - bx * 32, dequant(kl, f.lead, U));
      }
    }
  }
}

// The global inputs of one tile's parameters (lane-owned rows and columns).
struct TileLoads {
  float inv[BN / 32], zero[BN / 32], hz[BN / 32], hr[BN / 32];
  int rs[BN / 32], cs[BM / 32], lead[2];
  int gs[BN / 32], pr[BN / 32];  // NB = 0: group size and output row
};

template <int NB>
__device__ __forceinline__ void tile_loads(const GemmArgs &g, const Item &t, int lane,
                                           TileLoads &L) {
  constexpr int NBD = NB > 1 ? NB : 1;
#pragma unroll
  for (int i = 0; i < BN / 32; ++i) {
    const int64_t k = t.n0 + lane + 32 * i;
    const bool kv = k < g.N;
    const int64_t ri = g.kind == FQT_PTQ ? 0 : (kv ? k : 0);
    L.inv[i] = kv ? __ldg(g.inv_s + ri) : 0.0f;
    L.zero[i] = kv ? __ldg(g.zero + ri) : 0.0f;
    if (NB > 1) {
      L.hz[i] = kv ? __ldg(g.hz + k) : 0.0f;
      L.hr[i] = kv ? __ldg(g.hr + k) : 0.0f;
      L.rs[i] = 0;
    } else {
      L.hz[i] = L.hr[i] = 0.0f;
      L.rs[i] = kv ? __ldg(g.row_sum + k) : 0;
    }
    if (NB == 0) {
      L.gs[i] = kv ? __ldg(g.gsize + k) : 1;
      L.pr[i] = kv ? __ldg(g.perm + k) : 0;
    } else {
      L.gs[i] = 1;
      L.pr[i] = 0;
    }
  }
#pragma unroll
  for (int i = 0; i < BM / 32; ++i) {
    const int64_t j = t.m0 + lane + 32 * i;
    L.cs[i] = j < g.M ? __ldg(g.col_sum_w + j) : 0;
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {  // BN / NB <= 64 blocks per tile
    const int b = lane + 32 * u;
    L.lead[u] = 0;
    if (NB > 1 && b < BN / NBD) {
      const int64_t kb = t.n0 / NBD + b;
      L.lead[u] = kb * NBD < g.N ? __ldg(g.lead + kb) : 0;
    }
  }
}

// Parameter loader of grad_X (one warp): for every tile of this CTA, in
// order, the per-row terms of its rows and the column sums of its columns go
// into a parameter stage ahead of the epilogue warps that use them.  The
// global loads of the next tile are in flight while this tile's are used.
template <int NB, int FORM, bool PAIR>
__device__ __forceinline__ void gradx_params(const GemmArgs &g, uint8_t *smem, uint64_t *pfull,
                                             uint64_t *pempty, volatile int *abort_flag,
                                             int lane) {
  uint32_t *raw_mask = reinterpret_cast<uint32_t *>(smem + kOffRaw);
  const float inv_sw = *g.inv_sw, zw = *g.zero_w;
  const ff y = two_sum((float)g.ow, zw);
  const int Cn = (int)g.K;
  TileLoads cur, nxt;
  Item t, tn;
  bool have = cta_item<PAIR>(g, 0, t);
  if (have) tile_loads<NB>(g, t, lane, cur);
  for (int64_t local = 0; have && !*abort_flag; ++local) {
    const bool more = cta_item<PAIR>(g, local + 1, tn);
    if (more) tile_loads<NB>(g, tn, lane, nxt);
    const int s = (int)(local % kParStages);
    const uint32_t wrap = (uint32_t)(local / kParStages);
    const bool got = mbar_wait(&pempty[s], (wrap & 1u) ^ 1u, g.status);
    if (!__all_sync(0xffffffffu, got)) { *abort_flag = 1; break; }
    uint8_t *P = smem + kOffPar + (size_t)s * kParBytes;
    const RowPar kp{reinterpret_cast<float *>(P)};
    int *leads = reinterpret_cast<int *>(P + kParLeads);
    int *msum = reinterpret_cast<int *>(P + kParMsum);
    int *cs = reinterpret_cast<int *>(P + kParCs);
    float mabs = 0.0f;
    float mrow[BN / 32];
#pragma unroll
    for (int i = 0; i < BN / 32; ++i) {
      const int64_t k = t.n0 + lane + 32 * i;
      float sc = 0.0f, A = 0.0f, B = 0.0f, m = 0.0f;
      if (k < g.N) {
        sc = __fmul_rn(inv_sw, cur.inv[i]);
        const ff x = two_sum((float)g.og, cur.zero[i]);
        m = rintf(x.h);
        float hd, hR;
        if (NB > 1) {
          hd = cur.hz[i];
          hR = cur.hr[i];
        } else {
          // R = sum_c (a + m); rounding relative to R itself suffices for a
          // row-constant term
          hd = ff_round(fast_two_sum(__fsub_rn(x.h, m), x.l));
          hR = __fadd_rn((float)(cur.rs[i] - Cn * g.og), __fmul_rn((float)Cn, m));
        }
        A = __fmul_rn(sc, hd);
        B = __fmul_rn(sc, __fmaf_rn(hR, y.h, __fmul_rn(hR, y.l)));
        if (NB == 0 && (cur.gs[i] > 1 || !(fabsf(m) <= g.raw_mmax))) {
          // finished by the group pass: the exact integer product P alone
          sc = 1.0f;
          A = B = m = 0.0f;
        }
      }
      kp.set(lane + 32 * i, sc, A, B, m);
      mabs = fmaxf(mabs, fabsf(m));
      mrow[i] = m;
    }
    if constexpr (NB == 0) {
#pragma unroll
      for (int i = 0; i < BN / 32; ++i)
        leads[lane + 32 * i] = min(max(cur.pr[i], 0), (int)(g.N - 1));
    }
    if constexpr (NB > 1) {
      // sums of m over each block (the fp32 form's S = sum P + CWc sum m)
      constexpr int SEG = NB > 32 ? 32 : NB;
#pragma unroll
      for (int i = 0; i < BN / 32; ++i) {
        float v = mrow[i];
#pragma unroll
        for (int off = 1; off < SEG; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        mrow[i] = v;
      }
      if constexpr (NB <= 32) {
#pragma unroll
        for (int i = 0; i < BN / 32; ++i)
          if (lane % NB == 0) msum[(32 * i + lane) / NB] = (int)mrow[i];
      } else if (lane == 0) {
#pragma unroll
        for (int b = 0; b < BN / NB; ++b) {
          float v = 0.0f;
#pragma unroll
          for (int i = 0; i < NB / 32; ++i) v += mrow[b * (NB / 32) + i];
          msum[b] = (int)v;
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (lane + 32 * u < BN / NB) leads[lane + 32 * u] = cur.lead[u];
    }
#pragma unroll
    for (int i = 0; i < BM / 32; ++i) cs[lane + 32 * i] = cur.cs[i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
      mabs = fmaxf(mabs, __shfl_xor_sync(0xffffffffu, mabs, off));
    // a tile with a row offset beyond its forms (FORM 2: the fp32 form;
    // otherwise the int32 form, which holds more) keeps the exact products P
    // (unit row terms); its bit sends it to the CTA's final pass
    // (gradx_raw_fix)
    const bool raw = NB != 0 && !(mabs <= (FORM == 2 ? g.flt_mmax : g.i32_mmax));
    if (raw) {
#pragma unroll
      for (int i = 0; i < BN / 32; ++i) kp.set(lane + 32 * i, 1.0f, 0.0f, 0.0f, 0.0f);
      if (lane == 0 && local < kMaxLocalTiles) raw_mask[local >> 5] |= 1u << (local & 31);
    }
    // 1: the fp32 form, 2: the int32 form, 0: raw
    if (lane == 0)
      *reinterpret_cast<int *>(P + kParFlag) =
          NB == 0 || (FORM == 2 && !raw) || (FORM == 1 && mabs <= g.flt_mmax) ? 1
          : raw                                                             ? 0
                                                                            : 2;
    __syncwarp();
    if (lane == 0) mbar_arrive(&pfull[s]);
    cur = nxt;
    t = tn;
    have = more;
  }
}

template <int NB, int FORM, bool PAIR>
__device__ __forceinline__ void gradx_epilogue(const GemmArgs &g, uint8_t *smem,
                                               uint8_t *ring, uint64_t *accf,
                                               uint64_t *acce, uint64_t *pfull,
                                               uint64_t *pempty, uint32_t tmem,
                                               const CUtensorMap *tmOut,
                                               volatile int *abort_flag, int warp,
                                               int lane) {
  const int ew = warp - kGemmWarpEpi0;
  const int q = warp & 3;     // TMEM lane quadrant: columns j = 32q .. 32q + 31
  const int set = ew >> 2;    // the tiles (every g.sets-th one) this warp serves
  const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
  const float zw = *g.zero_w;
  const int Cn = (int)g.K;
  HhConst hc = {{0.0f, 0.0f}, {0.0f, 0.0f}};
  if (NB > 1) hc = hh_const(NB);
  bool ok = true;
  // this CTA's tiles local = set, set + g.sets, ...
  for (int64_t local = set; set < g.sets; local += g.sets) {
    Item t;
    if (!cta_item<PAIR>(g, local, t) || *abort_flag) break;
    const int buf = (int)(local & (g.nacc - 1));
    const uint32_t acc = lane_base + (uint32_t)(buf * BN);
    // int32 running sums (two accumulators only): columns 256 + 128 buf
    const uint32_t ints = lane_base + (uint32_t)(2 * BN + buf * BN);
    const int64_t nchunks = (t.kb1 - t.kb0 + g.kc_blocks - 1) / g.kc_blocks;
    const bool active = t.m0 + q * 32 < g.M;  // warp-uniform
    const int s = (int)(local % kParStages);
    const bool gotp = mbar_wait(&pfull[s], (uint32_t)(local / kParStages) & 1u, g.status);
    if (!__all_sync(0xffffffffu, gotp)) { ok = false; break; }
    const uint8_t *P = smem + kOffPar + (size_t)s * kParBytes;
    const RowPar kp{reinterpret_cast<float *>(const_cast<uint8_t *>(P))};
    const int *leads = reinterpret_cast<const int *>(P + kParLeads);
    const int *msum = reinterpret_cast<const int *>(P + kParMsum);
    const int cs = reinterpret_cast<const int *>(P + kParCs)[q * 32 + lane];
    const int tform = *reinterpret_cast<const int *>(P + kParFlag);  // 1 fp32, 2 int32, 0 raw
    const float cwc = (float)(cs - Cn * g.ow);
    const float U = __fmaf_rn((float)Cn, zw, (float)cs);
    for (int64_t c = 0; c < nchunks; ++c) {
      // every tile has nchunks chunks: the use count of this accumulator
      // before chunk c of this tile gives the phase
      const uint32_t par = (uint32_t)(((local / g.nacc) * nchunks + c) & 1);
      const bool got = !*abort_flag && mbar_wait(&accf[buf], par, g.status);
      if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
      tc_fence_after();
      const bool last_chunk = c + 1 == nchunks;
      if (!last_chunk && active) {
        // exact chunk boundary: fold the chunk into the int32 running sum
#pragma unroll 1
        for (int grp = 0; grp < BN / 32; ++grp) {
          uint32_t r[32];
          tmem_ld32_nw(acc + (uint32_t)(grp * 32), r);
          tmem_wait_ld(r);
          if (c > 0) {
            uint32_t sr[32];
            tmem_ld32_nw(ints + (uint32_t)(grp * 32), sr);
            tmem_wait_ld(sr);
#pragma unroll
            for (int i = 0; i < 32; ++i)
              r[i] = (uint32_t)(__float2int_rn(__uint_as_float(r[i])) + (int)sr[i]);
          } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) r[i] = (uint32_t)__float2int_rn(__uint_as_float(r[i]));
          }
          tmem_st32(ints + (uint32_t)(grp * 32), r);
        }
        tmem_wait_st();
      }
      if (!last_chunk || !active) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) acc_release<PAIR>(&acce[buf]);
        continue;
      }
      const bool multi = c > 0;
      if constexpr (NB == 0) {
        gradx_tile_f<0, PAIR>(g, t, acc, kp, leads, msum, hc, cwc, U, &acce[buf], q, lane, false);
      } else {
        if constexpr (FORM == 2) {
          // a tile outside the fp32 form has unit row terms (kq = (1, 0, 0, 0)):
          // the one-row epilogue stores its exact products P for gradx_raw_fix
          gradx_tile_f<NB, PAIR>(g, t, acc, kp, leads, msum, hc, cwc, U, &acce[buf], q, lane,
                           tform != 1);
        } else if (FORM == 1 && tform == 1) {
          gradx_tile_f<NB, PAIR>(g, t, acc, kp, leads, msum, hc, cwc, U, &acce[buf], q, lane, false);
        } else {
          gradx_tile<NB, PAIR>(g, t, acc, ints, multi, kp, leads, hc, cwc, U, &acce[buf], q, lane,
                         tform == 0);
        }
      }
    }
    // the parameter stage is free again
    __syncwarp();
    if (lane == 0) mbar_arrive(&pempty[s]);
    if (!ok) break;
  }
  if (!ok) *abort_flag = 1;
}

// ---------------------------------------------------------------------------
// Split-K partial epilogue: each warp owns TMEM lanes 32q .. 32q + 31 (rows)
// and 64 columns, stored as two 32 x 32 int32 boxes (3-D tensor map over
// splits x M x N) from a ring of boxes.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void partial_epilogue(const GemmArgs &g, uint8_t *ring,
                                                 uint64_t *accf, uint64_t *acce,
                                                 uint32_t tmem, const CUtensorMap *tmOut,
                                                 volatile int *abort_flag, int warp,
                                                 int lane) {
  const int ew = warp - kGemmWarpEpi0;
  const int q = warp & 3;
  const int hcol = ew >> 2;  // column half: 64 * hcol .. +63
  uint8_t *myring = ring + (size_t)ew * g.ring * kBoxBytes;
  int nbox = 0;
  const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
  const uint32_t int_cols = lane_base + (uint32_t)(2 * BN + hcol * 64);
  int buf = 0;
  uint32_t aph = 0u;  // bit b: phase parity of accumulator b
  bool ok = true;
  for (int64_t it = blockIdx.x; it < g.n_items && !*abort_flag; it += gridDim.x) {
    const Item t = decode_item(g, it);
    const int64_t nchunks = (t.kb1 - t.kb0 + g.kc_blocks - 1) / g.kc_blocks;
    for (int64_t c = 0; c < nchunks; ++c) {
      const bool got = !*abort_flag && mbar_wait(&accf[buf], (aph >> buf) & 1u, g.status);
      if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
      tc_fence_after();
      const uint32_t accb = lane_base + (uint32_t)(buf * BN + hcol * 64);
      const bool last = c + 1 == nchunks;
#pragma unroll
      for (int grp = 0; grp < 2; ++grp) {
        uint32_t r[32];
        tmem_ld32_nw(accb + (uint32_t)(grp * 32), r);
        tmem_wait_ld(r);
        if (c > 0) {
          uint32_t s[32];
          tmem_ld32_nw(int_cols + (uint32_t)(grp * 32), s);
          tmem_wait_ld(s);
#pragma unroll
          for (int j = 0; j < 32; ++j)
            r[j] = (uint32_t)(__float2int_rn(__uint_as_float(r[j])) + (int)s[j]);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) r[j] = (uint32_t)__float2int_rn(__uint_as_float(r[j]));
        }
        if (!last) {
          tmem_st32(int_cols + (uint32_t)(grp * 32), r);
          continue;
        }
        if (grp == 1) {  // this accumulator is no longer read
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acce[buf]);
        }
        uint8_t *tile = myring + (size_t)(nbox % g.ring) * kBoxBytes;
        if (nbox >= g.ring) {
          if (lane == 0) bulk_wait_read(g.ring - 1);
          __syncwarp();
        }
#pragma unroll
        for (int j4 = 0; j4 < 8; ++j4)
          *reinterpret_cast<uint4 *>(tile + sw128_off(lane, j4)) =
              make_uint4(r[4 * j4], r[4 * j4 + 1], r[4 * j4 + 2], r[4 * j4 + 3]);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          tma_store_3d(tmOut, (int32_t)(t.n0 + hcol * 64 + grp * 32), (int32_t)(t.m0 + q * 32),
                       t.split, tile);
          bulk_commit();
        }
        ++nbox;
      }
      if (!last) {
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce[buf]);
      }
      aph ^= 1u << buf;
      buf ^= 1;
    }
    if (!ok) break;
  }
  if (!ok) *abort_flag = 1;
  if (lane == 0) bulk_wait_all();
  __syncwarp();
}

// ---------------------------------------------------------------------------
// Byte operands of the split-K partials (both MN-major: K rows of 128 codes).
// TMA lands each operand's 128 x 64 byte tile in the stage (128-byte rows,
// 128-byte swizzle); kCvtWarps converter warps widen it into the fp16 carrier
// tile the MMA reads (two 64-wide swizzle atoms, as the fp16 boxes would
// land), code - 2^(b-1) exactly, rows past the end of the reduction as 0
// (a zero byte would widen to -2^(b-1)), then fence the writes for the
// tensor core and release the stage to the MMA issuer.
// ---------------------------------------------------------------------------
constexpr int kCvtWarps = 6;

// Shared-memory offsets of a converter thread's chunks (at most 3 of the
// 512 16-byte chunks of a 128 x 64 byte tile): the byte chunk, and the two
// fp16 chunks it widens into.
struct CvtSlots {
  int n;
  uint32_t src[3], dst0[3], dst1[3];
  int row[3];
};

__device__ __forceinline__ CvtSlots cvt_slots(int t) {
  CvtSlots o;
  o.n = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int c = t + i * kCvtWarps * 32;
    const int r = c >> 3, j = c & 7, cc = (j & 3) * 2;
    const uint32_t base = (uint32_t)((j >> 2) * (kTileBytes / 2) + r * 128);
    o.src[i] = (uint32_t)(r * 128 + ((j ^ (r & 7)) << 4));
    o.dst0[i] = base + (uint32_t)((cc ^ (r & 7)) << 4);
    o.dst1[i] = base + (uint32_t)(((cc + 1) ^ (r & 7)) << 4);
    o.row[i] = r;
    if (c < 512) o.n = i + 1;
  }
  return o;
}

// codes 16j .. 16j + 15 of a row: fp16 chunks 2 (j mod 4) and 2 (j mod 4) + 1
// of swizzle atom j / 4; rows from rows_valid on are 0
__device__ __forceinline__ void widen_tile(const uint8_t *src, uint8_t *dst, int rows_valid,
                                           __half2 bias, const CvtSlots &o) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (i >= o.n) break;
    uint4 lo = make_uint4(0u, 0u, 0u, 0u), hi = lo;
    if (o.row[i] < rows_valid) {
      const uint4 v = *reinterpret_cast<const uint4 *>(src + o.src[i]);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
      uint32_t h[8];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t a = __byte_perm(w[k], 0x6464u, 0x4140);
        const uint32_t b = __byte_perm(w[k], 0x6464u, 0x4342);
        __half2 x = __hsub2(*reinterpret_cast<const __half2 *>(&a), bias);
        __half2 y = __hsub2(*reinterpret_cast<const __half2 *>(&b), bias);
        h[2 * k] = *reinterpret_cast<uint32_t *>(&x);
        h[2 * k + 1] = *reinterpret_cast<uint32_t *>(&y);
      }
      lo = make_uint4(h[0], h[1], h[2], h[3]);
      hi = make_uint4(h[4], h[5], h[6], h[7]);
    }
    *reinterpret_cast<uint4 *>(dst + o.dst0[i]) = lo;
    *reinterpret_cast<uint4 *>(dst + o.dst1[i]) = hi;
  }
}

// Converter warp cw of kCvtWarps: byte stage su (ring of g.ustages) into
// carrier stage sf (ring of g.stages), in the producer's K-block order.
static __device__ __noinline__ void partial_convert(const GemmArgs &g, uint8_t *ops, uint8_t *uops,
                                             uint64_t *full, uint64_t *empty, uint64_t *cvt,
                                             uint64_t *fempty, volatile int *abort_flag, int cw,
                                             int lane) {
  const CvtSlots slots = cvt_slots(cw * 32 + lane);
  const __half2 bias_a = __half2half2(__int2half_rn(1024 + (1 << (g.bw - 1))));
  const __half2 bias_b = __half2half2(__int2half_rn(1024 + (1 << (g.b2 - 1))));
  int su = 0, sf = 0;
  uint32_t phu = 0, phf = 0;
  for (int64_t it = blockIdx.x; it < g.n_items && !*abort_flag; it += gridDim.x) {
    const Item tt = decode_item(g, it);
    for (int64_t kb = tt.kb0; kb < tt.kb1; ++kb) {
      // the byte tiles have landed, and the MMA is done with the carrier stage
      bool got = mbar_wait(&full[su], phu, g.status);
      got = got && mbar_wait(&fempty[sf], phf ^ 1u, g.status);
      if (!__all_sync(0xffffffffu, got)) { *abort_flag = 1; return; }
      const uint8_t *us = uops + (size_t)su * kTileBytes;
      uint8_t *fs = ops + (size_t)sf * 2 * kTileBytes;
      const int64_t left = g.K - kb * BK;
      const int rows_valid = left >= BK ? BK : (int)(left > 0 ? left : 0);
      widen_tile(us, fs, rows_valid, bias_a, slots);
      widen_tile(us + kTileBytes / 2, fs + kTileBytes, rows_valid, bias_b, slots);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&cvt[sf]);    // the carrier stage is ready for the MMA
        mbar_arrive(&empty[su]);  // the byte stage is free for the next loads
      }
      if (++su == g.ustages) { su = 0; phu ^= 1u; }
      if (++sf == g.stages) { sf = 0; phf ^= 1u; }
    }
  }
}

// ---------------------------------------------------------------------------
// Roles of a CTA pair (PAIR)
// ---------------------------------------------------------------------------
// TMA producer: this CTA's 128 rows of A and its 128 of the super tile's 256
// columns of B; the leader's full barrier counts the bytes of both CTAs.
template <int MODE>
__device__ __forceinline__ void produce_pair(const GemmArgs &g, const CUtensorMap &tmA,
                                             const CUtensorMap &tmB, uint8_t *ops,
                                             uint64_t *full, uint64_t *empty,
                                             volatile int *abort_flag, int &s, uint32_t &ph) {
  const int rank = (int)(blockIdx.x & 1);
  Item t;
  for (int64_t local = 0; cta_item<true>(g, local, t) && !*abort_flag; local += 2) {
    const int32_t m0 = (int32_t)t.m0, n0 = (int32_t)t.n0 + rank * BN;
    // implicit im2col (see the single-CTA producer)
    int cimg = 0, cyb = 0, ccg[2] = {0, 0}, ckx[2] = {0, 0}, cky[2] = {0, 0};
    bool cval[2] = {false, false};
    if (MODE == MODE_PARTIAL && g.conv) {
      cimg = (int)(t.kb0 / g.cybi);
      cyb = (int)(t.kb0 - (int64_t)cimg * g.cybi);
      for (int h = 0; h < 2; ++h) {
        const int d = n0 + 64 * h;
        const int tap = d / g.cin;
        ccg[h] = d - tap * g.cin;
        cky[h] = tap / g.ckw;
        ckx[h] = tap - cky[h] * g.ckw;
        cval[h] = d < g.N;
      }
    }
    for (int64_t kb = t.kb0; kb < t.kb1; ++kb) {
      if (!mbar_wait(&empty[s], ph ^ 1u, g.status)) { *abort_flag = 1; return; }
      if (rank == 0) mbar_expect_tx(&full[s], (uint32_t)(4 * kTileBytes));
      const uint32_t bar = leader_addr(&full[s]);
      uint8_t *sa = ops + (size_t)(2 * s) * kTileBytes;
      uint8_t *sb = sa + kTileBytes;
      const int32_t kc = (int32_t)(kb * BK);
      if (MODE == MODE_PARTIAL && g.conv) {
        const int oy0 = cyb * g.crpb;
        tma_load_4d_pair(sa, &tmA, m0, 0, oy0, cimg, bar);
        tma_load_4d_pair(sa + kTileBytes / 2, &tmA, m0 + 64, 0, oy0, cimg, bar);
        for (int h = 0; h < 2; ++h) {
          if (cval[h])
            tma_load_4d_pair(sb + h * (kTileBytes / 2), &tmB, ccg[h], ckx[h] - g.cpad,
                             oy0 + cky[h] - g.cpad, cimg, bar);
          else  // past the last tap: a box outside the tensor (zeros)
            tma_load_4d_pair(sb + h * (kTileBytes / 2), &tmB, 0, 0, g.cih + g.coh + 8, cimg, bar);
        }
        if (++cyb == g.cybi) { cyb = 0; ++cimg; }
      } else {
        // K-major: one 64 x 128 box; MN-major: two 64 (MN) x 64 (K) boxes
        if (g.a_kmajor) {
          tma_load_2d_pair(sa, &tmA, kc, m0, bar);
        } else {
          tma_load_2d_pair(sa, &tmA, m0, kc, bar);
          tma_load_2d_pair(sa + kTileBytes / 2, &tmA, m0 + 64, kc, bar);
        }
        if (g.b_kmajor) {
          tma_load_2d_pair(sb, &tmB, kc, n0, bar);
        } else {
          tma_load_2d_pair(sb, &tmB, n0, kc, bar);
          tma_load_2d_pair(sb + kTileBytes / 2, &tmB, n0 + 64, kc, bar);
        }
      }
      if (++s == g.stages) { s = 0; ph ^= 1u; }
    }
  }
}

// MMA issuer (one lane of the leader): the exact chunks of the super tiles
// alternate between the two 256-column accumulators.
__device__ __forceinline__ void issue_pair(const GemmArgs &g, uint8_t *ops, uint64_t *full,
                                           uint64_t *empty, uint64_t *accf, uint64_t *acce,
                                           uint64_t *drain, uint32_t tmem,
                                           volatile int *abort_flag) {
  int s = 0, b = 0;
  uint32_t ph = 0, aph = 0u;  // bit b of aph: phase parity of accumulator b
  const uint32_t idesc = make_idesc(!g.a_kmajor, !g.b_kmajor, 2 * BM, 2 * BN);
  const uint64_t a_step = g.a_kmajor ? 2u : (2048u >> 4);
  const uint64_t b_step = g.b_kmajor ? 2u : (2048u >> 4);
  Item t;
  bool ok = true;
  for (int64_t local = 0; ok && cta_item<true>(g, local, t) && !*abort_flag; local += 2) {
    for (int64_t c0 = t.kb0; ok && c0 < t.kb1; c0 += g.kc_blocks) {
      const int64_t c1 = min(t.kb1, c0 + g.kc_blocks);
      const uint32_t par = ((aph >> b) & 1u) ^ 1u;
      ok = mbar_wait(&acce[2 * b], par, g.status) && mbar_wait(&acce[2 * b + 1], par, g.status);
      if (!ok) break;
      tc_fence_after();
      const uint32_t dt = tmem + (uint32_t)(b * 2 * BN);
      for (int64_t kb = c0; kb < c1; ++kb) {
        if (!mbar_wait(&full[s], ph, g.status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t a_addr = smem_u32(ops + (size_t)(2 * s) * kTileBytes);
        const uint32_t b_addr = a_addr + (uint32_t)kTileBytes;
        const uint64_t da =
            g.a_kmajor ? sw128_desc(a_addr) : sw128_desc_mn(a_addr, g.mn_lbo, g.mn_sbo);
        const uint64_t db =
            g.b_kmajor ? sw128_desc(b_addr) : sw128_desc_mn(b_addr, g.mn_lbo, g.mn_sbo);
#pragma unroll
        for (int k = 0; k < BK / 16; ++k)
          umma_f16_pair(dt, da + a_step * k, db + b_step * k, idesc, (kb > c0 || k > 0) ? 1u : 0u);
        umma_commit_pair(&empty[s]);
        if (++s == g.stages) { s = 0; ph ^= 1u; }
      }
      umma_commit_pair(&accf[2 * b]);
      umma_commit_pair(&accf[2 * b + 1]);
      aph ^= 1u << b;
      b ^= 1;
    }
  }
  if (!ok) *abort_flag = 1;
  // every MMA has completed before tensor memory is released
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(drain))
      : "memory");
  mbar_wait(drain, 0, g.status);
}

// Split-K partials of a pair: set h (warps 4 h ..) owns the 128 columns of
// half h; a thread keeps its row's 128 int32 running sums in registers, adds
// each exact chunk to them and at the end stores four 32 x 32 boxes, the
// partials or, with one split (g.fuse), grad_W dequantized as k_reduce would.
// (With ll_to_float's range test and conversions per output the dequantization
// took 9 of the 60.5 us of 1024 x 4096 over 8192 rows, now 2.)
// Column terms of a super tile in shared memory: ka cb (int64) and cb - Kn mb
// (fp32) per column, written by the 256 threads together.
// WIDE: the same for k_gemm_wide (columns past g.wn are not stored).
template <bool WIDE>
__device__ __forceinline__ void partial_epilogue_pair(const GemmArgs &g, uint8_t *smem,
                                                      uint8_t *ring, uint64_t *accf,
                                                      uint64_t *acce, uint32_t tmem,
                                                      const CUtensorMap *tmOut,
                                                      volatile int *abort_flag, int warp,
                                                      int lane) {
  const int ew = warp - kGemmWarpEpi0, q = warp & 3, h = ew >> 2;
  uint8_t *box = ring + (size_t)ew * kBoxBytes;
  const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * BN);
  long long *col_i = reinterpret_cast<long long *>(smem + kOffPar);          // [256]
  float *col_f = reinterpret_cast<float *>(smem + kOffPar + 256 * 8);        // [256]
  const ReduceArgs &r = g.red;
  float sab = 0.0f, kdd = 0.0f, da = 0.0f, db = 0.0f;
  int64_t ka = 0, kb = 0, k0 = 0, ma = 0, mb = 0;
  if (g.fuse) {
    const float za = *r.zero_a, zb = *r.zero_b;
    sab = (*r.inv_a) * (*r.inv_b);
    ma = __float2int_rn(-za);
    mb = __float2int_rn(-zb);
    da = za + (float)ma;
    db = zb + (float)mb;
    kdd = ll_to_float(r.Kn) * da * db;
    ka = r.oa - ma;
    kb = r.ob - mb;
    k0 = r.Kn * ka * kb - ka * r.Kn * r.ob - kb * r.Kn * r.oa;
  }
  uint32_t cc = 0;  // exact chunks so far
  bool dead = false;
  bool stored = false;
  Item t;
  // the same trip count in all eight warps (they meet at named barriers)
  for (int64_t local = 0; WIDE ? wide_item(g, local + h, t) : cta_item<true>(g, local + h, t);
       local += 2) {
    dead = dead || *abort_flag;
    float rt = 0.0f;
    int64_t Ia = 0;
    bool wide = false;
    if (g.fuse) {
      const int64_t d = t.n0 - h * BN + ew * 32 + lane;  // one column each
      const int64_t cb = d < g.N ? r.cs_b[d] : 0;
      asm volatile("bar.sync 1, 256;" ::: "memory");  // the last item's terms are read
      col_i[ew * 32 + lane] = ka * cb;
      col_f[ew * 32 + lane] = ll_to_float(cb - r.Kn * mb);
      const int64_t c = t.m0 + q * 32 + lane;
      const int64_t ca = c < g.M ? r.cs_a[c] : 0;
      rt = db * ll_to_float(ca - r.Kn * ma);
      Ia = kb * ca + k0;
      // every |I| below 2^45?  (|P| < 2^31)
      const int64_t lim = (int64_t)1 << 43;
      const int64_t kac = ka * cb;
      const uint32_t far = kac >= lim || kac <= -lim || Ia >= lim || Ia <= -lim;
      uint32_t any;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\t"
          "setp.ne.u32 p, %1, 0;\n\t"
          "bar.red.or.pred q, 1, 256, p;\n\t"
          "selp.u32 %0, 1, 0, q;\n\t}"
          : "=r"(any)
          : "r"(far)
          : "memory");
      wide = any != 0u;
    }
    int sum[BN];
#pragma unroll
    for (int j = 0; j < BN; ++j) sum[j] = 0;
    const int64_t nchunks = (t.kb1 - t.kb0 + g.kc_blocks - 1) / g.kc_blocks;
    for (int64_t c = 0; c < nchunks; ++c, ++cc) {
      const int b = (int)(cc & 1u), buf = 2 * b + h;
      bool got = !dead && !*abort_flag && mbar_wait(&accf[buf], (cc >> 1) & 1u, g.status);
      got = __all_sync(0xffffffffu, got);
      if (!got) {
        dead = true;
        break;
      }
      tc_fence_after();
      const uint32_t acc = lane_base + (uint32_t)(b * 2 * BN);
#pragma unroll
      for (int grp = 0; grp < BN / 32; ++grp) {
        uint32_t v[32];
        tmem_ld32_nw(acc + (uint32_t)(grp * 32), v);
        tmem_wait_ld(v);
        if (grp == BN / 32 - 1) {  // the accumulator has been read in full
          tc_fence_before();
          __syncwarp();
          if (lane == 0) acc_release<!WIDE>(&acce[buf]);
        }
#pragma unroll
        for (int j = 0; j < 32; ++j)
          sum[grp * 32 + j] += __float2int_rn(__uint_as_float(v[j]));
      }
    }
    if (dead) {
      *abort_flag = 1;
      continue;
    }
#pragma unroll
    for (int grp = 0; grp < BN / 32; ++grp) {
      if (WIDE && h * BN + grp * 32 >= g.wn) break;
      uint32_t o[32];
      if (g.fuse) {
        const int c0 = h * BN + grp * 32;
        if (!wide) {
#pragma unroll
          for (int j = 0; j < 32; ++j)
            o[j] = __float_as_uint(i45_to_float((int64_t)sum[grp * 32 + j] + (col_i[c0 + j] + Ia)));
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j)
            o[j] = __float_as_uint(ll_to_float((int64_t)sum[grp * 32 + j] + (col_i[c0 + j] + Ia)));
        }
#pragma unroll
        for (int j = 0; j < 32; ++j)
          o[j] = __float_as_uint(sab * (__uint_as_float(o[j]) + rt + da * col_f[c0 + j] + kdd));
      } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) o[j] = (uint32_t)sum[grp * 32 + j];
      }
      if (stored) {
        if (lane == 0) bulk_wait_read(0);
        __syncwarp();
      }
#pragma unroll
      for (int j4 = 0; j4 < 8; ++j4)
        *reinterpret_cast<uint4 *>(box + sw128_off(lane, j4)) =
            make_uint4(o[4 * j4], o[4 * j4 + 1], o[4 * j4 + 2], o[4 * j4 + 3]);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0 && t.m0 < g.M && t.n0 < g.N) {
        int32_t col = (int32_t)(t.n0 + grp * 32);
        if (WIDE && g.taps) {  // tile = (kernel row, 64 channels), atom = tap of the row
          const int j = h * BN + grp * 32, tile = (int)(t.n0 - h * BN) / g.wn;
          const int gpr = g.cin / 64, ky = tile / gpr;
          col = (ky * g.taps + j / 64) * g.cin + (tile - ky * gpr) * 64 + j % 64;
        }
        tma_store_3d(tmOut, col, (int32_t)(t.m0 + q * 32), t.split, box);
        bulk_commit();
      }
      stored = true;
    }
  }
  if (lane == 0) bulk_wait_read(0);  // shared memory is read before the CTA ends
  __syncwarp();
}

// The tiles of this CTA left raw by the fp32-form epilogue (defined with the
// group fix-up, whose arithmetic it shares).
template <int NB, bool PAIR>
__device__ __noinline__ void gradx_raw_fix(const GemmArgs &g, const uint32_t *raw_mask, int ew,
                                           int nwarps, int lane, bool p_bits);

// PAIR: the CTAs of a cluster of two work as one tensor-core pair
// (cta_group::2): super tiles of 256 x 256, each CTA staging its 128 rows of
// A and its 128 columns of B per K block, so that a staged byte and a ring
// hand-over feed twice the MMA work of a CTA on its own and the instruction
// is 256 columns wide (1843 against 1487 TFLOP/s at 128).  The leader (rank
// 0) issues the MMAs for both and counts both CTAs' copies; its commits
// release the stages and hand over the accumulators in both.  Each CTA's
// tensor memory holds two accumulators of 256 columns for its 128 rows,
// drained as four of 128 by the same epilogue sets.
template <int MODE, int NB, int FORM, bool PAIR = false>
__global__ void __launch_bounds__(GemmLayout<MODE, FORM, NB, PAIR>::threads, 1)
    k_gemm(const __grid_constant__ CUtensorMap tmA,
           const __grid_constant__ CUtensorMap tmB,
           const __grid_constant__ CUtensorMap tmOut, const GemmArgs g) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // 1024-byte alignment of the shared-window address (swizzle atoms)
  uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kOffBar);
  const int nstages = g.stages;
  const bool u8ops = MODE == MODE_PARTIAL && g.u8 != 0;
  const int ustages = u8ops ? g.ustages : 0;
  uint8_t *ops = smem + kFixedBytes;                                // carrier stages
  uint8_t *uops = ops + (size_t)nstages * 2 * kTileBytes;          // byte stages
  uint8_t *ring = uops + (size_t)ustages * kTileBytes;             // output boxes
  uint64_t *full = bars, *empty = bars + kMaxStages;
  uint64_t *accf = bars + 2 * kMaxStages, *acce = accf + 4;
  uint64_t *pfull = acce + 4, *pempty = pfull + 4, *drain = pempty + 4;
  // byte operands: carrier stage widened (converters -> MMA), carrier stage
  // consumed (MMA -> converters); full / empty then serve the byte ring
  uint64_t *cvt = bars + 2 * kMaxStages + 17, *fempty = cvt + kMaxStages;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + kNumBars);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  // grad_X: one accumulator per item, served by 4 epilogue warps (one per
  // lane quadrant); partials: accumulators alternate per chunk, 8 warps each
  constexpr bool kPerItem = MODE == MODE_GRADX;
  // grad_X with several exact chunks per tile (two accumulators, each tile on
  // its own): the operand ring carries two tiles at a time, chunk by chunk,
  // so that the fold of one tile's chunk overlaps the other tile's MMAs
  // (FORM 2 runs one exact chunk per tile: never pairs)
  const bool pairs = FORM != 2 && kPerItem && g.nacc == 2;
  const int64_t gstep = (pairs ? 2 : 1) * (int64_t)gridDim.x;
  constexpr uint32_t kEpiArrivals = PAIR ? 8u : kPerItem ? 4u : (uint32_t)kPartialEpiWarps;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    const int nring = u8ops ? ustages : nstages;
    for (int i = 0; i < nring; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], u8ops ? kCvtWarps : 1);
    }
    for (int i = 0; u8ops && i < nstages; ++i) {
      mbar_init(&cvt[i], kCvtWarps);
      mbar_init(&fempty[i], 1);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(&accf[i], 1);
      mbar_init(&acce[i], kEpiArrivals);
      mbar_init(&pfull[i], 1);
      mbar_init(&pempty[i], 4);  // the 4 epilogue warps of the consuming set
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (MODE == MODE_GRADX && NB != 0)
    for (int i = threadIdx.x; i < (int)(kRawMaskBytes / 4); i += blockDim.x)
      reinterpret_cast<uint32_t *>(smem + kOffRaw)[i] = 0u;
  if (PAIR && warp == kWarpMma) {
    asm volatile(
        "tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
            smem_u32(tmem_slot)),
        "r"(kTmemCols)
        : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  } else if (warp == kWarpMma) {
    asm volatile(
        "tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
            smem_u32(tmem_slot)),
        "r"(kTmemCols)
        : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();  // the peer's barriers exist
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  using LY = GemmLayout<MODE, FORM, NB, PAIR>;

  auto fail = [&]() { *abort_flag = 1; };

  // Every warp of a warpgroup executes the same setmaxnreg, and each role's
  // code follows its own warpgroup's setmaxnreg.
  if (warp >= kGemmWarpEpi0) {
    if constexpr (LY::regs_epi > 0)
      asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(LY::regs_epi));
    if (MODE == MODE_GRADX) {
      gradx_epilogue<NB, FORM, PAIR>(g, smem, ring, accf, acce, pfull, pempty, tmem, &tmOut,
                               abort_flag, warp, lane);
      if constexpr (NB != 0) {
        // every epilogue warp arrives here once; then the tiles left raw
        // (their products stored by this CTA: fp32 values in FORM 2, int32
        // bit patterns otherwise) are finished
        asm volatile("bar.sync 1, %0;" ::"r"(32 * 4 * LY::sets) : "memory");
        if (!*abort_flag)
          gradx_raw_fix<NB, PAIR>(g, reinterpret_cast<const uint32_t *>(smem + kOffRaw),
                            warp - kGemmWarpEpi0, 4 * LY::sets, lane, FORM != 2);
      }
    }
    else if constexpr (PAIR)
      partial_epilogue_pair<false>(g, smem, ring, accf, acce, tmem, &tmOut, abort_flag, warp, lane);
    else if (warp < kGemmWarpEpi0 + kPartialEpiWarps)
      partial_epilogue(g, ring, accf, acce, tmem, &tmOut, abort_flag, warp, lane);
    else if (u8ops)  // the four warps after the partial epilogue
      partial_convert(g, ops, uops, full, empty, cvt, fempty, abort_flag,
                      2 + warp - (kGemmWarpEpi0 + kPartialEpiWarps), lane);
  } else {
  if constexpr (LY::regs_ctl > 0)
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(LY::regs_ctl));
  if (warp == kWarpTma) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      if constexpr (PAIR) {
        produce_pair<MODE>(g, tmA, tmB, ops, full, empty, abort_flag, s, ph);
      } else if (pairs) {
        bool ok = true;
        for (int64_t it = blockIdx.x; ok && it < g.n_items && !*abort_flag; it += gstep) {
          Item tt[2];
          const int nu = group_items(g, it, pairs, tt);
          const int64_t nch = (tt[0].kb1 - tt[0].kb0 + g.kc_blocks - 1) / g.kc_blocks;
          for (int64_t c = 0; ok && c < nch; ++c) {
            for (int u = 0; ok && u < nu; ++u) {
              const Item &t = tt[u];
              const int64_t c0 = t.kb0 + c * g.kc_blocks, c1 = min(t.kb1, c0 + g.kc_blocks);
              for (int64_t kb = c0; kb < c1; ++kb) {
                if (!mbar_wait(&empty[s], ph ^ 1u, g.status)) { fail(); ok = false; break; }
                mbar_expect_tx(&full[s], (uint32_t)(2 * kTileBytes));
                uint8_t *sa = ops + (size_t)(2 * s) * kTileBytes;
                uint8_t *sb = sa + kTileBytes;
                const int32_t kc = (int32_t)(kb * BK);
                // K-major: one 64 x 128 box; MN-major: two 64 (MN) x 64 (K) boxes
                if (g.a_kmajor) {
                  tma_load_2d(sa, &tmA, kc, (int32_t)t.m0, &full[s]);
                } else {
                  tma_load_2d(sa, &tmA, (int32_t)t.m0, kc, &full[s]);
                  tma_load_2d(sa + kTileBytes / 2, &tmA, (int32_t)t.m0 + 64, kc, &full[s]);
                }
                if (g.b_kmajor) {
                  tma_load_2d(sb, &tmB, kc, (int32_t)t.n0, &full[s]);
                } else {
                  tma_load_2d(sb, &tmB, (int32_t)t.n0, kc, &full[s]);
                  tma_load_2d(sb + kTileBytes / 2, &tmB, (int32_t)t.n0 + 64, kc, &full[s]);
                }
                if (++s == nstages) { s = 0; ph ^= 1u; }
              }
            }
          }
        }
      } else {
        for (int64_t it = blockIdx.x; it < g.n_items && !*abort_flag; it += gridDim.x) {
          const Item t = decode_item(g, it);
          // implicit im2col: the item's two (tap, channel group) columns of
          // X~ and its first block's (image, row group), then advanced per
          // K block without divisions
          int cimg = 0, cyb = 0, ccg[2] = {0, 0}, ckx[2] = {0, 0}, cky[2] = {0, 0};
          bool cval[2] = {false, false};
          if (MODE == MODE_PARTIAL && g.conv) {
            cimg = (int)(t.kb0 / g.cybi);
            cyb = (int)(t.kb0 - (int64_t)cimg * g.cybi);
            for (int h = 0; h < 2; ++h) {
              const int d = (int)t.n0 + 64 * h;
              const int tap = d / g.cin;
              ccg[h] = d - tap * g.cin;
              cky[h] = tap / g.ckw;
              ckx[h] = tap - cky[h] * g.ckw;
              cval[h] = d < g.N;
            }
          }
          for (int64_t kb = t.kb0; kb < t.kb1; ++kb) {
            if (!mbar_wait(&empty[s], ph ^ 1u, g.status)) { fail(); break; }
            const int32_t kc = (int32_t)(kb * BK);
            if (u8ops) {
              // byte operands (MN-major), into the byte ring: one 128 (MN) x
              // 64 (K) byte box each
              uint8_t *ua = uops + (size_t)s * kTileBytes;
              mbar_expect_tx(&full[s], (uint32_t)kTileBytes);
              tma_load_2d(ua, &tmA, (int32_t)t.m0, kc, &full[s]);
              tma_load_2d(ua + kTileBytes / 2, &tmB, (int32_t)t.n0, kc, &full[s]);
              if (++s == ustages) { s = 0; ph ^= 1u; }
              continue;
            }
            uint8_t *sa = ops + (size_t)(2 * s) * kTileBytes;
            uint8_t *sb = sa + kTileBytes;
            mbar_expect_tx(&full[s], (uint32_t)(2 * kTileBytes));
            if (MODE == MODE_PARTIAL && g.conv) {
              // implicit im2col: K block kb = output rows rpb yb .. of image
              // img, slots 0 .. pw - 1 of each; Q_b1 rows at those pixels,
              // X~ columns n0 .. n0 + 127 = (tap, 64 channels) pairs read at
              // the tap's offset (outside the input: zeros, the padding)
              const int oy0 = cyb * g.crpb;
              tma_load_4d(sa, &tmA, (int32_t)t.m0, 0, oy0, cimg, &full[s]);
              tma_load_4d(sa + kTileBytes / 2, &tmA, (int32_t)t.m0 + 64, 0, oy0, cimg, &full[s]);
              for (int h = 0; h < 2; ++h) {
                if (cval[h])
                  tma_load_4d(sb + h * (kTileBytes / 2), &tmB, ccg[h], ckx[h] - g.cpad,
                              oy0 + cky[h] - g.cpad, cimg, &full[s]);
                else  // past the last tap: a box outside the tensor (zeros)
                  tma_load_4d(sb + h * (kTileBytes / 2), &tmB, 0, 0, g.cih + g.coh + 8, cimg,
                              &full[s]);
              }
              if (++cyb == g.cybi) { cyb = 0; ++cimg; }
              if (++s == nstages) { s = 0; ph ^= 1u; }
              continue;
            }
            // K-major: one 64 x 128 box; MN-major: two 64 (MN) x 64 (K) boxes
            if (g.a_kmajor) {
              tma_load_2d(sa, &tmA, kc, (int32_t)t.m0, &full[s]);
            } else {
              tma_load_2d(sa, &tmA, (int32_t)t.m0, kc, &full[s]);
              tma_load_2d(sa + kTileBytes / 2, &tmA, (int32_t)t.m0 + 64, kc, &full[s]);
            }
            if (g.b_kmajor) {
              tma_load_2d(sb, &tmB, kc, (int32_t)t.n0, &full[s]);
            } else {
              tma_load_2d(sb, &tmB, (int32_t)t.n0, kc, &full[s]);
              tma_load_2d(sb + kTileBytes / 2, &tmB, (int32_t)t.n0 + 64, kc, &full[s]);
            }
            if (++s == nstages) { s = 0; ph ^= 1u; }
          }
        }
      }
      // every issued load lands before the CTA exits: in normal operation
      // the MMAs have consumed them all; after an abort, give in-flight
      // copies time to complete
      if (*abort_flag) {
        sleep_ns(200000);
      } else {
        const int pstages = u8ops ? ustages : nstages;
        for (int i = 0; i < pstages; ++i) {
          if (!mbar_wait(&empty[s], ph ^ 1u, g.status)) break;
          if (++s == pstages) { s = 0; ph ^= 1u; }
        }
      }
    }
  } else if (warp == kWarpMma) {
    // ------------------------------------------------------------ MMA issuer
    if (PAIR) {
      if (lane == 0 && (blockIdx.x & 1) == 0)
        issue_pair(g, ops, full, empty, accf, acce, drain, tmem, abort_flag);
    } else if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      int buf = 0;
      uint32_t aph = 0u;  // bit b: phase parity of accumulator b
      const uint32_t idesc = make_idesc(!g.a_kmajor, !g.b_kmajor);
      // start-address step of one K = 16 slice: 32 bytes inside a K-major
      // swizzle row, two 8-row K atoms (2048 bytes) for MN-major
      const uint64_t a_step = g.a_kmajor ? 2u : (2048u >> 4);
      const uint64_t b_step = g.b_kmajor ? 2u : (2048u >> 4);
      if (pairs) {
        int64_t local = 0;
        bool ok = true;
        for (int64_t it = blockIdx.x; ok && it < g.n_items && !*abort_flag; it += gstep) {
          Item tt[2];
          const int nu = group_items(g, it, pairs, tt);
          const int64_t nch = (tt[0].kb1 - tt[0].kb0 + g.kc_blocks - 1) / g.kc_blocks;
          for (int64_t c = 0; ok && c < nch && !*abort_flag; ++c) {
            for (int u = 0; ok && u < nu; ++u) {
              const Item &t = tt[u];
              if (kPerItem) buf = (int)((local + u) & (g.nacc - 1));
              const int64_t c0 = t.kb0 + c * g.kc_blocks, c1 = min(t.kb1, c0 + g.kc_blocks);
              if (!mbar_wait(&acce[buf], ((aph >> buf) & 1u) ^ 1u, g.status)) {
                fail();
                ok = false;
                break;
              }
              tc_fence_after();
              const uint32_t dt = tmem + (uint32_t)(buf * BN);
              for (int64_t kb = c0; kb < c1; ++kb) {
                if (!mbar_wait(&full[s], ph, g.status)) { fail(); ok = false; break; }
                tc_fence_after();
                const uint32_t a_addr = smem_u32(ops + (size_t)(2 * s) * kTileBytes);
                const uint32_t b_addr = a_addr + (uint32_t)kTileBytes;
                const uint64_t da = g.a_kmajor ? sw128_desc(a_addr)
                                               : sw128_desc_mn(a_addr, g.mn_lbo, g.mn_sbo);
                const uint64_t db = g.b_kmajor ? sw128_desc(b_addr)
                                               : sw128_desc_mn(b_addr, g.mn_lbo, g.mn_sbo);
  #pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                  umma_f16(dt, da + a_step * k, db + b_step * k, idesc,
                           (kb > c0 || k > 0) ? 1u : 0u);
                umma_commit(&empty[s]);
                if (++s == nstages) { s = 0; ph ^= 1u; }
              }
              umma_commit(&accf[buf]);
              aph ^= 1u << buf;
              if (!kPerItem) buf ^= 1;
            }
          }
          local += nu;
        }
      } else {
        int64_t local = 0;
        for (int64_t it = blockIdx.x; it < g.n_items && !*abort_flag; it += gridDim.x, ++local) {
          const Item t = decode_item(g, it);
          if (kPerItem) buf = (int)(local & (g.nacc - 1));
          for (int64_t c0 = t.kb0; c0 < t.kb1 && !*abort_flag; c0 += g.kc_blocks) {
            const int64_t c1 = min(t.kb1, c0 + g.kc_blocks);
            if (!mbar_wait(&acce[buf], ((aph >> buf) & 1u) ^ 1u, g.status)) { fail(); break; }
            tc_fence_after();
            const uint32_t dt = tmem + (uint32_t)(buf * BN);
            for (int64_t kb = c0; kb < c1; ++kb) {
              // byte operands: the carrier stage once the converter warps
              // widened it
              if (!mbar_wait(u8ops ? &cvt[s] : &full[s], ph, g.status)) { fail(); break; }
              tc_fence_after();
              const uint32_t a_addr = smem_u32(ops + (size_t)(2 * s) * kTileBytes);
              const uint32_t b_addr = a_addr + (uint32_t)kTileBytes;
              const uint64_t da = g.a_kmajor ? sw128_desc(a_addr)
                                             : sw128_desc_mn(a_addr, g.mn_lbo, g.mn_sbo);
              const uint64_t db = g.b_kmajor ? sw128_desc(b_addr)
                                             : sw128_desc_mn(b_addr, g.mn_lbo, g.mn_sbo);
  #pragma unroll
              for (int k = 0; k < BK / 16; ++k)
                umma_f16(dt, da + a_step * k, db + b_step * k, idesc,
                         (kb > c0 || k > 0) ? 1u : 0u);
              umma_commit(u8ops ? &fempty[s] : &empty[s]);
              if (++s == nstages) { s = 0; ph ^= 1u; }
            }
            umma_commit(&accf[buf]);
            aph ^= 1u << buf;
            if (!kPerItem) buf ^= 1;
          }
        }
      }
      // every MMA this thread issued has completed before TMEM is released
      // (after an abort the epilogue may have stopped waiting for them)
      umma_commit(drain);
      mbar_wait(drain, 0, g.status);
    }
  } else if (warp == kGemmWarpPar) {
    if (MODE == MODE_GRADX) gradx_params<NB, FORM, PAIR>(g, smem, pfull, pempty, abort_flag, lane);
    else if (u8ops) partial_convert(g, ops, uops, full, empty, cvt, fempty, abort_flag, 0, lane);
  } else if (MODE == MODE_PARTIAL && u8ops && warp == kGemmWarpPar + 1) {
    partial_convert(g, ops, uops, full, empty, cvt, fempty, abort_flag, 1, lane);
  }
  }

  tc_fence_before();
  __syncthreads();
  // neither CTA of a pair leaves while the other may still reach its memory
  if constexpr (PAIR) cluster_sync();
  if (warp == kWarpMma) {
    __syncwarp();
    tc_fence_after();
    if constexpr (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                   "r"(kTmemCols)
                   : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                   "r"(kTmemCols)
                   : "memory");
  }
}

// Arguments of the passes that finish grad_X rows left as exact products:
// the adaptive groups (fqt_gemm.cu) and the raw tiles of k_gemm.
struct FixArgs {
  float *out;
  int64_t N, D;
  int C, og, ow, bw, b2;
  const float *inv_s, *zero, *hz, *hr;
  const int32_t *row_sum, *perm, *gstart;
  const float *inv_sw, *zero_w;
  const int32_t *col_sum_w;
  float raw_mmax;
  int small_p;  // every |P| < 2^22: the fp32 block sums apply
  float mmax_nb[33];  // groups of nb <= 32 rows: largest |m| of the fp32 form
  int32_t *list, *list_big;
  int *count, *count_big;
  // fixed blocks (gradx_raw_fix): block size, per-tensor Q_b2 metadata
  // (PTQ) and the lead row of every block
  int nbk, per_tensor;
  const int32_t *lead;
  int p_bits;  // the stored products are int32 bit patterns (else fp32 values)
  int *status;
};

// Per-row terms of the epilogue: scale, the offsets (hd, hR) and m.
struct RowTerms {
  float sc, hd, hR, m;
};

__device__ __forceinline__ float zero_of(const FixArgs &f, int64_t k) {
  return f.zero[f.per_tensor ? 0 : k];
}

__device__ __forceinline__ RowTerms row_terms(const FixArgs &f, int64_t k, float inv_sw,
                                              bool reflected) {
  RowTerms t;
  t.sc = __fmul_rn(inv_sw, f.inv_s[f.per_tensor ? 0 : k]);
  const ff x = two_sum((float)f.og, zero_of(f, k));
  t.m = rintf(x.h);
  // BHQ rows (no row sums here) read their offsets from hz, hr even for a
  // one-row block, where they are the unreflected d and R
  if (reflected || !f.row_sum) {
    t.hd = f.hz[k];
    t.hR = f.hr[k];
  } else {
    t.hd = ff_round(fast_two_sum(__fsub_rn(x.h, t.m), x.l));
    t.hR = __fadd_rn((float)(f.row_sum[k] - f.C * f.og), __fmul_rn((float)f.C, t.m));
  }
  return t;
}

// Any group (or a single row left raw): rows visited one by one; the fp32
// form where it is exact, else int64 integer parts and float-float.  The
// lead row is row `lead` of the group (0 for the stored groups); rows are
// perm[k] of grad_X, or k itself without perm.
static __device__ __noinline__ void fix_group_general(const FixArgs &f, int64_t k0, int nb, int64_t j,
                                               bool jv, const float (&cwc)[4],
                                               const int (&cwi)[4], const float (&U)[4],
                                               float inv_sw, const ff &y, int lead) {
  const int lane = threadIdx.x & 31;
  const int Cn = f.C;
  const bool refl = nb >= 2;
  // the fp32 form: |P| < 2^22 and |I| (2 + sqrt(nb)) < 2^24 for every row
  bool fast = refl && f.small_p && !f.p_bits;
  auto pint = [&](float v) -> long long {
    return f.p_bits ? (long long)__float_as_int(v) : (long long)__float2int_rn(v);
  };
  if (fast) {
    const double lim = 16777216.0 / (2.0 + sqrt((double)nb));
    const double mmax = floor(lim / ((double)Cn * (double)(1 << (f.bw - 1)))) -
                        (double)(1 << (f.b2 - 1)) - 1.0;
    for (int r = lane; r < nb; r += 32) {
      const float m = rintf(two_sum((float)f.og, zero_of(f, k0 + r)).h);
      if (!((double)fabsf(m) <= mmax)) fast = false;
    }
    fast = __all_sync(0xffffffffu, fast);
  }
  auto prow = [&](int r) -> float * {
    int64_t pr = f.perm ? (int64_t)f.perm[k0 + r] : k0 + r;
    if (pr < 0 || pr >= f.N) pr = 0;
    return f.out + pr * f.D + j;
  };
  if (fast) {
    const HhConst hc = hh_const(nb);
    uint32_t sb[4] = {0u, 0u, 0u, 0u};
    int msum = 0, Ip[4] = {0, 0, 0, 0};
    for (int r = 0; r < nb; ++r) {
      const float m = rintf(two_sum((float)f.og, zero_of(f, k0 + r)).h);
      msum += (int)m;
      if (!jv) continue;
      const float4 P = *reinterpret_cast<const float4 *>(prow(r));
      const float pv[4] = {P.x, P.y, P.z, P.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        sb[c] += magic_bits(pv[c]);
        if (r == lead) Ip[c] = magic_int(pv[c]) + (int)m * cwi[c];
      }
    }
    BlockFixF bf[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int S = (int)(sb[c] - (uint32_t)nb * kMagicBits) + cwi[c] * msum;
      bf[c] = block_fix_f(hc, S, Ip[c]);
    }
    for (int r = 0; r < nb; ++r) {
      const RowTerms t = row_terms(f, k0 + r, inv_sw, true);
      const float A = __fmul_rn(t.sc, t.hd);
      const float B = __fmul_rn(t.sc, __fmaf_rn(t.hR, y.h, __fmul_rn(t.hR, y.l)));
      const float4 kq = make_float4(t.sc, A, B, t.m);
      if (!jv) continue;
      float *po = prow(r);
      const float4 P = *reinterpret_cast<const float4 *>(po);
      const float pv[4] = {P.x, P.y, P.z, P.w};
      float o4[4];
#pragma unroll
      for (int c = 0; c < 4; ++c)
        o4[c] = r == lead ? dequant(kq, bf[c].lead, U[c])
                       : dequant(kq, reflect_f(pv[c], kq, cwc[c], bf[c]), U[c]);
      __stcs(reinterpret_cast<float4 *>(po), make_float4(o4[0], o4[1], o4[2], o4[3]));
    }
  } else {
    // int64 integer parts I = P + m CWc, float-float reflection
    long long S[4] = {0, 0, 0, 0}, Ipl[4] = {0, 0, 0, 0};
    for (int r = 0; r < nb && jv; ++r) {
      const long long m = __float2ll_rn(rintf(two_sum((float)f.og, zero_of(f, k0 + r)).h));
      const float4 P = *reinterpret_cast<const float4 *>(prow(r));
      const float pv[4] = {P.x, P.y, P.z, P.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const long long I = pint(pv[c]) + m * cwi[c];
        S[c] += I;
        if (r == lead) Ipl[c] = I;
      }
    }
    ff rS[4], beta[4];
    if (refl) {
      const HhConst hc = hh_const(nb);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        rS[c] = ff_mul(hc.rho, ff_from_int(S[c]));
        beta[c] = ff_mul(hc.kap, ff_add(rS[c], ff_neg(ff_from_int(Ipl[c]))));
      }
    }
    for (int r = 0; r < nb && jv; ++r) {
      const RowTerms t = row_terms(f, k0 + r, inv_sw, refl);
      float *po = prow(r);
      const float4 P = *reinterpret_cast<const float4 *>(po);
      const float pv[4] = {P.x, P.y, P.z, P.w};
      const long long m = __float2ll_rn(t.m);
      float o4[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const ff I = ff_from_int(pint(pv[c]) + m * cwi[c]);
        ff v = !refl ? I : (r == lead ? rS[c] : ff_add(I, ff_neg(beta[c])));
        v = ff_add(v, two_prod(t.hd, U[c]));
        v = ff_add(v, ff_mul({t.hR, 0.0f}, y));
        o4[c] = __fmul_rn(t.sc, ff_round(v));
      }
      __stcs(reinterpret_cast<float4 *>(po), make_float4(o4[0], o4[1], o4[2], o4[3]));
    }
  }
}

// Tiles of a fixed-block grad_X (or of the forward) in the fp32 form that the
// contraction left raw (a row offset m beyond the form): after its last
// tile, every epilogue warp of the CTA takes every nwarps-th (tile, block)
// unit of the CTA's raw tiles -- each lane 4 of the tile's 128 columns --
// with the arithmetic of fix_group_general (int64 integer parts and
// float-float where the fp32 form is not exact).  NB = 1: one row per unit.
template <int NB, bool PAIR>
__device__ __noinline__ void gradx_raw_fix(const GemmArgs &g, const uint32_t *raw_mask, int ew,
                                           int nwarps, int lane, bool p_bits) {
  constexpr int NBD = NB > 1 ? NB : 1;
  constexpr int BPT = BN / NBD;  // units per tile
  int64_t n_local =
      PAIR ? 2 * ((g.n_items - (int64_t)(blockIdx.x >> 1) + (gridDim.x >> 1) - 1) /
                  (int64_t)(gridDim.x >> 1))
           : (g.n_items - (int64_t)blockIdx.x + gridDim.x - 1) / (int64_t)gridDim.x;
  if (n_local > kMaxLocalTiles) n_local = kMaxLocalTiles;
  const int nwords = (int)((n_local + 31) / 32);
  bool any = false;
  for (int w = 0; w < nwords; ++w) any |= raw_mask[w] != 0u;
  if (!any) return;
  FixArgs f;
  memset(&f, 0, sizeof(f));
  f.out = g.out;
  f.N = g.N;
  f.D = g.M;
  f.C = (int)g.K;
  f.og = g.og;
  f.ow = g.ow;
  f.bw = g.bw;
  f.b2 = g.b2;
  f.inv_s = g.inv_s;
  f.zero = g.zero;
  f.hz = g.hz;
  f.hr = g.hr;
  f.row_sum = NB > 1 ? nullptr : g.row_sum;
  f.inv_sw = g.inv_sw;
  f.zero_w = g.zero_w;
  f.col_sum_w = g.col_sum_w;
  f.small_p = g.small_p;
  f.p_bits = p_bits;
  f.nbk = NB;
  f.per_tensor = g.kind == FQT_PTQ;
  f.lead = g.lead;
  f.status = g.status;
  const float inv_sw = *g.inv_sw, zw = *g.zero_w;
  const ff y = two_sum((float)g.ow, zw);
  const int Cn = (int)g.K;
  int64_t u = 0;
  for (int w = 0; w < nwords; ++w) {
    uint32_t bits = raw_mask[w];
    while (bits) {
      const int l = w * 32 + __ffs(bits) - 1;
      bits &= bits - 1u;
      Item t;
      if (!cta_item<PAIR>(g, l, t)) continue;
      for (int b = 0; b < BPT; ++b, ++u) {
        if ((int)(u % nwarps) != ew) continue;
        const int64_t k0 = t.n0 + (int64_t)b * NBD;
        if (k0 >= g.N) continue;
        const int nb = (int)min((int64_t)NBD, g.N - k0);
        const int64_t j = t.m0 + lane * 4;
        const bool jv = j < g.M;
        float cwc[4], U[4];
        int cwi[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int cs = jv ? g.col_sum_w[j + c] : 0;
          cwc[c] = (float)(cs - Cn * g.ow);
          cwi[c] = (int)cwc[c];
          U[c] = __fmaf_rn((float)Cn, zw, (float)cs);
        }
        int lead = NBD > 1 ? g.lead[k0 / NBD] : 0;
        if (lead < 0 || lead >= nb) lead = 0;
        fix_group_general(f, k0, nb, j, jv, cwc, cwi, U, inv_sw, y, lead);
      }
    }
  }
}


// ---------------------------------------------------------------------------
// Host helpers of the launchers
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t,
                                  void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                         cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// Tensor map of an fp16 carrier matrix stored row-major as outer x inner,
// box of box_inner x box_outer elements, 128-byte swizzle (the UMMA layout).
inline bool make_map_f16(CUtensorMap *m, const void *base, uint64_t inner,
                         uint64_t outer, uint32_t box_inner, uint32_t box_outer) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {inner * 2};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void *>(base), dims,
            strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

inline int exact_chunk_blocks(int a_bits, int b_bits) {
  // centred magnitudes <= 2^(b-1): partial sums stay below 2^24
  const int lg = 26 - a_bits - b_bits;
  int64_t kc = (int64_t)1 << (lg < 0 ? 0 : lg);
  int64_t blocks = kc / BK;
  if (blocks < 1) blocks = 1;
  if (blocks > (1 << 20)) blocks = 1 << 20;
  return (int)blocks;
}

inline bool aligned16(const void *p) {
  return (reinterpret_cast<uintptr_t>(p) & 15u) == 0;
}

typedef void (*GemmKernel)(CUtensorMap, CUtensorMap, CUtensorMap, GemmArgs);

// Split-K partials of one or two 64-row atoms of A against up to 256 columns
// of B (fqt_gemm_pair.cu).
size_t gemm_wide_smem(uint32_t b_bytes, int stages);
__global__ void k_gemm_wide(const __grid_constant__ CUtensorMap tmA,
                            const __grid_constant__ CUtensorMap tmB,
                            const __grid_constant__ CUtensorMap tmOut, const GemmArgs g);

// The pair instance of a mode, block size and epilogue form (fqt_gemm_pair.cu).
GemmKernel gemm_pair_kernel(int mode, int nb, int form);

}  // namespace fqt
