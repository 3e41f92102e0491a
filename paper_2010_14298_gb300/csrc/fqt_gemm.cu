// fqt_gemm.cu -- the low-bit contractions of the FQT backward (Eq. 6, App. E)
// on the 5th-generation tensor cores of sm_103a.
//
// sm_103a has no tcgen05.mma kind::i8, so the integer codes ride in fp16:
// the quantizers emit every code centred, c - 2^(b-1) (|.| <= 128), as an
// exact fp16 value; products are exact and the fp32 accumulator in tensor
// memory stays exact while every partial sum is below 2^24 in magnitude.
// The reduction is therefore cut into exact chunks of K_c = 2^(26 - bA - bB)
// terms; between chunks the epilogue warps fold the accumulator into an
// int32 running sum kept in tensor memory (tcgen05.st).
//
// k_gemm and its epilogues are in fqt_gemm_core.cuh (warp roles there), the
// CTA-pair instances and k_gemm_wide in fqt_gemm_pair.cu; here are the
// single-CTA instances, the plans and the choice between them, k_reduce,
// k_gradw, the padding sums and the adaptive groups' fix-up.
// Every mbarrier wait is bounded; a wait that runs out records FQT_ETIMEOUT
// and the CTA winds down.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <algorithm>
#include <string.h>

#include "fqt_common.cuh"
#include "fqt_gemm_core.cuh"
#include "fqt_internal.h"

namespace fqt {

// ---------------------------------------------------------------------------
// Split-K reduction (int64) and the grad_W / raw epilogues
// ---------------------------------------------------------------------------
// A thread sums four consecutive outputs of one row (r.vec; else one output)
// over every `groups`-th split, one 16-byte load per split, coalesced across
// the warp and four in flight; the groups of an output meet in shared memory
// and the first dequantizes.  Few outputs with many splits were a chain of
// loads in a handful of CTAs: 256 x 64 over 76 splits 11.2 us with one group,
// 5.6 with eight; 112 x 80 over 152 splits 16.6 -> 6.2 us; 1008 x 2048 in one
// split (no 64-bit division or conversion per output) 12.0 -> 9.4 us.  With
// two groups and few splits the meeting costs more than it hides (1200 x 336
// over 5: 5.4 us with one group, 7.2 with two).
constexpr int kRedThreads = 256, kRedGroups = 8;

__global__ void __launch_bounds__(kRedThreads) k_reduce(const ReduceArgs r, int groups) {
  __shared__ long long part_s[kRedThreads][4];
  const int64_t total = r.M * r.N;
  const bool vec = r.vec != 0;
  const int W = vec ? 4 : 1;
  const int64_t units = vec ? total >> 2 : total;
  // per-tensor terms: z = -m + d with m an integer
  const bool deq = r.out_i64 == nullptr;
  const float za = deq ? *r.zero_a : 0.0f, zb = deq ? *r.zero_b : 0.0f;
  const float sab = deq ? (*r.inv_a) * (*r.inv_b) : 0.0f;
  const int64_t ma = __float2int_rn(-za), mb = __float2int_rn(-zb);
  const float da = za + (float)ma, db = zb + (float)mb;
  const int64_t ob = r.ob;
  const int64_t code_pad = r.pad_a ? (int64_t)*r.code_zero - ob : 0;
  const float kdd = ll_to_float(r.Kn) * da * db;
  // I = sum (a - ma)(b - mb) = P + ka cb + kb ca + k0, exact, from the
  // centred product P (ca, cb the code column sums)
  const int64_t ka = r.oa - ma, kb = ob - mb;
  const int64_t k0 = r.Kn * ka * kb - ka * r.Kn * ob - kb * r.Kn * r.oa;
  const int upc = kRedThreads / groups;  // units per CTA and step
  const int ul = (int)threadIdx.x & (upc - 1), grp = (int)threadIdx.x / upc;
  for (int64_t u0 = (int64_t)blockIdx.x * upc; u0 < units; u0 += (int64_t)gridDim.x * upc) {
    const int64_t u = u0 + ul, idx = u * W;
    long long P[4] = {0, 0, 0, 0};
    if (u < units && vec) {
      const int4 *src = reinterpret_cast<const int4 *>(r.part + idx);
      const int64_t step = total >> 2;
      int sp = grp;
      for (; sp + 3 * groups < r.splits; sp += 4 * groups) {
        int4 x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = __ldcs(src + (int64_t)(sp + i * groups) * step);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          P[0] += x[i].x;
          P[1] += x[i].y;
          P[2] += x[i].z;
          P[3] += x[i].w;
        }
      }
      for (; sp < r.splits; sp += groups) {
        const int4 x = __ldcs(src + (int64_t)sp * step);
        P[0] += x.x;
        P[1] += x.y;
        P[2] += x.z;
        P[3] += x.w;
      }
    } else if (u < units) {
      for (int sp = grp; sp < r.splits; sp += groups)
        P[0] += __ldcs(r.part + (int64_t)sp * total + idx);
    }
    if (groups > 1) {
      __syncthreads();  // the last step's sums are read
#pragma unroll
      for (int i = 0; i < 4; ++i) part_s[threadIdx.x][i] = P[i];
      __syncthreads();
      if (grp == 0)
        for (int g = 1; g < groups; ++g)
#pragma unroll
          for (int i = 0; i < 4; ++i) P[i] += part_s[g * upc + ul][i];
    }
    if (grp != 0 || u >= units) continue;
    if (!deq) {
      for (int i = 0; i < W; ++i) r.out_i64[idx + i] = P[i];
      continue;
    }
    const int64_t c = total < ((int64_t)1 << 32) ? (int64_t)((uint32_t)idx / (uint32_t)r.N)
                                                 : idx / r.N;
    const int64_t d0 = idx - c * r.N;
    const int64_t ca = r.cs_a[c];
    // row term db (ca - Kn ma) of this thread's row
    const float rt = db * ll_to_float(ca - r.Kn * ma);
    const int64_t Ia = kb * ca + k0;
    float o[4];
    for (int i = 0; i < W; ++i) {
      const int64_t d = d0 + i;
      const int64_t cb = r.cs_b[d];
      long long Pi = P[i];
      if (r.pad_a) Pi += code_pad * r.pad_a[(int64_t)((uint32_t)d / (uint32_t)r.cin) * r.M + c];
      const int64_t I = Pi + ka * cb + Ia;
      const float f = (uint64_t)(I + ((int64_t)1 << 44)) < ((uint64_t)1 << 45) ? i45_to_float(I)
                                                                               : ll_to_float(I);
      o[i] = sab * (f + rt + da * ll_to_float(cb - r.Kn * mb) + kdd);
    }
    if (vec)
      *reinterpret_cast<float4 *>(r.out_f32 + idx) = make_float4(o[0], o[1], o[2], o[3]);
    else
      r.out_f32[idx] = o[0];
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
// 4-D map of NHWC-ordered fp16 carriers (c, w, h, n) with boxes of 64
// channels x bw pixels x bh rows x 1 image, 128-byte swizzle: the image of a
// (bw bh) x 64 MN-major operand tile (one 128-byte row per pixel).
static bool make_map_f16_box4(CUtensorMap *m, const void *base, uint64_t n, uint64_t h,
                              uint64_t w, uint64_t c, uint32_t bw, uint32_t bh) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[4] = {c, w, h, n};
  cuuint64_t strides[3] = {c * 2, w * c * 2, h * w * c * 2};
  cuuint32_t box[4] = {64, bw, bh, 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void *>(base), dims, strides,
            box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tensor map of MN-major byte codes stored as outer (K) rows of inner (MN)
// bytes: 128 x 64 boxes (one 128-byte row per K row), 128-byte swizzle.
static bool make_map_u8(CUtensorMap *m, const void *base, uint64_t inner, uint64_t outer) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {inner};
  cuuint32_t box[2] = {128, BK};
  cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(base), dims, strides, box,
            es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Output tensor map: fp32 M x N (grad_X) or int32 splits x M x N
// (partials), 32 x 32 boxes with 128-byte swizzle.
static bool make_map_out(CUtensorMap *m, void *base, bool is_int, uint64_t cols,
                         uint64_t rows, uint64_t depth) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {cols, rows, depth};
  cuuint64_t strides[2] = {cols * 4, cols * rows * 4};
  cuuint32_t box[3] = {32, 32, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(m, is_int ? CU_TENSOR_MAP_DATA_TYPE_INT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
            is_int ? 3 : 2, base, dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_NONE,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Split-K plan for an M x N output reduced over K.
struct SplitPlan {
  int m_tiles, n_tiles, splits;
  int64_t ks_blocks, kb_total;
};

// pair: super tiles of 256 x 256 for CTA pairs.
static SplitPlan plan_splits(int64_t M, int64_t N, int64_t K, int a_bits,
                             int b_bits, int num_sms, bool allow_split, bool pair = false) {
  SplitPlan p;
  const int64_t tm = pair ? 2 * BM : BM, tn = pair ? 2 * BN : BN;
  if (pair) num_sms /= 2;
  p.m_tiles = (int)((M + tm - 1) / tm);
  p.n_tiles = (int)((N + tn - 1) / tn);
  p.kb_total = (K + BK - 1) / BK;
  if (p.kb_total < 1) p.kb_total = 1;
  int splits = 1;
  if (allow_split) {
    // as many splits as keep every (tile, split) item in one wave of CTAs
    const int64_t tiles = (int64_t)p.m_tiles * p.n_tiles;
    splits = (int)(num_sms / tiles);
    if (splits < 1) splits = 1;
    // int32 partials: a split reduces at most 2^31 / 2^(a+b-2) terms
    const int64_t max_terms = ((int64_t)1 << 31) >> (a_bits + b_bits - 2);
    const int64_t min_splits = (K + max_terms - 1) / max_terms;
    if (splits < min_splits) splits = (int)min_splits;
    if (splits > p.kb_total) splits = (int)p.kb_total;
    if (splits < 1) splits = 1;
  }
  p.ks_blocks = (p.kb_total + splits - 1) / splits;
  p.splits = (int)((p.kb_total + p.ks_blocks - 1) / p.ks_blocks);
  return p;
}

// The plan of k_gemm_wide: the tile width (128, 192 or 256 columns) whose waves
// take least, or `fixed` columns.  A K block takes 0.25 to 0.4 us (0.3 of 192
// columns where one copy serves the taps of a kernel row), an item 8 us beside
// them (its 128 x 256 sums).
static double wide_plan(int64_t M, int64_t N, int64_t K, int a_bits, int b_bits, int num_sms,
                        int fixed, SplitPlan *best, int *wn) {
  double least = 1e300;
  for (int w = fixed ? fixed : 128; w <= (fixed ? fixed : 256); w += 64) {
    SplitPlan p;
    p.m_tiles = (int)((M + BM - 1) / BM);
    p.n_tiles = (int)((N + w - 1) / w);
    p.kb_total = std::max<int64_t>(1, (K + BK - 1) / BK);
    const int64_t tiles = (int64_t)p.m_tiles * p.n_tiles;
    int64_t splits = std::max<int64_t>(1, num_sms / tiles);
    const int64_t max_terms = ((int64_t)1 << 31) >> (a_bits + b_bits - 2);
    splits = std::max(splits, (K + max_terms - 1) / max_terms);
    splits = std::min(splits, p.kb_total);
    p.ks_blocks = (p.kb_total + splits - 1) / splits;
    p.splits = (int)((p.kb_total + p.ks_blocks - 1) / p.ks_blocks);
    const int64_t waves = (tiles * p.splits + num_sms - 1) / num_sms;
    const double t = (double)waves * ((double)p.ks_blocks * ((fixed ? 60.0 : 100.0) + 1.2 * w) + 8000.0) +
                     (double)M * (double)N * 8.0 / 5000.0 * p.splits;
    if (t < least) {
      least = t;
      *best = p;
      *wn = w;
    }
  }
  return least;
}

// The single-CTA plan's time on the same scale.
static double single_time(const SplitPlan &p, int64_t M, int64_t N, int num_sms) {
  const int64_t waves =
      ((int64_t)p.m_tiles * p.n_tiles * p.splits + num_sms - 1) / num_sms;
  return (double)waves * (410.0 * (double)p.ks_blocks + 5000.0) +
         (double)M * (double)N * 8.0 / 5000.0 * p.splits;
}

// The k_gradw plan for grad_W of C x D over K rows, or splits = 0 when the
// shape does not fit it.
struct WPlan {
  int mt, ncb, Cn, stages, splits;
  int64_t ks_blocks, kb_total;
  size_t smem;
};

static WPlan gradw_plan(int64_t K, int64_t C, int64_t D, int b1, int bx, int num_sms);

// An implicit im2col grad_W takes k_gradw (one exact chunk per K range)
// unless its plan would need more than two ranges per SM (wide operands,
// e.g. the shift quantizer's 12-bit shifted codes); plain operands take the
// split-K tile kernel, whose ranges fold several exact chunks.
static bool use_gradw(const WPlan &w, int num_sms) {
  return w.splits > 0 && w.splits <= 2 * num_sms;
}

size_t gemm_workspace_bytes(int64_t N, int64_t C, int64_t D) {
  // grad_W: M = C, N = D, K = N, by either kernel; the operand bits run from
  // 2 (Q_b1) to 12 (shifted 8-bit codes of the shift quantizer)
  const int nsm = device_sm_count();
  int64_t splits = 0;
  for (int b = 2; b <= 12; ++b) {
    const WPlan w = gradw_plan(N, C, D, b, 8, nsm);
    int64_t sp = use_gradw(w, nsm) ? w.splits : plan_splits(C, D, N, b, 8, nsm, true).splits;
    // an implicit im2col operand pads each image's output rows to blocks of
    // 64 slots: at most 2.4 N slots (ow = 9 in blocks of 4 rows of 16)
    const int64_t Kp = (N * 5 + 1) / 2;
    const int64_t sc = plan_splits(C, D, Kp, b, 8, nsm, true).splits;
    if (sc > sp) sp = sc;
    // CTA pairs (more than 128 rows of grad_W)
    const int64_t s2 = C > BM ? plan_splits(C, D, Kp, b, 8, nsm, true, true).splits : 0;
    if (s2 > sp) sp = s2;
    if (C <= BM && D > BN) {
      SplitPlan wp;
      int wn;
      for (const int64_t K : {N, Kp})  // the widest tiles have the most splits
        for (const int fixed : {0, 2 * BN}) {
          wide_plan(C, D, K, b, 8, nsm, fixed, &wp, &wn);
          if (wp.splits > sp) sp = wp.splits;
        }
    }
    if (sp > splits) splits = sp;
  }
  // + the padding table of an implicit im2col X~ (C x taps, taps <= D)
  const size_t bytes = (size_t)splits * (size_t)C * (size_t)D * 4 + (size_t)C * D * 4;
  return (bytes + 255) & ~(size_t)255;
}

// Whether a contraction takes CTA pairs: p the plan of single CTAs, q that of
// pairs.  A K block takes about 0.4 us in either (128 x 128 for a CTA, 256 x
// 256 for a pair), so the one with clearly fewer K blocks in its longest
// chain of waves is taken.  Measured, 8192 tokens 1024 <-> 4096: grad_X 92 ->
// 57 us and 86 -> 54 us, forward 86 -> 55 us, grad_W 119 -> 63 us with its
// reduction fused.
// grad_X and the forward: below `min_kb` K blocks per tile the epilogue and
// its stores bound both, which a pair does not speed up: four with the fp32
// form (50176 x 256 x 2304: 130 -> 122 us), eight with the int32 one (53910 x
// 352 x 400, six K blocks: 86.6 -> 90.1 us).
static bool pair_faster(const SplitPlan &p, const SplitPlan &q, int num_sms, int min_kb) {
  const int64_t one = ((int64_t)p.m_tiles * p.n_tiles + num_sms - 1) / num_sms;
  const int64_t two = ((int64_t)q.m_tiles * q.n_tiles + num_sms / 2 - 1) / (num_sms / 2);
  return q.kb_total >= min_kb && 10 * two * (q.ks_blocks + 3) < 9 * one * (p.ks_blocks + 3);
}

// grad_W: a pair's item costs about 12 us beside its K blocks (a CTA's 5: the
// pair drains 128 x 256 sums per CTA), and every split writes and reads back
// its partials; the pair has to be ahead by 15% (53910 x 352 x 400, 19 splits
// of 45 K blocks against 12 of 71: 37.3 us against 41.1 with its reduction).
static bool pair_faster_w(const SplitPlan &p, const SplitPlan &q, int64_t C, int64_t D,
                          int num_sms) {
  const int64_t one = ((int64_t)p.m_tiles * p.n_tiles * p.splits + num_sms - 1) / num_sms;
  const int64_t two =
      ((int64_t)q.m_tiles * q.n_tiles * q.splits + num_sms / 2 - 1) / (num_sms / 2);
  const double red = (double)C * (double)D * 8.0 / 5000.0;  // ns per split
  const double t1 = (double)one * (410.0 * (double)p.ks_blocks + 5000.0) + red * p.splits;
  const double t2 =
      (double)two * (400.0 * (double)q.ks_blocks + 12000.0) + (q.splits > 1 ? red * q.splits : 0.0);
  return t2 < 0.85 * t1;
}

// The kernel instance of a mode, BHQ block size (1 = no reflection) and
// product representation (fp32-exact or int32).
// The epilogue form (see GemmLayout) of a contraction whose fp32 form holds
// rows with |m| <= mmax, for codes of b bits.  A row whose values straddle 0
// has z' in [-(2^b - 1), 0], so |m| <= 2^(b-1): with mmax at least that, only
// rows of one sign far from 0 leave the form, and form 2 finishes them in a
// final pass; otherwise many tiles can, and form 1 keeps both paths.
// The largest row offset |m| of the int32 form for a reduction over C with
// codes of bw (W~) and b bits and blocks of nb rows: every |I| (2 + sqrt(nb))
// below 2^31 with |I| <= C 2^(bw-1) (2^(b-1) + |m|); -1 when none.
static float int32_form_mmax(int64_t C, int bw, int b, int nb) {
  const double lim = nb <= 1 ? 2147483647.0 : 2147483647.0 / (2.0 + sqrt((double)nb));
  const double m = floor(lim / ((double)C * (double)(1 << (bw - 1)))) - (double)(1 << (b - 1)) - 1.0;
  return m >= 0.0 ? (float)m : -1.0f;
}

static int epilogue_form(bool flt, double mmax, int b) {
  if (!flt) return 0;
  return mmax >= (double)(1 << (b - 1)) ? 2 : 1;
}

static GemmKernel gemm_kernel(int mode, int nb, int form) {
  if (mode == MODE_PARTIAL) return k_gemm<MODE_PARTIAL, 1, 0>;
#define FQT_GX(NBV)                                                          \
  case NBV:                                                                  \
    return form == 2   ? k_gemm<MODE_GRADX, NBV, 2>                           \
           : form == 1 ? k_gemm<MODE_GRADX, NBV, 1>                           \
                       : k_gemm<MODE_GRADX, NBV, 0>;
  switch (nb) {
    case 0:  // adaptive BHQ groups: fp32 form only (raw rows go to the group pass)
      return form == 2 ? k_gemm<MODE_GRADX, 0, 2> : nullptr;
    FQT_GX(1)
    FQT_GX(2)
    FQT_GX(4)
    FQT_GX(8)
    FQT_GX(16)
    FQT_GX(32)
    FQT_GX(64)
    FQT_GX(128)
  }
#undef FQT_GX
  return nullptr;
}

static thread_local LastPlan g_last_plan[2];

const LastPlan &last_plan(int which) { return g_last_plan[which]; }

// Launches the contraction of fp16 carrier operands: A is M x K (stored
// M x K if a_kmajor, else K x M), B is the K x N operand (stored N x K if
// b_kmajor, else K x N).  Partials: out is splits x M x N int32.  grad_X:
// out is the N x M fp32 transpose (rows of dH x columns of W~).
static fqt_status run_gemm(const void *A, int a_kmajor, int a_bits, const void *Bm,
                           int b_kmajor, int b_bits, int64_t M, int64_t N, int64_t K,
                           const SplitPlan &p, GemmArgs &g, void *out, int mode, int nb,
                           int form, cudaStream_t st, bool pair = false, int wide = 0) {
  const bool partial = mode == MODE_PARTIAL;
  // byte operands (g.u8): split-K partials of MN-major operands only
  if (g.u8 && (!partial || a_kmajor || b_kmajor)) return FQT_EUNSUPPORTED;
  CUtensorMap ta, tb;
  bool ok;
  if (g.u8) {
    ok = make_map_u8(&ta, A, (uint64_t)M, (uint64_t)K) &&
         make_map_u8(&tb, Bm, (uint64_t)N, (uint64_t)K);
  } else if (g.conv) {
    // implicit im2col (split-K partials, both MN-major): Q_b1 as (C, ow, oh,
    // n), the NHWC codes as (cin, iw, ih, n)
    if (!partial || a_kmajor || b_kmajor) return FQT_EUNSUPPORTED;
    ok = make_map_f16_box4(&ta, A, (uint64_t)g.cnimg, (uint64_t)g.coh, (uint64_t)g.cow,
                           (uint64_t)M, (uint32_t)g.cpw, (uint32_t)g.crpb) &&
         make_map_f16_box4(&tb, Bm, (uint64_t)g.cnimg, (uint64_t)g.cih, (uint64_t)g.ciw,
                           (uint64_t)g.cin, (uint32_t)(g.cpw + (g.taps ? g.taps - 1 : 0)),
                           (uint32_t)g.crpb);
  } else {
    ok = a_kmajor ? make_map_f16(&ta, A, (uint64_t)K, (uint64_t)M, BK, BM)
                  : make_map_f16(&ta, A, (uint64_t)M, (uint64_t)K, 64, BK);
    ok = ok && (b_kmajor ? make_map_f16(&tb, Bm, (uint64_t)K, (uint64_t)N, BK, BN)
                         : make_map_f16(&tb, Bm, (uint64_t)N, (uint64_t)K, 64, BK));
  }
  CUtensorMap to;
  ok = ok && (partial ? make_map_out(&to, out, true, (uint64_t)N, (uint64_t)M,
                                     (uint64_t)p.splits)
                      : make_map_out(&to, out, false, (uint64_t)M, (uint64_t)N, 1));
  if (!ok) return cuda_fail(cudaErrorInvalidValue, "tensor map encode");
  GemmKernel kern = pair ? gemm_pair_kernel(mode, nb, form) : gemm_kernel(mode, nb, form);
  if (!kern) return FQT_EUNSUPPORTED;
  g_last_plan[partial] = {wide ? PLAN_WIDE : pair ? PLAN_PAIR : PLAN_SINGLE, partial ? 0 : form,
                          p.splits, g.fuse, wide ? g.taps : 0};
  const bool four = !partial && form == 2;  // GemmLayout: four epilogue sets
  using LP = GemmLayout<1, 0, 1, true>;
  const int threads = partial && pair ? LP::threads
                      : four          ? GemmLayout<0, 2>::threads
                                      : GemmLayout<0, 0>::threads;
  if (partial && pair) {  // the register split, as below
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return cuda_fail(e, "gemm attributes");
    if (fa.numRegs * LP::threads < 128 * LP::regs_ctl + 256 * LP::regs_epi)
      return FQT_EUNSUPPORTED;
  }
  if (four) {
    // the register split needs the launch's registers per thread: with fewer,
    // setmaxnreg.inc would wait for registers that do not exist
    using L16 = GemmLayout<0, 2, 16>;
    using L32 = GemmLayout<0, 2, 32>;
    const int64_t need = nb <= 16 ? 128 * L16::regs_ctl + 32 * 4 * L16::sets * L16::regs_epi
                                  : 128 * L32::regs_ctl + 32 * 4 * L32::sets * L32::regs_epi;
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return cuda_fail(e, "gemm attributes");
    if ((int64_t)fa.numRegs * L16::threads < need) return FQT_EUNSUPPORTED;
  }
  // the fp32 form: four epilogue sets for tiles bound by their output, three
  // for long reductions; the code bits for the final pass over raw tiles
  // (a pair's accumulators change over two at a time: all four sets)
  g.sets = (four && (pair || (K + BK - 1) / BK <= 2)) ? 4 : 3;
  g.bw = a_bits;
  g.b2 = b_bits;
  g.small_p = (K << (a_bits + b_bits - 2)) < ((int64_t)1 << 22);
  // HBM-bound output tiles (grad_X): deep store ring; long reductions
  // (split-K partials): deep operand ring
  // byte operands: two carrier stages fed by a ring of six byte stages
  g.stages = partial ? (g.u8 ? 2 : 5) : 2;
  g.ustages = g.u8 ? 6 : 0;
  g.ring = partial ? 1 : 0;  // grad_X stores straight from registers
  // grad_X tiles with a long reduction (K of many blocks: a contraction that
  // is tensor-bound rather than bound by its output) keep more operand
  // stages in flight
  if (!partial && (K + BK - 1) / BK > 2) {
    while (g.stages < kMaxStages && gemm_smem_bytes(g.stages + 1, g.ring) <= 227 * 1024)
      ++g.stages;
  }
  if (!partial) g.out = static_cast<float *>(out);
  // grad_X with one exact chunk per tile: four accumulators in rotation, so
  // the next tile of each epilogue set is ready when it finishes the last;
  // otherwise two, and the other half of tensor memory holds running sums
  g.nacc = (!partial && exact_chunk_blocks(a_bits, b_bits) >= (K + BK - 1) / BK) ? 4 : 2;
  // Several exact chunks per tile (two accumulators): one epilogue set per
  // accumulator, so that each accumulator's chunks are drained by one set in
  // order.  An mbarrier parity wait cannot tell a phase from the one two
  // phases later; with three sets, the set of tile L + 2 could start waiting
  // on accumulator L mod 2 while tile L's chunks still pass through it (the
  // parameter ring holds that set back only until tile L - 4 is done).  With
  // one chunk per tile, tile L's parameters wait for tile L - 4 (the same
  // accumulator of four) to be drained, which is enough.
  if (!partial && g.nacc == 2) g.sets = 2;
  g.m_fast = partial ? 0 : 1;
  g.M = M;
  g.N = N;
  g.K = K;
  g.a_kmajor = a_kmajor;
  g.b_kmajor = b_kmajor;
  g.mn_lbo = (uint32_t)(kTileBytes / 2);  // second 64-wide MN atom column
  g.mn_sbo = 1024;                        // next 8-row K atom
  g.kc_blocks = exact_chunk_blocks(a_bits, b_bits);
  g.m_tiles = p.m_tiles;
  g.n_tiles = p.n_tiles;
  g.splits = p.splits;
  g.ks_blocks = p.ks_blocks;
  g.kb_total = p.kb_total;
  g.n_items = (int64_t)p.m_tiles * p.n_tiles * p.splits;
  if (wide) {  // k_gemm_wide: the threads and registers of a pair's partials
    g.wn = wide;
    g.stages = kMaxStages;
    uint32_t bb = (uint32_t)(g.taps ? g.crpb * (g.cpw + g.taps - 1) : wide) * 128u;
    bb = (bb + 1023u) & ~1023u;
    while (g.stages > 2 && gemm_wide_smem(bb, g.stages) > 227 * 1024) --g.stages;
    const size_t smem = gemm_wide_smem(bb, g.stages);
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, k_gemm_wide);
    if (e != cudaSuccess) return cuda_fail(e, "wide gemm attributes");
    if (fa.numRegs * LP::threads < 128 * LP::regs_ctl + 256 * LP::regs_epi)
      return FQT_EUNSUPPORTED;
    e = cudaFuncSetAttribute(k_gemm_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "wide gemm shared-memory attribute");
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(g.n_items, device_sm_count()));
    k_gemm_wide<<<(int)grid, LP::threads, smem, st>>>(ta, tb, to, g);
    return cuda_fail(cudaGetLastError(), "wide gemm launch");
  }
  const size_t smem = gemm_smem_bytes(g.stages, g.ring, g.ustages);
  const cudaError_t ea =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (ea != cudaSuccess) return cuda_fail(ea, "gemm shared-memory attribute");
  const int nsm = device_sm_count();
  if (pair) {
    int64_t pairs = g.n_items < nsm / 2 ? g.n_items : nsm / 2;
    if (pairs < 1) pairs = 1;
    // two tiles per super tile
    if (!partial && 2 * ((g.n_items + pairs - 1) / pairs) > kMaxLocalTiles)
      return FQT_EUNSUPPORTED;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(2 * pairs));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cuda_fail(cudaLaunchKernelEx(&cfg, kern, ta, tb, to, g), "gemm pair launch");
  }
  int64_t grid = g.n_items < nsm ? g.n_items : nsm;
  if (grid < 1) grid = 1;
  // the raw-tile bits of a CTA cover kMaxLocalTiles of its tiles
  if (!partial && nb != 0 && (g.n_items + grid - 1) / grid > kMaxLocalTiles)
    return FQT_EUNSUPPORTED;
  kern<<<(int)grid, threads, smem, st>>>(ta, tb, to, g);
  return cuda_fail(cudaGetLastError(), "gemm launch");
}

// u8 codes -> fp16 carriers code - off (debug path only)
__global__ void k_u8_to_f16(const uint8_t *__restrict__ src, uint16_t *dst,
                            int64_t n, int off) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const __half h = __int2half_rn((int)src[i] - off);
    dst[i] = *reinterpret_cast<const uint16_t *>(&h);
  }
}

static void launch_reduce(ReduceArgs r, cudaStream_t st) {
  const int64_t total = r.M * r.N;
  auto a16 = [](const void *q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
  r.vec = (r.N & 3) == 0 && a16(r.part) && (r.out_i64 || a16(r.out_f32));
  const int64_t units = r.vec ? total >> 2 : total;
  // groups of splits until the GPU has about 512 threads per SM
  const int64_t nsm = device_sm_count();
  int groups = 1;
  while (groups < kRedGroups && groups * 2 <= r.splits && units * groups < nsm * 512) groups *= 2;
  const int64_t upc = kRedThreads / groups;
  int64_t grid = (units + upc - 1) / upc;
  const int64_t cap = nsm * 8;
  if (grid > cap) grid = cap;
  if (grid < 1) grid = 1;
  k_reduce<<<(int)grid, kRedThreads, 0, st>>>(r, groups);
}

static size_t round256(size_t v) { return (v + 255) & ~(size_t)255; }

size_t debug_workspace_bytes(int64_t M, int64_t N, int64_t K) {
  const SplitPlan p = plan_splits(M, N, K, 8, 8, device_sm_count(), true);
  return kGemmOffset + round256((size_t)p.splits * (size_t)M * (size_t)N * 4) +
         round256((size_t)M * (size_t)K * 2) + round256((size_t)N * (size_t)K * 2);
}

fqt_status debug_int_gemm(const uint8_t *A, int a_kmajor, int a_bits,
                          const uint8_t *Bm, int b_kmajor, int b_bits, int64_t M,
                          int64_t N, int64_t K, int64_t *out, void *ws,
                          size_t ws_bytes, cudaStream_t st) {
  if (!A || !Bm || !out || M <= 0 || N <= 0 || K <= 0) return FQT_EINVAL;
  if (a_bits < 2 || a_bits > 8 || b_bits < 2 || b_bits > 8) return FQT_EINVAL;
  // TMA: the row pitch of each stored operand must be a multiple of 16 bytes
  if ((a_kmajor ? K : M) % 8 || (b_kmajor ? K : N) % 8 || N % 4) return FQT_EUNSUPPORTED;
  if (M > INT32_MAX || N > INT32_MAX || K > INT32_MAX) return FQT_EUNSUPPORTED;
  const SplitPlan p = plan_splits(M, N, K, a_bits, b_bits, device_sm_count(), true);
  const size_t part_bytes = round256((size_t)p.splits * (size_t)M * (size_t)N * 4);
  const size_t need = kGemmOffset + part_bytes + round256((size_t)M * K * 2) +
                      round256((size_t)N * K * 2);
  if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < need)
    return FQT_EWORKSPACE;
  char *w = static_cast<char *>(ws);
  int32_t *part = reinterpret_cast<int32_t *>(w + kGemmOffset);
  uint16_t *a16 = reinterpret_cast<uint16_t *>(w + kGemmOffset + part_bytes);
  uint16_t *b16 = reinterpret_cast<uint16_t *>(w + kGemmOffset + part_bytes +
                                               round256((size_t)M * K * 2));
  const int nsm = device_sm_count();
  k_u8_to_f16<<<nsm * 4, 256, 0, st>>>(A, a16, M * K, 1 << (a_bits - 1));
  k_u8_to_f16<<<nsm * 4, 256, 0, st>>>(Bm, b16, N * K, 1 << (b_bits - 1));
  GemmArgs g;
  memset(&g, 0, sizeof(g));
  g.status = reinterpret_cast<int *>(ws);
  fqt_status s = run_gemm(a16, a_kmajor, a_bits, b16, b_kmajor, b_bits, M, N, K, p,
                          g, part, MODE_PARTIAL, 1, false, st);
  if (s != FQT_OK) return s;
  ReduceArgs r;
  memset(&r, 0, sizeof(r));
  r.part = part;
  r.splits = p.splits;
  r.M = M;
  r.N = N;
  r.out_i64 = out;
  launch_reduce(r, st);
  return cuda_fail(cudaGetLastError(), "split-K reduce launch");
}

// The same contraction with both operands MN-major byte codes (A stored
// K x M, B stored K x N) read as bytes and widened on chip: the path grad_W
// takes with byte operands.
fqt_status debug_int_gemm_u8(const uint8_t *A, int a_bits, const uint8_t *Bm, int b_bits,
                             int64_t M, int64_t N, int64_t K, int64_t *out, void *ws,
                             size_t ws_bytes, cudaStream_t st) {
  if (!A || !Bm || !out || M <= 0 || N <= 0 || K <= 0) return FQT_EINVAL;
  if (a_bits < 2 || a_bits > 8 || b_bits < 2 || b_bits > 8) return FQT_EINVAL;
  // TMA: byte rows of a multiple of 16 bytes, 16-byte aligned bases
  if (M % 16 || N % 16) return FQT_EUNSUPPORTED;
  if (M > INT32_MAX || N > INT32_MAX || K > INT32_MAX) return FQT_EUNSUPPORTED;
  if (!aligned16(A) || !aligned16(Bm)) return FQT_EINVAL;
  const SplitPlan p = plan_splits(M, N, K, a_bits, b_bits, device_sm_count(), true);
  const size_t part_bytes = round256((size_t)p.splits * (size_t)M * (size_t)N * 4);
  if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < kGemmOffset + part_bytes)
    return FQT_EWORKSPACE;
  int32_t *part = reinterpret_cast<int32_t *>(static_cast<char *>(ws) + kGemmOffset);
  GemmArgs g;
  memset(&g, 0, sizeof(g));
  g.status = reinterpret_cast<int *>(ws);
  g.u8 = 1;
  fqt_status s = run_gemm(A, 0, a_bits, Bm, 0, b_bits, M, N, K, p, g, part, MODE_PARTIAL, 1,
                          false, st);
  if (s != FQT_OK) return s;
  ReduceArgs r;
  memset(&r, 0, sizeof(r));
  r.part = part;
  r.splits = p.splits;
  r.M = M;
  r.N = N;
  r.out_i64 = out;
  launch_reduce(r, st);
  return cuda_fail(cudaGetLastError(), "split-K reduce launch");
}

// ---------------------------------------------------------------------------
// grad_W with one CTA per range of K rows and all of C x D (when C <= 256
// and ceil(D / 128) C <= 512 TMEM columns): out^T (D x C) = X~^T Q_b1 over
// the range, as ceil(D / 128) tiles of M = 128 (D) by N = C.  Every k-block
// of 64 rows loads X~'s rows (all D columns) and Q_b1's rows once, both
// contiguous in memory, and issues one MMA group per D tile into its own
// TMEM accumulator.  The range is one exact chunk (<= 2^(26 - b1 - bx)
// terms); the epilogue writes int32 partials [split][C][D] that k_reduce
// sums in int64.
// ---------------------------------------------------------------------------
constexpr int kWThreads = 320;  // TMA, MMA, 8 epilogue warps
constexpr int kWBK = 32;           // rows of K per stage (two K = 16 MMA steps)
constexpr size_t kWBox = 64 * kWBK * 2;  // one 64-wide fp16 box of a stage

struct WArgs {
  int64_t K;          // rows of dH / X
  int C, D, Cn;       // Cn: C rounded up to 16 (MMA N)
  int mt, ncb;        // D tiles of 128, 64-wide boxes of Q_b1
  int splits;
  int64_t ks_blocks, kb_total;
  int stages;
  int32_t *part;      // [splits][C][D]
  int *status;
  // implicit im2col operand (stride 1): X~ is read as 4-D boxes of an NHWC
  // tensor at shifted pixel coordinates; padding comes back as zero carriers
  int conv, ih, iw, oh, ow, cin, kh, kw, pad, taps;
};

__host__ __device__ constexpr uint32_t make_idesc_mn_n(int n) {
  // A and B MN-major, D fp32, M = 128, N = n
  return (1u << 4) | (1u << 15) | (1u << 16) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(BM >> 4) << 24);
}

// The int32 value of an fp32 holding an exact integer of magnitude <= 2^24,
// from its bits (no conversion instruction).
__device__ __forceinline__ int exact_f2i(float x) {
  const uint32_t bits = __float_as_uint(x);
  const uint32_t e = (bits >> 23) & 0xFFu;
  const uint32_t sig = (bits & 0x7FFFFFu) | 0x800000u;
  const uint32_t mag = e >= 150u ? sig << (e - 150u) : __funnelshift_rc(sig, 0u, 150u - e);
  return (bits >> 31) ? -(int)mag : (int)mag;
}

__global__ void __launch_bounds__(kWThreads, 1)
    k_gradw(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmQ,
            const WArgs w) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
  uint64_t *full = bars, *empty = bars + kMaxStages, *accf = empty + kMaxStages,
           *acce = accf + 1, *drain = acce + 1;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  uint8_t *ops = smem + 1024;
  const size_t xbytes = (size_t)w.mt * 2 * kWBox;  // per D tile: two 64-wide boxes
  const size_t stage_bytes = xbytes + (size_t)w.ncb * kWBox;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < w.stages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    mbar_init(accf, 1);
    mbar_init(acce, kPartialEpiWarps);
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == kWarpMma) {
    asm volatile(
        "tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
            smem_u32(tmem_slot)),
        "r"(kTmemCols)
        : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int64_t n_items = w.splits;

  if (warp == kWarpTma) {
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      // implicit im2col: the pixel position advances per K block; the D
      // boxes walk (channel group, tap) without divisions
      for (int64_t it = blockIdx.x; it < n_items && !*abort_flag; it += gridDim.x) {
        const int64_t kb0 = it * w.ks_blocks, kb1 = min(w.kb_total, kb0 + w.ks_blocks);
        int ox0 = 0, oy = 0, nimg = 0;
        if (w.conv) {
          const int64_t p0 = kb0 * kWBK, t = p0 / w.ow;
          ox0 = (int)(p0 - t * w.ow);
          oy = (int)(t % w.oh);
          nimg = (int)(t / w.oh);
        }
        for (int64_t kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(&empty[s], ph ^ 1u, w.status)) { *abort_flag = 1; break; }
          mbar_expect_tx(&full[s], (uint32_t)stage_bytes);
          uint8_t *sx = ops + (size_t)s * stage_bytes;
          uint8_t *sq = sx + xbytes;
          const int32_t kc = (int32_t)(kb * kWBK);
          if (w.conv) {
            // 32 output pixels of one output row (ow % 32 == 0); box (64 channels
            // of one tap) x 32 pixels read at the tap's offset
            int cg = 0, kx = 0, ky = 0;
            for (int m = 0; m < 2 * w.mt; ++m) {
              if (ky < w.kh)
                tma_load_4d(sx + (size_t)m * kWBox, &tmX, cg, ox0 + kx - w.pad,
                            oy + ky - w.pad, nimg, &full[s]);
              else  // past the last tap: a box outside the tensor (zeros)
                tma_load_4d(sx + (size_t)m * kWBox, &tmX, 0, 0, w.ih + w.oh + 8, nimg,
                            &full[s]);
              cg += 64;
              if (cg == w.cin) {
                cg = 0;
                if (++kx == w.kw) {
                  kx = 0;
                  ++ky;
                }
              }
            }
            ox0 += kWBK;
            if (ox0 == w.ow) {
              ox0 = 0;
              if (++oy == w.oh) {
                oy = 0;
                ++nimg;
              }
            }
          } else {
            for (int m = 0; m < w.mt; ++m) {
              tma_load_2d(sx + (size_t)m * 2 * kWBox, &tmX, m * 128, kc, &full[s]);
              tma_load_2d(sx + (size_t)m * 2 * kWBox + kWBox, &tmX, m * 128 + 64, kc, &full[s]);
            }
          }
          for (int cb = 0; cb < w.ncb; ++cb)
            tma_load_2d(sq + (size_t)cb * kWBox, &tmQ, cb * 64, kc, &full[s]);
          if (++s == w.stages) { s = 0; ph ^= 1u; }
        }
      }
      if (*abort_flag) {
        sleep_ns(200000);
      } else {
        for (int i = 0; i < w.stages; ++i) {
          if (!mbar_wait(&empty[s], ph ^ 1u, w.status)) break;
          if (++s == w.stages) { s = 0; ph ^= 1u; }
        }
      }
    }
  } else if (warp == kWarpMma) {
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0, eph = 0;
      const uint32_t idesc = make_idesc_mn_n(w.Cn);
      for (int64_t it = blockIdx.x; it < n_items && !*abort_flag; it += gridDim.x) {
        const int64_t kb0 = it * w.ks_blocks, kb1 = min(w.kb_total, kb0 + w.ks_blocks);
        if (!mbar_wait(acce, eph ^ 1u, w.status)) { *abort_flag = 1; break; }
        eph ^= 1u;
        tc_fence_after();
        for (int64_t kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(&full[s], ph, w.status)) { *abort_flag = 1; break; }
          tc_fence_after();
          const uint32_t x_addr = smem_u32(ops + (size_t)s * stage_bytes);
          const uint32_t q_addr = x_addr + (uint32_t)xbytes;
          const uint64_t dq = sw128_desc_mn(q_addr, (uint32_t)kWBox, 1024);
          for (int m = 0; m < w.mt; ++m) {
            const uint64_t dx =
                sw128_desc_mn(x_addr + (uint32_t)(m * 2 * kWBox), (uint32_t)kWBox, 1024);
#pragma unroll
            for (int k = 0; k < kWBK / 16; ++k)
              umma_f16(tmem + (uint32_t)(m * w.Cn), dx + (2048u >> 4) * k, dq + (2048u >> 4) * k,
                       idesc, (kb > kb0 || k > 0) ? 1u : 0u);
          }
          umma_commit(&empty[s]);
          if (++s == w.stages) { s = 0; ph ^= 1u; }
        }
        umma_commit(accf);
      }
      // every MMA this thread issued has completed before TMEM is released
      umma_commit(drain);
      mbar_wait(drain, 0, w.status);
    }
  } else {
    // epilogue: warp (q, h) takes the D tiles m = h, h + 2, ...; a thread owns
    // output column d = 128 m + 32 q + lane of grad_W^T
    const int q = warp & 3, h = (warp - kWarpEpi0) >> 2;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
    uint32_t aph = 0;
    for (int64_t it = blockIdx.x; it < n_items && !*abort_flag; it += gridDim.x) {
      const bool got = mbar_wait(accf, aph, w.status);
      if (!__all_sync(0xffffffffu, got)) { *abort_flag = 1; break; }
      aph ^= 1u;
      tc_fence_after();
      int32_t *pp = w.part + it * (int64_t)w.C * w.D;
      for (int m = h; m < w.mt; m += 2) {
        const int d = m * 128 + q * 32 + lane;
        for (int c0 = 0; c0 < w.Cn; c0 += 32) {
          uint32_t r[32];
          tmem_ld32_nw(lane_base + (uint32_t)(m * w.Cn + c0), r);
          tmem_wait_ld(r);
          if (d < w.D) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (c0 + i < w.C) pp[(int64_t)(c0 + i) * w.D + d] = exact_f2i(__uint_as_float(r[i]));
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce);
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

static WPlan gradw_plan(int64_t K, int64_t C, int64_t D, int b1, int bx, int num_sms) {
  WPlan p;
  memset(&p, 0, sizeof(p));
  if (C <= 0 || C > 256 || C % 16 || D <= 0 || D % 8 || K <= 0) return p;
  p.Cn = (int)C;
  p.mt = (int)((D + 127) / 128);
  if ((int64_t)p.mt * p.Cn > (int64_t)kTmemCols) return p;
  p.ncb = (int)((C + 63) / 64);
  const size_t stage = (size_t)p.mt * 2 * kWBox + (size_t)p.ncb * kWBox;
  p.stages = (int)((220 * 1024 - 1024 - 1024) / stage);
  if (p.stages > kMaxStages) p.stages = kMaxStages;
  if (p.stages < 2) {
    p.splits = 0;
    return p;
  }
  p.smem = 1024 + (size_t)p.stages * stage + 1024;
  p.kb_total = (K + kWBK - 1) / kWBK;
  const int64_t kc = exact_chunk_blocks(b1, bx) * (BK / kWBK);  // k-blocks per exact chunk
  int64_t splits = (p.kb_total + kc - 1) / kc;     // every range one exact chunk
  if (splits < num_sms) splits = num_sms;
  if (splits > p.kb_total) splits = p.kb_total;
  p.ks_blocks = (p.kb_total + splits - 1) / splits;
  p.splits = (int)((p.kb_total + p.ks_blocks - 1) / p.ks_blocks);
  return p;
}

// 4-D map of NHWC fp16 carriers (c, w, h, n), boxes of 64 channels x 32
// pixels of one image row, 128-byte swizzle: the same shared-memory image as
// a 64 x 32 box of the im2col matrix.
static bool make_map_f16_nhwc(CUtensorMap *m, const void *base, uint64_t n, uint64_t h,
                              uint64_t w, uint64_t c) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[4] = {c, w, h, n};
  cuuint64_t strides[3] = {c * 2, w * c * 2, h * w * c * 2};
  cuuint32_t box[4] = {64, (cuuint32_t)kWBK, 1, 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void *>(base), dims, strides,
            box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static fqt_status run_gradw(const uint16_t *X16, const uint16_t *Q16, int64_t K, int C, int D,
                            const WPlan &p, int32_t *part, int *status, cudaStream_t st,
                            const int32_t *conv = nullptr) {
  CUtensorMap tx, tq;
  bool ok = conv ? make_map_f16_nhwc(&tx, X16, (uint64_t)conv[0], (uint64_t)conv[1],
                                     (uint64_t)conv[2], (uint64_t)conv[3])
                 : make_map_f16(&tx, X16, (uint64_t)D, (uint64_t)K, 64, kWBK);
  ok = ok && make_map_f16(&tq, Q16, (uint64_t)C, (uint64_t)K, 64, kWBK);
  if (!ok) return cuda_fail(cudaErrorInvalidValue, "tensor map encode");
  WArgs w;
  memset(&w, 0, sizeof(w));
  w.K = K;
  w.C = C;
  w.D = D;
  w.Cn = p.Cn;
  w.mt = p.mt;
  w.ncb = p.ncb;
  w.splits = p.splits;
  w.ks_blocks = p.ks_blocks;
  w.kb_total = p.kb_total;
  w.stages = p.stages;
  w.part = part;
  w.status = status;
  if (conv) {
    w.conv = 1;
    w.ih = conv[1];
    w.iw = conv[2];
    w.cin = conv[3];
    w.kh = conv[4];
    w.kw = conv[5];
    w.pad = conv[6];
    w.oh = conv[1] + 2 * conv[6] - conv[4] + 1;
    w.ow = conv[2] + 2 * conv[6] - conv[5] + 1;
    w.taps = conv[4] * conv[5];
  }
  const cudaError_t ea =
      cudaFuncSetAttribute(k_gradw, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
  if (ea != cudaSuccess) return cuda_fail(ea, "grad_W shared-memory attribute");
  g_last_plan[1] = {PLAN_GRADW, 0, p.splits, 0, 0};
  const int nsm = device_sm_count();
  const int grid = p.splits < nsm ? p.splits : nsm;
  k_gradw<<<grid, kWThreads, p.smem, st>>>(tx, tq, w);
  return cuda_fail(cudaGetLastError(), "grad_W launch");
}

// H = X~ W~^T (Sec. 2.1): the grad_X kernel with the roles renamed -- M = C
// (rows of W~, K-major), N = rows of X~, K = D; the row terms of X~ take the
// place of Q_b2's (PTQ: one scale, one zero, the row sums), W~'s row sums the
// place of the column sums over the contraction.
fqt_status linear_forward(const fqt_qtensor *qx, const fqt_qtensor *qw, float *H, void *ws,
                          size_t ws_bytes, cudaStream_t st) {
  if (!qx || !qw || !H) return FQT_EINVAL;
  if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < kHeaderBytes)
    return FQT_EWORKSPACE;
  if (qx->kind != FQT_PTQ || qw->kind != FQT_PTQ) return FQT_EINVAL;
  const int64_t Nr = qx->rows, D = qx->cols, C = qw->rows;
  if (qw->cols != D || Nr < 0) return FQT_EINVAL;
  if (Nr == 0) return FQT_OK;
  if (!qx->codes_f16 || !qw->codes_f16 || !qx->row_sum || !qw->row_sum || !qx->inv_s ||
      !qx->zero || !qw->inv_s || !qw->zero)
    return FQT_EINVAL;
  if (C % 16 || D % 16) return FQT_EUNSUPPORTED;
  if (D > 8192) return FQT_EUNSUPPORTED;
  if (!aligned16(qx->codes_f16) || !aligned16(qw->codes_f16) || !aligned16(H)) return FQT_EINVAL;
  const int nsm = device_sm_count();
  const SplitPlan p = plan_splits(C, Nr, D, qw->bits, qx->bits, nsm, false);
  // no reflection: with P exact (one chunk) the fp32 form holds for all m
  const int64_t kc_terms = (int64_t)exact_chunk_blocks(qw->bits, qx->bits) * BK;
  const double mmax = 1e30;
  const bool flt = D <= kc_terms;
  GemmArgs g;
  memset(&g, 0, sizeof(g));
  g.status = reinterpret_cast<int *>(ws);
  g.kind = FQT_PTQ;
  g.og = 1 << (qx->bits - 1);
  g.ow = 1 << (qw->bits - 1);
  g.inv_s = qx->inv_s;
  g.zero = qx->zero;
  g.row_sum = qx->row_sum;
  g.col_sum_w = qw->row_sum;
  g.inv_sw = qw->inv_s;
  g.zero_w = qw->zero;
  g.flt_mmax = flt ? (float)mmax : -1.0f;
  g.i32_mmax = int32_form_mmax(D, qw->bits, qx->bits, 1);
  const SplitPlan pp = plan_splits(C, Nr, D, qw->bits, qx->bits, nsm, false, true);
  const bool pair = flt && pair_faster(p, pp, nsm, 4);
  return run_gemm(qw->codes_f16, 1, qw->bits, qx->codes_f16, 1, qx->bits, C, Nr, D,
                  pair ? pp : p, g, H, MODE_GRADX, 1, epilogue_form(flt, mmax, qx->bits), st,
                  pair);
}

// ---------------------------------------------------------------------------
// Implicit im2col X~ (stride 1): per tap (ky, kx), the sum over the output
// pixels whose input pixel (oy + ky - pad, ox + kx - pad) lies in the padding
// of the A operand's carriers (C per row), for the padding correction of
// k_reduce.  Only output pixels in the top / bottom pad rows or the left /
// right pad columns can read padding, and whether they do depends only on
// which of those rows and columns they sit in: (2 pad + 1)^2 classes (the
// inside class never).  A CTA (a run of images, a group of channels) adds
// each border pixel's carriers into its class in shared memory (16-byte
// loads, four in flight per thread), then adds each tap's share, the classes
// whose row or column reads padding, into the sums.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int pad_class(int y, int p, int n) {
  return y < p ? y : (y >= n - p ? 2 * p - (n - 1 - y) : p);
}

// the one output row (column) of border class r, or -1 for the inside class
__device__ __forceinline__ int pad_class_row(int r, int p, int n) {
  return r < p ? r : (r > p ? n - 1 - (2 * p - r) : -1);
}

__global__ void __launch_bounds__(256) k_conv_padsum(const uint16_t *__restrict__ A16, int C,
                                                     int ch_group, int64_t nimg, int imgs_per_cta,
                                                     int h, int w, int kw, int pad, int oh,
                                                     int ow, int taps, int32_t *pad_a) {
  extern __shared__ int cls_s[];  // classes x ch_group
  const int cc = 2 * pad + 1, ncls = cc * cc;
  const int64_t img0 = (int64_t)blockIdx.x * imgs_per_cta;
  const int nim = (int)min((int64_t)imgs_per_cta, nimg - img0);
  const int ch0 = (int)blockIdx.y * ch_group, nch = min(ch_group, C - ch0);
  for (int i = threadIdx.x; i < ncls * ch_group; i += blockDim.x) cls_s[i] = 0;
  __syncthreads();
  const int top = min(pad, oh), nbot = oh - max(top, oh - pad), full_rows = top + nbot;
  const int left = min(pad, ow), nright = ow - max(left, ow - pad), side = left + nright;
  const int full_px = full_rows * ow;
  const int npx = full_px + (oh - full_rows) * side;  // the pixel counts of one image fit int
  const int octs = nch / 8, per_img = npx * octs, items = nim * per_img;
  const uint16_t *base = A16 + (img0 * oh) * (int64_t)ow * C + ch0;
  for (int i0 = threadIdx.x; i0 < items; i0 += 4 * blockDim.x) {
    uint4 v[4];
    int k[4], oc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int it = i0 + u * (int)blockDim.x;
      k[u] = -1;
      oc[u] = 0;
      v[u] = make_uint4(0u, 0u, 0u, 0u);
      if (it < items) {
        const int im = it / per_img, rem = it - im * per_img, t = rem / octs;
        oc[u] = rem - t * octs;
        int oy, ox;
        if (t < full_px) {
          const int r = t / ow;
          oy = r < top ? r : oh - nbot + (r - top);
          ox = t - r * ow;
        } else {
          const int q = t - full_px, r = q / side, cq = q - r * side;
          oy = top + r;
          ox = cq < left ? cq : ow - nright + (cq - left);
        }
        k[u] = pad_class(oy, pad, oh) * cc + pad_class(ox, pad, ow);
        v[u] = __ldg(reinterpret_cast<const uint4 *>(
            base + (((int64_t)im * oh + oy) * ow + ox) * C + oc[u] * 8));
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (k[u] < 0) continue;
      const uint32_t wds[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&wds[q]));
        int *dst = &cls_s[k[u] * ch_group + oc[u] * 8 + 2 * q];
        if ((int)f.x) atomicAdd(dst, (int)f.x);
        if ((int)f.y) atomicAdd(dst + 1, (int)f.y);
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nch * taps; i += blockDim.x) {
    const int ch = i / taps, tap = i - ch * taps, ky = tap / kw, kx = tap - ky * kw;
    int v = 0;
    for (int ry = 0; ry < cc; ++ry) {
      const int yr = pad_class_row(ry, pad, oh);
      const bool row_out = yr >= 0 && (yr + ky - pad < 0 || yr + ky - pad >= h);
      for (int rx = 0; rx < cc; ++rx) {
        const int xr = pad_class_row(rx, pad, ow);
        const bool col_out = xr >= 0 && (xr + kx - pad < 0 || xr + kx - pad >= w);
        if (row_out || col_out) v += cls_s[(ry * cc + rx) * ch_group + ch];
      }
    }
    if (v) atomicAdd(&pad_a[(int64_t)tap * C + ch0 + ch], v);
  }
}

// Channels per CTA of k_conv_padsum: a multiple of 8 whose class sums fit
// 40 KB of shared memory (0: the padding is too wide, pad > 17).
static int padsum_group(int C, int pad) {
  const int ncls = (2 * pad + 1) * (2 * pad + 1);
  int grp = (40960 / (ncls * 4)) / 8 * 8;
  if (grp < 8) return 0;
  return grp < C ? grp : C;
}

// ---------------------------------------------------------------------------
// Adaptive BHQ groups (App. D.5).  After the contraction, the grad_X rows of
// every group of two or more rows -- and of single rows whose offset m is
// too large for the fp32 form -- hold the exact integer products P.  This
// pass adds the offsets and applies the group's inverse Householder
// reflection, the second of the two sparse-dense products Sec. 4.3 counts,
// with the arithmetic of the fused epilogue: fp32 where every magnitude is
// exact (block sums off the fp32 bits), int64 / float-float otherwise.
// k_grp_list collects the groups that need it; k_grp_fix gives a warp one
// (group, 128 columns) unit, each lane 4 consecutive columns, and
// k_grp_fix_big a CTA to each group of more than 32 rows.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_grp_list(const FixArgs f) {
  const int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool need = false;
  if (gi < f.N) {
    const int64_t k0 = f.gstart[gi];
    if (k0 < f.N) {
      const int64_t k1 = f.gstart[gi + 1];
      if (k1 - k0 > 32) {
        // a CTA of its own (k_grp_fix_big)
        const int slot = atomicAdd(f.count_big, 1);
        f.list_big[slot] = (int32_t)gi;
      } else if (k1 - k0 >= 2) {
        need = true;
      } else if (k1 - k0 == 1) {
        const float m = rintf(two_sum((float)f.og, f.zero[k0]).h);
        need = !(fabsf(m) <= f.raw_mmax);
      }
    }
  }
  const unsigned ball = __ballot_sync(0xffffffffu, need);
  if (!ball) return;
  const int lane = threadIdx.x & 31;
  int base = 0;
  if (lane == 0) base = atomicAdd(f.count, __popc(ball));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (need) f.list[base + __popc(ball & ((1u << lane) - 1u))] = (int32_t)gi;
}

// Groups of more than 32 rows: a CTA each, its warps taking every NW-th
// row (kBigBatch rows in flight per warp) with the int64 integer parts and
// float-float reflection of fix_group_general; the block sums S go through
// shared memory in warp order.
constexpr int kBigFixWarps = 16, kBigBatch = 4;

__global__ void __launch_bounds__(kBigFixWarps * 32) k_grp_fix_big(const FixArgs f) {
  constexpr int NW = kBigFixWarps;
  __shared__ long long s_part[NW][128];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nchunk = (int)((f.D + 127) / 128);
  const int nunits = *f.count_big;
  const float inv_sw = *f.inv_sw, zw = *f.zero_w;
  const ff y = two_sum((float)f.ow, zw);
  const int Cn = f.C;
  for (int u = blockIdx.x; u < nunits; u += gridDim.x) {
    const int64_t gi = f.list_big[u];
    if (gi < 0 || gi >= f.N) {
      if (threadIdx.x == 0) record_status(f.status, FQT_EINVAL);
      continue;
    }
    const int64_t k0 = f.gstart[gi];
    int64_t k1 = f.gstart[gi + 1];
    if (k1 > f.N) k1 = f.N;
    if (k0 < 0 || k1 - k0 < 2) continue;
    const int nb = (int)(k1 - k0);
    const HhConst hc = hh_const(nb);
    auto prow = [&](int r) -> int64_t {
      int64_t pr = f.perm[k0 + r];
      return pr < 0 || pr >= f.N ? 0 : pr;
    };
    for (int ch = 0; ch < nchunk; ++ch) {
      const int64_t j = (int64_t)ch * 128 + lane * 4;
      const bool jv = j < f.D;
      int cwi[4];
      float U[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int cs = jv ? f.col_sum_w[j + c] : 0;
        cwi[c] = cs - Cn * f.ow;
        U[c] = __fmaf_rn((float)Cn, zw, (float)cs);
      }
      // ---- pass 1: S = sum_k I_k, I = P + m CWc ----
      long long S[4] = {0, 0, 0, 0};
      for (int r0 = warp; r0 < nb; r0 += NW * kBigBatch) {
        float4 P[kBigBatch];
        long long m[kBigBatch];
#pragma unroll
        for (int b = 0; b < kBigBatch; ++b) {
          const int r = r0 + b * NW;
          const bool v = r < nb && jv;
          m[b] = v ? __float2ll_rn(rintf(two_sum((float)f.og, f.zero[k0 + r]).h)) : 0;
          P[b] = v ? *reinterpret_cast<const float4 *>(f.out + prow(r) * f.D + j)
                   : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int b = 0; b < kBigBatch; ++b) {
          S[0] += (long long)__float2int_rn(P[b].x) + m[b] * cwi[0];
          S[1] += (long long)__float2int_rn(P[b].y) + m[b] * cwi[1];
          S[2] += (long long)__float2int_rn(P[b].z) + m[b] * cwi[2];
          S[3] += (long long)__float2int_rn(P[b].w) + m[b] * cwi[3];
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) s_part[warp][lane * 4 + c] = S[c];
      // the lead row's integer parts (row 0 of the group)
      long long Ipl[4] = {0, 0, 0, 0};
      if (jv) {
        const long long m0 = __float2ll_rn(rintf(two_sum((float)f.og, f.zero[k0]).h));
        const float4 P0 = *reinterpret_cast<const float4 *>(f.out + prow(0) * f.D + j);
        Ipl[0] = (long long)__float2int_rn(P0.x) + m0 * cwi[0];
        Ipl[1] = (long long)__float2int_rn(P0.y) + m0 * cwi[1];
        Ipl[2] = (long long)__float2int_rn(P0.z) + m0 * cwi[2];
        Ipl[3] = (long long)__float2int_rn(P0.w) + m0 * cwi[3];
      }
      __syncthreads();
      ff rS[4], beta[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        long long tot = 0;
        for (int w = 0; w < NW; ++w) tot += s_part[w][lane * 4 + c];
        rS[c] = ff_mul(hc.rho, ff_from_int(tot));
        beta[c] = ff_mul(hc.kap, ff_add(rS[c], ff_neg(ff_from_int(Ipl[c]))));
      }
      // every warp has read the lead row and the sums before any row is
      // overwritten, and before the next chunk reuses s_part
      __syncthreads();
      // ---- pass 2: offsets and the inverse reflection ----
      for (int r0 = warp; r0 < nb; r0 += NW * kBigBatch) {
        float4 P[kBigBatch];
        int64_t pr[kBigBatch];
#pragma unroll
        for (int b = 0; b < kBigBatch; ++b) {
          const int r = r0 + b * NW;
          const bool v = r < nb && jv;
          pr[b] = v ? prow(r) : 0;
          P[b] = v ? *reinterpret_cast<const float4 *>(f.out + pr[b] * f.D + j)
                   : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int b = 0; b < kBigBatch; ++b) {
          const int r = r0 + b * NW;
          if (r >= nb || !jv) continue;
          const RowTerms t = row_terms(f, k0 + r, inv_sw, true);
          const long long m = __float2ll_rn(t.m);
          const float pv[4] = {P[b].x, P[b].y, P[b].z, P[b].w};
          float o4[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const ff I = ff_from_int((long long)__float2int_rn(pv[c]) + m * cwi[c]);
            ff v = r == 0 ? rS[c] : ff_add(I, ff_neg(beta[c]));
            v = ff_add(v, two_prod(t.hd, U[c]));
            v = ff_add(v, ff_mul({t.hR, 0.0f}, y));
            o4[c] = __fmul_rn(t.sc, ff_round(v));
          }
          __stcs(reinterpret_cast<float4 *>(f.out + pr[b] * f.D + j),
                 make_float4(o4[0], o4[1], o4[2], o4[3]));
        }
      }
    }
  }
}

// Groups of 2 .. 32 rows in the fp32 form: lane r loads the per-row terms
// of row r once; the rows' products are read 8 at a time (independent
// loads) and, for groups of up to 8 rows, kept in registers for the
// second pass.  Most groups have two to four rows: steps past the last are
// left out for the whole warp instead of lane by lane (49292 of 131072 rows
// of 576, 227 MB read and written: 97 -> 90 us; bound by the chain of each
// chunk, load, sums, store).
constexpr int kFixBatch = 8;

__device__ __forceinline__ float4 ld_row4(const FixArgs &f, int pr, int64_t j, bool jv) {
  return jv ? *reinterpret_cast<const float4 *>(f.out + (int64_t)pr * f.D + j)
            : make_float4(0.f, 0.f, 0.f, 0.f);
}

__global__ void __launch_bounds__(256, 4) k_grp_fix(const FixArgs f) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int nchunk = (int)((f.D + 127) / 128);
  const int64_t nunits = (int64_t)*f.count;
  const float inv_sw = *f.inv_sw, zw = *f.zero_w;
  const ff y = two_sum((float)f.ow, zw);
  const int Cn = f.C;
  for (int64_t u = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < nunits;
       u += nw) {
    const int64_t gi = f.list[u];
    if (gi < 0 || gi >= f.N) {
      if (lane == 0) record_status(f.status, FQT_EINVAL);
      continue;
    }
    const int64_t k0 = f.gstart[gi];
    int64_t k1 = f.gstart[gi + 1];
    if (k1 > f.N) k1 = f.N;
    if (k0 < 0 || k1 <= k0) continue;
    const int nb = (int)(k1 - k0);
    // ---- per-row terms, lane r for row r (groups of up to 32 rows) ----
    bool fast = nb >= 2 && nb <= 32 && f.small_p;
    float4 kq = make_float4(0.f, 0.f, 0.f, 0.f);
    int pr = 0;
    if (fast) {
      const float mmax = f.mmax_nb[nb];
      bool ok = true;
      if (lane < nb) {
        const RowTerms t = row_terms(f, k0 + lane, inv_sw, true);
        kq = make_float4(t.sc, __fmul_rn(t.sc, t.hd),
                         __fmul_rn(t.sc, __fmaf_rn(t.hR, y.h, __fmul_rn(t.hR, y.l))), t.m);
        ok = fabsf(t.m) <= mmax;
        const int p = f.perm[k0 + lane];
        pr = p < 0 || p >= f.N ? 0 : p;
      }
      fast = __all_sync(0xffffffffu, ok);
    }
    int msum = (int)kq.w;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) msum += __shfl_xor_sync(0xffffffffu, msum, off);
    const float mp = __shfl_sync(0xffffffffu, kq.w, 0);
    const HhConst hc = hh_const(nb >= 2 ? nb : 2);
    for (int ch = 0; ch < nchunk; ++ch) {
      const int64_t j = (int64_t)ch * 128 + lane * 4;
      const bool jv = j < f.D;
      float cwc[4], U[4];
      int cwi[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int cs = jv ? f.col_sum_w[j + c] : 0;
        cwc[c] = (float)(cs - Cn * f.ow);
        cwi[c] = (int)cwc[c];
        U[c] = __fmaf_rn((float)Cn, zw, (float)cs);
      }
      if (!fast) {
        fix_group_general(f, k0, nb, j, jv, cwc, cwi, U, inv_sw, y, 0);
        continue;
      }
      // ---- pass 1: block sums S = sum P + CWc sum m, lead I_p ----
      uint32_t sb[4] = {0u, 0u, 0u, 0u};
      float4 Pb[kFixBatch];
      float4 P0 = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int r0 = 0; r0 < nb; r0 += kFixBatch) {
#pragma unroll
        for (int b = 0; b < kFixBatch; ++b) {
          if (r0 + b >= nb) break;
          Pb[b] = ld_row4(f, __shfl_sync(0xffffffffu, pr, (r0 + b) & 31), j, jv);
        }
#pragma unroll
        for (int b = 0; b < kFixBatch; ++b) {
          if (r0 + b >= nb) break;
          sb[0] += magic_bits(Pb[b].x);
          sb[1] += magic_bits(Pb[b].y);
          sb[2] += magic_bits(Pb[b].z);
          sb[3] += magic_bits(Pb[b].w);
        }
        if (r0 == 0) P0 = Pb[0];
      }
      const float p0[4] = {P0.x, P0.y, P0.z, P0.w};
      BlockFixF bf[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int S = (int)(sb[c] - (uint32_t)nb * kMagicBits) + cwi[c] * msum;
        bf[c] = block_fix_f(hc, S, magic_int(p0[c]) + (int)mp * cwi[c]);
      }
      // ---- pass 2: offsets and the inverse reflection ----
      for (int r0 = 0; r0 < nb; r0 += kFixBatch) {
        if (nb > kFixBatch) {
#pragma unroll
          for (int b = 0; b < kFixBatch; ++b) {
            const int prb = __shfl_sync(0xffffffffu, pr, (r0 + b) & 31);
            Pb[b] = r0 + b < nb ? ld_row4(f, prb, j, jv) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
        }
#pragma unroll
        for (int b = 0; b < kFixBatch; ++b) {
          const int r = r0 + b;
          if (r >= nb) break;
          const int src = r & 31;
          const float4 q = make_float4(__shfl_sync(0xffffffffu, kq.x, src),
                                       __shfl_sync(0xffffffffu, kq.y, src),
                                       __shfl_sync(0xffffffffu, kq.z, src),
                                       __shfl_sync(0xffffffffu, kq.w, src));
          const int prb = __shfl_sync(0xffffffffu, pr, src);
          if (!jv) continue;
          const float pv[4] = {Pb[b].x, Pb[b].y, Pb[b].z, Pb[b].w};
          float o4[4];
#pragma unroll
          for (int c = 0; c < 4; ++c)
            o4[c] = r == 0 ? dequant(q, bf[c].lead, U[c])
                           : dequant(q, reflect_f(pv[c], q, cwc[c], bf[c]), U[c]);
          __stcs(reinterpret_cast<float4 *>(f.out + (int64_t)prb * f.D + j),
                 make_float4(o4[0], o4[1], o4[2], o4[3]));
        }
      }
    }
  }
}

fqt_status linear_backward(const fqt_qtensor *q_b2, const fqt_qtensor *q_b1,
                           const fqt_qtensor *qx, const fqt_qtensor *qw,
                           float *grad_X, float *grad_W, void *ws,
                           size_t ws_bytes, cudaStream_t st) {
  if (!grad_X && !grad_W) return FQT_OK;
  if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u)) return FQT_EWORKSPACE;
  int *status = reinterpret_cast<int *>(ws);
  const int nsm = device_sm_count();
  if (grad_X) {
    if (!q_b2 || !qw || !q_b2->codes_f16 || !qw->codes_f16 || !qw->col_sum ||
        !q_b2->inv_s || !q_b2->zero || !qw->inv_s || !qw->zero)
      return FQT_EINVAL;
    // BHQ with block 0: the adaptive groups of App. D.5 (NB = 0 kernels)
    const bool adapt = q_b2->kind == FQT_BHQ && q_b2->block == 0;
    const int nb = adapt ? 0 : (q_b2->kind == FQT_BHQ && q_b2->block > 1 ? q_b2->block : 1);
    if (nb > 1 && (!q_b2->lead || !q_b2->hz || !q_b2->hr)) return FQT_EINVAL;
    if (nb <= 1 && !q_b2->row_sum) return FQT_EINVAL;
    if (adapt && (!q_b2->perm || !q_b2->gstart || !q_b2->gsize || !q_b2->hz || !q_b2->hr))
      return FQT_EINVAL;
    if (nb > 128 || (nb & (nb - 1))) return FQT_EINVAL;
    const int64_t Nr = q_b2->rows, C = q_b2->cols, D = qw->cols;
    if (qw->rows != C || qw->kind != FQT_PTQ) return FQT_EINVAL;
    if (C % 16 || D % 16) return FQT_EUNSUPPORTED;
    if (C > 8192) return FQT_EUNSUPPORTED;  // int32 epilogue bound
    if (!aligned16(q_b2->codes_f16) || !aligned16(qw->codes_f16) || !aligned16(grad_X))
      return FQT_EINVAL;
    if (Nr > 0) {
      // transposed: M = D (columns of W~), N = rows of dH, K = C
      const SplitPlan p = plan_splits(D, Nr, C, qw->bits, q_b2->bits, nsm, false);
      // fp32 form of the integer parts I = P + m CWc: one exact chunk,
      // |P| < 2^22 and |I| (2 + sqrt(nb)) < 2^24 (|I| < 2^24 without
      // reflection) for every row offset |m| <= mmax, with
      // |I| <= C 2^(bw-1) (2^(b-1) + |m|)
      // Without reflection (nb = 1) and with P exact (one chunk), fma(m,
      // CWc, P) is the correctly rounded exact I for every row offset: the
      // value the integer forms round to, so the fp32 form holds for all m.
      const int64_t kc_terms = (int64_t)exact_chunk_blocks(qw->bits, q_b2->bits) * BK;
      const double lim = nb <= 1 ? 16777216.0 : 16777216.0 / (2.0 + sqrt((double)nb));
      const double mmax = nb == 1 ? 1e30
                                  : floor(lim / ((double)C * (double)(1 << (qw->bits - 1)))) -
                                        (double)(1 << (q_b2->bits - 1)) - 1.0;
      const int64_t pmax = C << (qw->bits + q_b2->bits - 2);
      // the block sums of the reflection read |P| < 2^22 off the fp32 bits
      const bool flt = C <= kc_terms && mmax >= 0.0 && (nb <= 1 || pmax < ((int64_t)1 << 22));
      // the adaptive groups need the fp32 form (rows are scattered by perm)
      if (adapt && !flt) return FQT_EUNSUPPORTED;
      const size_t list_bytes = group_list_bytes(Nr);
      if (adapt && ws_bytes < kGemmOffset + list_bytes) return FQT_EWORKSPACE;
      GemmArgs g;
      memset(&g, 0, sizeof(g));
      g.status = status;
      g.kind = q_b2->kind;
      g.og = 1 << (q_b2->bits - 1);
      g.ow = 1 << (qw->bits - 1);
      g.inv_s = q_b2->inv_s;
      g.zero = q_b2->zero;
      g.row_sum = q_b2->row_sum;
      g.lead = q_b2->lead;
      g.hz = q_b2->hz;
      g.hr = q_b2->hr;
      g.flt_mmax = flt ? (float)mmax : -1.0f;
      g.i32_mmax = int32_form_mmax(C, qw->bits, q_b2->bits, nb);
      g.col_sum_w = qw->col_sum;
      g.inv_sw = qw->inv_s;
      g.zero_w = qw->zero;
      g.perm = q_b2->perm;
      g.gsize = q_b2->gsize;
      g.raw_mmax = (float)mmax;
      const SplitPlan pp = plan_splits(D, Nr, C, qw->bits, q_b2->bits, nsm, false, true);
      const int form = adapt ? 2 : epilogue_form(flt, mmax, q_b2->bits);
      const bool pair = C <= kc_terms && gemm_pair_kernel(MODE_GRADX, nb, form) &&
                        pair_faster(p, pp, nsm, form == 2 ? 4 : 8);
      fqt_status s = run_gemm(qw->codes_f16, 0, qw->bits, q_b2->codes_f16, 1, q_b2->bits,
                              D, Nr, C, pair ? pp : p, g, grad_X, MODE_GRADX, nb, form, st, pair);
      if (s != FQT_OK) return s;
      if (adapt) {
        FixArgs f;
        memset(&f, 0, sizeof(f));
        f.out = grad_X;
        f.N = Nr;
        f.D = D;
        f.C = (int)C;
        f.og = g.og;
        f.ow = g.ow;
        f.bw = qw->bits;
        f.b2 = q_b2->bits;
        f.inv_s = q_b2->inv_s;
        f.zero = q_b2->zero;
        f.hz = q_b2->hz;
        f.hr = q_b2->hr;
        f.row_sum = q_b2->row_sum;
        f.perm = q_b2->perm;
        f.gstart = q_b2->gstart;
        f.inv_sw = qw->inv_s;
        f.zero_w = qw->zero;
        f.col_sum_w = qw->col_sum;
        f.raw_mmax = (float)mmax;
        f.small_p = pmax < ((int64_t)1 << 22);
        for (int n = 2; n <= 32; ++n) {
          const double l = 16777216.0 / (2.0 + sqrt((double)n));
          f.mmax_nb[n] = (float)(floor(l / ((double)C * (double)(1 << (qw->bits - 1)))) -
                                 (double)(1 << (q_b2->bits - 1)) - 1.0);
        }
        char *lw = static_cast<char *>(ws) + kGemmOffset;
        f.count = reinterpret_cast<int *>(lw);
        f.count_big = reinterpret_cast<int *>(lw + 4);
        f.list = reinterpret_cast<int32_t *>(lw + 256);
        f.list_big = reinterpret_cast<int32_t *>(lw + 256 + (((size_t)Nr * 4 + 255) & ~(size_t)255));
        f.status = status;
        cudaError_t e = cudaMemsetAsync(f.count, 0, 2 * sizeof(int), st);
        if (e != cudaSuccess) return cuda_fail(e, "group list clear");
        k_grp_list<<<(int)((Nr + 255) / 256), 256, 0, st>>>(f);
        k_grp_fix_big<<<nsm * 2, kBigFixWarps * 32, 0, st>>>(f);
        k_grp_fix<<<nsm * 8, 256, 0, st>>>(f);
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "group fix-up launch");
      }
    }
  }
  if (grad_W) {
    const fqt_qtensor *qa = q_b1 ? q_b1 : q_b2;
    // the shift quantizer feeds grad_W itself: its codes on the common scale
    const bool shifted = qa && qa->kind == FQT_SHIFT;
    // byte operands: both code sets given as bytes only (no fp16 carriers);
    // the split-K kernel widens them on chip
    const bool bytes = qa && qx && !shifted && !qa->codes_f16 && !qx->codes_f16 && qa->codes &&
                       qx->codes && qx->conv[0] == 0;
    if (!qa || !qx || (!qx->codes_f16 && !bytes) || !qx->col_sum || !qx->inv_s || !qx->zero)
      return FQT_EINVAL;
    if (shifted ? (!qa->shift_f16 || !qa->shift_col_sum || !qa->shift_scale)
                : ((!qa->codes_f16 && !bytes) || !qa->col_sum || !qa->inv_s || !qa->zero))
      return FQT_EINVAL;
    if ((!shifted && qa->kind != FQT_PTQ) || qx->kind != FQT_PTQ) return FQT_EINVAL;
    const void *A16 = bytes ? (const void *)qa->codes
                            : shifted ? (const void *)qa->shift_f16 : (const void *)qa->codes_f16;
    const void *X16 = bytes ? (const void *)qx->codes : (const void *)qx->codes_f16;
    // |shifted code| <= 16 (2^(b-1) - 1) < 2^(b+3): b + 4 bits of centred magnitude
    const int a_bits = shifted ? qa->bits + 4 : qa->bits;
    // an implicit im2col operand (its padding is corrected in the reduction)
    const bool conv = qx->conv[0] > 0;
    const int x_bits = qx->bits;
    const int64_t Nr = qa->rows, C = qa->cols, D = qx->cols;
    if (qx->rows != Nr) return FQT_EINVAL;
    if (C % 16 || D % 16) return FQT_EUNSUPPORTED;
    if (!aligned16(A16) || !aligned16(X16)) return FQT_EINVAL;
    if (conv) {
      const int32_t *g = qx->conv;
      const int64_t oh = (int64_t)g[1] + 2 * g[6] - g[4] + 1, ow = (int64_t)g[2] + 2 * g[6] - g[5] + 1;
      if (oh <= 0 || ow <= 0 || (int64_t)g[0] * oh * ow != Nr || (int64_t)g[4] * g[5] * g[3] != D)
        return FQT_EINVAL;
      // 64-channel boxes; rows of up to 64 pixels (the tile kernel) or of a
      // multiple of 32 (k_gradw)
      if (g[3] % 64 || (ow > 64 && ow % kWBK)) return FQT_EUNSUPPORTED;
      if (padsum_group((int)C, g[6]) == 0) return FQT_EUNSUPPORTED;
    }
    // An implicit im2col operand with output rows of at most 64 pixels takes
    // the split-K tile kernel too: K blocks of 64 slots are rpb = 64 / pw
    // whole output rows of pw (the power of two >= ow) slots, the slots past
    // ow and the rows past oh zero in Q_b1 (out of its bounds), so K runs over
    // n ceil(oh / rpb) 64 slots.
    int cpw = 0, crpb = 0, cybi = 0;
    int64_t Kt = Nr;
    if (conv) {
      const int32_t *g = qx->conv;
      const int ow = g[2] + 2 * g[6] - g[5] + 1, oh = g[1] + 2 * g[6] - g[4] + 1;
      if (ow <= 64 && !bytes) {
        cpw = 8;
        while (cpw < ow) cpw *= 2;
        crpb = 64 / cpw;
        cybi = (oh + crpb - 1) / crpb;
        Kt = (int64_t)g[0] * cybi * 64;
      }
    }
    const bool conv_tile = cpw > 0;
    SplitPlan p = plan_splits(C, D, Kt, a_bits, x_bits, nsm, true);
    // gemm_workspace_bytes counts the splits of N rows and of 2.5 N slots: tiny
    // images, which pad far beyond, and plans in between that round to more
    // splits than either (675 pixels in 960 slots: 15 against 14) take the
    // splits that fit
    const int64_t pad_bytes = conv ? C * qx->conv[4] * qx->conv[5] * 4 : 0;
    if (conv_tile &&
        (2 * Kt > 5 * Nr ||
         (int64_t)kGemmOffset + p.splits * C * D * 4 + pad_bytes > (int64_t)ws_bytes)) {
      const int64_t fit = plan_splits(C, D, (Nr * 5 + 1) / 2, a_bits, 8, nsm, true).splits;
      if (p.splits > fit) {
        p.ks_blocks = (p.kb_total + fit - 1) / fit;
        p.splits = (int)((p.kb_total + p.ks_blocks - 1) / p.ks_blocks);
      }
    }
    const WPlan wp = Nr > 0 ? gradw_plan(Nr, C, D, a_bits, x_bits, nsm) : WPlan{};
    // k_gradw serves the implicit im2col operand with wider output rows (4-D
    // boxes of 32 pixels of one row, ow % 32 == 0); plain matrices take the
    // split-K tile kernel, which measured faster wherever both apply (e.g.
    // 66.7 against 110.8 us on a 200704 x 128 x 512 layer) and widens byte
    // operands
    const bool w_ok = use_gradw(wp, nsm) && conv && !conv_tile;
    if (conv && Nr > 0 && !w_ok && !conv_tile) return FQT_EUNSUPPORTED;
    // CTA pairs where their plan is faster and its partials fit the workspace
    bool pair = false;
    if (Nr > 0 && !w_ok && !bytes && C > BM) {
      const SplitPlan pp = plan_splits(C, D, Kt, a_bits, x_bits, nsm, true, true);
      pair = pair_faster_w(p, pp, C, D, nsm) &&
             (int64_t)kGemmOffset + pp.splits * C * D * 4 + pad_bytes <= (int64_t)ws_bytes;
      if (pair) p = pp;
    }
    // At most one tile of rows: wide tiles, where their plan is ahead by 10%
    // and its partials fit; an implicit im2col operand of kw = 2 to 4 taps a
    // row then reads its pixels once per kernel row.  An explicit operand gains
    // nothing at 64 x 576 over 131072 rows (41 and 42 us with the reduction): its
    // time is counted as at least that of reading it, which keeps such shapes
    // here.  (That is not what they wait for: 168 MB at 60% of the DRAM peak, the
    // tensor pipe at 25%, each CTA's chain of 69 K blocks at 0.5 us.)
    int wide = 0, row_taps = 0;
    if (Nr > 0 && !w_ok && !bytes && C <= BM && D > BN) {
      SplitPlan wp;
      int wn;
      row_taps = conv && qx->conv[5] >= 2 && qx->conv[5] <= 4 ? qx->conv[5] : 0;
      double t = wide_plan(C, D, Kt, a_bits, x_bits, nsm, 64 * row_taps, &wp, &wn);
      double ts = single_time(p, C, D, nsm);
      if (!conv) {
        const double mem = (double)Kt * (double)(C + D) * 2.0 / 6500.0;
        t = std::max(t, mem + 8000.0);
        ts = std::max(ts, mem + 5000.0);
      }
      if (t < 0.9 * ts &&
          (int64_t)kGemmOffset + wp.splits * C * D * 4 + pad_bytes <= (int64_t)ws_bytes) {
        wide = wn;
        p = wp;
      }
    }
    // one split: the epilogue dequantizes, no partials and no reduction
    const bool fuse = (pair || wide) && p.splits == 1 && !conv && aligned16(grad_W);
    const int splits = w_ok ? wp.splits : p.splits;
    const size_t pbytes = (size_t)splits * (size_t)C * (size_t)D * 4;
    const int taps = conv ? qx->conv[4] * qx->conv[5] : 0;
    const size_t need = kGemmOffset + pbytes + (conv ? (size_t)C * taps * 4 : 0);
    if (ws_bytes < need) return FQT_EWORKSPACE;
    int32_t *part = reinterpret_cast<int32_t *>(static_cast<char *>(ws) + kGemmOffset);
    int32_t *pad_a = reinterpret_cast<int32_t *>(static_cast<char *>(ws) + kGemmOffset + pbytes);
    if (conv && Nr > 0) {
      const int32_t *g = qx->conv;
      const int oh = g[1] + 2 * g[6] - g[4] + 1, ow = g[2] + 2 * g[6] - g[5] + 1;
      cudaError_t e = cudaMemsetAsync(pad_a, 0, (size_t)C * taps * 4, st);
      if (e != cudaSuccess) return cuda_fail(e, "padding sums clear");
      const int grp = padsum_group((int)C, g[6]);
      if (conv_lines_supported(oh, ow, (int)C, g[4], g[5], g[6])) {
        const fqt_status ls = launch_conv_lines(static_cast<const uint16_t *>(A16), g[0], oh, ow,
                                                (int)C, pad_a, nullptr, 0, st);
        if (ls != FQT_OK) return ls;
      } else if (g[6] > 0) {  // without padding no tap reads any
        // about 16 loads per thread: runs of images whose border pixels
        // (bounded by the pad rows and columns) fill a CTA
        const int pd = g[6];
        const int64_t border = (int64_t)std::min(oh, 2 * pd) * ow +
                               (int64_t)std::max(0, oh - 2 * pd) * std::min(ow, 2 * pd);
        const int64_t items = std::max<int64_t>(1, border * (grp / 8));
        const int64_t per = std::max<int64_t>(1, (256 * 16) / items);
        const int ipc = (int)std::min<int64_t>(per, g[0]);
        const dim3 grid((unsigned)((g[0] + ipc - 1) / ipc), (unsigned)((C + grp - 1) / grp));
        const int ncls = (2 * pd + 1) * (2 * pd + 1);
        k_conv_padsum<<<grid, 256, sizeof(int) * (size_t)ncls * grp, st>>>(
            static_cast<const uint16_t *>(A16), (int)C, grp, g[0], ipc, g[1], g[2], g[5], pd, oh,
            ow, taps, pad_a);
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "padding sums launch");
      }
    }
    ReduceArgs r;
    memset(&r, 0, sizeof(r));
    r.part = part;
    r.splits = Nr > 0 ? splits : 1;
    r.M = C;
    r.N = D;
    r.out_f32 = grad_W;
    r.Kn = Nr;
    // shifted codes are their own carriers (offset 0, zero point 0)
    r.oa = shifted ? 0 : 1 << (qa->bits - 1);
    r.ob = 1 << (qx->bits - 1);
    r.cs_a = shifted ? qa->shift_col_sum : qa->col_sum;
    r.cs_b = qx->col_sum;
    if (conv) {
      r.pad_a = pad_a;
      r.code_zero = qx->col_sum + D;
      r.taps = taps;
      r.cin = qx->conv[3];
    }
    r.inv_a = shifted ? qa->shift_scale : qa->inv_s;
    r.zero_a = shifted ? qa->shift_scale + 1 : qa->zero;
    r.inv_b = qx->inv_s;
    r.zero_b = qx->zero;
    if (Nr > 0 && w_ok) {
      fqt_status s = run_gradw(qx->codes_f16, static_cast<const uint16_t *>(A16), Nr, (int)C,
                               (int)D, wp, part, status, st, conv ? qx->conv : nullptr);
      if (s != FQT_OK) return s;
    } else if (Nr > 0) {
      GemmArgs g;
      memset(&g, 0, sizeof(g));
      g.status = status;
      g.u8 = bytes ? 1 : 0;
      if (conv_tile) {
        const int32_t *cv = qx->conv;
        g.conv = 1;
        g.taps = wide ? row_taps : 0;
        g.cpw = cpw;
        g.crpb = crpb;
        g.cybi = cybi;
        g.cnimg = cv[0];
        g.cih = cv[1];
        g.ciw = cv[2];
        g.cin = cv[3];
        g.ckw = cv[5];
        g.cpad = cv[6];
        g.coh = cv[1] + 2 * cv[6] - cv[4] + 1;
        g.cow = cv[2] + 2 * cv[6] - cv[5] + 1;
      }
      g.fuse = fuse ? 1 : 0;
      g.red = r;
      fqt_status s = run_gemm(A16, 0, a_bits, X16, 0, qx->bits, C, D, Kt, p, g,
                              fuse ? (void *)grad_W : (void *)part, MODE_PARTIAL, 1, 0, st, pair, wide);
      if (s != FQT_OK) return s;
      if (fuse) return FQT_OK;
    } else {
      const cudaError_t e = cudaMemsetAsync(part, 0, (size_t)C * D * 4, st);
      if (e != cudaSuccess) return cuda_fail(e, "partial clear");
    }
    launch_reduce(r, st);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "split-K reduce launch");
  }
  return FQT_OK;
}

// ---------------------------------------------------------------------------
// grad_W without a caller-provided workspace.
//
// Some callers cannot allocate device memory at the point where they need
// the backward: for example a serving or training loop whose memory budget
// is frozen after warm-up, or a plain C host that has no allocator of its
// own to hand (and must not call cudaMalloc, which can synchronise the
// device and stall other streams).  For them the split-K partials of grad_W
// live in a fixed array inside the library.  Every GPU that loads the
// library holds it until the process exits; all calls on a device share it.
// ---------------------------------------------------------------------------
constexpr size_t kFixedPartialBytes = (size_t)8 << 20;  // 8 MiB of int32 partials
static __device__ __align__(256) unsigned char
    g_fixed_scratch[kHeaderBytes + kFixedPartialBytes];

// Device address of g_fixed_scratch on the current device, looked up once
// per device (the host-side symbol is only a stand-in for it).
static fqt_status fixed_scratch_address(void **out) {
  static void *addr[64] = {nullptr};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "get device");
  if (dev < 0 || dev >= 64) return FQT_EUNSUPPORTED;
  if (!addr[dev]) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_fixed_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "fixed scratch address");
    addr[dev] = p;
  }
  *out = addr[dev];
  return FQT_OK;
}

fqt_status grad_w_fixed_scratch(const fqt_qtensor *qa, const fqt_qtensor *qx,
                                float *grad_W, cudaStream_t st) {
  if (!grad_W || !qa || !qx || !qa->codes_f16 || !qx->codes_f16 || !qa->col_sum ||
      !qx->col_sum || !qa->inv_s || !qa->zero || !qx->inv_s || !qx->zero)
    return FQT_EINVAL;
  if (qa->kind != FQT_PTQ || qx->kind != FQT_PTQ) return FQT_EINVAL;
  // an implicit im2col operand stores NHWC codes, not the Nr x D matrix the
  // tile kernel below reads: refuse it before anything is enqueued
  if (qa->conv[0] > 0 || qx->conv[0] > 0) return FQT_EUNSUPPORTED;
  const int64_t Nr = qa->rows, C = qa->cols, D = qx->cols;
  if (qx->rows != Nr || Nr < 0) return FQT_EINVAL;
  if (C % 16 || D % 16) return FQT_EUNSUPPORTED;
  if (!aligned16(qa->codes_f16) || !aligned16(qx->codes_f16)) return FQT_EINVAL;
  // the partials of every split must fit the fixed array
  const size_t per_split = (size_t)C * (size_t)D * 4;
  if (per_split == 0 || per_split > kFixedPartialBytes) return FQT_EWORKSPACE;
  const int max_splits = (int)(kFixedPartialBytes / per_split);
  SplitPlan p = plan_splits(C, D, Nr, qa->bits, qx->bits, device_sm_count(), true);
  if (p.splits > max_splits) {
    // fewer, longer splits; each must stay within the int32 partial bound
    const int64_t max_terms = ((int64_t)1 << 31) >> (qa->bits + qx->bits - 2);
    p.ks_blocks = (p.kb_total + max_splits - 1) / max_splits;
    if (p.ks_blocks * BK > max_terms) return FQT_EWORKSPACE;
    p.splits = (int)((p.kb_total + p.ks_blocks - 1) / p.ks_blocks);
  }
  void *base = nullptr;
  fqt_status s = fixed_scratch_address(&base);
  if (s != FQT_OK) return s;
  // the status word keeps the first condition recorded since the last
  // fqt_fixed_scratch_sync_status (it is zero when the library loads); the
  // partials are fully rewritten by every split, so nothing else needs clearing
  int *status = static_cast<int *>(base);
  int32_t *part = reinterpret_cast<int32_t *>(static_cast<char *>(base) + kHeaderBytes);
  if (Nr == 0) {
    const cudaError_t e = cudaMemsetAsync(grad_W, 0, per_split, st);
    return cuda_fail(e, "grad_W clear");
  }
  GemmArgs g;
  memset(&g, 0, sizeof(g));
  g.status = status;
  s = run_gemm(qa->codes_f16, 0, qa->bits, qx->codes_f16, 0, qx->bits, C, D, Nr, p, g,
               part, MODE_PARTIAL, 1, false, st);
  if (s != FQT_OK) return s;
  ReduceArgs r;
  memset(&r, 0, sizeof(r));
  r.part = part;
  r.splits = p.splits;
  r.M = C;
  r.N = D;
  r.out_f32 = grad_W;
  r.Kn = Nr;
  r.oa = 1 << (qa->bits - 1);
  r.ob = 1 << (qx->bits - 1);
  r.cs_a = qa->col_sum;
  r.cs_b = qx->col_sum;
  r.inv_a = qa->inv_s;
  r.zero_a = qa->zero;
  r.inv_b = qx->inv_s;
  r.zero_b = qx->zero;
  launch_reduce(r, st);
  return cuda_fail(cudaGetLastError(), "split-K reduce launch");
}

// Status word of the fixed array (its first int): the device-side conditions
// of fqt_grad_w_fixed_scratch calls land there, as they land in a caller's
// workspace for the other calls.
fqt_status fixed_scratch_status(int **out) {
  void *base = nullptr;
  const fqt_status s = fixed_scratch_address(&base);
  if (s == FQT_OK) *out = static_cast<int *>(base);
  return s;
}

// ---------------------------------------------------------------------------
// A wait on an mbarrier that nothing arrives at, bounded by limit_ns: the
// same bounded wait the contraction kernels use, made to run out on purpose
// so that the timeout path (FQT_ETIMEOUT in the status word, the kernel
// returns, the context stays usable) can be checked.  No bulk copy or
// tensor-core operation is in flight.
// ---------------------------------------------------------------------------
__global__ void k_wait_nothing(int *status, uint64_t limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_wait_limit(&bar, 0, status, limit_ns);
}

fqt_status debug_wait_timeout(void *ws, size_t ws_bytes, uint64_t limit_ns,
                              cudaStream_t st) {
  if (limit_ns > 10000000000ull) return FQT_EINVAL;  // at most 10 s
  int *status = nullptr;
  if (ws) {
    if (ws_bytes < kHeaderBytes || ((uintptr_t)ws & 255)) return FQT_EWORKSPACE;
    status = static_cast<int *>(ws);
  } else {
    const fqt_status s = fixed_scratch_status(&status);
    if (s != FQT_OK) return s;
  }
  k_wait_nothing<<<1, 32, 0, st>>>(status, limit_ns);
  return cuda_fail(cudaGetLastError(), "wait test launch");
}

}  // namespace fqt

namespace fqt {

// ---------------------------------------------------------------------------
// Dense tensor-core rates of this GPU, the denominators of the contractions'
// rooflines (kind 0: tcgen05 kind::f16, fp16 x fp16 -> fp32; kind 1: tcgen05
// kind::f8f6f4, e4m3 x e4m3 -> fp32; kind 2: warp-level mma.sync m16n8k32
// u8 x s8 -> s32).  tcgen05 kind::i8 does not assemble for sm_103a.  One CTA
// per SM: one thread issues `iters` rounds of four back-to-back M128 N256
// MMAs (K 16 each for f16, 32 for e4m3, i.e. one 128-byte row of operands)
// into one TMEM accumulator, then waits (bounded) for them to drain.
// Operands are zero: the rates do not depend on the values.
// ---------------------------------------------------------------------------
constexpr int kPeakN = 256;

__device__ __forceinline__ void umma_f8(uint32_t tmem_d, uint64_t a_desc, uint64_t b_desc,
                                        uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__global__ void __launch_bounds__(128, 1) k_peak_umma(int kind, int64_t iters, int *status) {
  extern __shared__ __align__(1024) uint8_t peak_raw[];
  uint8_t *ops = peak_raw + ((1024u - (smem_u32(peak_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tslot;
  const int warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < (int)(kTileBytes + 2 * kTileBytes) / 16; i += blockDim.x)
    reinterpret_cast<uint4 *>(ops)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_barrier_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tslot)),
                 "r"((uint32_t)kPeakN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tslot;
  if (threadIdx.x == 0) {
    // A: 128 rows x 128 bytes, B: 256 rows x 128 bytes, K-major, 128-byte swizzle
    const uint64_t da = sw128_desc(smem_u32(ops));
    const uint64_t db = sw128_desc(smem_u32(ops + kTileBytes));
    // D fp32; A, B fp16 (kind::f16) or e4m3 (kind::f8f6f4, format 0); K-major
    const uint32_t idesc =
        (1u << 4) | ((uint32_t)(kPeakN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
    for (int64_t it = 0; it < iters; ++it) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (kind == 0)
          umma_f16(tmem, da + 2 * k, db + 2 * k, idesc, (it | k) ? 1u : 0u);
        else
          umma_f8(tmem, da + 2 * k, db + 2 * k, idesc, (it | k) ? 1u : 0u);
      }
    }
    umma_commit(&bar);
    mbar_wait(&bar, 0, status);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)kPeakN)
                 : "memory");
  }
}

// mma.sync u8 x s8 -> s32 (m16n8k32): eight independent accumulators per warp
__global__ void __launch_bounds__(256) k_peak_imma(int64_t iters, int *sink) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t a0 = 0x01010101u * (lane & 7), a1 = a0 ^ 0x02020202u, a2 = a0 ^ 0x04040404u,
                 a3 = a0 ^ 0x08080808u, b0 = 0x03030303u, b1 = 0x05050505u;
  int acc[8][4];
#pragma unroll
  for (int c = 0; c < 8; ++c)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[c][i] = 0;
  for (int64_t it = 0; it < iters; ++it) {
#pragma unroll
    for (int c = 0; c < 8; ++c)
      asm volatile(
          "mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
          "{%8, %9}, {%0, %1, %2, %3};"
          : "+r"(acc[c][0]), "+r"(acc[c][1]), "+r"(acc[c][2]), "+r"(acc[c][3])
          : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  }
  int s = 0;
#pragma unroll
  for (int c = 0; c < 8; ++c) s += acc[c][0] + acc[c][1] + acc[c][2] + acc[c][3];
  if (s == 0x7fffffff) *sink = s;  // keeps the accumulators live
}

fqt_status debug_mma_peak(int kind, int64_t iters, double *ops_out, void *ws, size_t ws_bytes,
                          cudaStream_t st) {
  if (kind < 0 || kind > 2 || iters <= 0 || iters > ((int64_t)1 << 32) || !ops_out)
    return FQT_EINVAL;
  if (!ws || ws_bytes < kHeaderBytes || ((uintptr_t)ws & 255)) return FQT_EWORKSPACE;
  int *status = static_cast<int *>(ws);
  const int nsm = device_sm_count();
  if (kind <= 1) {
    const size_t smem = 3 * kTileBytes + 1024;
    cudaError_t e = cudaFuncSetAttribute(k_peak_umma, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "peak attribute");
    k_peak_umma<<<nsm, 128, smem, st>>>(kind, iters, status);
    const double k_per = kind == 0 ? 16.0 : 32.0;
    *ops_out = 2.0 * BM * kPeakN * k_per * 4.0 * (double)iters * nsm;
  } else {
    const int ctas = nsm * 4;
    k_peak_imma<<<ctas, 256, 0, st>>>(iters, status + 1);
    *ops_out = 2.0 * 16 * 8 * 32 * 8.0 * (double)iters * ctas * 8;
  }
  return cuda_fail(cudaGetLastError(), "peak launch");
}

}  // namespace fqt

namespace fqt {

}  // namespace fqt
