// fqt_codes.cu -- the gradient quantizers as a statistics pass and a code pass
// over dH (Sec. 3.3, 4.1, 4.2, App. D.4), with Q_b1 (App. E) in the code pass:
//   PTQ       k_range (fqt_quant.cu), k_codes
//   PSQ       k_row_stats (a row per sample), k_codes
//   PSQ with a sample per image: k_sample_part, k_sample_finish, k_codes
//   BHQ, fixed blocks of 4, 8 or 16 rows: k_bhq_stats, k_codes; of 32, 64 or
//             128 rows: k_bhq_stats_big, k_codes (grad_X's offsets: k_codes
//             where its units hold whole blocks, else k_bhq_offsets in
//             fqt_quant.cu)
// Rows may have any multiple of 8 columns up to kCodesMaxCols (BHQ: 4096).
//
// Stochastic rounding runs on the fp32 pipe (two entries per instruction up to
// v): with U = 128 + u 2^-16 (u the 16-bit uniform, exact in fp32),
// floor(v + u 2^-16) = floor(rd(v + U)) - 128 because rounding down never
// crosses an integer, and a second round-down addition of 2^23 + 0x6400 - 128
// leaves 0x4B006400 + code in the bits: code = floor(v + u 2^-16) =
// (floor(v 2^16) + u) >> 16, the rule of sr_code16.  The low half of those
// bits is the fp16 number 1024 + code, so one byte permutation packs two
// codes, one packed minimum caps them at B (v exceeds B by rounding at most)
// and one packed subtraction makes them carriers; column and row sums add the
// packed codes as two 16-bit lanes.
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>
#include <string.h>
#include <algorithm>

#include "fqt_common.cuh"
#include "fqt_internal.h"

namespace fqt {

// ---------------------------------------------------------------------------
// Minima and maxima
// ---------------------------------------------------------------------------
// minimum / maximum that hand on a NaN
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float min3_nan(float a, float b, float c) {
  float r;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
struct MinNan {
  __device__ float operator()(float a, float b) const { return min_nan(a, b); }
};
struct MaxNan {
  __device__ float operator()(float a, float b) const { return max_nan(a, b); }
};

// ---------------------------------------------------------------------------
// Eight consecutive entries (an oct), kept as loaded
// ---------------------------------------------------------------------------
template <typename T>
struct Oct;

template <>
struct Oct<float> {
  float v[8];
  __device__ __forceinline__ void load(const float *p) {
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    const float4 b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = 0.0f;
  }
  __device__ __forceinline__ f32x2 pair(int i) const { return pack2(v[2 * i], v[2 * i + 1]); }
  __device__ __forceinline__ float min8() const {
    return min_nan(min3_nan(min3_nan(min3_nan(v[0], v[1], v[2]), v[3], v[4]), v[5], v[6]), v[7]);
  }
  __device__ __forceinline__ float max8() const {
    return max_nan(max3_nan(max3_nan(max3_nan(v[0], v[1], v[2]), v[3], v[4]), v[5], v[6]), v[7]);
  }
};

template <>
struct Oct<__nv_bfloat16> {
  uint32_t w[4];
  __device__ __forceinline__ void load(const __nv_bfloat16 *p) {
    const uint4 a = __ldg(reinterpret_cast<const uint4 *>(p));
    w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] = 0u;
  }
  __device__ __forceinline__ f32x2 pair(int i) const {
    return pack2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xFFFF0000u));
  }
  __device__ __forceinline__ float min8() const {
    uint32_t a, b, c;
    asm("min.NaN.bf16x2 %0, %1, %2;" : "=r"(a) : "r"(w[0]), "r"(w[1]));
    asm("min.NaN.bf16x2 %0, %1, %2;" : "=r"(b) : "r"(w[2]), "r"(w[3]));
    asm("min.NaN.bf16x2 %0, %1, %2;" : "=r"(c) : "r"(a), "r"(b));
    return min_nan(__uint_as_float(c << 16), __uint_as_float(c & 0xFFFF0000u));
  }
  __device__ __forceinline__ float max8() const {
    uint32_t a, b, c;
    asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(a) : "r"(w[0]), "r"(w[1]));
    asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(b) : "r"(w[2]), "r"(w[3]));
    asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(c) : "r"(a), "r"(b));
    return max_nan(__uint_as_float(c << 16), __uint_as_float(c & 0xFFFF0000u));
  }
};

// Reduces R rows (v[s] of row s in each of the row's L lanes, R <= L powers of
// two) by halving: a lane keeps half of the rows and hands the other half to
// its partner, so the whole takes 2 R - 1 + log2(L / R) shuffles instead of
// R log2 L.  The lane at place o of the L ends with row o / (L / R).
template <int R, int L, class Op>
__device__ __forceinline__ float reduce_rows(float (&v)[R], Op op) {
  const int lane = threadIdx.x & 31;
  int n = R;
#pragma unroll
  for (int off = L / 2; off >= 1; off /= 2) {
    if (n > 1) {
      n /= 2;
      const bool up = (lane & off) != 0;
#pragma unroll
      for (int i = 0; i < R / 2; ++i)
        if (i < n) {
          const float send = up ? v[i] : v[i + n];
          const float keep = up ? v[i + n] : v[i];
          v[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, off));
        }
    } else {
      v[0] = op(v[0], __shfl_xor_sync(0xffffffffu, v[0], off));
    }
  }
  return v[0];
}

template <int FROM, class Op>
__device__ __forceinline__ float xor_reduce_f(float v, Op op) {
#pragma unroll
  for (int off = FROM; off < 32; off <<= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, off));
  return v;
}

// Sum over the lanes of a row (offsets below TO) or over the rows of a warp
// (offsets from FROM up).
template <int FROM, int TO>
__device__ __forceinline__ int xor_add(int v) {
#pragma unroll
  for (int off = FROM; off < TO; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// The (min, max) of a CTA, NaN when any entry is not finite, into *out.
template <int WARPS>
__device__ __forceinline__ void cta_range(float mn, float mx, float2 (&red)[WARPS],
                                          float2 *out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  mn = xor_reduce_f<1>(mn, MinNan());
  mx = xor_reduce_f<1>(mx, MaxNan());
  if (lane == 0) red[warp] = make_float2(mn, mx);
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < (int)(blockDim.x >> 5); ++i) {
      mn = min_nan(mn, red[i].x);
      mx = max_nan(mx, red[i].y);
    }
    // an empty share leaves (inf, -inf)
    const bool bad = isnan(mn) || isnan(mx) || mn == -INFINITY || mx == INFINITY;
    *out = bad ? make_float2(NAN, NAN) : make_float2(mn, mx);
  }
}

// Clears what the code pass accumulates into.
__device__ __forceinline__ void clear_sums(const QuantArgs &a) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = g; i < a.C; i += stride) {
    if (a.csum1) a.csum1[i] = 0;
    if (a.csum2) a.csum2[i] = 0;
  }
  if (a.code_split > 1)
    for (int64_t i = g; i < a.N; i += stride) {
      if (a.rsum1) a.rsum1[i] = 0;
      if (a.rsum2) a.rsum2[i] = 0;
    }
}

// Named barrier of one team of TEAM warps (ids 1..8; 0 is __syncthreads).
template <int TEAM>
__device__ __forceinline__ void team_sync(int team) {
  if constexpr (TEAM > 1)
    asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(32 * TEAM) : "memory");
}

constexpr int kTeamRows = 16;  // rows of a block when TEAM > 1 (LPR = 32, STEPS <= 16)

// Per-block results of the statistics pass, read by the code pass: lead row
// p (as an integer bit pattern), s1, s2 and rho = 1/sqrt(nb) (0 for a block
// of one row or of zeros), followed in the workspace by w_j for every block.
struct BhqBlock {
  float p, s1, s2, rho;
};

// How the reflection's column sums w_j = sum_k e_k s_k h_kj are rounded, the
// rows in ascending order but for W_FOLDED: fma of the product e_k s_k;
// W_FMA: fma of e_k and the rounded s_k h_kj (as k_quant2); W_ADD: rounded
// products, added, and the block scalars in fp64 (as k_quant).  A shape keeps
// one order whichever kernels serve it, so its codes do not depend on the
// workspace.
enum { W_FOLDED = 0, W_FMA = 1, W_ADD = 2 };

// w2 += e s x for one pair of columns, in the given order.  (W_ADD in scalar
// operations: a packed sum of a packed product came out as one rounding.)
__device__ __forceinline__ f32x2 w_add(int order, float e, float s, f32x2 x, f32x2 w2) {
  const f32x2 t = mul2(pack2(s, s), x);
  if (order == W_FMA) return fma2(pack2(e, e), t, w2);
  float ta, tb, wa, wb;
  unpack2(t, ta, tb);
  unpack2(w2, wa, wb);
  return pack2(__fadd_rn(wa, __fmul_rn(e, ta)), __fadd_rn(wb, __fmul_rn(e, tb)));
}

// Workspace bytes of the two-pass BHQ quantizer for blocks of at least 4
// rows: the per-block record and the C column sums w of every block.
size_t bhq_pass_bytes(int64_t N, int64_t C) {
  const int64_t nblk = (N + 3) / 4;
  return (size_t)nblk * sizeof(BhqBlock) + (size_t)nblk * (size_t)C * sizeof(float) + 512;
}

// ---------------------------------------------------------------------------
// Statistics pass of BHQ (the first of the two passes over dH): for every
// block its row statistics, lead row, lambda1, lambda2, s1, s2 (App. D.4),
// the reflection's column sums w_j = sum_k e_k s_k h_kj and the row minima
// z'_k of T = Q diag(s) H (Sec. 4.2), plus the per-CTA (min, max) of the whole
// tensor (the range of Q_b1; NaN marks a non-finite input).
//
// A team of TEAM warps holds a block of nb rows in registers as loaded (bf16
// two to a register): each warp a slab of 8 LPR columns (H slabs one after
// another, the first one or ones read again from L2 for w and z'), lane l oct
// l % LPR of row l / LPR of each of the STEPS row groups.  Columns past C
// repeat the last oct, which changes no minimum or maximum and is not stored.
// What bounds it: HBM reads, once the per-block arithmetic is short enough to
// hide behind them with the 8 to 12 warps per SM that the held blocks leave
// room for (it took 2353 warp instructions per block of 16 x 256): row
// reductions by halving (47 shuffles per block of 16 rows instead of 240),
// three-input minima, NaN carried by the minima instead of a multiply-add per
// entry, f32x2 products, 12 warps instead of 8.  802816 x 256 fp32 (822 MB):
// 224 -> 144 us (5.7 TB/s), 50176 x 256: 22 -> 16 us, 8192 x 4096 bf16 (one
// block per SM at a time): 43 -> 31 us, 131072 x 64: 14.6 -> 12.2 us.
// ---------------------------------------------------------------------------
template <typename T, int LPR, int STEPS, int TEAM, int H, int WARPS, int MINB>
__global__ void __launch_bounds__(32 * WARPS, MINB)
    k_bhq_stats(const QuantArgs a, BhqBlock *__restrict__ bst, float *__restrict__ wsum,
                float2 *__restrict__ part, int order) {
  static_assert(TEAM == 1 || (LPR == 32 && STEPS <= kTeamRows), "team layout");
  static_assert(H == 1 || TEAM == 8, "column parts only for a full team");
  static_assert(WARPS % TEAM == 0, "whole teams");
  constexpr int RS = 32 / LPR, TPC = WARPS / TEAM;
  constexpr int ROWL = LPR / STEPS;  // lanes that end with the same row
  constexpr int XW = TEAM > 1 ? WARPS : 1;
  __shared__ float2 xs_mm[XW][kTeamRows];
  __shared__ float xs_tm[XW][kTeamRows];
  __shared__ BhqScale xs_sc[TPC];
  __shared__ float2 red[WARPS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int team = warp / TEAM, wi = warp - team * TEAM;
  const int nb = a.block, C = a.C;
  const int sub = lane / LPR, o = lane - sub * LPR;
  const int kown = sub + RS * (o / ROWL);  // this lane's row after a reduction
  auto col_of = [&](int h) { return ((h * TEAM + wi) * LPR + o) * 8; };
  const float fB2 = (float)((1u << a.bits) - 1u);
  clear_sums(a);
  float gmn = INFINITY, gmx = -INFINITY;
  const int64_t nblocks = (a.N + nb - 1) / nb;
  const int64_t tstride = (int64_t)gridDim.x * TPC;
  const T *const hp = reinterpret_cast<const T *>(a.h);
  for (int64_t blk = (int64_t)blockIdx.x * TPC + team; blk < nblocks; blk += tstride) {
    const int64_t r0 = blk * nb;
    const int nrows = (int)min((int64_t)nb, a.N - r0);
    Oct<T> x[STEPS];
    auto load_part = [&](int h) {
      const int c = min(col_of(h), C - 8);
#pragma unroll
      for (int s = 0; s < STEPS; ++s) {
        const int k = sub + RS * s;
        if (k < nrows) x[s].load(hp + (r0 + k) * C + c);
        else x[s].clear();
      }
    };
    // ---- row statistics ----
    float rmn = INFINITY, rmx = -INFINITY;  // of row kown
#pragma unroll 1
    for (int h = 0; h < H; ++h) {
      load_part(h);
      float v[STEPS];
#pragma unroll
      for (int s = 0; s < STEPS; ++s) v[s] = x[s].min8();
      rmn = min_nan(rmn, reduce_rows<STEPS, LPR>(v, MinNan()));
#pragma unroll
      for (int s = 0; s < STEPS; ++s) v[s] = x[s].max8();
      rmx = max_nan(rmx, reduce_rows<STEPS, LPR>(v, MaxNan()));
    }
    if constexpr (TEAM > 1) {
      if (o % ROWL == 0) xs_mm[warp][kown] = make_float2(rmn, rmx);
      team_sync<TEAM>(team);
#pragma unroll
      for (int w2 = 0; w2 < TEAM; ++w2) {
        const float2 m = xs_mm[team * TEAM + w2][kown];
        rmn = min_nan(rmn, m.x);
        rmx = max_nan(rmx, m.y);
      }
    }
    const bool rv = kown < nrows;
    if (rv) {
      gmn = min_nan(gmn, rmn);
      gmx = max_nan(gmx, rmx);
    }
    // ---- lead row (largest ||h_k||_inf, lowest index on ties), lambda2;
    // norms are >= 0, so their bits order as integers ----
    const uint32_t key = rv ? __float_as_uint(fmaxf(fabsf(rmn), fabsf(rmx))) : 0u;
    const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
    const int p = (int)__reduce_min_sync(0xffffffffu, rv && key == kmax ? (uint32_t)kown : 0u - 1u) &
                  (nb - 1);
    const uint32_t k2 = __reduce_max_sync(0xffffffffu, kown != p ? key : 0u);
    const float np = __uint_as_float(kmax), lam2 = 2.0f * __uint_as_float(k2);
    // range of the lead row, from a lane that owns it
    const int plane = (p % RS) * LPR + (p / RS) * ROWL;
    const float pmin = __shfl_sync(0xffffffffu, rmn, plane);
    const float pmax = __shfl_sync(0xffffffffu, rmx, plane);
    // ---- block scalars s1, s2 (App. D.4) and the reflection ----
    BhqScale sc;
    if (LPR < 32 || order != W_ADD) {
      sc = bhq_scale(np, __fsub_rn(pmax, pmin), lam2, nrows, fB2);
    } else if constexpr (TEAM == 1) {
      sc = bhq_scale_f64(np, __fsub_rn(pmax, pmin), lam2, nrows, a.bits);
    } else {  // in one warp: the fp64 pipe takes 16 cycles per instruction
      if (wi == 0) {
        sc = bhq_scale_f64(np, __fsub_rn(pmax, pmin), lam2, nrows, a.bits);
        if (lane == 0) xs_sc[team] = sc;
      }
      team_sync<TEAM>(team);
      sc = xs_sc[team];
    }
    const float s1f = sc.s1, s2f = sc.s2, rho = sc.rho, kap = sc.kap;
    const float el = __fmul_rn(kap * (rho - 1.0f), s1f), eo = __fmul_rn(kap * rho, s2f);
    float tmn = INFINITY;  // z' of row kown
    // the last part read is still in registers; the others are read again
#pragma unroll 1
    for (int h = H - 1; h >= 0; --h) {
      if (h != H - 1) load_part(h);
      // w_j = sum_k e_k s_k h_kj over the block (lane: its 8 columns)
      f32x2 w2[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) w2[i] = pack2(0.0f, 0.0f);
      if (LPR < 32 || order == W_FOLDED) {
#pragma unroll
        for (int s = 0; s < STEPS; ++s) {
          const float e = sub + RS * s == p ? el : eo;
          const f32x2 e2 = pack2(e, e);
#pragma unroll
          for (int i = 0; i < 4; ++i) w2[i] = fma2(e2, x[s].pair(i), w2[i]);
        }
      } else {
#pragma unroll
        for (int s = 0; s < STEPS; ++s) {
          const float e = kap * (s == p ? rho - 1.0f : rho), sk = s == p ? s1f : s2f;
#pragma unroll
          for (int i = 0; i < 4; ++i) w2[i] = w_add(order, e, sk, x[s].pair(i), w2[i]);
        }
      }
      float w[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) unpack2(w2[i], w[2 * i], w[2 * i + 1]);
      if constexpr (LPR < 32) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int off = LPR; off < 32; off <<= 1)
            w[j] += __shfl_xor_sync(0xffffffffu, w[j], off);
#pragma unroll
        for (int i = 0; i < 4; ++i) w2[i] = pack2(w[2 * i], w[2 * i + 1]);
      }
      // ---- row minima of T; the code pass recomputes each t_kj with this
      // same sequence of roundings, so z'_k is exactly its row minimum ----
      float v[STEPS];
#pragma unroll
      for (int s = 0; s < STEPS; ++s) {
        const bool lead = sub + RS * s == p;
        const float sk = lead ? s1f : s2f, nck = lead ? 1.0f - rho : -rho;
        const f32x2 sk2 = pack2(sk, sk), nc2 = pack2(nck, nck);
        float t[8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          unpack2(fma2(nc2, w2[i], mul2(sk2, x[s].pair(i))), t[2 * i], t[2 * i + 1]);
        v[s] = min_nan(
            min3_nan(min3_nan(min3_nan(t[0], t[1], t[2]), t[3], t[4]), t[5], t[6]), t[7]);
      }
      tmn = min_nan(tmn, reduce_rows<STEPS, LPR>(v, MinNan()));
      if (sub == 0 && col_of(h) < C) {
        float *wd = wsum + blk * (int64_t)C + col_of(h);
        *reinterpret_cast<float4 *>(wd) = make_float4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<float4 *>(wd + 4) = make_float4(w[4], w[5], w[6], w[7]);
      }
    }
    if constexpr (TEAM > 1) {
      if (o % ROWL == 0) xs_tm[warp][kown] = tmn;
      team_sync<TEAM>(team);
#pragma unroll
      for (int w2 = 0; w2 < TEAM; ++w2) tmn = min_nan(tmn, xs_tm[team * TEAM + w2][kown]);
    }
    // ---- outputs: each row from its first lane ----
    if (wi == 0) {
      if (o % ROWL == 0 && rv) {
        const float sk = kown == p ? s1f : s2f;
        a.inv2[r0 + kown] = sk > 0.0f ? __fdiv_rn(1.0f, sk) : 0.0f;
        a.zero2[r0 + kown] = tmn;
      }
      if (lane == 0) {
        bst[blk] = BhqBlock{__int_as_float(p), s1f, s2f, rho};
        a.lead2[blk] = p;
      }
    }
  }
  cta_range(gmn, gmx, red, part + blockIdx.x);
}

// ---------------------------------------------------------------------------
// The same statistics pass for blocks of 32, 64 or 128 rows, which registers
// do not hold: a CTA per block reads it three times, the second and third from
// L1 or L2: rows over warps for the row ranges (LPR lanes a row, four rows in
// flight), pairs of columns over threads for w, the rows in order, and rows
// over warps again for z'.
// What bounds it: the latency of the three passes at a block per CTA.  53910 x
// 352 bf16 in blocks of 64 (38 MB), with the code pass: k_range and k_quant2,
// one staged pass with the range pass before it, 127 -> 80 us; 50176 x 256
// fp32 in blocks of 32: 108 -> 52, 2471 x 208: 17 -> 14, 8192 x 2048: 152 -> 74
// (fp64 block scalars, about 10 us of them).
// ---------------------------------------------------------------------------
constexpr int kBigRows = 128;

template <typename T>
__device__ __forceinline__ f32x2 load_pair(const T *p) {
  if constexpr (sizeof(T) == 4) {
    const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
    return pack2(v.x, v.y);
  } else {
    const uint32_t v = __ldg(reinterpret_cast<const uint32_t *>(p));
    return pack2(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u));
  }
}

template <typename T, int LPR>
__global__ void __launch_bounds__(256, 3)
    k_bhq_stats_big(const QuantArgs a, BhqBlock *__restrict__ bst, float *__restrict__ wsum,
                    float2 *__restrict__ part, int order) {
  constexpr int RS = 32 / LPR, U = 4, WR = 8 * RS;  // rows of the CTA at a time
  extern __shared__ __align__(16) float wcol[];     // C column sums
  __shared__ float2 mm_s[kBigRows];
  __shared__ BhqScale sc_s;
  __shared__ float2 red[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sub = lane / LPR, o = lane - sub * LPR;
  const int nb = a.block, C = a.C, CO = C / 8;
  const float fB2 = (float)((1u << a.bits) - 1u);
  const T *const hp = reinterpret_cast<const T *>(a.h);
  clear_sums(a);
  float gmn = INFINITY, gmx = -INFINITY;
  const int64_t nblocks = (a.N + nb - 1) / nb;
  for (int64_t blk = blockIdx.x; blk < nblocks; blk += gridDim.x) {
    const int64_t r0 = blk * nb;
    const int nrows = (int)min((int64_t)nb, a.N - r0);
    const T *const hb = hp + r0 * C;
    // ---- row ranges (rows past the last repeat it) ----
    for (int q = warp * RS + sub; q - sub < nrows; q += U * WR) {
      float mn[U], mx[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        mn[u] = INFINITY;
        mx[u] = -INFINITY;
      }
      for (int c = o; c < CO; c += LPR) {
        Oct<T> x[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          x[u].load(hb + (int64_t)min(q + u * WR, nrows - 1) * C + c * 8);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          mn[u] = min_nan(mn[u], x[u].min8());
          mx[u] = max_nan(mx[u], x[u].max8());
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
#pragma unroll
        for (int off = LPR >> 1; off > 0; off >>= 1) {
          mn[u] = min_nan(mn[u], __shfl_xor_sync(0xffffffffu, mn[u], off));
          mx[u] = max_nan(mx[u], __shfl_xor_sync(0xffffffffu, mx[u], off));
        }
        gmn = min_nan(gmn, mn[u]);
        gmx = max_nan(gmx, mx[u]);
        if (o == 0 && q + u * WR < nrows) mm_s[q + u * WR] = make_float2(mn[u], mx[u]);
      }
    }
    __syncthreads();
    // ---- lead row and scalars, in every warp ----
    uint32_t key[kBigRows / 32], best = 0u, second = 0u, at = 0xFFFFFFFFu;
#pragma unroll
    for (int i = 0; i < kBigRows / 32; ++i) {
      const int k = 32 * i + lane;
      key[i] = 0u;
      if (k < nrows) key[i] = __float_as_uint(fmaxf(fabsf(mm_s[k].x), fabsf(mm_s[k].y)));
      best = max(best, key[i]);
    }
    best = __reduce_max_sync(0xffffffffu, best);
#pragma unroll
    for (int i = kBigRows / 32 - 1; i >= 0; --i)
      if (32 * i + lane < nrows && key[i] == best) at = 32 * i + lane;
    const int p = (int)__reduce_min_sync(0xffffffffu, at) & (nb - 1);
#pragma unroll
    for (int i = 0; i < kBigRows / 32; ++i)
      if (32 * i + lane != p) second = max(second, key[i]);
    second = __reduce_max_sync(0xffffffffu, second);
    const float np = __uint_as_float(best), lam1 = __fsub_rn(mm_s[p].y, mm_s[p].x);
    const float lam2 = 2.0f * __uint_as_float(second);
    BhqScale sc;
    if (order != W_ADD) {
      sc = bhq_scale(np, lam1, lam2, nrows, fB2);
    } else {  // in one warp (fp64)
      if (warp == 0) {
        sc = bhq_scale_f64(np, lam1, lam2, nrows, a.bits);
        if (lane == 0) sc_s = sc;
      }
      __syncthreads();
      sc = sc_s;
    }
    // ---- w ----
    const float el = sc.kap * (sc.rho - 1.0f), eo = sc.kap * sc.rho;
    for (int c = tid * 2; c < C; c += 512) {
      f32x2 w2 = pack2(0.0f, 0.0f);
      for (int k0 = 0; k0 < nrows; k0 += 16) {
        f32x2 x[16];
#pragma unroll
        for (int k = 0; k < 16; ++k)
          x[k] = load_pair(hb + (int64_t)min(k0 + k, nrows - 1) * C + c);
#pragma unroll
        for (int k = 0; k < 16; ++k)
          if (k0 + k < nrows) {
            const bool lead = k0 + k == p;
            w2 = w_add(order, lead ? el : eo, lead ? sc.s1 : sc.s2, x[k], w2);
          }
      }
      float2 w;
      unpack2(w2, w.x, w.y);
      *reinterpret_cast<float2 *>(wcol + c) = w;
      *reinterpret_cast<float2 *>(wsum + blk * (int64_t)C + c) = w;
    }
    __syncthreads();
    // ---- row minima of T (see k_bhq_stats) ----
    for (int q = warp * RS + sub; q - sub < nrows; q += U * WR) {
      float mn[U];
      f32x2 sk2[U], nc2[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        mn[u] = INFINITY;
        const bool lead = q + u * WR == p;
        const float sk = lead ? sc.s1 : sc.s2, nck = lead ? 1.0f - sc.rho : -sc.rho;
        sk2[u] = pack2(sk, sk);
        nc2[u] = pack2(nck, nck);
      }
      for (int c = o; c < CO; c += LPR) {
        Oct<T> x[U];
        Oct<float> w;
#pragma unroll
        for (int u = 0; u < U; ++u)
          x[u].load(hb + (int64_t)min(q + u * WR, nrows - 1) * C + c * 8);
#pragma unroll
        for (int i = 0; i < 2; ++i)
          *reinterpret_cast<float4 *>(&w.v[4 * i]) =
              *reinterpret_cast<const float4 *>(wcol + c * 8 + 4 * i);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          float t[8];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            unpack2(fma2(nc2[u], w.pair(i), mul2(sk2[u], x[u].pair(i))), t[2 * i], t[2 * i + 1]);
          mn[u] = min_nan(
              mn[u],
              min_nan(min3_nan(min3_nan(min3_nan(t[0], t[1], t[2]), t[3], t[4]), t[5], t[6]),
                      t[7]));
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
#pragma unroll
        for (int off = LPR >> 1; off > 0; off >>= 1)
          mn[u] = min_nan(mn[u], __shfl_xor_sync(0xffffffffu, mn[u], off));
        const int k = q + u * WR;
        if (o == 0 && k < nrows) {
          const float sk = k == p ? sc.s1 : sc.s2;
          a.inv2[r0 + k] = sk > 0.0f ? __fdiv_rn(1.0f, sk) : 0.0f;
          a.zero2[r0 + k] = mn[u];
        }
      }
    }
    if (tid == 0) {
      bst[blk] = BhqBlock{__int_as_float(p), sc.s1, sc.s2, sc.rho};
      a.lead2[blk] = p;
    }
    __syncthreads();  // the tables are reused
  }
  cta_range(gmn, gmx, red, part + blockIdx.x);
}

// ---------------------------------------------------------------------------
// Statistics pass of PSQ with one sample per row: each row's s = B / R and
// z = min (srec: s, z, 1/s, s z), and the (min, max) of the tensor.  LPR lanes
// share a row, a lane taking its octs o, o + LPR, ...
// ---------------------------------------------------------------------------
template <typename T, int LPR>
__global__ void __launch_bounds__(256) k_row_stats(const QuantArgs a, float4 *__restrict__ srec,
                                                   float2 *__restrict__ part) {
  constexpr int RS = 32 / LPR, U = 4;
  __shared__ float2 red[8];
  const int lane = threadIdx.x & 31;
  const int sub = lane / LPR, o = lane - sub * LPR, CO = a.C / 8;
  const uint32_t B = (1u << a.bits) - 1u;
  const T *const hp = reinterpret_cast<const T *>(a.h);
  clear_sums(a);
  float gmn = INFINITY, gmx = -INFINITY;
  const int64_t warps = (int64_t)gridDim.x * 8;
  for (int64_t g = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); g * RS < a.N; g += warps) {
    const int64_t row = g * RS + sub;
    const bool rv = row < a.N;
    const T *h = hp + (rv ? row : 0) * a.C;
    float mn = INFINITY, mx = -INFINITY;
    for (int c = o; c < CO; c += U * LPR) {
      Oct<T> x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) x[u].load(h + (int64_t)min(c + u * LPR, CO - 1) * 8);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        mn = min_nan(mn, x[u].min8());
        mx = max_nan(mx, x[u].max8());
      }
    }
#pragma unroll
    for (int off = LPR >> 1; off > 0; off >>= 1) {
      mn = min_nan(mn, __shfl_xor_sync(0xffffffffu, mn, off));
      mx = max_nan(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    }
    if (rv) {
      gmn = min_nan(gmn, mn);
      gmx = max_nan(gmx, mx);
      if (o == 0) {
        const float s = affine_scale(mn, mx, B);
        srec[row] = make_float4(s, mn, __fdiv_rn(1.0f, s), __fmul_rn(s, mn));
      }
    }
  }
  cta_range(gmn, gmx, red, part + blockIdx.x);
}

// ---------------------------------------------------------------------------
// Per-sample PSQ (fqt_quantize_grad_samples; Sec. 4.1 with a sample = R
// consecutive rows of dH, an image's output pixels): k_sample_part takes the
// (min, max) of chunks of kSampleChunk rows' worth of entries inside one
// sample; k_sample_finish reduces each sample's chunks to s = B / R(h_i),
// z = min h_i (affine_scale, as the row quantizer), 1 / s and s z, and leaves
// per-CTA (min, max) of the whole tensor (the range of Q_b1).  The code pass
// (k_codes) then rounds and packs.
// ---------------------------------------------------------------------------
constexpr int kSampleChunkElems = 16384;

template <typename T>
__global__ void __launch_bounds__(256) k_sample_part(const QuantArgs a, int64_t sample_elems,
                                                     int chunks_per_sample, float2 *cpart) {
  __shared__ float2 red[8];
  __shared__ int redi[8];
  const int64_t ch = blockIdx.x;
  const int64_t smp = ch / chunks_per_sample;
  const int64_t e0 = smp * sample_elems + (ch - smp * chunks_per_sample) * kSampleChunkElems;
  const int64_t e1 = min(smp * sample_elems + sample_elems, e0 + kSampleChunkElems);
  const T *h = reinterpret_cast<const T *>(a.h);
  float mn = INFINITY, mx = -INFINITY, nanacc = 0.0f;
  for (int64_t e = e0 + (int64_t)threadIdx.x * 8; e < e1; e += (int64_t)blockDim.x * 8) {
    float x[8];
    load_oct(h + e, x);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      mn = fminf(mn, x[j]);
      mx = fmaxf(mx, x[j]);
      nanacc = fmaf(x[j], 0.0f, nanacc);
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, off));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    nanacc += __shfl_xor_sync(0xffffffffu, nanacc, off);
  }
  if (lane == 0) {
    red[warp] = make_float2(mn, mx);
    redi[warp] = isnan(nanacc) ? 1 : 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int bad = 0;
    for (int i = 0; i < 8; ++i) {
      mn = fminf(mn, red[i].x);
      mx = fmaxf(mx, red[i].y);
      bad |= redi[i];
    }
    cpart[ch] = bad ? make_float2(NAN, NAN) : make_float2(mn, mx);
  }
}

__global__ void __launch_bounds__(256) k_sample_finish(const QuantArgs a, int64_t nsamples,
                                                       int chunks_per_sample,
                                                       const float2 *cpart, float4 *srec,
                                                       float2 *part) {
  __shared__ float2 red[8];
  __shared__ int redi[8];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t B = (1u << a.bits) - 1u;
  float mn = INFINITY, mx = -INFINITY;
  int bad = 0;
  if (i < nsamples) {
    for (int k = 0; k < chunks_per_sample; ++k) {
      const float2 p = cpart[i * chunks_per_sample + k];
      bad |= isnan(p.x);
      mn = fminf(mn, p.x);
      mx = fmaxf(mx, p.y);
    }
    const float s = affine_scale(mn, mx, B);
    srec[i] = make_float4(s, mn, __fdiv_rn(1.0f, s), __fmul_rn(s, mn));
  }
  // the CTA's (min, max) of the whole tensor, for Q_b1
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, off));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    bad |= __shfl_xor_sync(0xffffffffu, bad, off);
  }
  if (lane == 0) {
    red[warp] = make_float2(mn, mx);
    redi[warp] = bad;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) {
      mn = fminf(mn, red[w].x);
      mx = fmaxf(mx, red[w].y);
      bad |= redi[w];
    }
    mn = fminf(mn, red[0].x);
    mx = fmaxf(mx, red[0].y);
    bad |= redi[0];
    part[blockIdx.x] = bad ? make_float2(NAN, NAN) : make_float2(mn, mx);
  }
  // the code pass accumulates column sums (and, split, row sums) into these
  for (int64_t k = i; k < a.C; k += (int64_t)gridDim.x * blockDim.x) {
    if (a.csum1) a.csum1[k] = 0;
    if (a.csum2) a.csum2[k] = 0;
  }
  if (a.code_split > 1)
    for (int64_t k = i; k < a.N; k += (int64_t)gridDim.x * blockDim.x) {
      if (a.rsum1) a.rsum1[k] = 0;
      if (a.rsum2) a.rsum2[k] = 0;
    }
}

// Workspace bytes of the per-sample quantizer: chunk partials and records.
size_t sample_pass_bytes(int64_t N, int64_t C, int64_t rows_per_sample) {
  if (rows_per_sample < 1) return 0;
  const int64_t ns = N / rows_per_sample;
  const int64_t cps = (rows_per_sample * C + kSampleChunkElems - 1) / kSampleChunkElems;
  return (size_t)(ns * cps) * sizeof(float2) + (size_t)ns * sizeof(float4) + 512;
}

// ---------------------------------------------------------------------------
// Code pass (the second pass over dH), fused with Q_b1: per entry
//   BHQ   v = t - z'_k, t = s_k h_kj - c_k w_j (c_k = rho - 1 on the lead
//         row, rho elsewhere) as the statistics pass computed it,
//   PSQ   v = s_i (h - z_i) with the scalars of sample i = row /
//         rows_per_sample (srec), written per row as well,
//   PTQ   v = s (h - min H),
// stochastic rounding of v (Q_b2) and of s (h - min H) (Q_b1), fp16 carriers
// (and optional bytes), row sums of Q_b2 and column sums of the grad_W code
// set.  A lane owns two octs of a row, o and o + LPR of a slab of 16 LPR
// columns (one coalesced access each; octs past C are computed on a repeated
// oct and dropped); a warp takes units of `urows` rows and 1 / code_split of
// the row's slabs, walks those slabs one after another and, inside a slab,
// the unit's rows 32 / LPR at a time, issuing the loads of its next row before
// it rounds the current one.  A block's w_j and scalars stay in registers
// while the lane's rows belong to it.  A row's parts meet only in its row sums
// (atomic when code_split > 1).  Units shrink with the tensor, down to 8 rows
// and one slab, until there are enough for every warp of the GPU (on the
// smallest tensors down to 2 rows).
// What bounds it: HBM on the largest tensors (802816 x 256 BHQ-5, 822 MB read
// and as much written: 322 -> 305 us, 5.6 TB/s), the issue slots and the
// integer pipe (two Philox streams) on those that L2 holds: packed operations,
// stepped offsets and column sums kept over the units took it from 42 to 34
// warp instructions per 32 entries, units of 8 rows fill the GPU: 50176 x 256
// 33 -> 25 us, 8192 x 4096 bf16 70 -> 50 us, 8192 x 1024 bf16 PTQ-8 (k_quant2
// before) 29 -> 16 us.  Staging the rows through shared memory three deep
// (cp.async) instead of one row ahead in registers was slower (397 us on the
// first shape).  grad_X's BHQ offsets of a unit that holds whole blocks are
// computed from the row sums at its end: 305 -> 312 us on the first shape, and
// no k_bhq_offsets (13 us).
// ---------------------------------------------------------------------------
constexpr int kCodeRows = 32;
constexpr int kCodesMaxCols = 8192;
enum { CODES_BHQ = 0, CODES_PSQ = 1, CODES_PTQ = 2 };

constexpr float kSrMagic = 8414080.0f;  // 2^23 + 0x6400 - 128

// Two codes SR(v) as fp16 1024 + min(code, B) (cap: 1024 + B in both halves);
// U = 128 + u 2^-16 for the two 16-bit uniforms of a Philox word.
__device__ __forceinline__ uint32_t sr_codes2(f32x2 v, uint32_t word, __half2 cap) {
  float a, b;
  unpack2(v, a, b);
  a = __fadd_rd(__fadd_rd(a, __uint_as_float(0x43000000u | (word & 0xFFFFu))), kSrMagic);
  b = __fadd_rd(__fadd_rd(b, __uint_as_float(__byte_perm(word, 0x43000000u, 0x7632))), kSrMagic);
  const uint32_t h = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x5410);
  const __half2 m = __hmin2(*reinterpret_cast<const __half2 *>(&h), cap);
  return *reinterpret_cast<const uint32_t *>(&m);
}

// Eight codes (packed pairs of 1024 + code) as carriers code - off and bytes.
__device__ __forceinline__ void store_oct(uint16_t *f, uint8_t *c, const uint32_t *h,
                                          __half2 bias) {
  if (f) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __half2 v = __hsub2(*reinterpret_cast<const __half2 *>(&h[i]), bias);
      w[i] = *reinterpret_cast<const uint32_t *>(&v);
    }
    *reinterpret_cast<uint4 *>(f) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  if (c)
    *reinterpret_cast<uint2 *>(c) =
        make_uint2(__byte_perm(h[0], h[1], 0x6420), __byte_perm(h[2], h[3], 0x6420));
}

// PLAIN: both code sets as carriers only and no row sums of Q_b1, the call of
// a training step; other outputs are tested for at run time.
template <typename T, int LPR, int MODE, bool PLAIN>
__global__ void __launch_bounds__(256, 2)
    k_codes(const QuantArgs a, const BhqBlock *__restrict__ bst, const float *__restrict__ wsum,
            int lg_nb, const float4 *__restrict__ srec, int rows_per_sample, int lg_urows) {
  constexpr int RS = 32 / LPR, SLAB = 16 * LPR;
  __shared__ float2 red[8];
  __shared__ int redi[8];
  __shared__ int rs_s[8][2][kCodeRows];
  extern __shared__ int csum_s[];  // C column sums of the grad_W code set
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int C = a.C, CO = C / 8;
  const int sub = lane / LPR, o = lane - sub * LPR;

  // ---- global range (Q_b1 scale) from the first pass's partials ----
  float gmin = INFINITY, gmax = -INFINITY;
  int bad = 0;
  for (int i = tid; i < a.npart; i += blockDim.x) {
    const float2 p = a.part[i];
    bad |= isnan(p.x);
    gmin = fminf(gmin, p.x);
    gmax = fmaxf(gmax, p.y);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    gmin = fminf(gmin, __shfl_xor_sync(0xffffffffu, gmin, off));
    gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, off));
    bad |= __shfl_xor_sync(0xffffffffu, bad, off);
  }
  if (lane == 0) {
    red[warp] = make_float2(gmin, gmax);
    redi[warp] = bad;
  }
  for (int i = tid; i < C; i += blockDim.x) csum_s[i] = 0;
  __syncthreads();
  gmin = red[0].x;
  gmax = red[0].y;
  bad = redi[0];
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
    gmin = fminf(gmin, red[w].x);
    gmax = fmaxf(gmax, red[w].y);
    bad |= redi[w];
  }
  if (bad) {
    if (blockIdx.x == 0 && tid == 0) record_status(a.status, FQT_ENONFINITE);
    return;
  }
  const uint32_t B2 = (1u << a.bits) - 1u;
  const float s_g1 = affine_scale(gmin, gmax, 255u);
  const float s_g2 = MODE == CODES_PTQ ? affine_scale(gmin, gmax, B2) : 0.0f;
  const bool has_b1 = PLAIN || a.c1 != nullptr || a.f1 != nullptr;
  uint8_t *const c1 = PLAIN ? nullptr : a.c1, *const c2 = PLAIN ? nullptr : a.c2;
  if (blockIdx.x == 0 && tid == 0) {
    if (has_b1) {
      a.inv1[0] = __fdiv_rn(1.0f, s_g1);
      a.zero1[0] = __fmul_rn(s_g1, gmin);
    }
    if (MODE == CODES_PTQ) {
      a.inv2[0] = __fdiv_rn(1.0f, s_g2);
      a.zero2[0] = __fmul_rn(s_g2, gmin);
    }
  }
  int32_t *const csum_g = has_b1 ? a.csum1 : a.csum2;
  PhiloxKeys key;
#pragma unroll
  for (int i = 0; i < 20; ++i) key.k[i] = a.round_keys[i];
  const __half2 bias2 = __half2half2(__int2half_rn(1024 + (int)((B2 + 1u) >> 1)));
  const __half2 bias1 = __half2half2(__int2half_rn(1024 + 128));
  const __half2 cap2 = __half2half2(__int2half_rn(1024 + (int)B2));
  const __half2 cap1 = __half2half2(__int2half_rn(1024 + 255));
  const f32x2 ng2 = pack2(-gmin, -gmin), sg1 = pack2(s_g1, s_g1);
  const bool want_rs1 = !PLAIN && has_b1 && a.rsum1 != nullptr;
  const T *const h = reinterpret_cast<const T *>(a.h);
  const int nbm = (1 << lg_nb) - 1;

  const int urows = 1 << lg_urows;
  const int64_t nchunks = (a.N + urows - 1) >> lg_urows;
  const int lg_split = a.code_split > 1 ? __ffs(a.code_split) - 1 : 0;
  const int split = 1 << lg_split;
  // slabs per column part, rounded up (a last part may be empty)
  const int part_cols = (((C + SLAB - 1) / SLAB + split - 1) >> lg_split) * SLAB;
  const int64_t nunits = nchunks << lg_split;
  const bool one_slab = C <= SLAB;
  const int64_t wstride = (int64_t)gridDim.x * (blockDim.x >> 5);
  // column sums of the current slab, two 16-bit lanes a word (at most 255 rows
  // per lane between flushes); kept over the units when a row is one slab
  uint32_t cs[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) cs[j] = 0u;
  int cs_rows = 0;
  auto flush_cs = [&](int c0) {
    if (csum_g) {
      const int ca = c0 + o * 8, cb = ca + 8 * LPR;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int lo = xor_add<LPR, 32>((int)(cs[j] & 0xFFFFu));
        const int hi = xor_add<LPR, 32>((int)(cs[j] >> 16));
        const int col = (j < 4 ? ca : cb - 8) + 2 * j;
        if (sub == 0 && (j < 4 ? ca : cb) < C) {
          if (lo) atomicAdd(&csum_s[col], lo);
          if (hi) atomicAdd(&csum_s[col + 1], hi);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) cs[j] = 0u;
    cs_rows = 0;
  };
  for (int64_t u = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp; u < nunits;
       u += wstride) {
    // from the end of dH, which the first pass left in L2
    const int64_t ch = nchunks - 1 - (u >> lg_split);
    const int cpart = (int)u & (split - 1);
    const int64_t row0 = ch << lg_urows;
    const int rows = (int)min((int64_t)urows, a.N - row0);
    rs_s[warp][0][lane] = 0;
    rs_s[warp][1][lane] = 0;
    __syncwarp();
    const int c_end = min(C, (cpart + 1) * part_cols);
#pragma unroll 1
    for (int c0 = cpart * part_cols; c0 < c_end; c0 += SLAB) {
      const int ca = c0 + o * 8, cb = ca + 8 * LPR;  // this lane's two octs
      const bool va = ca < C, vb = cb < C;
      const int la = min(ca, C - 8), lb = min(cb, C - 8);
      if (cs_rows + kCodeRows > 255) flush_cs(c0);  // (kept only over one slab)
      cs_rows += kCodeRows / RS;
      int cur_blk = -1;  // block of the unit's rows, or sample
      f32x2 w[8];
      float sk_l = 0.0f, sk_o = 0.0f, ck_l = 0.0f, ck_o = 0.0f;
      int p_lead = -1;
      // offset of this lane's row in dH and the code sets, stepped per row group
      int64_t e = (row0 + sub) * C + la;
      const int dab = lb - la;
      const int64_t estep = (int64_t)RS * C;
      // the first row's loads; every later row's are issued one row ahead
      Oct<T> xa, xb;
      float zn = 0.0f;
      float4 sn = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      xa.clear();
      xb.clear();
      if (sub < rows) {
        xa.load(h + e);
        xb.load(h + e + dab);
        if (MODE == CODES_BHQ) zn = a.zero2[row0 + sub];
        if (MODE == CODES_PSQ && rows_per_sample == 1) sn = srec[row0 + sub];
      }
#pragma unroll 1
      for (int rr = sub; rr < rows + sub; rr += RS, e += estep) {  // one trip count per warp
        const bool valid = rr < rows;  // the LPR lanes of a row agree
        f32x2 x[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          x[j] = xa.pair(j);
          x[4 + j] = xb.pair(j);
        }
        const float zr = zn;
        if (MODE == CODES_PSQ && rows_per_sample == 1) {
          sk_l = sn.x;
          ck_l = sn.y;
          sk_o = sn.z;
          ck_o = sn.w;
        }
        if (rr + RS < rows) {
          const T *r = h + e + estep;
          xa.load(r);
          xb.load(r + dab);
          if (MODE == CODES_BHQ) zn = a.zero2[row0 + rr + RS];
          if (MODE == CODES_PSQ && rows_per_sample == 1) sn = srec[row0 + rr + RS];
        }
        uint32_t acc1 = 0u, acc2 = 0u;  // sums of codes, two 16-bit lanes
        uint32_t acc1b = 0u, acc2b = 0u;
        if (valid) {
          if (MODE == CODES_BHQ || (MODE == CODES_PSQ && rows_per_sample > 1)) {
            // (a unit starts on a block: its rows are a multiple of RS and of nb
            // or inside one)
            const int blk = MODE == CODES_PSQ ? (int)((row0 + rr) / rows_per_sample)
                                              : (int)((row0 + rr) >> lg_nb);
            if (blk != cur_blk) {  // a new block (sample): its w_j and scalars
              if constexpr (MODE == CODES_PSQ) {
                const float4 sr = srec[blk];  // s, z, inv_s, zero of the sample
                sk_l = sr.x;
                ck_l = sr.y;
                sk_o = sr.z;
                ck_o = sr.w;
              } else {
                const BhqBlock bs = bst[blk];
                p_lead = __float_as_int(bs.p);
                sk_l = bs.s1;
                sk_o = bs.s2;
                ck_l = 1.0f - bs.rho;  // -c_k
                ck_o = -bs.rho;
                Oct<float> wa, wb;
                const float *wp = wsum + (int64_t)blk * C + la;
                wa.load(wp);
                wb.load(wp + dab);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  w[j] = wa.pair(j);
                  w[4 + j] = wb.pair(j);
                }
              }
              cur_blk = blk;
            }
          }
          if (MODE == CODES_PSQ && o == 0 && c0 == 0) {
            a.inv2[row0 + rr] = sk_o;
            a.zero2[row0 + rr] = ck_o;
          }
          const uint64_t qa = (uint64_t)e >> 3, qb = (uint64_t)(e + dab) >> 3;
          uint32_t c[8];
          if (has_b1) {
            const uint4 ua = philox_oct(qa, 1u, key), ub = philox_oct(qb, 1u, key);
            const uint32_t uw[8] = {ua.x, ua.y, ua.z, ua.w, ub.x, ub.y, ub.z, ub.w};
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              c[j] = sr_codes2(mul2(add2(x[j], ng2), sg1), uw[j], cap1);
              cs[j] += c[j] - 0x64006400u;
            }
            if (va)
              store_oct(PLAIN || a.f1 ? a.f1 + e : nullptr, c1 ? c1 + e : nullptr, &c[0], bias1);
            if (vb)
              store_oct(PLAIN || a.f1 ? a.f1 + e + dab : nullptr, c1 ? c1 + e + dab : nullptr,
                        &c[4], bias1);
            if (want_rs1) {
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                acc1 += c[j] - 0x64006400u;
                acc1b += c[4 + j] - 0x64006400u;
              }
            }
          }
          const uint4 ua = philox_oct(qa, 0u, key), ub = philox_oct(qb, 0u, key);
          const uint32_t uw[8] = {ua.x, ua.y, ua.z, ua.w, ub.x, ub.y, ub.z, ub.w};
          const bool lead = MODE == CODES_BHQ && (((int)row0 + rr) & nbm) == p_lead;
          const float sk = MODE == CODES_BHQ ? (lead ? sk_l : sk_o)
                           : MODE == CODES_PSQ ? sk_l : s_g2;
          const float nc = MODE == CODES_BHQ ? (lead ? ck_l : ck_o) : 0.0f;
          const float sh = MODE == CODES_BHQ ? -zr : MODE == CODES_PSQ ? -ck_l : -gmin;
          const f32x2 sk2 = pack2(sk, sk), nc2 = pack2(nc, nc), sh2 = pack2(sh, sh);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            // BHQ: t - z'; PSQ, PTQ: s (h - z)
            const f32x2 v = MODE == CODES_BHQ ? add2(fma2(nc2, w[j], mul2(sk2, x[j])), sh2)
                                              : mul2(add2(x[j], sh2), sk2);
            c[j] = sr_codes2(v, uw[j], cap2);
            if (j < 4) acc2 += c[j] - 0x64006400u;
            else acc2b += c[j] - 0x64006400u;
          }
          if (!has_b1) {
#pragma unroll
            for (int j = 0; j < 8; ++j) cs[j] += c[j] - 0x64006400u;
          }
          if (va)
            store_oct(PLAIN || a.f2 ? a.f2 + e : nullptr, c2 ? c2 + e : nullptr, &c[0], bias2);
          if (vb)
            store_oct(PLAIN || a.f2 ? a.f2 + e + dab : nullptr, c2 ? c2 + e + dab : nullptr,
                      &c[4], bias2);
        }
        if (want_rs1) {
          const uint32_t t = (va ? acc1 : 0u) + (vb ? acc1b : 0u);
          const int r1 = xor_add<1, LPR>((int)((t & 0xFFFFu) + (t >> 16)));
          if (o == 0 && valid) rs_s[warp][1][rr] += r1;
        }
        const uint32_t t = (va ? acc2 : 0u) + (vb ? acc2b : 0u);
        const uint32_t rv = (t & 0xFFFFu) + (t >> 16);  // at most 16 x 255
        if constexpr (LPR == 32) {
          const int r2 = (int)__reduce_add_sync(0xffffffffu, rv);
          if (lane == 0 && valid) rs_s[warp][0][rr] += r2;
        } else if constexpr (LPR == 16) {  // two rows in one reduction (16 x 4080 < 2^16)
          const uint32_t r2 = __reduce_add_sync(0xffffffffu, sub ? rv << 16 : rv);
          if (o == 0 && valid) rs_s[warp][0][rr] += (int)(sub ? r2 >> 16 : r2 & 0xFFFFu);
        } else {
          const int r2 = xor_add<1, LPR>((int)rv);
          if (o == 0 && valid) rs_s[warp][0][rr] += r2;
        }
      }
      if (!one_slab) flush_cs(c0);
    }
    __syncwarp();
    // grad_X's offsets, where the unit holds whole blocks and whole rows
    if (MODE == CODES_BHQ && a.hz) {
      const bool kv = lane < rows;
      const int base = lane & ~nbm, nact = min(nbm + 1, rows - base);
      ff d = {0.0f, 0.0f};
      long long R = 0;
      int p = 0;
      if (kv) {
        bhq_offset_terms(a.zero2[row0 + lane], rs_s[warp][0][lane], C, 1 << (a.bits - 1), &d, &R);
        p = __float_as_int(bst[(row0 + lane) >> lg_nb].p);
      }
      ff sd = d;
      long long sR = R;
      bhq_offset_sums(&sd, &sR, nbm + 1);
      const ff dp = {__shfl_sync(0xffffffffu, d.h, base + p),
                     __shfl_sync(0xffffffffu, d.l, base + p)};
      const long long Rp = __shfl_sync(0xffffffffu, R, base + p);
      if (kv) {
        const float2 v = nact < 2 ? make_float2(ff_round(d), ff_round(ff_from_int(R)))
                                  : bhq_offset_reflect(d, R, sd, sR, dp, Rp, lane - base == p, nact);
        a.hz[row0 + lane] = v.x;
        a.hr[row0 + lane] = v.y;
      }
    }
    if (lane < rows) {
      if (split > 1) {
        if (a.rsum2) atomicAdd(&a.rsum2[row0 + lane], rs_s[warp][0][lane]);
        if (want_rs1) atomicAdd(&a.rsum1[row0 + lane], rs_s[warp][1][lane]);
      } else {
        if (a.rsum2) a.rsum2[row0 + lane] = rs_s[warp][0][lane];
        if (want_rs1) a.rsum1[row0 + lane] = rs_s[warp][1][lane];
      }
    }
    __syncwarp();
  }
  if (csum_g) {
    if (one_slab) flush_cs(0);
    __syncthreads();
    for (int i = tid; i < C; i += blockDim.x)
      if (csum_s[i]) atomicAdd(&csum_g[i], csum_s[i]);
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
// Lanes per row of the code pass: the widest slab of 16 LPR columns whose
// padded row is within 5% of the least padded one (idle lanes).
static int codes_lpr(int C) {
  int least = 1 << 30;
  auto padded = [&](int l) { return (C + 16 * l - 1) / (16 * l) * 16 * l; };
  for (int l = 4; l <= 32; l *= 2) least = std::min(least, padded(l));
  for (int l = 32; l > 4; l /= 2)
    if (padded(l) * 20 <= least * 21) return l;
  return 4;
}

// Rows per unit and column parts of the code pass: about 64 units per SM
// (four per warp), first by splitting wide rows into slabs, then by units of
// 16 and 8 rows, fewer where that leaves SMs idle.
static void codes_plan(QuantArgs &a, int lpr, int num_sms, int *lg_urows, int lg_nb = 0) {
  const int nslab = (a.C + 16 * lpr - 1) / (16 * lpr);
  const int64_t target = (int64_t)num_sms * 64;
  int lg = 5, split = 1;
  auto units = [&]() { return ((a.N + (1 << lg) - 1) >> lg) * (int64_t)split; };
  while (split < nslab && units() < target) split *= 2;
  while (lg > 3 && units() < target) --lg;
  // a small tensor: units of down to 2 rows (a warp's rows at a time at least)
  // until there are eight per SM, but for blocks that a unit holds.  256 x 1008
  // fp32 BHQ-5: 64 units of 8 rows on 8 SMs 11.4 us, 256 of 2 rows 5.7; 128 x
  // 256 8.0 -> 4.6; 2471 x 208 8.3 -> 5.8
  const int lg_min = std::max(1, 5 - (31 - __builtin_clz((unsigned)lpr)));
  while (lg > lg_min && !(lg_nb && lg_nb <= 3) &&
         units() < (int64_t)num_sms * 8)
    --lg;
  // units of whole blocks hold what grad_X's offsets need: three per warp are
  // still enough (131072 x 64: code pass 21.9 -> 22.9 us without 3.7 + 2.5 for
  // k_bhq_offsets and its gap)
  if (split == 1 && lg < lg_nb && lg_nb <= 5) {
    const int few = lg;
    lg = lg_nb;
    if (units() < (int64_t)num_sms * 48) lg = few;
  }
  a.code_split = split;
  *lg_urows = lg;
}

template <typename T, int LPR, int MODE>
static cudaError_t launch_codes_t(const QuantArgs &a, const BhqBlock *bst, const float *wsum,
                                  int lg_nb, const float4 *srec, int rps, int lg_urows,
                                  int num_sms, cudaStream_t st) {
  const bool plain = a.f1 && a.f2 && !a.c1 && !a.c2 && !a.rsum1;
  auto kern = plain ? k_codes<T, LPR, MODE, true> : k_codes<T, LPR, MODE, false>;
  const size_t smem = sizeof(int) * (size_t)a.C;
  const int64_t nunits = ((a.N + (1 << lg_urows) - 1) >> lg_urows) * a.code_split;
  // two CTAs of eight warps per SM (__launch_bounds__); four warps where the
  // units would leave SMs idle
  const int warps = nunits < (int64_t)num_sms * 8 ? 4 : 8;
  const int64_t grid =
      std::max<int64_t>(1, std::min<int64_t>((nunits + warps - 1) / warps, 2 * num_sms));
  kern<<<(int)grid, 32 * warps, smem, st>>>(a, bst, wsum, lg_nb, srec, rps, lg_urows);
  return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_codes(const QuantArgs &a, bool bf16, int lpr, const BhqBlock *bst,
                                const float *wsum, int lg_nb, const float4 *srec, int rps,
                                int lg_urows, int num_sms, cudaStream_t st) {
#define FQT_CODES(L)                                                                       \
  case L:                                                                                  \
    return bf16 ? launch_codes_t<__nv_bfloat16, L, MODE>(a, bst, wsum, lg_nb, srec, rps,   \
                                                         lg_urows, num_sms, st)            \
                : launch_codes_t<float, L, MODE>(a, bst, wsum, lg_nb, srec, rps, lg_urows, \
                                                 num_sms, st);
  switch (lpr) {
    FQT_CODES(4)
    FQT_CODES(8)
    FQT_CODES(16)
    FQT_CODES(32)
  }
#undef FQT_CODES
  return cudaErrorInvalidValue;
}

// PTQ: the range partials (a.part, a.npart) and cleared column sums come from
// k_range; `plan` first, so that it also clears the row sums of split rows.
bool ptq_pass_supported(int C) { return C % 8 == 0 && C <= kCodesMaxCols; }

void ptq_pass_plan(QuantArgs &a, int num_sms) {
  int lg;
  codes_plan(a, codes_lpr(a.C), num_sms, &lg);
}

fqt_status launch_ptq_codes(QuantArgs &a, bool bf16, int num_sms, cudaStream_t st) {
  const int lpr = codes_lpr(a.C);
  int lg;
  codes_plan(a, lpr, num_sms, &lg);
  return cuda_fail(launch_codes<CODES_PTQ>(a, bf16, lpr, nullptr, nullptr, 0, nullptr, 1, lg,
                                           num_sms, st),
                   "PTQ code pass launch");
}

// The per-sample PSQ with Q_b1: samples of rows_per_sample rows (one: the row
// quantizer, any C of the code pass; more: C % 8 == 0 and at most 2^20
// samples).  `scratch` (sample_pass_bytes) holds the samples' scalars.
bool psq_pass_supported(int C) { return C % 8 == 0 && C <= kCodesMaxCols; }

fqt_status launch_sample_passes(QuantArgs &a, bool bf16, int64_t rows_per_sample, int num_sms,
                                void *scratch, float2 *part, cudaStream_t st) {
  const int C = a.C;
  if (!psq_pass_supported(C)) return FQT_EUNSUPPORTED;
  const int64_t ns = a.N / rows_per_sample;
  if (rows_per_sample > 1 && ns > ((int64_t)1 << 20)) return FQT_EUNSUPPORTED;
  const int64_t se = rows_per_sample * C;
  const int cps = (int)((se + kSampleChunkElems - 1) / kSampleChunkElems);
  float2 *cpart = static_cast<float2 *>(scratch);
  float4 *srec = reinterpret_cast<float4 *>(
      (reinterpret_cast<uintptr_t>(cpart + ns * cps) + 255) & ~(uintptr_t)255);
  const int lpr = codes_lpr(C);
  int lg;
  codes_plan(a, lpr, num_sms, &lg);
  QuantArgs a2 = a;
  a2.part = part;
  cudaError_t e;
  if (rows_per_sample == 1) {
    // LPR lanes per row: at least one oct each, four in flight
    const int CO = C / 8;
    const int64_t rows_per_cta = 8 * (CO >= 32 ? 1 : CO >= 16 ? 2 : 4);
    const int64_t grid = std::min<int64_t>((a.N + rows_per_cta - 1) / rows_per_cta, 8 * num_sms);
#define FQT_RS(L)                                                                   \
  {                                                                                 \
    if (bf16) k_row_stats<__nv_bfloat16, L><<<(int)grid, 256, 0, st>>>(a, srec, part); \
    else k_row_stats<float, L><<<(int)grid, 256, 0, st>>>(a, srec, part);           \
  }
    if (CO >= 32) FQT_RS(32) else if (CO >= 16) FQT_RS(16) else FQT_RS(8)
#undef FQT_RS
    a2.npart = (int)grid;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "row statistics launch");
  } else {
    if (bf16)
      k_sample_part<__nv_bfloat16><<<(unsigned)(ns * cps), 256, 0, st>>>(a, se, cps, cpart);
    else
      k_sample_part<float><<<(unsigned)(ns * cps), 256, 0, st>>>(a, se, cps, cpart);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "sample statistics launch");
    const int fin = (int)((ns + 255) / 256);
    k_sample_finish<<<fin, 256, 0, st>>>(a, ns, cps, cpart, srec, part);
    a2.npart = fin;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "sample scalars launch");
  }
  return cuda_fail(launch_codes<CODES_PSQ>(a2, bf16, lpr, nullptr, nullptr, 0, srec,
                                           (int)rows_per_sample, lg, num_sms, st),
                   "sample code pass launch");
}

// The two-pass BHQ quantizer: the order of w of a shape, or -1 for the shapes
// that stay with the one-pass quantizers.  Powers of two from 64 to 4096
// columns with blocks of 16 (fp32: 4 and 8 too) fold e and s and add a warp's
// row groups last; the others keep the rounding of the one-pass quantizer that
// takes them without this scratch, whose rows are added in order, so a warp
// holds whole columns of them (200000 x 80 fp32 in blocks of 16: 179 us
// staged, 83 so).  Blocks of one and two rows stay with it, as do rows of
// fewer than 40 columns, most of whose lanes would be idle (200000 rows of 16
// in blocks of 16: 45 against 61 us, of 32 in blocks of 4: 60 against 70, of
// 24 in blocks of 64: 68 against 76; of 40 in blocks of 16: 95 against 63).
int bhq_pass_order(int C, int block, bool bf16) {
  if (C % 8 || C > 4096 || block < 4) return -1;
  if (C >= 64 && !(C & (C - 1)) && (block == 16 || (!bf16 && block < 16))) return W_FOLDED;
  if (C < 40) return -1;
  QuantArgs q;
  memset(&q, 0, sizeof(q));
  q.N = 1;
  q.C = C;
  q.kind = KIND_BHQ;
  q.block = block;
  int nth, grid;
  size_t smem;
  if (quant2_geometry(q, bf16, 1, &grid, &smem) == FQT_OK) return W_FMA;
  return quant_geometry(q, 1, &nth, &grid, &smem) == FQT_OK ? W_ADD : -1;
}

template <typename T, int LPR, int STEPS, int TEAM, int H>
static cudaError_t launch_stats(const QuantArgs &a, BhqBlock *bst, float *wsum, float2 *part,
                                int num_sms, int *grid_out, int order, cudaStream_t st) {
  // registers of the block per thread: 8 (fp32) or 4 per oct
  constexpr int data = STEPS * (sizeof(T) == 4 ? 8 : 4);
  constexpr int WARPS = data >= 64 ? (TEAM == 8 ? 8 : 12) : 8;
  constexpr int MINB = data >= 64 ? 1 : data > 16 ? 2 : 3;
  constexpr int TPC = WARPS / TEAM;
  const int64_t nblocks = (a.N + a.block - 1) / a.block;
  int64_t grid = std::min<int64_t>((nblocks + TPC - 1) / TPC, (int64_t)num_sms * MINB);
  if (grid < 1) grid = 1;
  *grid_out = (int)grid;
  k_bhq_stats<T, LPR, STEPS, TEAM, H, WARPS, MINB><<<(int)grid, 32 * WARPS, 0, st>>>(
      a, bst, wsum, part, order);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_stats_any(const QuantArgs &a, BhqBlock *bst, float *wsum, float2 *part,
                                    int num_sms, int *grid, int order, cudaStream_t st) {
  const int C = a.C, nb = a.block;
  if (nb > 16) {
    // a CTA per block, three per SM; the fewest lanes that hold a row
    const int64_t nblocks = (a.N + nb - 1) / nb;
    *grid = (int)std::max<int64_t>(1, std::min<int64_t>(nblocks, (int64_t)num_sms * 3));
    auto kern = C <= 64 ? k_bhq_stats_big<T, 8> : C <= 128 ? k_bhq_stats_big<T, 16>
                                                           : k_bhq_stats_big<T, 32>;
    kern<<<*grid, 256, sizeof(float) * (size_t)C, st>>>(a, bst, wsum, part, order);
    return cudaGetLastError();
  }
#define FQT_ST(L, S, TM, HH) \
  return launch_stats<T, L, S, TM, HH>(a, bst, wsum, part, num_sms, grid, order, st);
#define FQT_ST_NB(L, TM, HH)                                                     \
  {                                                                              \
    if (nb == 4) FQT_ST(L, L / 8, TM, HH)                                        \
    if (nb == 8) FQT_ST(L, L / 4, TM, HH)                                        \
    FQT_ST(L, L / 2, TM, HH)                                                     \
  }
  if (order == W_FOLDED && C <= 64) FQT_ST_NB(8, 1, 1)
  if (order == W_FOLDED && C <= 128) FQT_ST_NB(16, 1, 1)
  if (C <= 256) FQT_ST_NB(32, 1, 1)
  if (C <= 512) FQT_ST_NB(32, 2, 1)
  if (C <= 1024) FQT_ST_NB(32, 4, 1)
  if (C <= 2048) FQT_ST_NB(32, 8, 1)
  FQT_ST_NB(32, 8, 2)
#undef FQT_ST_NB
#undef FQT_ST
}

// Statistics pass, code pass and the grad_X offsets (k_bhq_offsets) of the
// fixed-block BHQ quantizer with Q_b1.  `scratch` (bhq_pass_bytes) holds the
// per-block records and column sums w between the passes; `part` receives
// the statistics pass's range partials, which the code pass reduces.
fqt_status launch_bhq_passes(QuantArgs &a, bool bf16, int num_sms, void *scratch,
                             float2 *part, cudaStream_t st) {
  const int order = a.kind == KIND_BHQ ? bhq_pass_order(a.C, a.block, bf16) : -1;
  if (order < 0) return FQT_EUNSUPPORTED;
  const int64_t nblocks = (a.N + a.block - 1) / a.block;
  BhqBlock *bst = static_cast<BhqBlock *>(scratch);
  float *wsum = reinterpret_cast<float *>(
      (reinterpret_cast<uintptr_t>(bst + nblocks) + 255) & ~(uintptr_t)255);
  const int lpr = codes_lpr(a.C);
  int lg;
  int lg_nb = 0;
  while ((1 << lg_nb) < a.block) ++lg_nb;
  codes_plan(a, lpr, num_sms, &lg, a.hz && a.hr ? lg_nb : 0);
  int grid1 = 0;
  cudaError_t e = bf16 ? launch_stats_any<__nv_bfloat16>(a, bst, wsum, part, num_sms, &grid1, order,
                                                          st)
                       : launch_stats_any<float>(a, bst, wsum, part, num_sms, &grid1, order, st);
  if (e != cudaSuccess) return cuda_fail(e, "BHQ statistics pass launch");
  QuantArgs a2 = a;
  a2.part = part;
  a2.npart = grid1;
  // a warp that holds whole rows of whole blocks has what the offsets need
  const bool fused = a.hz && a.hr && a.rsum2 && a2.code_split == 1 && lg_nb <= lg;
  if (!fused) a2.hz = a2.hr = nullptr;
  e = launch_codes<CODES_BHQ>(a2, bf16, lpr, bst, wsum, lg_nb, nullptr, 1, lg, num_sms, st);
  if (e != cudaSuccess) return cuda_fail(e, "BHQ code pass launch");
  if (a.hz && a.hr && !fused) {
    e = launch_bhq_offsets(a.zero2, a.rsum2, a.lead2, a.hz, a.hr, a.N, a.C, a.bits, a.block, st);
    if (e != cudaSuccess) return cuda_fail(e, "BHQ offsets launch");
  }
  return FQT_OK;
}

}  // namespace fqt
