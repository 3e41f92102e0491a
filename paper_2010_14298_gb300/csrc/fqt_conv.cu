// fqt_conv.cu -- grad_X of a stride-1 3 x 3 conv in NHWC with col2im fused.
//
// Sec. 2.1: a conv is a linear layer on im2col rows; grad_X is summed back
// over the taps, i.e. the transposed convolution dX[p, j] = sum over taps t
// and output channels c of Q_b2(dH)[o(p, t), c] W~[c, t, j], o(p, t) the
// output pixel that tap t of input pixel p reads (out of the image: no term).
// It needs the scale of Q_b2 to be the same for every output pixel of an
// image -- per tensor (PTQ) or per image (fqt_quantize_grad_samples) -- so
// that it factors out of the sum over taps.
//
// Contraction.  A tile is R whole image rows (or I whole small images) as one
// run of pixel slots of pitch P = W + 2: the dH carriers of its R + 2 rows
// with a zero column on either side (TMA's fill) land in shared memory once
// per 64 channels, one 128-byte row per slot.  In that run the output pixel a
// tap reads sits a constant number of slots away,
//   slot(o(p, t)) = slot(p) + (2 - ky) P + (2 - kx),
// so every tap's operand is the same shared tile at another start address
// (the 128-byte swizzle follows the address bits, so any row may start it):
// N = (R - 1) P + W <= 256 columns, M = C_in in tiles of 128, K = 9 C_out.
// The tile is read once instead of once per tap, and the tensor cores run
// 240-column instructions.  W~ (MN-major, column offset tap C_in) stays in
// shared memory for the whole launch where it fits (C_in <= 64, one 64-wide
// atom per tap), else it passes through a ring of 16 KB tiles.
//
// What bounds it: at 64 -> 64 channels the MMAs (C_in fills half of the 128
// lanes); the layer of 256 x 56 x 56 x 64 -> 64 takes 111 us (59 GFLOP, 205 MB
// of output), against 432 us for the earlier kernel, which loaded every tap's
// shifted box (dH nine times, W~ once per 112 pixels) through one ring.
//
// Dequantization.  With a, w the centred codes, the image's offset
// 2^(b-1) + z' = m + d and y = 2^(bw-1) + z_w, for the set T(p) of taps of
// p that read a pixel of the image:
//   V_pj = I_pj + y R_p + d U_T(j),  I_pj = P_pj + m CW_T(j),
//   R_p = sum_{t in T(p)} (row_sum[o(p, t)] - C 2^(b-1) + C m),
//   CW_T(j) = sum_{t in T} sum_c w_ctj,  U_T(j) = CW_T(j) + |T| C y,
// and dX = inv_sw inv_s V.  For k = 3, pad 1 the sets T are the nine border
// classes of p (top / middle / bottom row times left / middle / right
// column); the class tables CW, U of a tile come from W~'s column sums.
// ---------------------------------------------------------------------------
#include <algorithm>

#include "fqt_gemm_core.cuh"

namespace fqt {

constexpr int kCvMaxA = 9;       // W~ tiles in shared memory (ring or resident)
constexpr int kCvWarpPar = 4, kCvWarpEpi = 8;
constexpr int kCvThreads = 512;  // TMA, MMA, (two idle,) four parameter warps,
                                 // two sets of four epilogue warps
constexpr int kCvClasses = 9;
constexpr int kCvCols = 256;     // pixel slots per tile

struct ConvXArgs {
  int n, h, w, cin, cout;
  int pitch, rows, imgs;   // slots per image row, rows and images per tile
  int img_slots;           // (rows + 2) pitch
  int ncols;               // MMA columns (a multiple of 16)
  int tiles_per_img, m_tiles;
  int64_t n_items;
  int cbs;                 // blocks of 64 output channels
  int resident, a_stages;  // W~ kept for the launch; else tiles in the ring
  uint32_t a_bytes;        // bytes of one W~ tile
  uint32_t b_bytes, b_stride;  // bytes of one dH tile, and its stage
  int og, ow;              // 2^(b-1) of Q_b2, of W~
  const float *inv_s, *zero;  // Q_b2: per row (per image constant) or one entry
  int per_tensor;
  const int32_t *row_sum;  // Q_b2 row sums (codes), one per output pixel
  const float *inv_sw, *zero_w;
  const int32_t *col_sum_w;
  float *out;              // NHWC n h w cin
  int *status;
};

// Shared memory after the dH stages and the W~ tiles, per epilogue set: the
// pixel terms (bp, Ad, sc, m) and (output offset, class) of 256 slots, and the
// class tables of the tile's 128 channels.
constexpr size_t kCvSetBytes = kCvCols * (16 + 8) + 2 * kCvClasses * 128 * 4;
constexpr size_t kCvTailBytes = 2 * kCvSetBytes + 64 * 8 + 16;

__device__ __forceinline__ int conv_class(int y, int x, int h, int w) {
  const int cy = y == 0 ? 0 : (y == h - 1 ? 2 : 1);
  const int cx = x == 0 ? 0 : (x == w - 1 ? 2 : 1);
  return cy * 3 + cx;
}

// CW_T(j) and U_T(j) of one input channel for the nine border classes of a
// 3 x 3 stride-1 pad-1 conv (T = the taps whose output pixel exists).
__device__ __forceinline__ void conv_class_terms(const ConvXArgs &g, int j, const ff &y,
                                                 float *cw_s, float *u_s) {
  int cs[9];
#pragma unroll
  for (int t = 0; t < 9; ++t) cs[t] = j < g.cin ? __ldg(g.col_sum_w + t * g.cin + j) : 0;
#pragma unroll
  for (int cls = 0; cls < kCvClasses; ++cls) {
    const int cy = cls / 3, cx = cls % 3;
    long long cw = 0;
    int taps = 0;
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const int ky = t / 3, kx = t % 3;
      // top row (cy 0): the tap ky = 2 reads output row -1; bottom: ky = 0
      if ((cy == 0 && ky == 2) || (cy == 2 && ky == 0)) continue;
      if ((cx == 0 && kx == 2) || (cx == 2 && kx == 0)) continue;
      cw += (long long)cs[t] - (long long)g.cout * g.ow;
      ++taps;
    }
    cw_s[cls * 128] = ll_to_float(cw);
    // U = CW + |T| C y, rounded once from float-float
    const ff tcy = ff_mul({(float)(taps * g.cout), 0.0f}, y);
    u_s[cls * 128] = ff_round(ff_add(ff_from_int(cw), tcy));
  }
}

struct ConvTile {
  int m0, img, y0;
};

__device__ __forceinline__ ConvTile conv_tile(const ConvXArgs &g, int64_t it) {
  ConvTile t;
  const int64_t pt = it / g.m_tiles;
  t.m0 = (int)(it - pt * g.m_tiles) * BM;
  if (g.imgs > 1) {
    t.img = (int)pt * g.imgs;
    t.y0 = 0;
  } else {
    t.img = (int)(pt / g.tiles_per_img);
    t.y0 = (int)(pt - (int64_t)t.img * g.tiles_per_img) * g.rows;
  }
  return t;
}

__global__ void __launch_bounds__(kCvThreads, 1)
    k_gradx_nhwc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const ConvXArgs g) {
  extern __shared__ __align__(1024) uint8_t cv_raw[];
  uint8_t *smem = cv_raw + ((1024u - (smem_u32(cv_raw) & 1023u)) & 1023u);
  uint8_t *bst = smem;                                  // two dH stages
  uint8_t *ast = bst + 2 * (size_t)g.b_stride;          // W~ tiles
  uint8_t *sets = ast + (size_t)g.a_stages * g.a_bytes;
  uint64_t *bars = reinterpret_cast<uint64_t *>(sets + 2 * kCvSetBytes);
  uint64_t *afull = bars, *aempty = afull + kCvMaxA, *bfull = aempty + kCvMaxA,
           *bempty = bfull + 2, *accf = bempty + 2, *acce = accf + 2, *pfull = acce + 2,
           *pempty = pfull + 2, *drain = pempty + 2;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 64);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kCvMaxA; ++i) {
      mbar_init(&afull[i], 1);
      mbar_init(&aempty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bfull[i], 1);
      mbar_init(&bempty[i], 1);
      mbar_init(&accf[i], 1);
      mbar_init(&acce[i], 4);  // the four warps of the set
      mbar_init(&pfull[i], 4);  // the four parameter warps
      mbar_init(&pempty[i], 4);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    // ---------------------------------------------------------------- producer
    if (lane == 0) {
      int as = 0, bs = 0;
      uint32_t aph = 0, bph = 0;
      if (g.resident) {  // one barrier for all of W~
        mbar_expect_tx(&afull[0], 9u * (uint32_t)g.cbs * g.a_bytes);
        for (int i = 0; i < 9 * g.cbs; ++i)
          tma_load_2d(ast + (size_t)i * g.a_bytes, &tmA, (i % 9) * g.cin, (i / 9) * 64,
                      &afull[0]);
      }
      for (int64_t it = blockIdx.x; it < g.n_items && !*abort_flag; it += gridDim.x) {
        const ConvTile t = conv_tile(g, it);
        bool ok = true;
        for (int cb = 0; ok && cb < g.cbs; ++cb) {
          ok = mbar_wait(&bempty[bs], bph ^ 1u, g.status);
          if (!ok) break;
          mbar_expect_tx(&bfull[bs], g.b_bytes);
          tma_load_4d(bst + (size_t)bs * g.b_stride, &tmB, cb * 64, -1, t.y0 - 1, t.img,
                      &bfull[bs]);
          if (++bs == 2) { bs = 0; bph ^= 1u; }
          for (int k = 0; !g.resident && k < 9; ++k) {
            ok = mbar_wait(&aempty[as], aph ^ 1u, g.status);
            if (!ok) break;
            mbar_expect_tx(&afull[as], g.a_bytes);
            uint8_t *sa = ast + (size_t)as * g.a_bytes;
            // two 64-wide MN atoms of 64 output channels
            tma_load_2d(sa, &tmA, t.m0 + k * g.cin, cb * 64, &afull[as]);
            tma_load_2d(sa + kTileBytes / 2, &tmA, t.m0 + 64 + k * g.cin, cb * 64, &afull[as]);
            if (++as == g.a_stages) { as = 0; aph ^= 1u; }
          }
        }
        if (!ok) { *abort_flag = 1; break; }
      }
      if (*abort_flag) {
        sleep_ns(200000);  // copies in flight land before the CTA exits
      } else {
        for (int i = 0; i < 2; ++i) {
          if (!mbar_wait(&bempty[bs], bph ^ 1u, g.status)) break;
          if (++bs == 2) { bs = 0; bph ^= 1u; }
        }
        for (int i = 0; !g.resident && i < g.a_stages; ++i) {
          if (!mbar_wait(&aempty[as], aph ^ 1u, g.status)) break;
          if (++as == g.a_stages) { as = 0; aph ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    // -------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      int as = 0, bs = 0;
      uint32_t aph = 0, bph = 0, accph = 0;
      const uint32_t idesc = make_idesc(true, false, BM, g.ncols);  // A MN-major, B K-major
      bool ok = !g.resident || mbar_wait(&afull[0], 0, g.status);
      int64_t local = 0;
      for (int64_t it = blockIdx.x; ok && it < g.n_items && !*abort_flag;
           it += gridDim.x, ++local) {
        const int buf = (int)(local & 1);
        ok = mbar_wait(&acce[buf], ((accph >> buf) & 1u) ^ 1u, g.status);
        if (!ok) break;
        tc_fence_after();
        const uint32_t dt = tmem + (uint32_t)(buf * kCvCols);
        for (int cb = 0; ok && cb < g.cbs; ++cb) {
          ok = mbar_wait(&bfull[bs], bph, g.status);
          if (!ok) break;
          const uint32_t b_addr = smem_u32(bst + (size_t)bs * g.b_stride);
          for (int t = 0; t < 9; ++t) {
            const int slot_a = g.resident ? cb * 9 + t : as;
            if (!g.resident) {
              ok = mbar_wait(&afull[as], aph, g.status);
              if (!ok) break;
            }
            tc_fence_after();
            const int shift = (2 - t / 3) * g.pitch + 2 - t % 3;
            const uint64_t da = sw128_desc_mn(smem_u32(ast + (size_t)slot_a * g.a_bytes),
                                              (uint32_t)(kTileBytes / 2), 1024);
            const uint64_t db = sw128_desc(b_addr + (uint32_t)shift * 128u);
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
              umma_f16(dt, da + (2048u >> 4) * k, db + 2 * k, idesc,
                       (cb > 0 || t > 0 || k > 0) ? 1u : 0u);
            if (!g.resident) {
              umma_commit(&aempty[as]);
              if (++as == g.a_stages) { as = 0; aph ^= 1u; }
            }
          }
          umma_commit(&bempty[bs]);
          if (++bs == 2) { bs = 0; bph ^= 1u; }
        }
        umma_commit(&accf[buf]);
        accph ^= 1u << buf;
      }
      if (!ok) *abort_flag = 1;
      umma_commit(drain);  // every MMA has completed before TMEM is released
      mbar_wait(drain, 0, g.status);
    }
  } else if (warp >= kCvWarpPar && warp < kCvWarpEpi) {
    // -------------------------------------------------------------- parameters
    // the pixel terms and class tables of tile `local` for set local & 1, one
    // tile of each set ahead of its epilogue
    const int st = threadIdx.x - kCvWarpPar * 32;  // 0 .. 127
    const float inv_sw = *g.inv_sw, zw = *g.zero_w;
    const ff yy = two_sum((float)g.ow, zw);
    const int C = g.cout;
    int last_m0[2] = {-1, -1};
    int64_t local = 0;
    for (int64_t it = blockIdx.x; it < g.n_items && !*abort_flag; it += gridDim.x, ++local) {
      const int set = (int)(local & 1);
      const bool got = mbar_wait(&pempty[set], (uint32_t)((local >> 1) & 1) ^ 1u, g.status);
      if (!__all_sync(0xffffffffu, got)) { *abort_flag = 1; break; }
      uint8_t *tab = sets + (size_t)set * kCvSetBytes;
      float4 *px_f = reinterpret_cast<float4 *>(tab);                  // [256] bp, Ad, sc, m
      int2 *px_i = reinterpret_cast<int2 *>(tab + kCvCols * 16);       // [256] offset, class
      const ConvTile t = conv_tile(g, it);
      for (int sl = st; sl < g.ncols; sl += 128) {
        const int im = sl / g.img_slots, in = sl - im * g.img_slots;
        const int r = in / g.pitch, x = in - r * g.pitch, y = t.y0 + r, img = t.img + im;
        float4 f = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        int2 oc = make_int2(-1, 0);
        if (x < g.w && r < g.rows && y < g.h && img < g.n) {
          // scalars of Q_b2 (one scale per image or per tensor)
          const int64_t prow = (int64_t)img * g.h * g.w;
          const float inv = g.per_tensor ? g.inv_s[0] : g.inv_s[prow];
          const float z = g.per_tensor ? g.zero[0] : g.zero[prow];
          int rs[9], taps = 0;
#pragma unroll
          for (int k = 0; k < 9; ++k) {
            const int oy = y + 1 - k / 3, ox = x + 1 - k % 3;
            const bool v = oy >= 0 && oy < g.h && ox >= 0 && ox < g.w;
            rs[k] = v ? __ldg(g.row_sum + prow + (int64_t)oy * g.w + ox) : 0;
            taps += v;
          }
          const float sc = __fmul_rn(inv_sw, inv);
          const ff xo = two_sum((float)g.og, z);
          const float m = rintf(xo.h);
          const float dd = ff_round(fast_two_sum(__fsub_rn(xo.h, m), xo.l));
          // sum over the taps of row_sum - C og + C m
          long long R = (long long)taps * ((long long)C * (long long)m - (long long)C * g.og);
#pragma unroll
          for (int k = 0; k < 9; ++k) R += rs[k];
          const ff Rf = ff_from_int(R);
          f = make_float4(__fmul_rn(sc, ff_round(ff_mul(Rf, yy))), __fmul_rn(sc, dd), sc, m);
          oc = make_int2(((im * g.h + r) * g.w + x) * g.cin, conv_class(y, x, g.h, g.w) * 128);
        }
        px_f[sl] = f;
        px_i[sl] = oc;
      }
      if (t.m0 != last_m0[set]) {  // the class tables of this tile's 128 channels
        float *cw_s = reinterpret_cast<float *>(tab + kCvCols * 24);   // [9][128]
        conv_class_terms(g, t.m0 + st, yy, cw_s + st, cw_s + kCvClasses * 128 + st);
        last_m0[set] = t.m0;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&pfull[set]);
    }
  } else if (warp >= kCvWarpEpi) {
    // ---------------------------------------------------------------- epilogue
    // set s owns accumulator s and the tiles local = s, s + 2, ...; warp q
    // of the set reads TMEM lanes 32 q .. 32 q + 31 (input channels)
    const int set = (warp - kCvWarpEpi) >> 2, q = warp & 3;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(set * kCvCols);
    const uint8_t *tab = sets + (size_t)set * kCvSetBytes;
    const float4 *px_f = reinterpret_cast<const float4 *>(tab);
    const int2 *px_i = reinterpret_cast<const int2 *>(tab + kCvCols * 16);
    const int jl = q * 32 + lane;
    const float *cw_j = reinterpret_cast<const float *>(tab + kCvCols * 24) + jl;
    const float *u_j = cw_j + kCvClasses * 128;
    for (int64_t local = set;; local += 2) {
      const int64_t it = (int64_t)blockIdx.x + local * (int64_t)gridDim.x;
      if (it >= g.n_items || *abort_flag) break;
      const ConvTile t = conv_tile(g, it);
      const uint32_t par = (uint32_t)((local >> 1) & 1);  // this set's earlier tiles
      const bool got = mbar_wait(&pfull[set], par, g.status) &&
                       mbar_wait(&accf[set], par, g.status);
      if (!__all_sync(0xffffffffu, got)) { *abort_flag = 1; break; }
      tc_fence_after();
      if (t.m0 + q * 32 < g.cin) {  // warp-uniform (cin % 32 == 0)
        float *out = g.out + ((int64_t)t.img * g.h + t.y0) * g.w * g.cin + t.m0 + jl;
        // eight pixels per step, their terms loaded before any is used, so
        // that the shared-memory latencies overlap
#pragma unroll 1
        for (int c0 = 0; c0 < g.ncols; c0 += 8) {
          uint32_t v[8];
          tmem_ld8_nw(lane_base + (uint32_t)c0, v);
          int2 oc[8];
          float4 f[8];
          float cw[8], u[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            oc[i] = px_i[c0 + i];
            f[i] = px_f[c0 + i];
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            cw[i] = cw_j[oc[i].y];
            u[i] = u_j[oc[i].y];
          }
          tmem_wait_ld(v);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float I = __fmaf_rn(f[i].w, cw[i], __uint_as_float(v[i]));
            const float o = __fmaf_rn(f[i].z, I, __fmaf_rn(f[i].y, u[i], f[i].x));
            if (oc[i].x >= 0) __stcs(out + oc[i].x, o);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&acce[set]);
        mbar_arrive(&pempty[set]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
}

// dH carriers as (c, w, h, n): boxes of 64 channels x pitch x (rows + 2) x
// images, 128-byte swizzle, one 128-byte row per pixel slot.
static bool make_map_f16_tile(CUtensorMap *m, const void *base, uint64_t n, uint64_t h,
                              uint64_t w, uint64_t c, const ConvXArgs &g) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[4] = {c, w, h, n};
  cuuint64_t strides[3] = {c * 2, w * c * 2, h * w * c * 2};
  cuuint32_t box[4] = {64, (cuuint32_t)g.pitch, (cuuint32_t)(g.rows + 2), (cuuint32_t)g.imgs};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void *>(base), dims, strides,
            box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The tile of a geometry: as many rows (then whole images) as fit 256 columns
// and the dH stages, evened out over the image's tiles.  A slot past the
// columns' end may be read as an operand row (its column is unused): the W~
// tiles that follow the stages keep that inside shared memory.
static size_t conv_geometry(ConvXArgs &g) {
  const size_t total = 227 * 1024 - 1024 - kCvTailBytes;
  g.cbs = g.cout / 64;
  g.m_tiles = (g.cin + BM - 1) / BM;
  g.resident = g.cin <= 64 && g.cbs == 1;
  g.a_bytes = (uint32_t)(g.resident ? kTileBytes / 2 : kTileBytes);
  g.a_stages = g.resident ? 9 : 4;
  const size_t budget = (total - (size_t)g.a_stages * g.a_bytes) / 2 / 1024 * 1024;
  g.pitch = g.w + 2;
  const size_t row = (size_t)g.pitch * 128;
  int r = 1;
  while (r < g.h && r * g.pitch + g.w <= kCvCols && (r + 3) * row <= budget) ++r;
  if ((r + 2) * row > budget) return 0;
  g.tiles_per_img = (g.h + r - 1) / r;
  g.rows = (g.h + g.tiles_per_img - 1) / g.tiles_per_img;
  g.img_slots = (g.rows + 2) * g.pitch;
  g.imgs = 1;
  if (g.tiles_per_img == 1)
    while (g.imgs < g.n && g.imgs * g.img_slots + (g.rows - 1) * g.pitch + g.w <= kCvCols &&
           (g.imgs + 1) * (size_t)(g.rows + 2) * row <= budget)
      ++g.imgs;
  const int cols = (g.imgs - 1) * g.img_slots + (g.rows - 1) * g.pitch + g.w;
  g.ncols = (cols + 15) / 16 * 16;
  g.b_bytes = (uint32_t)((size_t)g.imgs * (g.rows + 2) * row);
  g.b_stride = (g.b_bytes + 1023u) / 1024u * 1024u;
  g.n_items = g.imgs > 1 ? (int64_t)((g.n + g.imgs - 1) / g.imgs)
                         : (int64_t)g.n * g.tiles_per_img;
  g.n_items *= g.m_tiles;
  return 1024 + 2 * (size_t)g.b_stride + (size_t)g.a_stages * g.a_bytes + kCvTailBytes;
}

// The status word is all that is used.  An earlier kernel kept two class tables
// of C_in floats here; callers allocate, and smaller workspaces are refused, as
// for it.
size_t conv_grad_x_ws_bytes(int64_t cin) {
  return kGemmOffset + 2 * (size_t)kCvClasses * (size_t)(cin > 0 ? cin : 0) * sizeof(float) + 256;
}

fqt_status conv_grad_x_nhwc(const fqt_qtensor *q2, const fqt_qtensor *qw, int64_t n, int64_t h,
                            int64_t w, int64_t cin, int k, int pad, float *out, void *ws,
                            size_t ws_bytes, cudaStream_t st) {
  if (!q2 || !qw || !out || n <= 0 || h <= 0 || w <= 0 || cin <= 0) return FQT_EINVAL;
  if (!q2->codes_f16 || !q2->row_sum || !q2->inv_s || !q2->zero || !qw->codes_f16 ||
      !qw->col_sum || !qw->inv_s || !qw->zero)
    return FQT_EINVAL;
  if (k != 3 || pad != 1 || h < 2 || w < 2 || w > 128) return FQT_EUNSUPPORTED;
  const int64_t cout = q2->cols;
  if (q2->rows != n * h * w || qw->rows != cout || qw->cols != 9 * cin) return FQT_EINVAL;
  if (cout % 64 || cin % 32) return FQT_EUNSUPPORTED;
  const bool per_tensor = q2->kind == FQT_PTQ;
  if (!per_tensor && !(q2->kind == FQT_PSQ && q2->rows_per_sample == h * w))
    return FQT_EUNSUPPORTED;  // the scale must be constant over every image's pixels
  if (qw->kind != FQT_PTQ || q2->conv[0] || qw->conv[0]) return FQT_EUNSUPPORTED;
  if (9 * cout > (int64_t)exact_chunk_blocks(q2->bits, qw->bits) * BK) return FQT_EUNSUPPORTED;
  if (!aligned16(q2->codes_f16) || !aligned16(qw->codes_f16) || !aligned16(out))
    return FQT_EINVAL;
  if (!ws || ((uintptr_t)ws & 255) || ws_bytes < conv_grad_x_ws_bytes(cin))
    return FQT_EWORKSPACE;
  ConvXArgs g;
  memset(&g, 0, sizeof(g));
  g.n = (int)n;
  g.h = (int)h;
  g.w = (int)w;
  g.cin = (int)cin;
  g.cout = (int)cout;
  const size_t smem = conv_geometry(g);
  if (smem == 0) return FQT_EUNSUPPORTED;
  CUtensorMap ta, tb;
  bool ok = make_map_f16(&ta, qw->codes_f16, (uint64_t)(9 * cin), (uint64_t)cout, 64, BK);
  ok = ok && make_map_f16_tile(&tb, q2->codes_f16, (uint64_t)n, (uint64_t)h, (uint64_t)w,
                               (uint64_t)cout, g);
  if (!ok) return cuda_fail(cudaErrorInvalidValue, "tensor map encode");
  g.og = 1 << (q2->bits - 1);
  g.ow = 1 << (qw->bits - 1);
  g.inv_s = q2->inv_s;
  g.zero = q2->zero;
  g.per_tensor = per_tensor ? 1 : 0;
  g.row_sum = q2->row_sum;
  g.inv_sw = qw->inv_s;
  g.zero_w = qw->zero;
  g.col_sum_w = qw->col_sum;
  g.out = out;
  g.status = reinterpret_cast<int *>(ws);
  const cudaError_t e =
      cudaFuncSetAttribute(k_gradx_nhwc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return cuda_fail(e, "conv grad_X shared-memory attribute");
  const int nsm = device_sm_count();
  const int64_t grid = g.n_items < nsm ? g.n_items : nsm;
  k_gradx_nhwc<<<(int)grid, kCvThreads, smem, st>>>(ta, tb, g);
  return cuda_fail(cudaGetLastError(), "conv grad_X launch");
}

// ---------------------------------------------------------------------------
// Border sums of a 3 x 3, pad 1, stride 1 conv operand (fp16 carriers of
// n x h x w pixels, h, w >= 2): the sums over the top and bottom rows and the
// left and right columns, per channel, and what the nine taps make of them.
//   pad_a (grad_W's padding correction, layout [9][c]): tap (ky, kx) reads
//     padding from the top (ky = 0) or bottom (ky = 2) output row and the left
//     (kx = 0) or right (kx = 2) column: row + column - corner.
//   col_sum (the im2col column sums of X~, layout [9][c]): tap (ky, kx) reads
//     every input pixel but the bottom (ky = 0) or top (ky = 2) row and the
//     right (kx = 0) or left (kx = 2) column: total - row - column + corner,
//     plus code(0) for every padding entry.  The centre tap's slot holds the
//     total when the kernel starts (the code pass sums it in registers), and
//     the first CTA of a channel group adds it and the constants to the
//     other eight.
// A thread owns one channel oct of one line, sums its pixels in registers
// (eight loads in flight; corners are the first and last pixel of a row) and
// meets the others in shared memory once; the kernels this replaces on 3 x 3
// convs went through shared-memory atomics per border pixel and formed every
// tap from nine classes in every CTA, one of them after reading all pixels:
// 20.5 and 19.6 us (256 x 14 x 14 x 256), 14.7 and 26.5 us (256 x 56 x 56 x
// 64); now 7.2 and 6.6 us, 6.5 and 6.3 us.  What is left is latency: the launch,
// one round of loads and the sums' atomics.
// ---------------------------------------------------------------------------
constexpr int kLineOcts = 64;  // channel octs per CTA

__global__ void __launch_bounds__(256) k_conv_lines(const uint16_t *__restrict__ f16, int C,
                                                    int64_t nimg, int imgs_per_cta, int h, int w,
                                                    int32_t *pad_a, int32_t *col_sum,
                                                    int centre) {
  __shared__ int sum_s[8 * kLineOcts * 8];  // top, bottom, left, right, TL, TR, BL, BR
  const int ch0 = (int)blockIdx.y * kLineOcts * 8;
  const int octs = min(kLineOcts, (C - ch0) / 8), nch = octs * 8;
  const int lanes = 256 / octs / 4;  // per line
  const int o = (int)threadIdx.x % octs, g = (int)threadIdx.x / octs;
  const int line = g & 3, l0 = g >> 2;
  const int64_t img0 = (int64_t)blockIdx.x * imgs_per_cta;
  const int nim = (int)min((int64_t)imgs_per_cta, nimg - img0);
  for (int i = threadIdx.x; i < 8 * nch; i += blockDim.x) sum_s[i] = 0;
  __syncthreads();
  if (l0 < lanes) {
    const uint16_t *base = f16 + img0 * h * (int64_t)w * C + ch0 + o * 8;
    const int len = line < 2 ? w : h;
    const int64_t first = line == 1 ? (int64_t)(h - 1) * w : line == 3 ? w - 1 : 0;
    const int64_t step = line < 2 ? 1 : w;
    int acc[8], ca[8], cz[8];  // the line, its first and its last pixels
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = ca[j] = cz[j] = 0;
    const int items = nim * len;
    for (int i0 = l0; i0 < items; i0 += 8 * lanes) {
      uint4 v[8];
      int px[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int it = i0 + u * lanes, im = it / len;
        px[u] = it < items ? it - im * len : -1;
        v[u] = make_uint4(0u, 0u, 0u, 0u);
        if (px[u] >= 0)
          v[u] = __ldg(reinterpret_cast<const uint4 *>(
              base + ((int64_t)im * h * w + first + px[u] * step) * C));
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint32_t w4[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
        const bool fa = px[u] == 0, fz = px[u] == len - 1;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&w4[q]));
          const int a = (int)f.x, b = (int)f.y;
          acc[2 * q] += a;
          acc[2 * q + 1] += b;
          if (fa) { ca[2 * q] += a; ca[2 * q + 1] += b; }
          if (fz) { cz[2 * q] += a; cz[2 * q + 1] += b; }
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (acc[j]) atomicAdd(&sum_s[line * nch + o * 8 + j], acc[j]);
      if (line < 2 && ca[j]) atomicAdd(&sum_s[(4 + 2 * line) * nch + o * 8 + j], ca[j]);
      if (line < 2 && cz[j]) atomicAdd(&sum_s[(5 + 2 * line) * nch + o * 8 + j], cz[j]);
    }
  }
  __syncthreads();
  const int64_t c9 = 9 * (int64_t)C;
  const int code0 = col_sum ? col_sum[c9] : 0;
  for (int ch = threadIdx.x; ch < nch; ch += blockDim.x) {
    int s[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) s[k] = sum_s[k * nch + ch];
    const int total = col_sum && blockIdx.x == 0 ? col_sum[4 * (int64_t)C + ch0 + ch] : 0;
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      if (t == 4) continue;
      const int ky = t / 3, kx = t % 3;
      // pad_a: the row (column) on the tap's own side; col_sum: the opposite
      const int flip = col_sum ? 1 : 0;
      const int ri = (ky >> 1) ^ flip, ci = (kx >> 1) ^ flip;  // 0 top / left, 1 bottom / right
      int v = 0;
      if (ky != 1) v += s[ri];
      if (kx != 1) v += s[2 + ci];
      if (ky != 1 && kx != 1) v -= s[4 + 2 * ri + ci];
      if (col_sum) {
        v = -v;
        if (blockIdx.x == 0) {
          const int64_t npad = nimg * ((ky != 1 ? w : 0) + (kx != 1 ? h : 0) -
                                       (ky != 1 && kx != 1 ? 1 : 0));
          v += total + (int)(npad * (code0 - centre));
        }
        if (v) atomicAdd(&col_sum[(int64_t)t * C + ch0 + ch], v);
      } else if (v) {
        atomicAdd(&pad_a[(int64_t)t * C + ch0 + ch], v);
      }
    }
  }
}

bool conv_lines_supported(int h, int w, int C, int kh, int kw, int pad) {
  return kh == 3 && kw == 3 && pad == 1 && h > 1 && w > 1 && C % 8 == 0;
}

// pad_a != NULL: the padding sums of Q_b1's carriers (h x w output pixels);
// else the column sums of X~ (col_sum, its centre tap holding the totals, the
// others 0, code(0) behind the ninth).
fqt_status launch_conv_lines(const uint16_t *f16, int64_t n, int h, int w, int C, int32_t *pad_a,
                             int32_t *col_sum, int centre, cudaStream_t st) {
  // about eight pixels of a line per thread
  const int octs = std::min(C / 8, kLineOcts), lanes = 256 / octs / 4;
  const int ipc = (int)std::min<int64_t>(std::max(1, 8 * lanes / std::max(h, w)), n);
  const dim3 grid((unsigned)((n + ipc - 1) / ipc),
                  (unsigned)((C / 8 + kLineOcts - 1) / kLineOcts));
  k_conv_lines<<<grid, 256, 0, st>>>(f16, C, n, ipc, h, w, pad_a, col_sum, centre);
  return cuda_fail(cudaGetLastError(), "conv border sums launch");
}

}  // namespace fqt
