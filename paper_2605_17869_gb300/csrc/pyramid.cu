// Gaussian scale space (§3.2, "GPU Pipeline Stages"): the launches of the level
// blurs (blur.cuh), the 2x magnified first octave (k_base_poly, a polyphase
// filter of the input, below) and the pyramid export.
#include "blur.cuh"

namespace sift {

namespace {

constexpr int kGenThreads = 320;  // k_base_generic

// Rows [y0 - R, y0 + rows - R) x columns [x0 - 16, x0 + 144) of the 2x bilinear
// magnification of the input:
// u[2k] = I[k], u[2k+1] = (I[k] + I[k+1]) / 2 (last sample clamped), rows of
// the magnified image formed after its columns.
__device__ __forceinline__ void stage_upsampled(const float *__restrict__ src, int spitch, int h,
                                                int w, int x0, int y0, int R, int rows,
                                                float *s_in) {
  const int H = 2 * h, W = 2 * w;
  const int xb = x0 - kBlurHalo;
  for (int idx = threadIdx.x; idx < rows * kSinW; idx += kGenThreads) {
    const int r = idx / kSinW, c = idx - r * kSinW;
    const int gy = refl101(y0 - R + r, H);
    const int iy = gy >> 1, fy = gy & 1;
    const int iy1 = min(iy + 1, h - 1);
    const float *ra = src + (long long)iy * spitch;
    const float *rb = src + (long long)iy1 * spitch;
    const int gx = refl101(xb + c, W);
    const int ix = gx >> 1, fx = gx & 1;
    const int ix1 = min(ix + 1, w - 1);
    const float a = __ldg(ra + ix);
    float v;
    if (!fy) {
      v = fx ? 0.5f * (a + __ldg(ra + ix1)) : a;
    } else {
      const float c0 = __ldg(rb + ix);
      v = fx ? 0.5f * (0.5f * (a + __ldg(ra + ix1)) + 0.5f * (c0 + __ldg(rb + ix1)))
             : 0.5f * (a + c0);
    }
    s_in[idx] = v;
  }
}

// The same output from scalar operations, for the generic kernel: row points
// at the output's first tap column s, odd tells the parity of s. Radius 0 has one
// tap only (the chains below take at least three).
__device__ __forceinline__ float row_tap_sum(const float *row, bool odd, int R, const float *w) {
  if (R == 0) return __fmul_rn(w[0], row[0]);
  float ax, ay;
  if (!odd) {
    ax = __fmul_rn(w[0], row[0]);
    ay = __fmul_rn(w[1], row[1]);
    for (int i = 1; i < R; i++) {
      ax = fmaf(w[2 * i], row[2 * i], ax);
      ay = fmaf(w[2 * i + 1], row[2 * i + 1], ay);
    }
    return __fadd_rn(fmaf(w[2 * R], row[2 * R], ax), ay);
  }
  ax = __fmul_rn(w[1], row[1]);
  ay = __fmul_rn(w[2], row[2]);
  for (int i = 1; i < R; i++) {
    ax = fmaf(w[2 * i + 1], row[2 * i + 1], ax);
    ay = fmaf(w[2 * i + 2], row[2 * i + 2], ay);
  }
  return __fadd_rn(fmaf(w[0], row[0], ax), ay);
}

// The base blur without a specialised kernel: the magnified input at radii
// that k_base_poly is not instantiated for (MODE 2), and radius 0 (MODE 1).
// Tiles of 128 x 32 outputs, the per-output order of operations of k_blur,
// plain loops.
template <int MODE>
__global__ void __launch_bounds__(kGenThreads) k_base_generic(const Desc *__restrict__ d, int R, BlurTaps tp) {
  pdl_trigger();
  pdl_wait();
  constexpr int TH = 32;
  const int ROWS = TH + 2 * R;
  extern __shared__ float4 smem4[];
  float *s_in = reinterpret_cast<float *>(smem4);
  float *s_v = s_in + ROWS * kSinW;
  const int n = d->n_img;
  const int *pre = d->base_pre[MODE - 1];
  const int total = pre[n];
  for (int t = blockIdx.x; t < total; t += gridDim.x) {
    const int b = find_owner(pre, n, t);
    const ImgDev &im = d->img[b];
    const OctDev od = d->oct[im.oct0];
    const int tiles_x = (od.W + kBlurTW - 1) / kBlurTW;
    const int lt = t - pre[b];
    const int ty = lt / tiles_x, tx = lt - ty * tiles_x;
    const int x0 = tx * kBlurTW, y0 = ty * TH;
    float *out = d->pyr + od.lvl;
    if (MODE == 1) {
      for (int idx = threadIdx.x; idx < ROWS * kSinW; idx += kGenThreads) {
        const int r = idx / kSinW, c = idx - r * kSinW;
        s_in[idx] = im.src[(long long)refl101(y0 - R + r, od.H) * im.spitch + refl101(x0 - kBlurHalo + c, od.W)];
      }
    } else {
      stage_upsampled(im.src, im.spitch, im.H, im.W, x0, y0, R, ROWS, s_in);
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < TH * kSinW; idx += kGenThreads) {
      const int v = idx / kSinW, c = idx - v * kSinW;
      float acc = tp.w[0] * s_in[v * kSinW + c];
      for (int j = 1; j <= 2 * R; j++) acc = fmaf(tp.w[j], s_in[(v + j) * kSinW + c], acc);
      s_v[idx] = acc;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < TH * kBlurTW; idx += kGenThreads) {
      const int v = idx / kBlurTW, k = idx - v * kBlurTW;
      const int y = y0 + v, x = x0 + k;
      const int sc = kBlurHalo + k - R;  // first tap column; its parity is that of x - R
      const float acc = row_tap_sum(s_v + v * kSinW + sc, (sc & 1) != 0, R, tp.w);
      if (y < od.H && x < od.pitch) out[(long long)y * od.pitch + x] = acc;
    }
    __syncthreads();
  }
}

int generic_smem_bytes(int R) { return (2 * 32 + 2 * R) * kSinW * (int)sizeof(float); }

// ------------------------------------------------- magnified base, polyphase
//
// The base level of a magnified first octave is G = g * U(I): U the 2x bilinear
// magnification (u[2k] = I[k], u[2k+1] = (I[k] + I[k+1]) / 2, last sample
// clamped), g the base Gaussian with reflect-101 on the magnified grid. Both
// are linear, so output sample 2k + p (p = 0, 1) of a row is a 2Q + 1 tap
// filter c_p of the input around k, with c_p[q] = sum_t g[t] * (weight of
// I[k + q] in u[2k + p + t]), Q = (R + 2) / 2. The reflection and the clamp
// are exact on an extended input I_e[i] = I[refl101(2i, 2n) / 2]
// (reflect-101 on the left, half-sample symmetric on the right, which is what
// the magnified grid's reflection maps back to). A tile of 128 x 32 outputs
// stages (64 + 2Q) x (16 + 2Q) input samples, filters its rows into 128
// columns at input-row resolution, then its columns into 32 rows: about 12
// FMAs per output against 22 for the two passes on the magnified grid, and no
// magnified window. Each output is the same fixed chain (sum over q
// ascending, rows then columns) whatever the tile.
constexpr int kPolyThreads = 256;
constexpr int kPolyMaxQ = kMaxR / 2 + 1;

struct PolyTaps {
  float c[2][2 * kPolyMaxQ + 1];
};

struct PolyTile {
  const float *src;
  float *out;
  int spitch, pitch, H, W, sh, sw, x0, y0;
};
__device__ __forceinline__ PolyTile poly_tile(const Desc *__restrict__ d, const int *pre, int t) {
  PolyTile g;
  const int b = find_owner(pre, d->n_img, t);
  const OctDev od = d->oct[b * kMaxOct];
  const ImgDev &im = d->img[b];
  g.src = im.src;
  g.spitch = im.spitch;
  g.sh = im.H;
  g.sw = im.W;
  g.out = d->pyr + od.lvl;
  g.pitch = od.pitch;
  g.H = od.H;
  g.W = od.W;
  const int tiles_x = (od.W + kBlurTW - 1) / kBlurTW;
  const int lt = t - pre[b];
  const int ty = lt / tiles_x, tx = lt - ty * tiles_x;
  g.x0 = tx * kBlurTW;
  g.y0 = ty * kBaseTileRows;
  return g;
}

template <int Q>
__global__ void __launch_bounds__(kPolyThreads) k_base_poly(const Desc *__restrict__ d, PolyTaps pt) {
  constexpr int NR = 16 + 2 * Q, NC = 64 + 2 * Q, NT = 2 * Q + 1;
  __shared__ float sI[NR * NC];
  __shared__ __align__(16) float sH[NR * kBlurTW];
  const int *pre = d->base_pre[1];
  const int total = pre[d->n_img];
  const int G = gridDim.x;
  for (int t = blockIdx.x; t < total; t += G) {
    if (t + G >= total) pdl_trigger();  // successors launch during this block's last tile
    const PolyTile g = poly_tile(d, pre, t);
    const int kx0 = g.x0 >> 1, ky0 = g.y0 >> 1;
    const int iyb = ky0 - Q, ixb = kx0 - Q;
    if (iyb >= 0 && iyb + NR <= g.sh && ixb >= 0 && ixb + NC <= g.sw) {
      // Interior: the window needs no reflection; warp w copies rows w, w + 8, ...
      const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
      for (int r = warp; r < NR; r += kPolyThreads / 32) {
        const float *srow = g.src + (long long)(iyb + r) * g.spitch + ixb;
        for (int c = lane; c < NC; c += 32) cp_async4(sI + r * NC + c, srow + c);
      }
    } else {
      for (int idx = threadIdx.x; idx < NR * NC; idx += kPolyThreads) {
        const int r = idx / NC, c = idx - r * NC;
        const int iy = refl101(2 * (iyb + r), g.H) >> 1;
        const int ix = refl101(2 * (ixb + c), g.W) >> 1;
        cp_async4(sI + idx, g.src + (long long)iy * g.spitch + ix);
      }
    }
    cp_async_wait_all();
    __syncthreads();
    // Rows: outputs 2j and 2j + 1 of input row r share the taps sI[r][j .. j + 2Q].
    for (int idx = threadIdx.x; idx < NR * (kBlurTW / 2); idx += kPolyThreads) {
      const int r = idx / (kBlurTW / 2), j = idx - r * (kBlurTW / 2);
      const float *row = sI + r * NC + j;
      float a = 0.f, b = 0.f;
#pragma unroll
      for (int q = 0; q < NT; q++) {
        const float v = row[q];
        a = fmaf(pt.c[0][q], v, a);
        b = fmaf(pt.c[1][q], v, b);
      }
      *reinterpret_cast<float2 *>(sH + r * kBlurTW + 2 * j) = make_float2(a, b);
    }
    __syncthreads();
    // Columns: output rows 2j and 2j + 1 of a 4-column group share the taps
    // sH[j .. j + 2Q][4 g4 .. 4 g4 + 3].
    for (int idx = threadIdx.x; idx < 16 * (kBlurTW / 4); idx += kPolyThreads) {
      const int j = idx / (kBlurTW / 4), g4 = idx - j * (kBlurTW / 4);
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
#pragma unroll
      for (int q = 0; q < NT; q++) {
        const float4 v = *reinterpret_cast<const float4 *>(sH + (j + q) * kBlurTW + 4 * g4);
        const float c0 = pt.c[0][q], c1 = pt.c[1][q];
        a.x = fmaf(c0, v.x, a.x);
        a.y = fmaf(c0, v.y, a.y);
        a.z = fmaf(c0, v.z, a.z);
        a.w = fmaf(c0, v.w, a.w);
        b.x = fmaf(c1, v.x, b.x);
        b.y = fmaf(c1, v.y, b.y);
        b.z = fmaf(c1, v.z, b.z);
        b.w = fmaf(c1, v.w, b.w);
      }
      const int X = g.x0 + 4 * g4, Y = g.y0 + 2 * j;
#pragma unroll
      for (int p = 0; p < 2; p++) {
        if (Y + p >= g.H) break;
        const float4 v = p ? b : a;
        float *o = g.out + (long long)(Y + p) * g.pitch + X;
        if (X + 3 < g.W) {
          *reinterpret_cast<float4 *>(o) = v;
        } else {
          if (X < g.W) o[0] = v.x;
          if (X + 1 < g.W) o[1] = v.y;
          if (X + 2 < g.W) o[2] = v.z;
        }
      }
    }
    __syncthreads();  // the next tile reuses sI and sH
  }
}

PolyTaps make_poly_taps(const BlurTaps &t, int R) {
  const int Q = (R + 2) / 2;
  PolyTaps p{};
  for (int ph = 0; ph < 2; ph++)
    for (int q = -Q; q <= Q; q++) {
      double c = 0.0;
      for (int tt = -R; tt <= R; tt++) {
        const int n = ph + tt;  // magnified offset from 2k
        double w = 0.0;
        if ((n & 1) == 0) w = (n / 2 == q) ? 1.0 : 0.0;
        else w = ((n - 1) / 2 == q || (n + 1) / 2 == q) ? 0.5 : 0.0;
        c += (double)t.w[tt + R] * w;
      }
      p.c[ph][q + Q] = (float)c;
    }
  return p;
}

}  // namespace


#define SIFT_FOR_EACH_POLY_R(X) X(5) X(7) X(8) X(10) X(13)

namespace {

// The radii of three scales per octave at sigma0 1.6, the base blurs' among them, are
// in this unit. A unit's code is loaded when the first of its kernels is asked for, which
// takes some 0.4 ms and more the larger it is, and each kernel 6 us on top. With the
// radii spread over four units of their own, a process's first sift_create took 3.7 ms
// (three units) against 2.6 now, its first sift_extract_noalloc 4.0 against 3.35 (2.35
// when one kernel with a runtime radius served the other radii).
BlurFn blur_fn(int R, int variant) {
  const bool rows64 = variant == BV_LVL64 || variant == BV_DEC64;
  switch (R) {
    case 5: return rows64 ? blur_instance64<5>(variant) : blur_instance<5>(variant);
    case 7: return rows64 ? blur_instance64<7>(variant) : blur_instance<7>(variant);
    case 8: return rows64 ? blur_instance64<8>(variant) : blur_instance<8>(variant);
    case 10: return rows64 ? blur_instance64<10>(variant) : blur_instance<10>(variant);
    case 13: return rows64 ? blur_instance64<13>(variant) : blur_instance<13>(variant);
    default: return rows64 ? blur_rest64(R, variant) : blur_rest(R, variant);
  }
}

int level_variant(int th_kind, bool m3, int storage) {
  if (storage == 1) return BV_DEC_R16;
  if (storage == 2) return m3 ? BV_DEC_H16 : BV_LVL_H16;
  if (th_kind == TK_BLUR64) return m3 ? BV_DEC64 : BV_LVL64;
  return m3 ? BV_DEC : BV_LVL;
}

cudaError_t launch_fn(const BlurFn &f, int grid, cudaStream_t s, bool pdl, const Desc *d, int oct,
                      int lvl, const BlurTaps &t) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = kThreads;
  cfg.dynamicSmemBytes = f.smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  if (pdl) {
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
  void *args[] = {&d, &oct, &lvl, const_cast<BlurTaps *>(&t)};
  return cudaLaunchKernelExC(&cfg, f.fn, args);
}

}  // namespace

int blur_tile_rows(int th_kind) { return tile_rows(th_kind); }

cudaError_t blur_set_attributes(unsigned radii, bool h16, bool rows64) {
  cudaError_t e = cudaSuccess;
  for (int R = 1; R <= kMaxR && e == cudaSuccess; R++)
    for (int v = (radii >> R & 1) ? 0 : BV_COUNT; v < BV_COUNT && e == cudaSuccess; v++) {
      if (!h16 && (v == BV_LVL_H16 || v == BV_DEC_R16 || v == BV_DEC_H16)) continue;
      if (!rows64 && (v == BV_LVL64 || v == BV_DEC64)) continue;
      const BlurFn f = blur_fn(R, v);
      e = cudaFuncSetAttribute(f.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, f.smem);
    }
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_base_generic<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, generic_smem_bytes(kMaxR));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_base_generic<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, generic_smem_bytes(kMaxR));
  return e;
}

cudaError_t launch_level_blur(const Desc *d, int oct, int lvl_out, int R, const BlurTaps &t,
                              int th_kind, int grid, cudaStream_t s, bool from_prev_octave,
                              bool pdl, int storage) {
  if (R < 1 || R > kMaxR || (storage != 0 && (th_kind == TK_BLUR64 || storage > 2 || (storage == 1 && !from_prev_octave))))
    return cudaErrorInvalidValue;  // binary16 octaves use the smaller tile
  // A programmatic dependent of the previous kernel on s, or (pdl false) a plain
  // launch that waits for everything before it (a branch after an event wait).
  return launch_fn(blur_fn(R, level_variant(th_kind, from_prev_octave, storage)), grid, s, pdl, d, oct, lvl_out, t);
}

namespace {
// The whole pyramid of image 0 copied out as dense H x W FP32 planes (binary16
// levels widened), octave by octave, level by level: a warp copies rows, 16 bytes
// per lane where the output row allows it, four loads in flight. One launch: it was
// one per level, 42 of them for 1920 x 1080, and the host's launches were the
// call's bound.
__global__ void __launch_bounds__(256) k_export(const Desc *__restrict__ d, float *__restrict__ out) {
  const int n_oct = d->img[0].n_oct, L = d->n_scales + 3;
  const int lane = threadIdx.x & 31;
  int o = 0, first = 0;  // octave of row r and its first row
  long long off = 0;     // the octave's offset in `out`
  OctDev od = d->oct[d->img[0].oct0];
  for (int r = blockIdx.x * 8 + (threadIdx.x >> 5);; r += gridDim.x * 8) {
    while (r - first >= L * od.H) {
      first += L * od.H;
      off += (long long)L * od.H * od.W;
      if (++o >= n_oct) return;
      od = d->oct[d->img[0].oct0 + o];
    }
    const int rr = r - first, l = rr / od.H, y = rr - l * od.H;
    const long long se = (long long)l * od.lstride + (long long)y * od.pitch;
    float *dst = out + off + (long long)rr * od.W;
    const float *lv = d->pyr + od.lvl;
    if (od.half) {
      const __half *src = reinterpret_cast<const __half *>(lv) + se;
#pragma unroll 4
      for (int c = lane; c < od.W; c += 32) dst[c] = __half2float(src[c]);
    } else if ((od.W & 3) == 0 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
      const float4 *src = reinterpret_cast<const float4 *>(lv + se);
#pragma unroll 4
      for (int c = lane; c < od.W / 4; c += 32) reinterpret_cast<float4 *>(dst)[c] = src[c];
    } else {
      const float *src = lv + se;
#pragma unroll 4
      for (int c = lane; c < od.W; c += 32) dst[c] = src[c];
    }
  }
}
}  // namespace

cudaError_t launch_export(const Desc *d, float *out, int n_sm, cudaStream_t s) {
  return launch_plain(k_export, n_sm * 8, 256, 0, s, d, out);
}

cudaError_t launch_base_blur(const Desc *d, int R, const BlurTaps &t, bool upsample, int grid,
                             cudaStream_t s) {
  if (!upsample && R > 0) return launch_fn(blur_fn(R, BV_BASE), grid, s, false, d, 0, 0, t);
#define CASE_R(RR) \
  case RR: return launch_plain(k_base_poly<(RR + 2) / 2>, grid, kPolyThreads, 0, s, d, make_poly_taps(t, RR));
  if (upsample) switch (R) {
      SIFT_FOR_EACH_POLY_R(CASE_R)
      default: return launch_plain(k_base_generic<2>, grid, kGenThreads, generic_smem_bytes(R), s, d, R, t);
    }
#undef CASE_R
  return launch_plain(k_base_generic<1>, grid, kGenThreads, generic_smem_bytes(R), s, d, R, t);
}

int blur_blocks_per_sm(int R, int th_kind, int mode, int storage) {
  int nb = 0;
  cudaError_t e = cudaErrorInvalidValue;
  auto occ = [&](const void *fn, int threads, int smem) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, threads, smem);
  };
  if (mode == 2) {
#define CASE_R(RR) \
  case RR: occ(reinterpret_cast<const void *>(k_base_poly<(RR + 2) / 2>), kPolyThreads, 0); break;
    switch (R) {
      SIFT_FOR_EACH_POLY_R(CASE_R)
      default: occ(reinterpret_cast<const void *>(k_base_generic<2>), kGenThreads, generic_smem_bytes(R));
    }
#undef CASE_R
  } else if (R == 0) {
    occ(reinterpret_cast<const void *>(k_base_generic<1>), kGenThreads, generic_smem_bytes(0));
  } else {
    const BlurFn f = blur_fn(R, mode == 1 ? (int)BV_BASE : level_variant(th_kind, mode == 3, storage));
    occ(f.fn, kThreads, f.smem);
  }
  return (e == cudaSuccess && nb > 0) ? nb : 1;
}

}  // namespace sift
