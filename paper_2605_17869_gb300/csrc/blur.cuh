// Separable Gaussian level blur (§3.2, "GPU Pipeline Stages"), 4-sigma
// truncation, reflect-101 borders: the kernel template, instantiated and launched by
// pyramid.cu (radii of the default scale space), blur_rest.cu and blur_rest64.cu (the
// others).
//
// One launch computes one pyramid level for every image of the batch: a
// persistent grid of ten-warp blocks walks a flattened queue of 128 x TH output
// tiles. A tile stages its (TH + 2R) x 160 input window in shared memory with
// cp.async (16-byte copies inside the image, reflect-101 element copies at its
// borders), runs the column pass (a thread: one column pair x V rows, packed
// two-lane FP32 FMAs) into a second shared buffer, then the row pass (a
// half-warp: one row, a lane: 8 adjacent outputs) and stores float4 rows.
//  * TH = 20, V = 5: the column pass is 80 pairs x 4 row blocks, one item per
//    thread, and the row pass 10 pairs of rows, one per warp, so that neither pass
//    leaves warps waiting at the two barriers of a tile. What bounds the kernel is
//    the L1 and shared-memory path (70-72% busy) with the waits at barriers and on
//    loads, not HBM (28-43% of its bandwidth) or the FMA pipe (41% at R = 5, 56% at
//    R = 13), so four blocks per SM matter more than the halo rows that a short tile
//    stages again (from L2). Measured when the tile was chosen, on the 64-image batch, 1024 x 768 x 4 images
//    at five scales per octave, and one 640 x 480 image (us per call): TH = 20: 2367
//    / 334 / 135; TH = 30: 2407 / 339 / 145; TH = 40 with 640 threads: 2433 / 360 /
//    148, with 320 threads and V = 10: 2425 / 407 / 147. A ring of rows marched down
//    a strip, which stages every row once, took 2550 (blocks of five warps) and 2377
//    (warps by themselves), and 160 on the single image.
//  * 8 outputs per lane read 2R + 8 values, 3 to 5 16-byte loads per 4 outputs
//    (4 outputs: 5 to 9), which was the tile's main load on shared memory. The
//    buffer keeps the even float4 groups of a row apart
//    from the odd ones, so that lanes two groups apart read without conflicts.
//
// Every output pixel is the same fixed-order chain of FP32 operations whatever
// the tile height: out(y, x) = sum_i w_i * c_i with c_i = sum_j w_j * in(y - R
// + j, x - R + i), each c_i summed over j ascending and the outer sum split into
// two ascending chains of alternate taps whose grouping depends only on the
// parity of x - R (row_pass_store). Results therefore do not depend on the
// tiling or on which other images share the launch.
#pragma once
#include "sift_dev.cuh"

namespace sift {

constexpr int kSinW = kBlurTW + 2 * kBlurHalo;  // 160 staged columns
constexpr int kPairs = kSinW / 2;               // 80 column pairs
constexpr int kThreads = 4 * kPairs;            // 10 warps: one column-pass item per thread
constexpr int kWarps = kThreads / 32;
constexpr int kNG = kSinW / 4;                  // 40 float4 column groups

__device__ __forceinline__ unsigned smem_u32(const void *p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(src));
}
__device__ __forceinline__ void cp_async16_u(unsigned dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src));
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32(dst)), "l"(src));
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// Element st of plane p, for planes of 4-byte (half false) or 2-byte elements.
__device__ __forceinline__ float *elem_ptr(float *p, long long st, bool half) {
  return half ? reinterpret_cast<float *>(reinterpret_cast<__half *>(p) + st) : p + st;
}

// How the staged window holds its values:
//   SK_F32  FP32 values;
//   SK_H16  binary16 values (a binary16 level, MODE 0);
//   SK_R16  FP32 values still to be rounded to binary16 (the decimated base of
//           the first binary16 octave, MODE 3 from an FP32 octave);
//   SK_P16  32-bit words whose low half is the binary16 value (the decimated
//           base of a later binary16 octave: the word holding sample 2x of a
//           binary16 row, copied whole by a 4-byte cp.async).
enum StageKind { SK_F32 = 0, SK_H16 = 1, SK_R16 = 2, SK_P16 = 3 };

template <int MODE, int ST> __host__ __device__ constexpr int stage_kind() {
  return ST == 0 ? SK_F32 : MODE == 0 ? SK_H16 : ST == 1 ? SK_R16 : SK_P16;
}

// Two adjacent staged elements (the first at an even index) as FP32; binary16
// values widen exactly, and SK_R16 rounds to binary16 first (what the level
// stores). p: the first one's address.
template <int KIND> __device__ __forceinline__ float2 staged_pair(const char *p) {
  if constexpr (KIND == SK_H16) {
    return __half22float2(*reinterpret_cast<const __half2 *>(p));
  } else if constexpr (KIND == SK_P16) {
    const uint2 w = *reinterpret_cast<const uint2 *>(p);
    const unsigned lo = __byte_perm(w.x, w.y, 0x5410);  // the two low halves
    return __half22float2(*reinterpret_cast<const __half2 *>(&lo));
  } else {
    const float2 f = *reinterpret_cast<const float2 *>(p);
    if constexpr (KIND == SK_R16) return __half22float2(__float22half2_rn(f));
    return f;
  }
}
template <int KIND> constexpr int staged_bytes() { return KIND == SK_H16 ? 2 : 4; }

// Shapes of one radius. Row pass: lane l of a half-warp reads float4 groups G0 +
// 2l .. G0 + 2l + NV - 1.
template <int R> struct BlurShape {
  static constexpr int OFF = (kBlurHalo - R) & 3;         // first tap's offset in the first group
  static constexpr int C0 = kBlurHalo - R - OFF;          // first column read by lane 0
  static constexpr int NV = (OFF + 8 + 2 * R + 3) / 4;    // groups read per lane
  static constexpr int G0 = C0 / 4;
  static constexpr int G1 = G0 + 30 + NV;                 // one past the last group read
  static_assert(G1 <= kNG, "the row pass stays inside the staged columns");
};
// Shared memory: the staging buffer (binary16 for a binary16 level, ST 2 with
// MODE 0) plus the column-pass output.
template <int R, int TH, int MODE, int ST> constexpr int blur_smem() {
  return (TH + 2 * R) * kSinW * (MODE == 0 && ST == 2 ? 2 : 4) + TH * kSinW * 4;
}
// Tile rows of a queue, and rows of a column-pass item of such a tile.
constexpr int tile_rows(int kind) { return kind == TK_BLUR64 ? 40 : 20; }
constexpr int item_rows(int th) { return th / 4; }

// MODE 0: level lvl_out from level lvl_out - 1 of octave `oct`.
// MODE 1: octave 0 level 0 from the input image.
// MODE 3: level 1 of octave `oct` > 0 from its level 0, decimated on the fly
//         from level S of octave oct - 1; level 0 itself is stored on the way.
struct alignas(16) TileGeo {
  const float *src;  // staging source: level lvl_out - 1 (MODE 0), the input (1),
                     // level S of the previous octave (3)
  float *out;        // level lvl_out of the tile's octave
  int pitch, H, W;   // the octave's pitch and size
  int vec;           // 16-byte aligned source rows
  int x0, y0;
  int spitch;        // source pitch (elements)
  int pad;
  float *out0;       // level 0 of the tile's octave (MODE 3 stores it)
};
// A tile's geometry from shared memory by 16-byte loads, once per tile (field by
// field, for the tile and for the next one's copies, it was a fifth of the R = 5
// kernel's shared-memory accesses).
template <int MODE> __device__ __forceinline__ TileGeo load_geo(const TileGeo *p) {
  const int4 *q = reinterpret_cast<const int4 *>(p);
  const int4 a = q[0], b = q[1], c = q[2];
  auto ptr = [](int lo, int hi) {
    return reinterpret_cast<float *>((unsigned long long)(unsigned)lo | (unsigned long long)(unsigned)hi << 32);
  };
  TileGeo g;
  g.src = ptr(a.x, a.y);
  g.out = ptr(a.z, a.w);
  g.pitch = b.x;
  g.H = b.y;
  g.W = b.z;
  g.vec = MODE == 0 ? 1 : b.w;
  g.x0 = c.x;
  g.y0 = c.y;
  g.spitch = MODE == 0 ? b.x : c.z;
  g.out0 = MODE == 3 ? p->out0 : nullptr;
  return g;
}

// Geometry of flattened tile t. Image b's octaves sit at fixed slots
// oct[b * kMaxOct + o], so no ImgDev read is needed for pyramid levels.
// ST: storage of the source and the output. 0: FP32 in and out; 1: FP32 source,
// binary16 output (the first level of octave 1 in the fp16 storage mode);
// 2: binary16 in and out (octaves above 1, and every level after the first of
// octave 1).
template <int TH, int MODE, int ST = 0>
__device__ __forceinline__ TileGeo tile_geo(const Desc *__restrict__ d, const int *pre, int oct,
                                            int lvl_out, int t) {
  TileGeo g;
  const int b = find_owner(pre, d->n_img, t);
  const OctDev od = d->oct[b * kMaxOct + oct];
  g.pitch = od.pitch;
  g.H = od.H;
  g.W = od.W;
  float *lv = d->pyr + od.lvl;
  g.out0 = lv;
  g.out = elem_ptr(lv, (long long)lvl_out * od.lstride, ST != 0);
  if (MODE == 0) {
    g.src = elem_ptr(lv, (long long)(lvl_out - 1) * od.lstride, ST == 2);
    g.spitch = od.pitch;
    g.vec = 1;
  } else if (MODE == 3) {
    const OctDev op = d->oct[b * kMaxOct + oct - 1];
    g.src = elem_ptr(d->pyr + op.lvl, (long long)d->n_scales * op.lstride, ST == 2);
    g.spitch = op.pitch;
    g.vec = 0;
  } else {
    const ImgDev &im = d->img[b];
    g.src = im.src;
    g.spitch = im.spitch;
    g.vec = im.src_vec_ok;
  }
  const int tiles_x = (od.W + kBlurTW - 1) / kBlurTW;
  const int lt = t - pre[b];
  const int ty = lt / tiles_x, tx = lt - ty * tiles_x;
  g.x0 = tx * kBlurTW;
  g.y0 = ty * TH;
  return g;
}

// Issue (without waiting) the copies of rows [y0 - R, y0 + TH + R) x columns
// [x0 - 16, x0 + 144) of a plain image (pyramid level or input) into s_in,
// reflect-101 at the borders.
// 16-byte path (16-byte aligned rows): thread t copies float4 column group
// t % 40 of rows t / 40, t / 40 + 8, ...; a group that crosses or lies past an
// image edge copies its four reflected columns one by one. Element path
// (unaligned input rows): thread t copies column t % 160 of rows t / 160,
// t / 160 + 2, .... Reflection is only computed where the window crosses an
// image edge.
__device__ __forceinline__ void stage_plain_issue(const float *__restrict__ src, int pitch, int H,
                                                  int W, bool vec_ok, int x0, int y0, int R,
                                                  int rows, float *s_in) {
  const int xb = x0 - kBlurHalo;
  const int yb = y0 - R;
  const bool yin = yb >= 0 && yb + rows <= H;
  const int tid = threadIdx.x;
  if (vec_ok) {
    constexpr int RPP = kThreads / kNG;  // rows per pass (8)
    const int g = tid % kNG, r0 = tid / kNG;
    const int c = xb + 4 * g;
    float *dst = s_in + r0 * kSinW + 4 * g;
    if (c >= 0 && c + 4 <= W) {
      const float *col = src + c;
      if (yin) {
        const float *p = col + (long long)(yb + r0) * pitch;
        for (int r = r0; r < rows; r += RPP, p += (long long)RPP * pitch, dst += RPP * kSinW)
          cp_async16(dst, p);
      } else {
        for (int r = r0; r < rows; r += RPP, dst += RPP * kSinW)
          cp_async16(dst, col + (long long)refl101(yb + r, H) * pitch);
      }
    } else {
      const int c0 = refl101(c, W), c1 = refl101(c + 1, W), c2 = refl101(c + 2, W),
                c3 = refl101(c + 3, W);
      for (int r = r0; r < rows; r += RPP, dst += RPP * kSinW) {
        const float *row = src + (long long)(yin ? yb + r : refl101(yb + r, H)) * pitch;
        cp_async4(dst, row + c0);
        cp_async4(dst + 1, row + c1);
        cp_async4(dst + 2, row + c2);
        cp_async4(dst + 3, row + c3);
      }
    }
  } else {
    constexpr int RPP = kThreads / kSinW;  // rows per pass (2)
    const int c = tid % kSinW, r0 = tid / kSinW;
    const float *col = src + refl101(xb + c, W);
    float *dst = s_in + r0 * kSinW + c;
    for (int r = r0; r < rows; r += RPP, dst += RPP * kSinW)
      cp_async4(dst, col + (long long)(yin ? yb + r : refl101(yb + r, H)) * pitch);
  }
}

// Issue the copies of the window of octave o > 0's level 0 without storing
// that level first: sample (y, x) of level 0 is sample (2y, 2x) of level S of
// octave o - 1, so the window is gathered from there (reflect-101 applied in
// octave o's own domain), element by element.
// DEC 2: src holds FP32 samples, spitch in floats. DEC 1: src is a binary16
// plane seen as 32-bit words (spitch in halves): word gy * spitch + gx holds
// halves 2 (gy * spitch + gx) and the next, the first of which is sample
// (2 gy, 2 gx) (SK_P16).
template <int DEC>
__device__ __forceinline__ void stage_decim_issue(const float *__restrict__ src, int spitch, int H,
                                                  int W, int x0, int y0, int R, int rows,
                                                  float *s_in) {
  const int xb = x0 - kBlurHalo, yb = y0 - R;
  const bool yin = yb >= 0 && yb + rows <= H;
  constexpr int RPP = kThreads / kSinW;  // rows per pass (2)
  const int c = threadIdx.x % kSinW, r0 = threadIdx.x / kSinW;
  const float *col = src + DEC * refl101(xb + c, W);
  float *dst = s_in + r0 * kSinW + c;
  for (int r = r0; r < rows; r += RPP, dst += RPP * kSinW)
    cp_async4(dst, col + (long long)(DEC * (yin ? yb + r : refl101(yb + r, H))) * spitch);
}

// Interior tile of a 16-byte aligned plane (no staged row or column outside
// the image): a fixed, fully unrolled copy schedule, thread t copying float4
// group t % 40 of rows t / 40 + 8 i, so the copies cost almost nothing but
// the copy instructions themselves.
template <int ROWS>
__device__ __forceinline__ void stage_interior(const float *__restrict__ src, int pitch, int xb,
                                               int yb, float *s_in) {
  constexpr int RPP = kThreads / kNG;  // 8
  constexpr int NIT = (ROWS + RPP - 1) / RPP;
  const int tid = threadIdx.x;
  const int g = tid % kNG, r0 = tid / kNG;
  const unsigned d0 = smem_u32(s_in + r0 * kSinW + 4 * g);
  const float *p = src + (long long)(yb + r0) * pitch + (xb + 4 * g);
  const long long step = (long long)RPP * pitch;
#pragma unroll
  for (int i = 0; i < NIT; i++)
    if (i + 1 < NIT || r0 + i * RPP < ROWS) cp_async16_u(d0 + i * RPP * kSinW * 4, p + i * step);
}

// The window of a binary16 level (MODE 0, ST 2), kept as binary16 in shared
// memory (rows of kSinW halves) and widened by the column pass. Every group of
// 8 columns that lies inside the image is one 16-byte cp.async copy (rows
// start on 64-byte boundaries and xb is a multiple of 16; a row outside the
// image is its reflect-101 row); a group that crosses or lies past a left or
// right edge is copied element by element through registers with reflect-101
// (cp.async has no 2-byte copy).
__device__ __forceinline__ void stage_half_issue(const TileGeo &g, int R, int rows, __half *s_in) {
  const __half *src = reinterpret_cast<const __half *>(g.src);
  const int xb = g.x0 - kBlurHalo, yb = g.y0 - R;
  constexpr int NG8 = kSinW / 8;  // 20 groups of 8 halves per row
  const bool yin = yb >= 0 && yb + rows <= g.H;
  for (int i = threadIdx.x; i < rows * NG8; i += kThreads) {
    const int r = i / NG8, c8 = i - r * NG8;
    const int gx = xb + 8 * c8;
    const __half *row = src + (long long)(yin ? yb + r : refl101(yb + r, g.H)) * g.spitch;
    __half *dst = s_in + r * kSinW + 8 * c8;
    if (gx >= 0 && gx + 8 <= g.W) {
      cp_async16(dst, row + gx);
    } else {
#pragma unroll
      for (int k = 0; k < 8; k++) dst[k] = row[refl101(gx + k, g.W)];
    }
  }
}

template <int R, int TH, int MODE, int ST = 0>
__device__ __forceinline__ void issue_stage(const TileGeo &g, float *dst) {
  constexpr int ROWS = TH + 2 * R;
  if constexpr (MODE == 0 && ST == 2) {
    stage_half_issue(g, R, ROWS, reinterpret_cast<__half *>(dst));
  } else if constexpr (MODE == 3) {  // FP32 samples (ST 0, 1) or binary16 words (ST 2)
    stage_decim_issue<ST == 2 ? 1 : 2>(g.src, g.spitch, g.H, g.W, g.x0, g.y0, R, ROWS, dst);
  } else {
    static_assert(ST == 0, "binary16 output is MODE 3 (ST 1) or MODE 0 / 3 (ST 2)");
    const int xb = g.x0 - kBlurHalo, yb = g.y0 - R;
    if (g.vec && xb >= 0 && xb + kSinW <= g.W && yb >= 0 && yb + ROWS <= g.H)
      stage_interior<ROWS>(g.src, g.spitch, xb, yb, dst);
    else
      stage_plain_issue(g.src, g.spitch, g.H, g.W, g.vec != 0, g.x0, g.y0, R, ROWS, dst);
  }
}

// Column pass: s_v[v][c] = sum_j w[j] * s_in[v + j][c], j = 0 .. 2R in order,
// for the column pairs the row pass reads. KIND: how s_in holds the window.
template <int R, int TH, int KIND>
__device__ __forceinline__ void col_pass(const float *s_in, float *s_v, const BlurTaps &tp) {
  using S = BlurShape<R>;
  constexpr int V = item_rows(TH), EB = staged_bytes<KIND>();
  const int rb = threadIdx.x / kPairs, c = 2 * (threadIdx.x - rb * kPairs);
  if (c < 4 * S::G0 || c >= 4 * S::G1) return;
  const char *src = reinterpret_cast<const char *>(s_in) + (rb * V * kSinW + c) * EB;
  float2 acc[V];
#pragma unroll
  for (int i = 0; i < V + 2 * R; i++) {
    const float2 f = staged_pair<KIND>(src + i * kSinW * EB);
#pragma unroll
    for (int v = 0; v < V; v++) {
      const int j = i - v;
      if (j == 0) acc[v] = __fmul2_rn(tp.wd[0], f);
      else if (j > 0 && j <= 2 * R) acc[v] = __ffma2_rn(tp.wd[j], f, acc[v]);
    }
  }
  // Group q = c / 4 of a row of s_v lies at (q >> 1) + 20 (q & 1).
  const int q = c >> 2;
  float *dst = s_v + rb * V * kSinW + 4 * ((q >> 1) + (q & 1) * (kNG / 2)) + (c & 3);
#pragma unroll
  for (int v = 0; v < V; v++) *reinterpret_cast<float2 *>(dst + v * kSinW) = acc[v];
}

// Store four adjacent outputs: FP32, or (DH) rounded to binary16.
template <bool DH>
__device__ __forceinline__ void store4(float *out, long long idx, float a, float b, float c, float e) {
  if (DH) {
    const __half2 lo = __floats2half2_rn(a, b), hi = __floats2half2_rn(c, e);
    uint2 u;
    u.x = *reinterpret_cast<const unsigned *>(&lo);
    u.y = *reinterpret_cast<const unsigned *>(&hi);
    *reinterpret_cast<uint2 *>(reinterpret_cast<__half *>(out) + idx) = u;
  } else {
    *reinterpret_cast<float4 *>(out + idx) = make_float4(a, b, c, e);
  }
}

// Row pass + store: out[y0 + v][x0 + k] from s_v[v][16 + k - R + i], i = 0..2R.
// The taps are taken two at a time by packed FMAs whose operand pairs are
// aligned (even, odd) column pairs of the row, so with s the output's first tap
// column (each lane of a packed FMA is an ordinary FP32 fma):
//   s even: a = (w0 v[s], w1 v[s+1]), a += (w2i, w2i+1)(v[s+2i], v[s+2i+1]) for
//           i = 1..R-1, out = fma(w2R, v[s+2R], a.x) + a.y;
//   s odd:  a = (w1 v[s+1], w2 v[s+2]), a += (w2i+1, w2i+2)(v[s+2i+1], v[s+2i+2])
//           for i = 1..R-1, out = fma(w0, v[s], a.x) + a.y.
// The parity of s is that of the output's column, so the order of operations
// is a fixed function of the pixel.
template <int R, int TH, bool DH>
__device__ __forceinline__ void row_pass_store(const float *s_v, float *out, int pitch, int H, int x0,
                                               int y0, const BlurTaps &tp) {
  using S = BlurShape<R>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int hl = lane >> 4, l = lane & 15;
  const int x = x0 + 8 * l;
  const bool xok = x < pitch;  // pitches are multiples of 32: all eight or none
  constexpr int IT = TH / (2 * kWarps);  // rows per half-warp
#pragma unroll 1
  for (int it = 0, v = 2 * warp + hl; it < IT; it++, v += 2 * kWarps) {
    const float4 *s4 = reinterpret_cast<const float4 *>(s_v + v * kSinW) + l;
    float in[S::NV * 4];
#pragma unroll
    for (int t = 0; t < S::NV; t++) {
      constexpr int G = S::G0;
      const float4 f = s4[((G + t) >> 1) + ((G + t) & 1) * (kNG / 2)];
      in[4 * t + 0] = f.x; in[4 * t + 1] = f.y; in[4 * t + 2] = f.z; in[4 * t + 3] = f.w;
    }
    float o[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int s = S::OFF + k;
      if ((s & 1) == 0) {
        float2 a = __fmul2_rn(tp.wp[0], make_float2(in[s], in[s + 1]));
#pragma unroll
        for (int i = 1; i < R; i++)
          a = __ffma2_rn(tp.wp[i], make_float2(in[s + 2 * i], in[s + 2 * i + 1]), a);
        o[k] = __fadd_rn(fmaf(tp.w[2 * R], in[s + 2 * R], a.x), a.y);
      } else {
        float2 a = __fmul2_rn(tp.wq[0], make_float2(in[s + 1], in[s + 2]));
#pragma unroll
        for (int i = 1; i < R; i++)
          a = __ffma2_rn(tp.wq[i], make_float2(in[s + 2 * i + 1], in[s + 2 * i + 2]), a);
        o[k] = __fadd_rn(fmaf(tp.w[0], in[s], a.x), a.y);
      }
    }
    if (y0 + v < H && xok) {
      const long long oi = (long long)(y0 + v) * pitch + x;
      store4<DH>(out, oi, o[0], o[1], o[2], o[3]);
      store4<DH>(out, oi + 4, o[4], o[5], o[6], o[7]);
    }
  }
}

// Store the tile's own rows / columns of the staged (decimated) level 0:
// FP32, or (DH) rounded to binary16 (exact for SK_P16 words, whose low
// halves are binary16 values already).
template <int R, int TH, bool DH, int KIND>
__device__ __forceinline__ void store_level0(const float *s_in, float *out0, int pitch, int H,
                                             int x0, int y0) {
  constexpr int K = KIND == SK_P16 ? SK_P16 : SK_F32;
  for (int q = threadIdx.x; q < TH * (kBlurTW / 4); q += kThreads) {
    const int v = q / (kBlurTW / 4), g = q - v * (kBlurTW / 4);
    const int y = y0 + v, x = x0 + 4 * g;
    if (y < H && x < pitch) {
      const char *p = reinterpret_cast<const char *>(s_in + (R + v) * kSinW + kBlurHalo + 4 * g);
      const float2 a = staged_pair<K>(p), b = staged_pair<K>(p + 8);
      store4<DH>(out0, (long long)y * pitch + x, a.x, a.y, b.x, b.y);
    }
  }
}

// The block's tiles are t0, t0 + grid, t0 + 2 grid, .... Their geometry is
// resolved 32 tiles at a time, one tile per lane of warp 0, into a ring of two
// 32-entry chunks in shared memory: the lanes' owner searches and descriptor
// loads overlap, and chunk m + 1 is filled half-way through chunk m, so no
// tile waits on a dependent chain of global loads.
// One staging buffer per block, but its copies run ahead: once the column pass
// of tile i has read the staged window, the block issues tile i + 1's copies
// into it and they land while the row pass of tile i runs. With three or four blocks per SM this measured faster than
// a second buffer with fewer blocks.
constexpr int kGeoChunk = 32;
template <int R, int TH, int MODE, int ST>
__global__ void __launch_bounds__(kThreads, TH == 20 ? 4 : 3)
    k_blur(const Desc *__restrict__ d, int oct, int lvl_out, BlurTaps tp) {
  constexpr int ROWS = TH + 2 * R;
  extern __shared__ float4 smem4[];
  __shared__ TileGeo geo[2 * kGeoChunk];
  // A binary16 level (MODE 0, ST 2) is staged as binary16: half the bytes.
  constexpr int KIND = stage_kind<MODE, ST>();
  constexpr bool H16 = KIND == SK_H16;
  float *s_in = reinterpret_cast<float *>(smem4);
  float *s_v = s_in + (H16 ? ROWS * kSinW / 2 : ROWS * kSinW);
  // The base blur of images kept at their size (MODE 1) takes the queue of
  // those images only.
  const int *pre = MODE == 1 ? d->base_pre[0] : d->tile_pre[TH == 20 ? TK_BLUR32 : TK_BLUR64][oct];
  const int total = pre[d->n_img];
  const int t0 = blockIdx.x, G = gridDim.x;
  if (t0 >= total) return;
  const int n_mine = (total - t0 + G - 1) / G;  // tiles of this block
  auto fill_chunk = [&](int m) {                // tiles 32 m .. 32 m + 31, by warp 0
    const int k = m * kGeoChunk + (int)threadIdx.x;
    if (k < n_mine) geo[k & (2 * kGeoChunk - 1)] = tile_geo<TH, MODE, ST>(d, pre, oct, lvl_out, t0 + k * G);
  };
  if (threadIdx.x < 32) fill_chunk(0);
  __syncthreads();
  pdl_wait();  // the source level is the previous kernel's output
  TileGeo g = load_geo<MODE>(&geo[0]);
  issue_stage<R, TH, MODE, ST>(g, s_in);
  for (int k = 0; k < n_mine; k++) {
    if (k + 1 == n_mine) pdl_trigger();  // successors launch during this block's last tile
    cp_async_wait_all();
    __syncthreads();
    if (MODE == 3) store_level0<R, TH, ST != 0, KIND>(s_in, g.out0, g.pitch, g.H, g.x0, g.y0);
    col_pass<R, TH, KIND>(s_in, s_v, tp);
    __syncthreads();
    TileGeo gn = g;
    if (k + 1 < n_mine) {
      gn = load_geo<MODE>(&geo[(k + 1) & (2 * kGeoChunk - 1)]);
      issue_stage<R, TH, MODE, ST>(gn, s_in);
    }
    row_pass_store<R, TH, ST != 0>(s_v, g.out, g.pitch, g.H, g.x0, g.y0, tp);
    g = gn;
    if (threadIdx.x < 32 && (k & (kGeoChunk - 1)) == kGeoChunk / 2)
      fill_chunk(k / kGeoChunk + 1);
    // No barrier here: the barrier after the next copy-wait orders every
    // warp's row pass (reads of s_v) before the next column pass writes s_v,
    // and the column pass (reads of s_in) before s_in is restaged.
  }
}

// The instances of one radius, by launch variant.
enum BlurVariant { BV_LVL, BV_DEC, BV_LVL_H16, BV_DEC_R16, BV_DEC_H16, BV_BASE, BV_LVL64, BV_DEC64, BV_COUNT };
struct BlurFn {
  const void *fn;
  int smem;
};
#define SIFT_BLUR_FN(TH, MODE, ST) \
  BlurFn{reinterpret_cast<const void *>(k_blur<R, TH, MODE, ST>), blur_smem<R, TH, MODE, ST>()}
template <int R> BlurFn blur_instance(int variant) {  // 20-row tiles
  switch (variant) {
    case BV_LVL: return SIFT_BLUR_FN(20, 0, 0);
    case BV_DEC: return SIFT_BLUR_FN(20, 3, 0);
    case BV_LVL_H16: return SIFT_BLUR_FN(20, 0, 2);
    case BV_DEC_R16: return SIFT_BLUR_FN(20, 3, 1);
    case BV_DEC_H16: return SIFT_BLUR_FN(20, 3, 2);
    default: return SIFT_BLUR_FN(20, 1, 0);
  }
}
template <int R> BlurFn blur_instance64(int variant) {  // 40-row tiles
  return variant == BV_LVL64 ? SIFT_BLUR_FN(40, 0, 0) : SIFT_BLUR_FN(40, 3, 0);
}
#undef SIFT_BLUR_FN
// Of a radius in 1 .. kMaxR that blur_fn (pyramid.cu) does not instantiate itself.
BlurFn blur_rest(int R, int variant);
BlurFn blur_rest64(int R, int variant);

}  // namespace sift
