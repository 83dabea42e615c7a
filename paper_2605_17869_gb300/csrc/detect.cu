// Detection (§3.2): DoG subtraction fused with the 26-neighbour extremum test
// and the contrast gate, compaction of candidates in canonical order, and
// sub-pixel refinement by a 3-D Taylor expansion solved with Cramer's rule.
//
// The DoG is never stored: every consumer recomputes D = G[i+1] - G[i] with the
// same single FP32 subtraction, so all stages see identical values.
//
// Candidates are first marked in a bitmap (30 pixels of a row and layer per word,
// by warp ballots), then compacted by a single-pass scan over bitmap words. The
// bitmap's memory order is (octave, layer, row, column), so the candidate list
// comes out in that canonical order independently of tile shapes or batch
// composition.
#include <algorithm>

#include "scan.cuh"
#include "sift_dev.cuh"

namespace sift {

namespace {

constexpr int kThreads = 256;
constexpr int kExtThreads = 128;  // extrema scan: four independent warps per block

// ------------------------------------------------------------ extrema scan

// 3-input maximum / minimum (one instruction on sm_100 and later).
__device__ __forceinline__ float max3f(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// One row of DoG values as the scan holds it, for the lane's columns x and x + 1:
// the maximum and minimum over columns x - 1 .. x + 1 and x .. x + 2 of each of
// the S + 2 DoG layers, and for the tested layers 1 .. S the values at columns
// x - 1 .. x + 2.
template <int S> struct ExtRow {
  float hx[S + 2][2], hn[S + 2][2];
  float l[S], c[S][2], r[S];
};

// DoG (one FP32 subtraction per value, as in every other stage) of one row from
// its S + 3 Gaussian levels, and the row's three-column maxima / minima: the two
// outer neighbours by warp shuffle (lane 0's left and lane 31's right one are
// meaningless; these lanes only supply neighbours).
template <int S>
__device__ __forceinline__ void ext_row(ExtRow<S> &R, const float2 (&g)[S + 3]) {
#pragma unroll
  for (int i = 0; i < S + 2; i++) {
    const float v0 = g[i + 1].x - g[i].x, v1 = g[i + 1].y - g[i].y;
    const float lf = __shfl_up_sync(0xffffffffu, v1, 1);
    const float rt = __shfl_down_sync(0xffffffffu, v0, 1);
    R.hx[i][0] = max3f(lf, v0, v1);
    R.hn[i][0] = min3f(lf, v0, v1);
    R.hx[i][1] = max3f(v0, v1, rt);
    R.hn[i][1] = min3f(v0, v1, rt);
    if (i >= 1 && i <= S) {
      R.l[i - 1] = lf;
      R.c[i - 1][0] = v0;
      R.c[i - 1][1] = v1;
      R.r[i - 1] = rt;
    }
  }
}

// The rows a warp has in flight: kExtRing rows x (S + 3) levels x 32 lanes in
// shared memory, filled by asynchronous copies (each lane copies and reads its
// own two columns); a row's slot is refilled as soon as it is read. Three, as the
// rows that the tests hold in turn, so that every slot is a fixed address.
constexpr int kExtRing = 3;

__device__ __forceinline__ void cp_async4_ca(unsigned dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8_ca(unsigned dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ unsigned lds32(unsigned a) {
  unsigned v;
  asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float2 lds64(unsigned a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Bits 0 .. 14 spread to the even bit positions 0 .. 28.
__device__ __forceinline__ unsigned spread15(unsigned v) {
  v = (v | (v << 8)) & 0x00ff00ffu;
  v = (v | (v << 4)) & 0x0f0f0f0fu;
  v = (v | (v << 2)) & 0x33333333u;
  return (v | (v << 1)) & 0x55555555u;
}

// Test row y (P, C, N: rows y - 1, y, y + 1) and write its bitmap words: pixel x
// of layer s is a candidate when it lies inside the border, |D| exceeds the
// pre-gate, and D is strictly above the maximum, or strictly below the minimum,
// of its 26 neighbours. Those extrema are separable: the 9 values of layer s +- 1
// reduce to max(hx(y - 1), hx(y), hx(y + 1)), the 8 of layer s to max(hx(y - 1),
// hx(y + 1), left, right). Lane s of the first S writes layer s + 1's two words
// (word: its address, two: whether the row has the second one).
// thr0, thr1: the pre-gate for the lane's columns, infinite where a column lies
// outside the border (no |D| is above it).
template <int S>
__device__ __forceinline__ void ext_test(const ExtRow<S> &P, const ExtRow<S> &C,
                                         const ExtRow<S> &N, bool yin, float thr0, float thr1,
                                         int lane, uint32_t *word, bool two) {
  // Rows where no pixel of the strip passes the border and pre-gate tests
  // in any layer have no candidate: skip the neighbour comparisons.
  bool gate = false;
#pragma unroll
  for (int s = 0; s < S; s++) gate |= (fabsf(C.c[s][0]) > thr0) | (fabsf(C.c[s][1]) > thr1);
  unsigned lo = 0u, hi = 0u;
  if (yin && __any_sync(0xffffffffu, gate)) {
    // First the extrema that may be shared with a neighbour: |c| above the gate and
    // c at least (at most) the maximum (minimum) over the 27 values, five
    // instructions per value; a row of the strip that has one (about one in six)
    // is then tested strictly, which takes nine.
    bool any = false;
#pragma unroll
    for (int k = 0; k < 2; k++) {
      float vx[S + 2], vn[S + 2];
#pragma unroll
      for (int i = 0; i < S + 2; i++) {
        vx[i] = max3f(P.hx[i][k], C.hx[i][k], N.hx[i][k]);
        vn[i] = min3f(P.hn[i][k], C.hn[i][k], N.hn[i][k]);
      }
#pragma unroll
      for (int s = 1; s <= S; s++) {
        const float c = C.c[s - 1][k];
        any |= ((c >= max3f(vx[s - 1], vx[s], vx[s + 1])) | (c <= min3f(vn[s - 1], vn[s], vn[s + 1]))) &
               (fabsf(c) > (k ? thr1 : thr0));
      }
    }
    if (__any_sync(0xffffffffu, any)) {
      bool ok[S][2];
#pragma unroll
      for (int k = 0; k < 2; k++) {
#pragma unroll
        for (int s = 1; s <= S; s++) {
          const float c = C.c[s - 1][k];
          const float lf = k ? C.c[s - 1][0] : C.l[s - 1], rt = k ? C.r[s - 1] : C.c[s - 1][1];
          float mx = max3f(max3f(P.hx[s][k], N.hx[s][k], lf), rt, max3f(P.hx[s - 1][k], C.hx[s - 1][k], N.hx[s - 1][k]));
          float mn = min3f(min3f(P.hn[s][k], N.hn[s][k], lf), rt, min3f(P.hn[s - 1][k], C.hn[s - 1][k], N.hn[s - 1][k]));
          mx = fmaxf(mx, max3f(P.hx[s + 1][k], C.hx[s + 1][k], N.hx[s + 1][k]));
          mn = fminf(mn, min3f(P.hn[s + 1][k], C.hn[s + 1][k], N.hn[s + 1][k]));
          ok[s - 1][k] = ((c > mx) | (c < mn)) & (fabsf(c) > (k ? thr1 : thr0));
        }
      }
      unsigned m0 = 0u, m1 = 0u;  // lane s: layer s + 1 at the lanes' first / second columns
#pragma unroll
      for (int s = 0; s < S; s++) {
        const unsigned b0 = __ballot_sync(0xffffffffu, ok[s][0]), b1 = __ballot_sync(0xffffffffu, ok[s][1]);
        m0 = lane == s ? b0 : m0;
        m1 = lane == s ? b1 : m1;
      }
      // Lanes 1 .. 15: columns 0 .. 29 of the strip; 16 .. 30: 30 .. 59.
      lo = spread15(m0 >> 1 & 0x7fffu) | spread15(m1 >> 1 & 0x7fffu) << 1;
      hi = spread15(m0 >> 16 & 0x7fffu) | spread15(m1 >> 16 & 0x7fffu) << 1;
    }
  }
  if (lane < S) {
    word[0] = lo;
    if (two) word[1] = hi;
  }
}

// A warp owns a strip of 2 kBmCols = 60 columns x ext_rows[oct] rows: lane l
// holds columns 60 tx - 2 + 2l and the next one, so lanes 1 .. 30 are the strip
// (two bitmap words per row and layer) and lanes 0 and 31 its neighbours. The
// warp streams down the strip: each image row's S + 3 levels are copied once, by
// 8 bytes per lane, kExtRing rows ahead, and every test is done from registers.
// The candidate decisions are exact comparisons of the same FP32 values, so they do
// not depend on the tiling. Bitmap words are written by ballots; no atomics.
// Two columns per lane share the copies, the loop, two of four shuffles per layer
// and the middle values of the three-column extrema. What bounds the scan is the
// ALU pipe (64%: three-input extrema and comparisons) together with HBM (62%, 73% of
// the measured copy; every level value read once) at 16 warps per SM, which 128 registers allow (12 warps at
// 150: 2 percent more per call on the 64-image batch); rings of 4 and 8 rows were no
// faster than 3. All scans of the 64-image batch: 545 us with one column per lane
// (4.9 warp instructions per pixel and warp row), 480 with two (3.5), 439 with the
// two-stage test of ext_test; of four 1024 x 768 images with five layers, whose
// one-column strips left 8 warps per SM, 333 -> 276 us per call.
// HALF: the octave's levels are binary16 (fp16 storage mode): a lane's two columns
// are one 32-bit word, widened when the row is read.
template <int S, bool HALF>
__global__ void __launch_bounds__(kExtThreads, S <= 3 ? 4 : S == 4 ? 3 : 2) k_extrema(const Desc *__restrict__ d, int oct) {
  constexpr int WPB = kExtThreads / 32;
  constexpr int PB = HALF ? 4 : 8;                       // bytes of a lane's pair
  constexpr int LB = 32 * PB, SB = (S + 3) * LB;         // of a level's and of a row's pairs
  __shared__ __align__(16) unsigned char ring[WPB * kExtRing * SB];
  const int n = d->n_img;
  const int *pre = d->tile_pre[TK_EXT][oct];
  const int total = pre[n];
  const int lane = threadIdx.x & 31;
  const unsigned my = static_cast<unsigned>(__cvta_generic_to_shared(ring)) +
                      (threadIdx.x >> 5) * (kExtRing * SB) + lane * PB;
  const int bord = d->border, th = d->ext_rows[oct];
  pdl_wait();
  for (int t = blockIdx.x * WPB + (threadIdx.x >> 5); t < total; t += gridDim.x * WPB) {
    if (t + gridDim.x * WPB >= total) pdl_trigger();  // this warp's last tile
    const int b = find_owner(pre, n, t);
    const OctDev od = d->oct[b * kMaxOct + oct];  // image b's octaves sit at fixed slots
    const int H = od.H, W = od.W;
    const long long pitch = od.pitch, ls = od.lstride;
    const int lt = t - pre[b];
    const int sx = (od.wpr + 1) / 2;  // strips per row
    const int ty = lt / sx, tx = lt - ty * sx;
    const int x = tx * (2 * kBmCols) - 2 + 2 * lane;
    const int y0 = ty * th, y1 = min(y0 + th, H);
    // G: the lane's pair of columns in row 0 of level 0; x is even and rows
    // start on 64-byte boundaries at least. Pairs past the row's padding and left
    // of the image are moved inside: no tested pixel has them as neighbours.
    constexpr int EB = HALF ? 2 : 4;
    const char *G = reinterpret_cast<const char *>(d->pyr + od.lvl) +
                    (long long)min(max(x, 0), (int)pitch - 2) * EB;
    const long long lb = ls * EB;
    const bool lx = lane >= 1 && lane <= kBmCols;
    const float thr0 = lx && x >= bord && x < W - bord ? d->prefilter : INFINITY;
    const float thr1 = lx && x + 1 >= bord && x + 1 < W - bord ? d->prefilter : INFINITY;
    const bool two = 2 * tx + 1 < od.wpr;
    uint32_t *bmw = d->bm + od.bm + ((long long)lane * H + y0) * od.wpr + 2 * tx;
    // Row k of the strip's sequence is image row y0 - 1 + k (clamped); it lives in
    // slot k % 3. One commit group per row, empty past the last one (y1), so that
    // the number of pending groups is fixed.
    auto issue = [&](int slot, int y) {
      if (y <= y1) {
        const char *p = G + (long long)min(max(y, 0), H - 1) * pitch * EB;
#pragma unroll
        for (int l = 0; l < S + 3; l++) {
          if (HALF) cp_async4_ca(my + slot * SB + l * LB, p + l * lb);
          else cp_async8_ca(my + slot * SB + l * LB, p + l * lb);
        }
      }
      cp_async_commit();
    };
    auto consume = [&](ExtRow<S> &R, int slot, int y) {  // image row y
      cp_async_wait<kExtRing - 1>();
      float2 g[S + 3];
#pragma unroll
      for (int l = 0; l < S + 3; l++) {
        if constexpr (HALF) {
          const unsigned w = lds32(my + slot * SB + l * LB);
          g[l] = __half22float2(*reinterpret_cast<const __half2 *>(&w));
        } else {
          g[l] = lds64(my + slot * SB + l * LB);
        }
      }
      ext_row<S>(R, g);
      issue(slot, y + kExtRing);  // into the slot just read (each lane rewrites only its own words)
    };
#pragma unroll
    for (int k = 0; k < kExtRing; k++) issue(k, y0 - 1 + k);
    ExtRow<S> A, B, C;
    consume(A, 0, y0 - 1);
    consume(B, 1, y0);
    // Rows rotate through A, B, C (previous, current, next) without copies; the
    // steps past the strip's last row test nothing.
    auto step = [&](const ExtRow<S> &Pr, const ExtRow<S> &Cu, ExtRow<S> &Nx, int slot, int y) {
      consume(Nx, slot, y + 1);
      if (y < y1) ext_test<S>(Pr, Cu, Nx, y >= bord && y < H - bord, thr0, thr1, lane, bmw, two);
      bmw += od.wpr;
    };
    for (int y = y0; y < y1; y += 3) {
      step(A, B, C, 2, y);
      step(B, C, A, 0, y + 1);
      step(C, A, B, 1, y + 2);
    }
    cp_async_wait<0>();  // no copy of this strip outlives it
    __syncwarp();
  }
}

// ----------------------------------------------------- bitmap compaction

// Candidate list of every image in canonical order (octave, layer, row,
// column), in one pass. Block g of G takes the contiguous range of bitmap
// chunks [C g / G, C (g + 1) / G):
//  1. it counts the set bits of its chunks (per chunk and warp, kept in
//     shared memory);
//  2. it takes the count of everything before its range from the
//     single-pass scan over blocks, so it only ever waits for blocks of lower
//     index, and at once publishes the global offset of every image that
//     starts in its range;
//  3. it writes its candidates chunk by chunk, each image's slots counted
//     from that image's start (published by the block that holds the image's
//     first chunk).
// The block with an image's last chunk writes the image's totals, and the
// last block forms the prefix of the candidate counts over the images.
constexpr int kCmpWarps = kThreads / 32;
constexpr int kMaxCh = 256;  // chunks per block whose counts are kept (more are recounted)

__device__ __forceinline__ int warp_sum_i(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ int bm_chunk_words(const Desc *__restrict__ d, const ImgDev &im, int c,
                                              int c0, uint32_t (&words)[kChunk / kThreads],
                                              long long *w0_out) {
  constexpr int WPT = kChunk / kThreads;
  const long long w0 = (long long)(c - c0) * kChunk + threadIdx.x * WPT;
  const uint32_t *bm = d->bm + im.bm_begin;
  int cnt = 0;
#pragma unroll
  for (int k = 0; k < WPT; k++) {
    words[k] = (w0 + k < im.bm_words) ? bm[w0 + k] : 0u;
    cnt += __popc(words[k]);
  }
  *w0_out = w0;
  return cnt;
}

__global__ void __launch_bounds__(kThreads) k_bm_compact(const Desc *__restrict__ d) {
  pdl_wait();
  __shared__ int tmp[kThreads / 32 + 1];
  __shared__ int s_w[kMaxCh][kCmpWarps];  // set bits per kept chunk and warp
  __shared__ int s_val;
  constexpr int WPT = kChunk / kThreads;  // words per thread
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // (no more blocks than chunks: a short list's look-back is short)
  const int n = d->n_img, C = d->n_bm_chunks, G = min((int)gridDim.x, C), g = blockIdx.x;
  if (g >= G) return;
  const LookbackCfg cfg{d->lb_epoch, d->lb_spins, d->lb_hold, d->lb_err};
  const int ca = (int)((long long)C * g / G), cb = (int)((long long)C * (g + 1) / G);
  const int kept = min(cb - ca, kMaxCh);
  // Owners of the range's chunks: found once, then advanced (the chunks are
  // contiguous and images are in order).
  const int b_lo = ca < cb ? find_owner(d->bmc_pre, n, ca) : 0;
  uint32_t words[WPT];
  long long w0;
  // 1. Counts.
  int over = 0;
  for (int c = ca, b = b_lo; c < cb; c++) {
    while (c >= d->bmc_pre[b + 1]) b++;
    const int cnt = bm_chunk_words(d, d->img[b], c, d->bmc_pre[b], words, &w0);
    if (c - ca < kMaxCh) {
      const int ws = warp_sum_i(cnt);
      if (lane == 0) s_w[c - ca][warp] = ws;
    } else {
      over += cnt;
    }
  }
  __syncthreads();
  int part = over;
  for (int k = threadIdx.x; k < kept; k += kThreads)
#pragma unroll
    for (int w = 0; w < kCmpWarps; w++) part += s_w[k][w];
  const int agg = block_sum(part, tmp);
  // 2. Offset of the range; starts of the images beginning in it.
  if (threadIdx.x < 32) {
    const int ex = lb_exclusive(d->lb_bm, 0, g, agg, cfg);
    if (threadIdx.x == 0) s_val = ex;
  }
  __syncthreads();
  const int base = s_val;
  __syncthreads();
  {
    int acc = base;
    for (int c = ca, b = b_lo; c < cb; c++) {
      while (c >= d->bmc_pre[b + 1]) b++;
      if (c == d->bmc_pre[b] && threadIdx.x == 0)
        lb_store(d->lb_start + b, lb_word(kLbInc, cfg.epoch, acc));
      int t = 0;
      if (c - ca < kMaxCh) {
#pragma unroll
        for (int w = 0; w < kCmpWarps; w++) t += s_w[c - ca][w];
      } else {  // uniform over the block
        t = block_sum(bm_chunk_words(d, d->img[b], c, d->bmc_pre[b], words, &w0), tmp);
      }
      acc += t;
    }
  }
  // 3. Candidates.
  int carry = base;         // global offset of chunk c
  int cur = -1, start = 0;  // image of the previous chunk, global offset of its first slot
  for (int c = ca, b = b_lo; c < cb; c++) {
    while (c >= d->bmc_pre[b + 1]) b++;
    const ImgDev &im = d->img[b];
    const int c0 = d->bmc_pre[b];
    const int cnt = bm_chunk_words(d, im, c, c0, words, &w0);
    int pre, tot;
    if (c - ca < kMaxCh) {
      const int incl = warp_incl_scan(cnt);
      int wb = 0;
      tot = 0;
#pragma unroll
      for (int w = 0; w < kCmpWarps; w++) {
        const int x = s_w[c - ca][w];
        wb += w < warp ? x : 0;
        tot += x;
      }
      pre = wb + incl - cnt;
    } else {  // uniform over the block
      pre = block_excl_scan(cnt, tmp, &tot);
    }
    if (b != cur) {  // uniform over the block
      cur = b;
      if (c == c0) {
        start = carry;
      } else {  // the image began in a lower block's range (only the range's first image)
        if (threadIdx.x < 32) {
          unsigned long long w = 0;
          lb_wait(d->lb_start, b, threadIdx.x == 0, cfg, &w);
          if (threadIdx.x == 0) s_val = lb_current(w, cfg.epoch) ? (int)(unsigned)w : carry;
        }
        __syncthreads();
        start = s_val;
        __syncthreads();
      }
    }
    const int rel = carry - start;  // image-relative offset of chunk c
    int slot = rel + pre;
    if (cnt) {
      // Octave of the thread's words: found once and advanced (the words are
      // contiguous). Offsets within an octave's bitmap fit 32 bits.
      int o = 0;
      OctDev od = d->oct[im.oct0];
      for (int k = 0; k < WPT; k++) {
        uint32_t wv = words[k];
        if (!wv) continue;
        // Locate octave / layer / row / word of this bitmap word.
        const long long wa = im.bm_begin + w0 + k;
        while (o + 1 < im.n_oct && wa >= d->oct[im.oct0 + o + 1].bm) {
          o++;
          od = d->oct[im.oct0 + o];
        }
        const unsigned rel_w = (unsigned)(wa - od.bm);
        const unsigned lw = (unsigned)od.H * (unsigned)od.wpr;
        const unsigned li = rel_w / lw;
        const unsigned r2 = rel_w - li * lw;
        const int layer = (int)li + 1;
        const int y = (int)(r2 / (unsigned)od.wpr);
        const int wx = (int)(r2 - (unsigned)y * (unsigned)od.wpr);
        while (wv) {
          const int bit = __ffs(wv) - 1;
          wv &= wv - 1;
          if (slot >= 0 && slot < im.cand_cap)
            d->cand[im.cand_off + slot] = make_int4(o, layer, y, wx * kBmCols + bit);
          slot++;
        }
      }
    }
    if (threadIdx.x == 0 && c == d->bmc_pre[b + 1] - 1) {
      const int total = max(0, rel + tot);
      const int nc = min(total, im.cand_cap);
      ImgCounters &k = d->cnt[b];
      k.n_cand_raw = total;
      k.n_cand = nc;
      k.flags = total > im.cand_cap ? TF_CAND : 0;
      lb_store(d->lb_img + b, lb_word(kLbInc, cfg.epoch, nc));
    }
    carry += tot;
  }
  if (g == G - 1 && threadIdx.x < 32) lb_image_prefix(d->lb_img, n, cfg, d->cand_flat);
}

// ------------------------------------------------------------ refinement

__device__ __forceinline__ float det3(float a00, float a01, float a02, float a10, float a11,
                                      float a12, float a20, float a21, float a22) {
  return a00 * (a11 * a22 - a12 * a21) - a01 * (a10 * a22 - a12 * a20) +
         a02 * (a10 * a21 - a11 * a20);
}

__device__ __forceinline__ int round_half_away(float v) {
  const float a = floorf(fabsf(v) + 0.5f);
  return (int)(v >= 0.f ? a : -a);
}

// Levels s - 1 .. s + 2 at rows y - 1 .. y + 1 and columns x - 1 .. x + 1 of
// an octave's level stack G (FP32, or binary16 widened: HF).
template <bool HF>
__device__ __forceinline__ void refine_window(const float *__restrict__ G, int s, int y, int x,
                                              long long ls, int pitch, float (&g)[4][3][3]) {
  const long long base = (long long)(s - 1) * ls + (long long)(y - 1) * pitch + (x - 1);
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int bb = 0; bb < 3; bb++)
#pragma unroll
      for (int cc = 0; cc < 3; cc++) g[a][bb][cc] = lvl_ld(G, HF, base + a * ls + bb * pitch + cc);
}

__global__ void __launch_bounds__(kThreads) k_refine(const Desc *__restrict__ d) {
  pdl_wait();
  const int n = d->n_img;
  const int total = d->cand_flat[n];
  const int S = d->n_scales, bord = d->border, iters = d->max_iter;
  const float T = d->contrast_thr, er = d->edge_ratio;
  // Runs of 32 consecutive candidates go to the warps in turn, block first
  // (run c to block c % G, warp (c / G) % 8): a few thousand candidates still
  // spread over every SM, and the lanes of a warp refine neighbouring
  // candidates (canonical order: same layer, nearby rows), whose 3 x 3 x 3
  // windows share cache sectors.
  const int lane = threadIdx.x & 31;
  const int NW = gridDim.x * (blockDim.x >> 5);
  for (int run = blockIdx.x + gridDim.x * (threadIdx.x >> 5); run * 32 < total; run += NW) {
    const int t = run * 32 + lane;
    if (t >= total) continue;
    const int b = find_owner(d->cand_flat, n, t);
    const ImgDev &im = d->img[b];
    const long long slot = im.cand_off + (t - d->cand_flat[b]);
    const int4 cd = d->cand[slot];
    const int o = cd.x;
    int s = cd.y, y = cd.z, x = cd.w;
    const OctDev od = d->oct[im.oct0 + o];
    const float *G = d->pyr + od.lvl;
    const bool hf = od.half != 0;
    const long long ls = od.lstride;
    const int pitch = od.pitch;
    int code = RC_NOCONV;
    float dX = 0.f, dY = 0.f, dS = 0.f, gx = 0.f, gy = 0.f, gs = 0.f, c = 0.f;
    float hxx = 0.f, hyy = 0.f, hxy = 0.f;
    bool conv = false;
    for (int it = 0; it < iters; it++) {
      // The 3 x 3 x 3 DoG neighbourhood of layers s - 1 .. s + 1: the four
      // Gaussian levels s - 1 .. s + 2 are each loaded once (36 values), and
      // DoG layer k is level k + 1 minus level k, one FP32 subtraction.
      float g[4][3][3];
      if (hf)
        refine_window<true>(G, s, y, x, ls, pitch, g);
      else
        refine_window<false>(G, s, y, x, ls, pitch, g);
      float v[3][3][3];
#pragma unroll
      for (int a = 0; a < 3; a++)
#pragma unroll
        for (int bb = 0; bb < 3; bb++)
#pragma unroll
          for (int cc = 0; cc < 3; cc++) v[a][bb][cc] = g[a + 1][bb][cc] - g[a][bb][cc];
      c = v[1][1][1];
      gx = 0.5f * (v[1][1][2] - v[1][1][0]);
      gy = 0.5f * (v[1][2][1] - v[1][0][1]);
      gs = 0.5f * (v[2][1][1] - v[0][1][1]);
      hxx = v[1][1][2] + v[1][1][0] - 2.0f * c;
      hyy = v[1][2][1] + v[1][0][1] - 2.0f * c;
      const float hss = v[2][1][1] + v[0][1][1] - 2.0f * c;
      hxy = 0.25f * (v[1][2][2] - v[1][2][0] - v[1][0][2] + v[1][0][0]);
      const float hxs = 0.25f * (v[2][1][2] - v[2][1][0] - v[0][1][2] + v[0][1][0]);
      const float hys = 0.25f * (v[2][2][1] - v[2][0][1] - v[0][2][1] + v[0][0][1]);
      const float det = det3(hxx, hxy, hxs, hxy, hyy, hys, hxs, hys, hss);
      if (det == 0.f) { code = RC_SINGULAR; break; }
      // Cramer's rule for H delta = -g.
      dX = det3(-gx, hxy, hxs, -gy, hyy, hys, -gs, hys, hss) / det;
      dY = det3(hxx, -gx, hxs, hxy, -gy, hys, hxs, -gs, hss) / det;
      dS = det3(hxx, hxy, -gx, hxy, hyy, -gy, hxs, hys, -gs) / det;
      if (!isfinite(dX) || !isfinite(dY) || !isfinite(dS)) { code = RC_SINGULAR; break; }
      const float m = fmaxf(fabsf(dX), fmaxf(fabsf(dY), fabsf(dS)));
      if (m < 0.5f) { conv = true; break; }
      if (m > 1e7f) { code = RC_BOUNDS; break; }
      x += round_half_away(dX);
      y += round_half_away(dY);
      s += round_half_away(dS);
      if (s < 1 || s > S || x < bord || x >= od.W - bord || y < bord || y >= od.H - bord) {
        code = RC_BOUNDS;
        break;
      }
    }
    float resp = 0.f;
    if (conv) {
      const float contrast = c + 0.5f * (gx * dX + gy * dY + gs * dS);
      resp = fabsf(contrast);
      if (resp < T) {
        code = RC_CONTRAST;
      } else {
        const float tr = hxx + hyy;
        const float dt = hxx * hyy - hxy * hxy;
        code = (dt <= 0.f || tr * tr * er >= (er + 1.f) * (er + 1.f) * dt) ? RC_EDGE : RC_KEEP;
      }
    }
    RefRec r;
    r.o = o; r.s = s; r.y = y; r.x = x;
    r.dx = dX; r.dy = dY; r.ds = dS; r.resp = resp;
    d->ref[slot] = r;
    d->code[slot] = code;
  }
}

}  // namespace

cudaError_t extrema_set_attributes() { return cudaSuccess; }

int compact_max_ctas() {
  int a = 0, b = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_bm_compact, kThreads, 0);
  if (e == cudaSuccess) e = cc_compact_occupancy(&b);
  return (e == cudaSuccess && a > 0 && b > 0) ? std::min(a, b) : 1;
}

int extrema_warps() { return kExtThreads / 32; }

int extrema_max_ctas(int n_scales) {
  int nb = 0;
  cudaError_t e = cudaErrorInvalidValue;
  switch (n_scales) {
    case 2: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_extrema<2, false>, kExtThreads, 0); break;
    case 3: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_extrema<3, false>, kExtThreads, 0); break;
    case 4: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_extrema<4, false>, kExtThreads, 0); break;
    case 5: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_extrema<5, false>, kExtThreads, 0); break;
    case 6: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_extrema<6, false>, kExtThreads, 0); break;
    default: break;
  }
  return (e == cudaSuccess && nb > 0) ? nb : 1;
}

cudaError_t launch_extrema(const Desc *d, int oct, int n_scales, int grid, cudaStream_t s, bool pdl,
                           bool half) {
#define EXT_CASE(SS)                                                                       \
  case SS:                                                                                 \
    if (half)                                                                              \
      return pdl ? launch_pdl(k_extrema<SS, true>, grid, kExtThreads, 0, s, d, oct)          \
                 : launch_plain(k_extrema<SS, true>, grid, kExtThreads, 0, s, d, oct);       \
    return pdl ? launch_pdl(k_extrema<SS, false>, grid, kExtThreads, 0, s, d, oct)           \
               : launch_plain(k_extrema<SS, false>, grid, kExtThreads, 0, s, d, oct);
  switch (n_scales) {
    EXT_CASE(2)
    EXT_CASE(3)
    EXT_CASE(4)
    EXT_CASE(5)
    EXT_CASE(6)
    default: return cudaErrorInvalidValue;
  }
#undef EXT_CASE
}

cudaError_t launch_bm_compact(const Desc *d, int grid, cudaStream_t s) {
  return launch_pdl(k_bm_compact, grid, kThreads, 0, s, d);
}

cudaError_t launch_refine(const Desc *d, int grid, cudaStream_t s) {
  return launch_pdl(k_refine, grid, kThreads, 0, s, d);
}

}  // namespace sift
