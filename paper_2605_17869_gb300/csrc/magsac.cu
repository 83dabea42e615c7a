// GPU MAGSAC++ homography verification (§3.6 "GPU MAGSAC++").
//
// Hypotheses: eight lanes per minimal sample of 4 correspondences fit the
// homography by the normalised DLT in FP64, one lane per point, then per triangle,
// per equation and per entry. Each image's 4 points are moved to centroid 0 and
// mean distance sqrt(2). The 8 x 8 system of the DLT with h33 = 1 is then solved by
// Gaussian elimination with partial pivoting (rows stay in their lanes, their
// positions are exchanged), and the
// result is de-normalised and scaled to H[2][2] = 1. A sample is degenerate
// (score +inf) in four cases:
//   - an index lies outside [0, n);
//   - three of its normalised points in either image span a triangle of area
//     below 1e-6;
//   - the system is singular, or its solution has |(h, 1)| above 1e9 (the unit
//     null vector's last entry below 1e-9);
//   - |H[2][2]| falls below 1e-12 of the largest entry.
//
// Scoring: one block per hypothesis sums the MAGSAC++ loss over all
// correspondences. The loss is the chi (4 degrees of freedom) likelihood
// marginalised over the noise sigma in [0, sigma_max], truncated at
// k sigma_max (k the 0.99 chi quantile), as an M-estimator loss:
//   rho(r) = P (s^2 gamma(5/2, x) + r^2 / 2 (Gamma(3/2, x) - Gamma(3/2, k^2 / 2))),
//   x = r^2 / (2 s^2), P = 2^(3/2) / (4 s), s = sigma_max; rho(k s) beyond.
// The incomplete gamma functions of half-integer order come from erfc and exp
// by the recurrence Gamma(a + 1, x) = a Gamma(a, x) + x^a e^-x, starting from
// Gamma(1/2, x) = sqrt(pi) erfc(sqrt(x)). The residual is the forward transfer
// error |pi(H x) - x'| in FP32. Each thread adds its correspondences in index
// order, and the block combines the threads in a fixed tree: the scores are
// bitwise reproducible.
//
// Selection: every block takes the smallest score (ties to the smaller index),
// the first one writes it out, and each marks its share of the inliers of its
// model (r <= k sigma_max).
#include <algorithm>
#include <cmath>

#include "sift_dev.cuh"

namespace sift {

namespace {

constexpr int kFitThreads = 32;  // four hypotheses per block: blocks spread over the SMs
constexpr int kScoreThreads = 256;
constexpr int kSelectThreads = 1024;

struct MagsacConst {
  float kk_s2;     // (k sigma_max)^2
  float inv_2s2;   // 1 / (2 sigma_max^2)
  float s2;        // sigma_max^2
  float pref;      // C(4) 2^(3/2) / sigma_max
  float g15_k;     // Gamma(3/2, k^2 / 2)
  float rho_max;   // rho(k sigma_max)
};

__device__ __forceinline__ float magsac_rho(float r2, const MagsacConst &c) {
  if (!(r2 < c.kk_s2)) return c.rho_max;  // beyond the truncation, +inf or NaN
  const float x = r2 * c.inv_2s2;
  const float sx = sqrtf(x), ex = expf(-x);
  const float g15 = 0.886226925452758f * erfcf(sx) + sx * ex;  // Gamma(3/2, x)
  const float g25 = 1.5f * g15 + x * sx * ex;                   // Gamma(5/2, x)
  const float l25 = 1.329340388179137f - g25;                   // gamma(5/2, x)
  return c.pref * (c.s2 * l25 + 0.5f * r2 * (g15 - c.g15_k));
}

// Squared forward transfer error of (a -> b) under H (row-major, FP32).
__device__ __forceinline__ float transfer_r2(const float *H, float2 a, float2 b) {
  const float q0 = fmaf(H[0], a.x, fmaf(H[1], a.y, H[2]));
  const float q1 = fmaf(H[3], a.x, fmaf(H[4], a.y, H[5]));
  const float q2 = fmaf(H[6], a.x, fmaf(H[7], a.y, H[8]));
  if (q2 == 0.f) return INFINITY;
  const float dx = q0 / q2 - b.x, dy = q1 / q2 - b.y;
  return dx * dx + dy * dy;
}

__device__ __forceinline__ double shfl_d(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// Column C of Gaussian elimination with partial pivoting on the 8 x 9 augmented
// system, one row per lane of the group g0 .. g0 + 7; pos is the row's position.
// The row at position >= C with the largest |m[C]| (the first on ties) becomes the
// pivot row and takes position C; the rows below are reduced. False (for the whole
// group) if the column is all zero (singular system).
template <int C>
__device__ __forceinline__ bool elim_step(double (&m)[9], int &pos, double &rinv, int g0, int lane) {
  // |m[C]| as an integer: the bits of non-negative doubles are ordered as they are.
  unsigned long long key = pos >= C ? (unsigned long long)__double_as_longlong(fabs(m[C])) : 0ull;
  int at = pos >= C ? pos : 8, src = lane;
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
    const int a2 = __shfl_xor_sync(0xffffffffu, at, o), s2 = __shfl_xor_sync(0xffffffffu, src, o);
    if (k2 > key || (k2 == key && a2 < at)) {
      key = k2;
      at = a2;
      src = s2;
    }
  }
  if (pos == C) pos = at;
  if (lane == src) pos = C;
  const double ri = 1.0 / shfl_d(m[C], src);
  if (lane == src) rinv = ri;
  const double f = m[C] * ri;
  const bool below = pos > C;
#pragma unroll
  for (int k = C + 1; k < 9; k++) {
    const double p = shfl_d(m[k], src);
    const double r = m[k] - f * p;
    m[k] = below ? r : m[k];
  }
  return key != 0ull;
}

// What bounds the fit is FP64: two lanes per cycle and SM, each operation some tens
// of cycles late. With a thread per hypothesis and one warp per SM it was a chain of
// about 650 dependent operations, 26 us for 1,500 hypotheses; eight lanes shorten
// the chain to about 250 and leave 12 us (both cold, under ncu). The arithmetic of a
// row is unchanged but for the back substitution, which takes its terms from the last
// unknown down.
__global__ void __launch_bounds__(kFitThreads) k_magsac_fit(const float2 *__restrict__ xa,
                                                            const float2 *__restrict__ xb, int n,
                                                            const int *__restrict__ samples,
                                                            int n_hyp, double *__restrict__ models,
                                                            int *__restrict__ valid) {
  const int lane = threadIdx.x & 31, s = lane & 7, g0 = lane & 24;
  const int hyp = blockIdx.x * (kFitThreads / 8) + (threadIdx.x >> 3);
  const int h = min(hyp, n_hyp - 1);  // every lane takes part in the shuffles
  auto group_any = [&](bool v) { return (__ballot_sync(0xffffffffu, v) >> g0 & 0xffu) != 0u; };
  // Lane s: point s & 3 of image a (s < 4) or b.
  const int idx = samples[4 * h + (s & 3)];
  const bool in = idx >= 0 && idx < n;
  bool bad = group_any(!in);
  const float2 pt = (s < 4 ? xa : xb)[in ? idx : 0];
  double x = pt.x, y = pt.y;
  const int im = g0 + (s & 4);  // the image's first lane
  double mx = 0.0, my = 0.0;
#pragma unroll
  for (int j = 0; j < 4; j++) {
    mx += shfl_d(x, im + j);
    my += shfl_d(y, im + j);
  }
  mx /= 4.0;
  my /= 4.0;
  const double dist = sqrt((x - mx) * (x - mx) + (y - my) * (y - my));
  double dsum = 0.0;
#pragma unroll
  for (int j = 0; j < 4; j++) dsum += shfl_d(dist, im + j);
  dsum /= 4.0;
  const double sc = dsum > 0.0 ? 1.4142135623730951 / dsum : 1.0;
  x = sc * x - sc * mx;
  y = sc * y - sc * my;
  {  // lane s: triangle s & 3 of its image: (0, 1, 2), (0, 1, 3), (0, 2, 3), (1, 2, 3)
    const int t = s & 3;
    const int ti = im + (t == 3), tj = im + (t < 2 ? 1 : 2), tm = im + (t == 0 ? 2 : 3);
    const double xi = shfl_d(x, ti), yi = shfl_d(y, ti);
    const double xj = shfl_d(x, tj), yj = shfl_d(y, tj);
    const double xm = shfl_d(x, tm), ym = shfl_d(y, tm);
    const double area = 0.5 * fabs((xj - xi) * (ym - yi) - (yj - yi) * (xm - xi));
    bad |= group_any(area < 1e-6);
  }
  // A h = 0 with h33 = 1: rows (x, y, 1, 0, 0, 0, -u x, -u y | u) and
  // (0, 0, 0, x, y, 1, -v x, -v y | v) (signs flipped from the DLT rows); lane s has
  // row s: correspondence s / 2, u for even s and v for odd.
  double m[9];
  {
    const int j = s >> 1;
    const double ax = shfl_d(x, g0 + j), ay = shfl_d(y, g0 + j);
    const double u = shfl_d(x, g0 + 4 + j), v = shfl_d(y, g0 + 4 + j);
    const bool odd = s & 1;
    const double q = odd ? v : u;
    m[0] = odd ? 0.0 : ax;
    m[1] = odd ? 0.0 : ay;
    m[2] = odd ? 0.0 : 1.0;
    m[3] = odd ? ax : 0.0;
    m[4] = odd ? ay : 0.0;
    m[5] = odd ? 1.0 : 0.0;
    m[6] = -q * ax;
    m[7] = -q * ay;
    m[8] = q;
  }
  int pos = s;
  double rinv = 0.0;
  bool ok8 = elim_step<0>(m, pos, rinv, g0, lane);
  ok8 &= elim_step<1>(m, pos, rinv, g0, lane);
  ok8 &= elim_step<2>(m, pos, rinv, g0, lane);
  ok8 &= elim_step<3>(m, pos, rinv, g0, lane);
  ok8 &= elim_step<4>(m, pos, rinv, g0, lane);
  ok8 &= elim_step<5>(m, pos, rinv, g0, lane);
  ok8 &= elim_step<6>(m, pos, rinv, g0, lane);
  ok8 &= elim_step<7>(m, pos, rinv, g0, lane);
  bad |= !ok8;
  // Back substitution: the row at position c gives h[c], which every row above it
  // subtracts at once.
  double hn[9];
  hn[8] = 1.0;
#pragma unroll
  for (int c = 7; c >= 0; c--) {
    const unsigned who = __ballot_sync(0xffffffffu, pos == c) >> g0 & 0xffu;
    hn[c] = shfl_d(m[8] * rinv, g0 + __ffs(who) - 1);
    m[8] -= m[c] * hn[c];  // (only the rows above are read again)
  }
  double nn = 1.0;
#pragma unroll
  for (int k = 0; k < 8; k++) nn += hn[k] * hn[k];
  bad |= !(nn <= 1e18);  // the null vector's h33 component below 1e-9 (or not finite)
  // H = Tb^-1 Hn Ta with Ta = [[sa, 0, -sa ax], [0, sa, -sa ay], [0, 0, 1]] and
  // Tb^-1 = [[1/sb, 0, bx], [0, 1/sb, by], [0, 0, 1]]. Lane s: entry s; all: entry 8.
  const double sa = shfl_d(sc, g0), ax = shfl_d(mx, g0), ay = shfl_d(my, g0);
  const double sb = shfl_d(sc, g0 + 4), bx = shfl_d(mx, g0 + 4), by = shfl_d(my, g0 + 4);
  auto third = [&](double a0, double a1, double a2) { return a2 - a0 * sa * ax - a1 * sa * ay; };  // of Hn Ta
  const int row = s / 3, col = s - 3 * row;
  const double a0 = row == 0 ? hn[0] : row == 1 ? hn[3] : hn[6];
  const double a1 = row == 0 ? hn[1] : row == 1 ? hn[4] : hn[7];
  const double a2 = row == 0 ? hn[2] : row == 1 ? hn[5] : hn[8];
  const double g8 = third(hn[6], hn[7], hn[8]);
  const double ge = col == 2 ? third(a0, a1, a2) : (col ? a1 : a0) * sa;
  const double gl = col == 2 ? g8 : (col ? hn[7] : hn[6]) * sa;  // the last row's entry of this column
  const double e = row == 2 ? ge : ge / sb + (row ? by : bx) * gl;
  double big = fmax(fabs(e), fabs(g8));
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
  bad |= !(fabs(g8) >= 1e-12 * big);
  if (hyp >= n_hyp) return;
  if (!bad) {
    const double inv = 1.0 / g8;
    models[9 * h + s] = e * inv;
    if (s == 7) models[9 * h + 8] = 1.0;
  }
  if (s == 0) valid[h] = bad ? 0 : 1;
}

__global__ void __launch_bounds__(kScoreThreads) k_magsac_score(const float2 *__restrict__ xa,
                                                                const float2 *__restrict__ xb,
                                                                int n, const double *__restrict__ models,
                                                                const int *__restrict__ valid,
                                                                int n_hyp, MagsacConst c,
                                                                float *__restrict__ scores) {
  pdl_wait();  // the models
  __shared__ float red[kScoreThreads / 32];
  const int tid = threadIdx.x;
  for (int h = blockIdx.x; h < n_hyp; h += gridDim.x) {
    if (!valid[h]) {  // block-uniform
      if (tid == 0) scores[h] = INFINITY;
      continue;
    }
    float H[9];
#pragma unroll
    for (int k = 0; k < 9; k++) H[k] = (float)models[9 * h + k];
    float acc = 0.f;
    for (int i = tid; i < n; i += kScoreThreads) acc += magsac_rho(transfer_r2(H, xa[i], xb[i]), c);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((tid & 31) == 0) red[tid >> 5] = acc;
    __syncthreads();
    if (tid == 0) {
      float s = red[0];
#pragma unroll
      for (int w = 1; w < kScoreThreads / 32; w++) s += red[w];
      scores[h] = s;
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void better(float &v, int &i, float v2, int i2) {
  if (v2 < v || (v2 == v && i2 < i)) {
    v = v2;
    i = i2;
  }
}

__global__ void __launch_bounds__(kSelectThreads) k_magsac_select(
    const float2 *__restrict__ xa, const float2 *__restrict__ xb, int n,
    const double *__restrict__ models, const float *__restrict__ scores, int n_hyp, MagsacConst c,
    double *__restrict__ H_out, int *__restrict__ best_out, float *__restrict__ score_out,
    unsigned char *__restrict__ inliers, float *__restrict__ scores_out) {
  __shared__ float sv[kSelectThreads / 32];
  __shared__ int si[kSelectThreads / 32];
  __shared__ float s_H[9];
  __shared__ int s_best;
  pdl_wait();  // the scores
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool first = blockIdx.x == 0;
  float v = INFINITY;
  int bi = 0x7fffffff;
  for (int h = tid; h < n_hyp; h += kSelectThreads) {
    const float s = scores[h];
    if (scores_out && first) scores_out[h] = s;
    better(v, bi, s, h);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float v2 = __shfl_xor_sync(0xffffffffu, v, o);
    const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
    better(v, bi, v2, i2);
  }
  if (lane == 0) {
    sv[warp] = v;
    si[warp] = bi;
  }
  __syncthreads();
  if (tid == 0) {
    float bv = sv[0];
    int b = si[0];
    for (int w = 1; w < kSelectThreads / 32; w++) better(bv, b, sv[w], si[w]);
    const int best = (bv < INFINITY) ? b : -1;
    s_best = best;
    if (first) {
      *best_out = best;
      *score_out = best >= 0 ? bv : INFINITY;
    }
    for (int k = 0; k < 9; k++) {
      const double e = best >= 0 ? models[9 * best + k] : 0.0;
      if (first) H_out[k] = e;
      s_H[k] = (float)e;
    }
  }
  __syncthreads();
  const int best = s_best;
  for (int i = blockIdx.x * kSelectThreads + tid; i < n; i += gridDim.x * kSelectThreads)
    inliers[i] = (best >= 0 && transfer_r2(s_H, xa[i], xb[i]) <= c.kk_s2) ? 1 : 0;
}

// Gamma(3/2, x) and gamma(5/2, x) in double (host), by the same recurrences.
double upper_g15(double x) { return 0.5 * std::sqrt(M_PI) * std::erfc(std::sqrt(x)) + std::sqrt(x) * std::exp(-x); }
double lower_g25(double x) {
  return 0.75 * std::sqrt(M_PI) - (1.5 * upper_g15(x) + x * std::sqrt(x) * std::exp(-x));
}

// k: the 0.99 quantile of the chi distribution with 4 degrees of freedom.
// P(chi^2_4 <= 2y) = 1 - e^-y (1 + y); Newton on e^-y (1 + y) = 0.01.
double chi4_quantile_099() {
  double y = 6.0;
  for (int it = 0; it < 60; it++) {
    const double f = std::exp(-y) * (1.0 + y) - 0.01;
    const double df = -std::exp(-y) * y;
    const double step = f / df;
    y -= step;
    if (std::fabs(step) < 1e-15 * y) break;
  }
  return std::sqrt(2.0 * y);
}

MagsacConst make_const(float sigma_max) {
  const double s = sigma_max, k = chi4_quantile_099();
  const double pref = 0.25 * std::pow(2.0, 1.5) / s;
  const double xk = 0.5 * k * k;
  MagsacConst c;
  c.kk_s2 = (float)(k * k * s * s);
  c.inv_2s2 = (float)(1.0 / (2.0 * s * s));
  c.s2 = (float)(s * s);
  c.pref = (float)pref;
  c.g15_k = (float)upper_g15(xk);
  c.rho_max = (float)(pref * (s * s * lower_g25(xk)));  // the r^2 term vanishes at k sigma_max
  return c;
}

}  // namespace

size_t magsac_workspace_bytes(int n_hyp) {
  return (size_t)n_hyp * (9 * sizeof(double) + sizeof(int) + sizeof(float)) + 256;
}

cudaError_t launch_magsac(const float *xa, const float *xb, int n, const int *samples, int n_hyp,
                          float sigma_max, void *ws, cudaStream_t s, double *H_out, int *best_out,
                          float *score_out, unsigned char *inliers, float *scores_out) {
  char *p = static_cast<char *>(ws);
  double *models = reinterpret_cast<double *>(p);
  int *valid = reinterpret_cast<int *>(p + (size_t)n_hyp * 9 * sizeof(double));
  float *scores = reinterpret_cast<float *>(p + (size_t)n_hyp * (9 * sizeof(double) + sizeof(int)));
  const MagsacConst c = make_const(sigma_max);
  const float2 *a = reinterpret_cast<const float2 *>(xa);
  const float2 *b = reinterpret_cast<const float2 *>(xb);
  int dev = 0, n_sm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e = launch_plain(k_magsac_fit, (n_hyp + kFitThreads / 8 - 1) / (kFitThreads / 8), kFitThreads, 0,
                               s, a, b, n, samples, n_hyp, models, valid);
  if (e != cudaSuccess) return e;
  const int grid = n_hyp < 8 * n_sm ? n_hyp : 8 * n_sm;
  e = launch_pdl(k_magsac_score, grid, kScoreThreads, 0, s, a, b, n, models, valid, n_hyp, c,
                   scores);
  if (e != cudaSuccess) return e;
  // Every block reads all scores, so more than one only where the points are many.
  // One block against this many (us, cold): 8,192 points and 1,500 hypotheses 12.8
  // against 8.9, 20,011 and 500 23.8 against 9.8, 65,536 and 500 66 against 8.5.
  const int sel = std::max(1, std::min({n_sm, n / (4 * kSelectThreads), n / n_hyp}));
  return launch_pdl(k_magsac_select, sel, kSelectThreads, 0, s, a, b, n, models, scores, n_hyp, c,
                      H_out, best_out, score_out, inliers, scores_out);
}

}  // namespace sift
