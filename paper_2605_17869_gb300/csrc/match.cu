// Symmetric ratio-test matcher (§3.4 "Descriptor Matching", first backend):
// the similarity matrix of two descriptor sets from fp16 tensor-core products,
// nearest neighbours in both directions, mutual consistency and Lowe's ratio
// test on both sides.
//
// The similarity matrix is a dense N x M x 128 contraction, so it runs on the
// 5th-generation tensor cores, and only its rows' best entries leave the SM. Both
// sets are first converted once to fp16 in the core-matrix layout the tensor core
// reads. One persistent grid then takes the work items of both directions, 256
// rows of one set against a run of 256-row tiles of the other:
//  * a control thread brings the rows (64 KB) and the tiles (64 KB each, two
//    buffers) to shared memory by bulk copies on mbarriers and issues, per tile
//    and 128-row half, 8 tcgen05.mma (M = 128, N = 256, K = 16, FP32 accumulation in
//    that half's 256 TMEM columns);
//  * four warps per half read the accumulators back with tcgen05.ld and keep each
//    row's best index and two best similarities in registers over the whole run,
//    while the tensor core works on the other half. 16 columns whose maxima beat no row's
//    second best are left at that (most are).
// Rows of 256 halve the tiles' traffic from L2 against rows of 128 (one SM's tensor
// core takes a 64 KB tile in about 1,000 cycles, close to what L2 gives it in that
// time). The last kernel merges the runs of each row in column order (ties keep the
// smaller index) and applies the mutual check and the ratio tests. The tensor core's
// accumulation order is fixed, so results are reproducible.
//
// What bounds it at 8192 x 7801: the minima and maxima of the read-back (the ALU
// pipe 47%, the tensor core about 40%), with two warps per scheduler; 53 us of the
// call's 61. Before, a grid of one-tile blocks per direction (2 x 61 us, nothing
// overlapped within a block), two merge kernels (2 x 20 us) and two conversions: 162
// us. A branch per similarity or per 8 of them instead of the network: 102 us.
#include <cuda_fp16.h>

#include <algorithm>

#include "sift_dev.cuh"

namespace sift {

namespace {

constexpr int kMM = 128;      // rows per accumulator (TMEM lanes)
constexpr int kMN = 256;      // rows per item and per tile (accumulator columns)
constexpr int kDim = 128;     // descriptor length (K)
constexpr int kEpiThreads = 256;                // two halves x four warps
constexpr int kMThreads = kEpiThreads + 32;     // and the control warp
constexpr int kSmemTile = kMN * kDim * 2;       // 64 KB of fp16
constexpr int kMatchSmem = 3 * kSmemTile;       // the item's rows, two tile buffers
constexpr unsigned kMaxPolls = 1u << 22;

__device__ __forceinline__ unsigned saddr(const void *p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor of a K-major operand without swizzle: 8 x 8
// fp16 core matrices of 128 contiguous bytes, the next core matrix along K at
// +128 bytes (leading byte offset), the next 8-row group at +2048 bytes (stride
// byte offset); bits 46-47 hold the descriptor version (1).
__device__ __forceinline__ unsigned long long smem_desc(unsigned addr) {
  const unsigned long long lbo = 128 >> 4, sbo = 2048 >> 4;
  return (unsigned long long)((addr >> 4) & 0x3FFFu) | (lbo << 16) | (sbo << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), A and
// B fp16 (formats 0), both K-major, N >> 3 in bits 17-22, M >> 4 in bits 24-28.
constexpr unsigned kIdesc = (1u << 4) | ((unsigned)(kMN >> 3) << 17) | ((unsigned)(kMM >> 4) << 24);

__device__ __forceinline__ void mbar_init(unsigned long long *m, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(m)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long *m) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(m)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *m, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(saddr(m)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded: false after kMaxPolls polls (each may suspend the thread briefly), or once
// another thread of the block has given up, which *abort records.
__device__ __forceinline__ bool mbar_wait(unsigned long long *m, unsigned parity, volatile int *abort) {
  for (unsigned i = 0; i < kMaxPolls; i++) {
    if (mbar_try_wait(m, parity)) return true;
    if ((i & 63) == 63 && *abort) return false;
  }
  *abort = 1;
  return false;
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Both descriptor sets (FP32, kDim per row, row-major) as fp16 core matrices in
// global memory, the layout the tensor core reads from shared memory: core
// matrix (row / 8, k / 8) at byte (row / 8) * 2048 + (k / 8) * 128, 8 rows x
// 16 bytes inside; rows n .. n_pad - 1 are zero. 256 rows are then 64 contiguous
// KB. Thread: 8 elements; a warp takes 8 rows x 4 groups of 8, so that it reads
// and writes whole 128-byte lines. err[1] is set if a value is
// not finite in fp16.
__global__ void __launch_bounds__(256) k_to_core_matrices(const float *__restrict__ A, int n_a, int pa,
                                                          unsigned char *dst_a, const float *__restrict__ B,
                                                          int n_b, int pb, unsigned char *dst_b, int *err) {
  int c = blockIdx.x * 256 + threadIdx.x;
  const bool second = c >= pa * (kDim / 8);
  if (second) c -= pa * (kDim / 8);
  if (second && c >= pb * (kDim / 8)) return;
  const float *src = second ? B : A;
  const int n = second ? n_b : n_a;
  unsigned char *dst = second ? dst_b : dst_a;
  const int w = c >> 5, lane = c & 31;
  const int row = (w >> 2) * 8 + (lane & 7), kg = (w & 3) * 4 + (lane >> 3);
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (row < n) {
    const float4 *p = reinterpret_cast<const float4 *>(src + (size_t)row * kDim + kg * 8);
    const float4 a = __ldg(p), b = __ldg(p + 1);
    const __half2 h0 = __floats2half2_rn(a.x, a.y), h1 = __floats2half2_rn(a.z, a.w);
    const __half2 h2 = __floats2half2_rn(b.x, b.y), h3 = __floats2half2_rn(b.z, b.w);
    v = make_uint4(*reinterpret_cast<const unsigned *>(&h0), *reinterpret_cast<const unsigned *>(&h1),
                   *reinterpret_cast<const unsigned *>(&h2), *reinterpret_cast<const unsigned *>(&h3));
    // An exponent of all ones: infinite or NaN.
    const auto odd = [](unsigned w) { return (w & 0x7c00u) == 0x7c00u || (w & 0x7c000000u) == 0x7c000000u; };
    if (odd(v.x) || odd(v.y) || odd(v.z) || odd(v.w)) err[1] = 1;
  }
  *reinterpret_cast<uint4 *>(dst + (size_t)(row >> 3) * 2048 + kg * 128 + (row & 7) * 16) = v;
}

__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long *m, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(m)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes,
                                         unsigned long long *m) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          saddr(dst)),
      "l"(src), "r"(bytes), "r"(saddr(m))
      : "memory");
}

// One direction of the search: rows of `rows` (n of them, core matrices) against
// the columns `cols` (m of them, `tiles` tiles of 256 in runs of MatchPlan::run).
// Results of run c and row i at [c * n_pad + i].
struct MatchSide {
  const unsigned char *rows, *cols;
  int n, m, n_pad, tiles, runs;
  int *best;
  float *s1, *s2;
};
struct MatchPlan {
  MatchSide side[2];
  int run;       // tiles per run
  int items[2];  // row blocks x runs of each side
};

__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// 32 accumulator columns of the warp's 32 rows, from column `col` of the tile.
__device__ __forceinline__ void tmem_ld32(unsigned (&v)[32], unsigned addr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, "
      "%30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
        "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(addr));
}

struct Top2 {
  float s1, s2;
  int b1;
};

// The row's best two over 32 more columns j0 .. j0 + 31, in column order: 16
// columns at a time, their maximum first (three-input maxima). Where no row of the
// warp has a maximum above its second best, which is the usual case after the first
// few hundred columns, that is all; else the 16 columns' best two come from a
// network of minima and maxima without branches, and where a best is new its first
// column is looked for. No value is NaN.
__device__ __forceinline__ void top2_update(Top2 &t, const unsigned (&v)[32], int j0) {
#pragma unroll
  for (int q = 0; q < 2; q++) {
    float e[16];
#pragma unroll
    for (int k = 0; k < 16; k++) e[k] = __uint_as_float(v[16 * q + k]);
    float m = fmax3(fmax3(e[0], e[1], e[2]), fmax3(e[3], e[4], e[5]), fmax3(e[6], e[7], e[8]));
    m = fmax3(m, fmax3(fmax3(e[9], e[10], e[11]), e[12], e[13]), fmaxf(e[14], e[15]));
    if (!__any_sync(0xffffffffu, m > t.s2)) continue;
    float a[8], b[8];  // best and second best of pairs, then of quadruples, ...
#pragma unroll
    for (int k = 0; k < 8; k++) {
      a[k] = fmaxf(e[2 * k], e[2 * k + 1]);
      b[k] = fminf(e[2 * k], e[2 * k + 1]);
    }
#pragma unroll
    for (int n = 4; n > 0; n >>= 1)
#pragma unroll
      for (int k = 0; k < n; k++) {
        b[k] = fmax3(fminf(a[k], a[k + n]), b[k], b[k + n]);
        a[k] = fmaxf(a[k], a[k + n]);
      }
    if (__any_sync(0xffffffffu, m > t.s1)) {
      int k1 = 15;
#pragma unroll
      for (int k = 14; k >= 0; k--) k1 = e[k] == m ? k : k1;
      t.b1 = m > t.s1 ? j0 + 16 * q + k1 : t.b1;
    }
    t.s2 = fmax3(fminf(t.s1, m), t.s2, b[0]);
    t.s1 = fmaxf(t.s1, m);
  }
}

// The same where a value may be NaN, which is never larger than another.
__device__ __forceinline__ void top2_update_nan(Top2 &t, const unsigned (&v)[32], int j0) {
#pragma unroll
  for (int k = 0; k < 32; k++) {
    const float e = __uint_as_float(v[k]);
    if (e > t.s1) {
      t.s2 = t.s1;
      t.s1 = e;
      t.b1 = j0 + k;
    } else if (e > t.s2) {
      t.s2 = e;
    }
  }
}

__global__ void __launch_bounds__(kMThreads, 1) k_match(const __grid_constant__ MatchPlan plan, int *err) {
  extern __shared__ __align__(128) unsigned char sm[];
  // full: a tile buffer's (0, 1) or the rows' (2) copy landed; done[h]: half h's
  // MMAs of a tile finished; drained[h]: its accumulators are read.
  __shared__ __align__(8) unsigned long long full[3], done[2], drained[2];
  __shared__ unsigned tmem_sh;
  __shared__ volatile int abort_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == kEpiThreads / 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_sh)),
                 "r"(2 * kMN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    abort_sh = 0;
    for (int i = 0; i < 3; i++) mbar_init(&full[i], 1);
    for (int h = 0; h < 2; h++) {
      mbar_init(&done[h], 1);
      mbar_init(&drained[h], 4);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();  // the core matrices
  const bool finite = err[1] == 0;  // no operand is infinite or NaN: no similarity is
  const unsigned tmem = tmem_sh;
  const int n_items = plan.items[0] + plan.items[1];
  unsigned tile = 0;  // tiles of this block so far: tile k is in buffer k & 1
  unsigned item_no = 0;
  unsigned copies[3] = {0, 0, 0}, commits[2] = {0, 0};  // issued by the control thread
  bool ok = true;
  for (int it = blockIdx.x; it < n_items && ok; it += gridDim.x, item_no++) {
    const int sd = it >= plan.items[0];
    const MatchSide &S = plan.side[sd];
    const int u = it - (sd ? plan.items[0] : 0);
    const int run = u % S.runs, r0 = (u / S.runs) * kMN;
    const int t0 = run * plan.run, nt = min(plan.run, S.tiles - t0);
    const bool two = r0 + kMM < S.n;  // rows in the second half
    if (warp == kEpiThreads / 32) {
      if (lane == 0) {
        auto copy = [&](int to, const unsigned char *from, int bar) {
          mbar_arrive_expect_tx(&full[bar], kSmemTile);
          bulk_g2s(sm + to * kSmemTile, from, kSmemTile, &full[bar]);
          copies[bar]++;
        };
        // The last tile's MMAs have finished: the rows and both buffers are free.
        auto last_tile_done = [&] {
          return tile == 0 || (mbar_wait(&done[0], (tile - 1) & 1, &abort_sh) &&
                               mbar_wait(&done[1], (tile - 1) & 1, &abort_sh));
        };
        ok = last_tile_done();
        if (ok) {
          copy(0, S.rows + (size_t)r0 * kDim * 2, 2);
          copy(1 + (tile & 1), S.cols + (size_t)t0 * kSmemTile, tile & 1);
          ok = mbar_wait(&full[2], item_no & 1, &abort_sh);
        }
        for (int t = 0; t < nt && ok; t++, tile++) {
          const unsigned buf = tile & 1;
          if (t + 1 < nt) {  // into the other buffer, which the previous tile's MMAs read
            ok = last_tile_done();
            if (!ok) break;
            copy(1 + (buf ^ 1), S.cols + (size_t)(t0 + t + 1) * kSmemTile, buf ^ 1);
          }
          ok = mbar_wait(&full[buf], (tile >> 1) & 1, &abort_sh);
          for (int h = 0; h < 2 && ok; h++) {
            if (tile > 0) ok = mbar_wait(&drained[h], (tile - 1) & 1, &abort_sh);
            if (!ok) break;
            tc_fence_after();
            if (h == 0 || two) {
#pragma unroll
              for (int kk = 0; kk < kDim / 16; kk++) {
                const unsigned long long da = smem_desc(saddr(sm) + h * (kSmemTile / 2) + kk * 256);
                const unsigned long long db = smem_desc(saddr(sm) + (1 + buf) * kSmemTile + kk * 256);
                asm volatile(
                    "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                    " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem + h * kMN),
                    "l"(da), "l"(db), "r"(kIdesc), "r"(kk)
                    : "memory");
              }
            }
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    saddr(&done[h]))
                : "memory");
            commits[h]++;
          }
        }
      }
      ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
    } else {
      const int h = warp >> 2;
      const unsigned taddr = tmem + ((unsigned)(32 * (warp & 3)) << 16) + h * kMN;
      Top2 best{-INFINITY, -INFINITY, -1};
      for (int t = 0; t < nt && ok; t++, tile++) {
        ok = __all_sync(0xffffffffu, mbar_wait(&done[h], tile & 1, &abort_sh));
        if (!ok) break;
        tc_fence_after();
        const int j0 = (t0 + t) * kMN;
        const int cols = min(kMN, S.m - j0);
        if (h == 0 || two) {
          unsigned va[32], vb[32];
          tmem_ld32(va, taddr);
#pragma unroll 1
          for (int c = 0; c < cols; c += 64) {
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            tmem_ld32(vb, taddr + c + 32);
            if (c + 32 > cols) {
#pragma unroll
              for (int k = 0; k < 32; k++) va[k] = c + k < cols ? va[k] : 0xff800000u;  // -inf
            }
            if (finite) top2_update(best, va, j0 + c);
            else top2_update_nan(best, va, j0 + c);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (c + 64 < cols) tmem_ld32(va, taddr + c + 64);
            if (c + 64 > cols) {
#pragma unroll
              for (int k = 0; k < 32; k++) vb[k] = c + 32 + k < cols ? vb[k] : 0xff800000u;
            }
            if (finite) top2_update(best, vb, j0 + c + 32);
            else top2_update_nan(best, vb, j0 + c + 32);
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&drained[h]);
      }
      const int row = r0 + h * kMM + 32 * (warp & 3) + lane;
      if (ok && row < S.n) {
        const size_t o = (size_t)run * S.n_pad + row;
        S.best[o] = best.b1;
        S.s1[o] = best.s1;
        S.s2[o] = best.s2;
      }
    }
  }
  if (!ok) {  // a wait gave up: flag, wait (again with a limit) for what is in flight, free, exit
    *err = 1;
    if (warp == kEpiThreads / 32 && lane == 0) {
      auto settle = [](unsigned long long *m, unsigned n) {
        for (unsigned p = 0; n > 0 && p < kMaxPolls && !mbar_try_wait(m, (n - 1) & 1); p++) {
        }
      };
      for (int i = 0; i < 3; i++) settle(&full[i], copies[i]);
      for (int h = 0; h < 2; h++) settle(&done[h], commits[h]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kEpiThreads / 32) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kMN)
                 : "memory");
  }
}

// Row i of a side: its runs merged in column order (ties keep the smaller index).
__device__ __forceinline__ Top2 merge_runs(const MatchSide &S, int i) {
  Top2 t{-INFINITY, -INFINITY, -1};
  for (int c = 0; c < S.runs; c++) {
    const size_t o = (size_t)c * S.n_pad + i;
    const float a1 = S.s1[o], a2 = S.s2[o];
    if (a1 > t.s1) {
      t.s2 = fmaxf(t.s1, a2);
      t.s1 = a1;
      t.b1 = S.best[o];
    } else {
      t.s2 = fmaxf(t.s2, a1);
    }
  }
  return t;
}

__device__ __forceinline__ float unit_distance(float s) { return sqrtf(fmaxf(0.f, 2.f - 2.f * s)); }

// Mutual nearest neighbours passing the ratio test on both sides; -1 else,
// -2 for every row if a bounded device wait gave up.
__global__ void __launch_bounds__(128) k_match_final(const __grid_constant__ MatchPlan plan, float ratio,
                                                     const int *err, int *out) {
  pdl_wait();
  const int i = blockIdx.x * 128 + threadIdx.x;
  const int n_a = plan.side[0].n, n_b = plan.side[1].n;
  if (i >= n_a) return;
  int m = -1;
  if (*err) {
    m = -2;
  } else if (n_a >= 2 && n_b >= 2) {
    const Top2 a = merge_runs(plan.side[0], i);
    if (a.b1 >= 0 && unit_distance(a.s1) < ratio * unit_distance(a.s2)) {
      const Top2 b = merge_runs(plan.side[1], a.b1);
      if (b.b1 == i && unit_distance(b.s1) < ratio * unit_distance(b.s2)) m = a.b1;
    }
  }
  out[i] = m;
}

}  // namespace

static inline size_t pad256(int n) { return (size_t)((n + kMN - 1) / kMN) * kMN; }
static inline size_t align256(size_t v) { return (v + 255) / 256 * 256; }

// Tiles per run: the items of both directions go to the SMs one at a time, so the
// run length that minimises waves x (tiles of a run + 1 for the item's own rows).
static int match_run(int n_a, int n_b, int n_sm) {
  const int ta = (int)(pad256(n_a) / kMN), tb = (int)(pad256(n_b) / kMN);
  int best = 1;
  long long cost = -1;
  for (int L = 1; L <= std::max(ta, tb); L++) {
    const long long items = (long long)ta * ((tb + L - 1) / L) + (long long)tb * ((ta + L - 1) / L);
    const long long c = (items + n_sm - 1) / n_sm * (L + 1);
    if (cost < 0 || c < cost) {
      cost = c;
      best = L;
    }
  }
  return best;
}

// Workspace: error word, both sets in core-matrix layout, per-run results of both
// directions.
size_t match_workspace_bytes(int n_a, int n_b, int n_sm) {
  const size_t pa = pad256(n_a), pb = pad256(n_b);
  const int L = match_run(n_a, n_b, n_sm);
  const size_t ra = (pb / kMN + L - 1) / L, rb = (pa / kMN + L - 1) / L;
  return 256 + align256(pa * kDim * 2) + align256(pb * kDim * 2) + align256(ra * pa * 12) +
         align256(rb * pb * 12);
}

cudaError_t match_set_attributes() {
  return cudaFuncSetAttribute(k_match, cudaFuncAttributeMaxDynamicSharedMemorySize, kMatchSmem);
}

cudaError_t launch_match(const float *A, int n_a, const float *B, int n_b, float ratio, void *ws,
                         int *out, int n_sm, cudaStream_t s) {
  if (n_a == 0) return cudaSuccess;
  if (n_b == 0) return cudaMemsetAsync(out, 0xff, (size_t)n_a * sizeof(int), s);  // -1: no pair
  const size_t pa = pad256(n_a), pb = pad256(n_b);
  char *w = static_cast<char *>(ws);
  int *err = reinterpret_cast<int *>(w);
  size_t o = 256;
  auto take = [&](size_t bytes) {
    char *p = w + o;
    o += align256(bytes);
    return p;
  };
  unsigned char *cm_a = reinterpret_cast<unsigned char *>(take(pa * kDim * 2));
  unsigned char *cm_b = reinterpret_cast<unsigned char *>(take(pb * kDim * 2));
  MatchPlan plan;
  plan.run = match_run(n_a, n_b, n_sm);
  for (int k = 0; k < 2; k++) {
    MatchSide &S = plan.side[k];
    S.rows = k ? cm_b : cm_a;
    S.cols = k ? cm_a : cm_b;
    S.n = k ? n_b : n_a;
    S.m = k ? n_a : n_b;
    S.n_pad = (int)(k ? pb : pa);
    S.tiles = (int)((k ? pa : pb) / kMN);
    S.runs = (S.tiles + plan.run - 1) / plan.run;
    const size_t e = (size_t)S.runs * S.n_pad;
    S.best = reinterpret_cast<int *>(take(e * 12));
    S.s1 = reinterpret_cast<float *>(S.best + e);
    S.s2 = S.s1 + e;
    plan.items[k] = S.n_pad / kMN * S.runs;
  }
  cudaError_t e = cudaMemsetAsync(err, 0, 2 * sizeof(int), s);
  if (e == cudaSuccess)
    e = launch_plain(k_to_core_matrices, (int)(((pa + pb) * (kDim / 8) + 255) / 256), 256, 0, s, A,
                               n_a, (int)pa, cm_a, B, n_b, (int)pb, cm_b, err);
  if (e == cudaSuccess)
    e = launch_pdl(k_match, std::min(n_sm, plan.items[0] + plan.items[1]), kMThreads, kMatchSmem, s, plan, err);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_match_final, (n_a + 127) / 128, 128, 0, s, plan, ratio, err, out);
}

}  // namespace sift
