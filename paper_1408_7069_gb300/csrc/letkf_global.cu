// The global ETKF (Section 3.1.1: one domain observing every slope, partition
// 1) for ensembles of more than 64 members (the paper's global curves reach
// m ~ 626, Section 5.1; from m = 101 on this path is faster than the one-CTA
// Jacobi, which also stops at 128 columns). The transform needs only
// A^-1/2 and A^-1 c, so the eigendecomposition is replaced by matrix products:
//   Gram     A = (m-1)/rho I + S^T S, c = S^T s (the split-K Gram of
//            letkf_domains.cu), s_A = |A|_F >= lambda_max
//   root     coupled Newton-Schulz on Y0 = A / s_A, Z0 = I:
//            T = a I - b Z Y, Y <- Y T, Z <- T Z, converging to
//            Y -> (A/s_A)^1/2 and Z -> (A/s_A)^-1/2, FP32 matrix products
//   mean     wbar = A^-1 c by iterative refinement: residual c - A wbar in
//            FP64, correction Z (Z r) / s_A in FP32
//   apply    P = X' sqrt((m-1) / s_A) Z over all state rows, Xa = xbar + X' wbar + P,
//            X' wbar in pairs of floats (FP64 took 1 us more at m = 101, 5 us at m = 626),
//            mean and spread. P's mean over the members is zero but for Z's rounding, which grows
//            with kappa, and the rounding of the slopes' means, part of whose error in
//            X' wbar it takes back: it is kept up to NR_KEEP and taken out beyond
//
// Scaled steps: the singular values x = sqrt(eig(Z Y)) start in [x_0, 1] with
// x_0 = sqrt(alpha / s_A), alpha = (m-1)/rho the smallest eigenvalue A can have.
// A step maps x -> (3 mu x - (mu x)^3) / 2; mu^2 = 3 / (1 + x_0 + x_0^2) makes
// both ends of the interval equal, so that the lower one grows by up to
// 1.5 sqrt(3) = 2.6 per step instead of 1.5, and the next interval is known
// without looking at the matrices (Chen & Chow's and Higham's scaled iterations).
// From x_0 = 0.003 (the prior draw's kappa of 1e5) ten steps reach 1 - 2^-21
// where the unscaled iteration took 26; a loop's kappa of 50 takes six.
//
// Everything between the Gram and the apply is one cooperative kernel: a grid
// barrier (about 1 us) per dependent stage instead of a launch, and the
// number of iterations is the device's own. (Forming only the upper triangle
// of these products of commuting symmetric matrices and mirroring it would
// halve the flops, but it breaks the coupling of the iteration: in FP32 at the
// prior draw's kappa ~ 1.5e5, m = 200, the symmetrised iteration overflows
// after 20 steps where the full one converges.)
#include <math.h>

#include "letkf_df.cuh"

namespace {

// acc += rows (4 floats at x of each of n columns, stride xs float4) times the 4
// columns at y (stride ys float4): packed FMAs over row pairs.
__device__ __forceinline__ void tile4x4(float2 (&acc)[4][2], float4 a, float4 b) {
  const float bj[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 bb = make_float2(bj[j], bj[j]);
    acc[j][0] = __ffma2_rn(make_float2(a.x, a.y), bb, acc[j][0]);
    acc[j][1] = __ffma2_rn(make_float2(a.z, a.w), bb, acc[j][1]);
  }
}

constexpr int NS_TILE = 64, NS_KT = 32, NS_THREADS = 256;

// C = A B, all row-major, M, N, K multiples of 64, leading dimensions multiples
// of 4 floats. A 64 x 64 tile per CTA, 4 x 4 outputs per thread; a warp's
// threads hold 8 x 4 of these tiles (a 16-byte shared load costs 2 clocks per eight
// different addresses: 4 clocks of loads against 4.3 of packed FMAs). The next 32-deep slice of A and B is
// loaded into registers (float4) while the current one, in shared memory (A
// transposed), is multiplied; a slice's sum is formed by itself and then added (the
// rounding of K / 32 + 32 additions instead of K: the analysis rows are much
// smaller than the terms).
__global__ void __launch_bounds__(NS_THREADS)
    ns_gemm_kernel(int K, const float *__restrict__ A, int lda, const float *__restrict__ B,
                   int ldb, float *__restrict__ C, int ldc) {
  __shared__ __align__(16) float As[NS_KT][NS_TILE + 4];
  __shared__ __align__(16) float Bs[NS_KT][NS_TILE + 4];
  lk_pdl_wait();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tr = (warp & 1) * 8 + (lane & 7), tc = (warp >> 1) * 4 + (lane >> 3);
  const int row0 = blockIdx.y * NS_TILE, col0 = blockIdx.x * NS_TILE;
  // slice loads: A 64 x 32 (two float4 per thread: row ar + 32 q, columns ak .. ak+3),
  // B 32 x 64 (two float4 per thread: row bk + 16 q, columns bc .. bc+3)
  const int ar = tid / 8, ak = (tid % 8) * 4;
  const int bk = tid / 16, bc = (tid % 16) * 4;
  float4 ra[2], rb[2];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      ra[q] = *reinterpret_cast<const float4 *>(A + (size_t)(row0 + ar + 32 * q) * lda + k0 + ak);
      rb[q] = *reinterpret_cast<const float4 *>(B + (size_t)(k0 + bk + 16 * q) * ldb + col0 + bc);
    }
  };
  auto store = [&]() {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int r = ar + 32 * q;
      As[ak + 0][r] = ra[q].x;
      As[ak + 1][r] = ra[q].y;
      As[ak + 2][r] = ra[q].z;
      As[ak + 3][r] = ra[q].w;
      *reinterpret_cast<float4 *>(&Bs[bk + 16 * q][bc]) = rb[q];
    }
  };
  float2 acc[4][2];                                  // sums over the slices so far
#pragma unroll
  for (int j = 0; j < 4; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
  load(0);
  for (int k0 = 0; k0 < K; k0 += NS_KT) {
    store();
    __syncthreads();
    if (k0 + NS_KT < K) load(k0 + NS_KT);
    float2 part[4][2];
#pragma unroll
    for (int j = 0; j < 4; ++j) part[j][0] = part[j][1] = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int k = 0; k < NS_KT; ++k)
      tile4x4(part, *reinterpret_cast<const float4 *>(&As[k][tr * 4]),
              *reinterpret_cast<const float4 *>(&Bs[k][tc * 4]));
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc[j][0] = __fadd2_rn(acc[j][0], part[j][0]);
      acc[j][1] = __fadd2_rn(acc[j][1], part[j][1]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 o = i & 1 ? make_float4(acc[0][i >> 1].y, acc[1][i >> 1].y, acc[2][i >> 1].y, acc[3][i >> 1].y)
                           : make_float4(acc[0][i >> 1].x, acc[1][i >> 1].x, acc[2][i >> 1].x, acc[3][i >> 1].x);
    *reinterpret_cast<float4 *>(C + (size_t)(row0 + tr * 4 + i) * ldc + col0 + tc * 4) = o;
  }
}

// ---------------------------------------------------------------------------
// The cooperative kernel
// ---------------------------------------------------------------------------
constexpr int NR_THREADS = 512, NR_WARPS = NR_THREADS / 32;
constexpr int NR_TILE = 32, NR_KT = 8, NR_STAGES = 3, NR_LD = NR_TILE + 4;
constexpr int NR_SLICE = 2 * NR_KT * NR_TILE;          // floats of a slice of A and B
constexpr int NR_PART = NR_TILE * NR_LD;               // floats of a warp's partial tile
// shared floats: every warp's slices, every warp's partial tile, the tile's sums
constexpr int NR_SMEM = NR_WARPS * (NR_STAGES * NR_SLICE + NR_PART) + NR_TILE * (NR_TILE + 1);
constexpr int NR_MAX_ITERS = 24, NR_REFINE = 8;
// What the iteration may leave of 1 - x at the interval's lower end: an error of Z as large in
// every direction without slopes, so no more than the products' rounding. (At 1e-5 the spread
// of a loop's update was wrong by up to 7e-6; the step that takes 1e-5 below this is the last.)
constexpr float NR_LEFT = 0x1p-21f;
// Largest last correction, relative to wbar, of corrections that ran out (a contraction
// takes the error below it); its word and wbar's in the barrier words.
constexpr float NR_CORRECTION = 1e-3f;
constexpr int NR_LAST = 16;
// s_A / alpha up to which P keeps its mean. Measured, error of the mean of Xa at m = 128,
// 320 and 70 (kept, taken out): 16-70 1.4-2.9e-8, 1.5-3.7e-8; 400-1000 3.6-7.8e-8, 4.0-8.5e-8;
// 1600-3900 4.4-17e-8, 4.5-16e-8; 2.2e4-5.5e4 8.7e-8-2.6e-6, 5.4e-8-2.0e-6; at 3e6 1e-3, 1e-4.
constexpr double NR_KEEP = 2e3;
constexpr unsigned NR_SPIN = 1u << 21;       // polls of a grid barrier (about a second)

struct NsArgs {
  const LkInst *insts;
  const double *gpart, *cpart;
  int kchunks, mpt;
  long long n_pad;
  double *A64, *c64, *w64, *part;            // part [grid]: sums of squares
  float *mat;                                // eight [n][n] matrices: Y, Y^T, Z, Z^T, twice
  float *T, *TT, *rv, *vv, *Xp, *xm;
  unsigned *sync;                            // [0] arrivals, [1] departures, [2] abort, [3] P
                                             // keeps its mean, [4 ..] per refinement: max |r|,
                                             // [NR_LAST ..] last correction, wbar (float bits)
  int *counters;
};

// All CTAs of the grid (co-resident: a cooperative launch) arrive, then leave. A
// wait that runs out raises the abort word, which every CTA then finds.
__device__ __forceinline__ bool grid_sync(const NsArgs &a, unsigned &target, unsigned *flag) {
  __syncthreads();
  if (threadIdx.x == 0) {
    target += gridDim.x;
    __threadfence();
    atomicAdd(a.sync, 1u);
    unsigned ok = 0;
    for (unsigned n = 0; n < NR_SPIN; ++n) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.sync) : "memory");
      if (v >= target) {
        ok = 1;
        break;
      }
      if ((n & 255u) == 255u && *reinterpret_cast<volatile unsigned *>(a.sync + 2)) break;
    }
    if (!ok) {
      atomicExch(a.sync + 2, 1u);
      atomicOr(a.counters, LK_BIT_TIMEOUT);
    }
    __threadfence();
    *flag = ok;
  }
  __syncthreads();
  return *flag != 0;
}

// ---------------------------------------------------------------------------
// A 32 x 32 output tile of A B, n x n, by one CTA: warp w takes the 8-deep slices
// w, w + 16, ... of the product on its own, three slices in flight (cp.async: the
// operands were written by other CTAs of this launch, so they come from L2), each
// lane 4 x 8 outputs (6 clocks of shared loads against 8.6 of packed FMAs per
// column and SM); the 16 partial tiles are added in warp order. No CTA barrier
// inside the product, and the next tile's first slices are on their way during the sums. A is read from its
// transpose, which every product of the iteration writes beside itself, so
// that both operands' slices are rows of 32.
// ---------------------------------------------------------------------------
struct NsTile {
  const float *AT, *B;
  int row0, col0;
};

__device__ __forceinline__ void ns_load(const NsTile &t, int n, int s, float *st) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int e = lane + 32 * j, k = e >> 3, c = (e & 7) * 4;
    const float *ga = t.AT + (size_t)(s * NR_KT + k) * n + t.row0 + c;
    const float *gb = t.B + (size_t)(s * NR_KT + k) * n + t.col0 + c;
    const unsigned sa = (unsigned)__cvta_generic_to_shared(st + k * NR_TILE + c);
    const unsigned sb = (unsigned)__cvta_generic_to_shared(st + (NR_KT + k) * NR_TILE + c);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(ga) : "memory");
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sb), "l"(gb) : "memory");
  }
}

// The first NR_STAGES - 1 slices of the warp (a group is committed for each, empty
// beyond the last slice).
__device__ __forceinline__ void ns_begin(const NsTile &t, int n, float *st) {
  const int warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NR_STAGES - 1; ++q) {
    const int s = warp + NR_WARPS * q;
    if (s * NR_KT < n) ns_load(t, n, s, st + q * NR_SLICE);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
}

// The product of a tile begun by ns_begin; `next` (if any) is begun before the
// sums. Returns this thread's two outputs: row tid / 16, columns 2 (tid % 16).
__device__ __forceinline__ float2 ns_tile(const NsTile &t, const NsTile *next, int n, float *smem) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float *st = smem + warp * NR_STAGES * NR_SLICE;
  float *part = smem + NR_WARPS * NR_STAGES * NR_SLICE;
  const int tr = lane & 7, tc = lane >> 3;
  float2 acc[2][4][2];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[h][j][0] = acc[h][j][1] = make_float2(0.f, 0.f);
  int buf = 0, ld = NR_STAGES - 1;
  for (int s = warp; s * NR_KT < n; s += NR_WARPS) {
    asm volatile("cp.async.wait_group %0;" ::"n"(NR_STAGES - 2) : "memory");
    __syncwarp();
    const int sn = s + NR_WARPS * (NR_STAGES - 1);
    if (sn * NR_KT < n) ns_load(t, n, sn, st + ld * NR_SLICE);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float4 *as = reinterpret_cast<const float4 *>(st + buf * NR_SLICE) + tr;
    const float4 *bs = reinterpret_cast<const float4 *>(st + buf * NR_SLICE + NR_KT * NR_TILE) + 2 * tc;
#pragma unroll
    for (int k = 0; k < NR_KT; ++k) {
      const float4 a = as[k * (NR_TILE / 4)];
      tile4x4(acc[0], a, bs[k * (NR_TILE / 4)]);
      tile4x4(acc[1], a, bs[k * (NR_TILE / 4) + 1]);
    }
    buf = buf + 1 == NR_STAGES ? 0 : buf + 1;
    ld = ld + 1 == NR_STAGES ? 0 : ld + 1;
  }
  __syncwarp();
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (next) ns_begin(*next, n, st);
  float *p = part + warp * NR_PART;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      *reinterpret_cast<float4 *>(p + (tr * 4 + i) * NR_LD + tc * 8 + 4 * h) =
          i & 1 ? make_float4(acc[h][0][i >> 1].y, acc[h][1][i >> 1].y, acc[h][2][i >> 1].y, acc[h][3][i >> 1].y)
                : make_float4(acc[h][0][i >> 1].x, acc[h][1][i >> 1].x, acc[h][2][i >> 1].x, acc[h][3][i >> 1].x);
  __syncthreads();
  float2 r = make_float2(0.f, 0.f);
#pragma unroll
  for (int w = 0; w < NR_WARPS; ++w)
    r = __fadd2_rn(r, *reinterpret_cast<const float2 *>(part + w * NR_PART + (tid >> 4) * NR_LD +
                                                       2 * (tid & 15)));
  return r;
}

// The tile's outputs (as ns_tile returned them, after the caller's epilogue) into C
// and, transposed, into CT. Two barriers: the sums are read, the tile is complete.
__device__ __forceinline__ void ns_write(float2 v, int n, int row0, int col0, float *C, float *CT,
                                         float *smem) {
  const int tid = threadIdx.x, r = tid >> 4, c = 2 * (tid & 15);
  float *R = smem + NR_WARPS * (NR_STAGES * NR_SLICE + NR_PART);
  R[r * (NR_TILE + 1) + c] = v.x;
  R[r * (NR_TILE + 1) + c + 1] = v.y;
  *reinterpret_cast<float2 *>(C + (size_t)(row0 + r) * n + col0 + c) = v;
  __syncthreads();
  *reinterpret_cast<float2 *>(CT + (size_t)(col0 + r) * n + row0 + c) =
      make_float2(R[c * (NR_TILE + 1) + r], R[(c + 1) * (NR_TILE + 1) + r]);
  __syncthreads();
}

__global__ void __launch_bounds__(NR_THREADS, 1) ns_root_kernel(NsArgs a) {
  extern __shared__ __align__(16) float smem[];
  __shared__ double red[NR_THREADS / 32];
  __shared__ unsigned flag;
  const LkInst &I = a.insts[0];
  const int n = a.mpt, m = I.m, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gw = blockIdx.x * (NR_THREADS / 32) + warp, nw = gridDim.x * (NR_THREADS / 32);
  const int nt = n / NR_TILE;
  const size_t nn = (size_t)n * n;
  float *st = smem + warp * NR_STAGES * NR_SLICE;
  unsigned target = 0;
  bool live = true;
  do {
    // ---- A (FP64) from the Gram's partial sums of its upper triangle, c, |A|_F ----
    double sq = 0.0;
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
      for (int j = i + tid; j < n; j += NR_THREADS) {
        double s = 0.0;
#pragma unroll 4
        for (int k = 0; k < a.kchunks; ++k) s += a.gpart[((size_t)k * n + i) * n + j];
        // (m-1)/rho on the diagonal, the padding included: the padding's
        // eigenvalues then sit with the smallest real ones
        if (i == j) s += I.alpha;
        a.A64[(size_t)i * n + j] = s;
        if (j > i) a.A64[(size_t)j * n + i] = s;
        sq = fma(i == j ? s : 2.0 * s, s, sq);
      }
      if (warp == 0) {
        double c = 0.0;
        for (int k = lane; k < a.kchunks; k += 32) c += a.cpart[(size_t)k * n + i];
        c = lk_warp_sum(c);
        if (lane == 0) {
          a.c64[i] = c;
          a.w64[i] = 0.0;
          a.rv[i] = (float)c;
        }
      }
    }
    sq = lk_warp_sum(sq);
    if (lane == 0) red[warp] = sq;
    if (blockIdx.x == 0 && tid < NR_REFINE) a.sync[4 + tid] = 0u;
    if (blockIdx.x == 0 && tid < 2) a.sync[NR_LAST + tid] = 0u;
    // the state rows' anomalies and means, a warp per row
    for (long long r = gw; r < a.n_pad; r += nw) {
      const bool real = r < 2LL * I.n_pts;
      const float *x = static_cast<const float *>(I.X) + r * m;
      float s = 0.f;
      if (real)
        for (int j = lane; j < m; j += 32) s += x[j];
      s = lk_warp_sum(s) / float(m);
      for (int j = lane; j < n; j += 32) a.Xp[r * n + j] = (real && j < m) ? x[j] - s : 0.f;
      if (lane == 0) a.xm[r] = s;
    }
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < NR_THREADS / 32; ++w) t += red[w];
      a.part[blockIdx.x] = t;
    }
    if (!(live = grid_sync(a, target, &flag))) break;
    // ---- Y = A / s_A, Z = I ----
    double fro = 0.0;
    for (int k = lane; k < (int)gridDim.x; k += 32) fro += __ldcg(a.part + k);
    fro = sqrt(lk_warp_sum(fro));
    const double inv = 1.0 / fro;
    if (blockIdx.x == 0 && tid == 0) a.sync[3] = inv * I.alpha * NR_KEEP >= 1.0;
    for (long long e = (long long)blockIdx.x * NR_THREADS + tid; e < (long long)n * n;
         e += (long long)gridDim.x * NR_THREADS) {
      const float y = (float)(__ldcg(a.A64 + e) * inv), z = e / n == e % n ? 1.f : 0.f;
      a.mat[e] = a.mat[nn + e] = y;                  // symmetric
      a.mat[2 * nn + e] = a.mat[3 * nn + e] = z;
    }
    if (!(live = grid_sync(a, target, &flag))) break;
    // ---- Newton-Schulz; x: the lower end of the interval ----
    float *cur = a.mat, *nxt = a.mat + 4 * nn;         // Y, Y^T, Z, Z^T
    float x = (float)sqrt(I.alpha * inv);
    for (int it = 0; x < 1.f - NR_LEFT && it < NR_MAX_ITERS; ++it) {
      const float mu2 = 3.f / (1.f + x + x * x), mu = sqrtf(mu2);
      const float ca = 1.5f * mu, cb = 0.5f * mu * mu2;
      auto first = [&](int t) {                      // Z Y
        return NsTile{cur + 3 * nn, cur, t / nt * NR_TILE, t % nt * NR_TILE};
      };
      auto second = [&](int t) {                     // Y T, then T Z
        const int u = t < nt * nt ? t : t - nt * nt;
        return NsTile{t < nt * nt ? cur + nn : a.TT, t < nt * nt ? a.T : cur + 2 * nn,
                      u / nt * NR_TILE, u % nt * NR_TILE};
      };
      NsTile now, next;
      if ((int)blockIdx.x < nt * nt) {
        now = first(blockIdx.x);
        ns_begin(now, n, st);
      }
      for (int t = blockIdx.x; t < nt * nt; t += gridDim.x) {
        const bool more = t + (int)gridDim.x < nt * nt;
        if (more) next = first(t + gridDim.x);
        const float2 p = ns_tile(now, more ? &next : nullptr, n, smem);
        const int r = now.row0 + (tid >> 4), c = now.col0 + 2 * (tid & 15);
        ns_write(make_float2((r == c ? ca : 0.f) - cb * p.x, (r == c + 1 ? ca : 0.f) - cb * p.y), n,
                 now.row0, now.col0, a.T, a.TT, smem);
        now = next;
      }
      if (!(live = grid_sync(a, target, &flag))) break;
      if ((int)blockIdx.x < 2 * nt * nt) {
        now = second(blockIdx.x);
        ns_begin(now, n, st);
      }
      for (int t = blockIdx.x; t < 2 * nt * nt; t += gridDim.x) {
        const bool more = t + (int)gridDim.x < 2 * nt * nt;
        if (more) next = second(t + gridDim.x);
        const float2 p = ns_tile(now, more ? &next : nullptr, n, smem);
        float *C = nxt + (t < nt * nt ? 0 : 2 * nn);
        ns_write(p, n, now.row0, now.col0, C, C + nn, smem);
        now = next;
      }
      if (!(live = grid_sync(a, target, &flag))) break;
      float *swap = cur;
      cur = nxt;
      nxt = swap;
      const float y = mu * x;
      x = fminf(1.f, 0.5f * y * (3.f - y * y));
    }
    const float *Y = cur, *Z = cur + 2 * nn, *ZT = cur + 3 * nn;
    if (!live) break;
    // ---- wbar = A^-1 c by refinement with A^-1 ~ Z Z / s_A; done when the residual
    // bounds the relative error of wbar by 1e-9, or after NR_REFINE corrections ----
    bool met = false;
    for (int rf = 0; rf < NR_REFINE; ++rf) {
      if (rf > 0) {                                  // r = c - A w (at first w = 0)
        for (int i = gw; i < n; i += nw) {
          double s = 0.0;
          for (int j = lane; j < n; j += 32)
            s = fma(__ldcg(a.A64 + (size_t)i * n + j), __ldcg(a.w64 + j), s);
          s = __ldcg(a.c64 + i) - lk_warp_sum(s);
          if (lane == 0) {
            a.rv[i] = (float)s;
            atomicMax(a.sync + 4 + rf, __float_as_uint(fabsf((float)s)));
          }
        }
      } else {
        for (int i = gw * 32 + lane; i < n; i += nw * 32)
          atomicMax(a.sync + 4, __float_as_uint(fabsf((float)__ldcg(a.c64 + i))));
      }
      if (!(live = grid_sync(a, target, &flag))) break;
      if (rf > 0 && __uint_as_float(__ldcg(a.sync + 4 + rf)) <=
                        1e-9f * (float)(I.alpha * inv) * __uint_as_float(__ldcg(a.sync + 4))) {
        met = true;
        break;
      }
      for (int i = gw; i < n; i += nw) {
        float s = 0.f;
        for (int j = lane; j < n; j += 32)
          s = fmaf(__ldcg(Z + (size_t)i * n + j), __ldcg(a.rv + j), s);
        s = lk_warp_sum(s);
        if (lane == 0) a.vv[i] = s;
      }
      if (!(live = grid_sync(a, target, &flag))) break;
      for (int i = gw; i < n; i += nw) {
        float s = 0.f;
        for (int j = lane; j < n; j += 32)
          s = fmaf(__ldcg(Z + (size_t)i * n + j), __ldcg(a.vv + j), s);
        s = lk_warp_sum(s);
        if (lane == 0) {
          const double d = (double)s * inv, w = __ldcg(a.w64 + i) + d;
          a.w64[i] = w;
          if (rf == NR_REFINE - 1) {
            atomicMax(a.sync + NR_LAST, __float_as_uint(fabsf((float)d)));
            atomicMax(a.sync + NR_LAST + 1, __float_as_uint(fabsf((float)w)));
          }
        }
      }
      if (!(live = grid_sync(a, target, &flag))) break;
    }
    if (!live) break;
    // Z Z is no inverse to FP32 any more from a condition of about 5e7 on, where Z Y still
    // passes for I: the corrections grow instead of shrinking, and the last one says so
    if (!met && blockIdx.x == 0 && tid == 0 &&
        !(__uint_as_float(__ldcg(a.sync + NR_LAST)) <=
          NR_CORRECTION * __uint_as_float(__ldcg(a.sync + NR_LAST + 1))))
      atomicOr(a.counters, LK_BIT_NOCONVERGE);
    // wbar as a pair of floats, in the refinement's vectors
    for (int i = gw * 32 + lane; i < n; i += nw * 32) {
      const Df w = df_of(__ldcg(a.w64 + i));
      a.rv[i] = w.h;
      a.vv[i] = w.l;
    }
    // ---- T = sqrt((m-1) / s_A) Z on the m x m block, zero elsewhere; the iteration
    // failed if Z Y strays from I by more than 1e-3 ----
    const float f = (float)sqrt((m - 1) * inv);
    float mx = 0.f;
    for (int t = blockIdx.x; t < nt * nt; t += gridDim.x) {
      const NsTile now{ZT, Y, t / nt * NR_TILE, t % nt * NR_TILE};
      ns_begin(now, n, st);
      const float2 p = ns_tile(now, nullptr, n, smem);
      __syncthreads();                               // the sums are read
      const int r = now.row0 + (tid >> 4), c = now.col0 + 2 * (tid & 15);
      const float e0 = fabsf(p.x - (r == c ? 1.f : 0.f)), e1 = fabsf(p.y - (r == c + 1 ? 1.f : 0.f));
      if (!(e0 <= 1e-3f) || !(e1 <= 1e-3f)) mx = 1.f;
      const float2 z = __ldcg(reinterpret_cast<const float2 *>(Z + (size_t)r * n + c));
      *reinterpret_cast<float2 *>(a.T + (size_t)r * n + c) =
          make_float2(r < m && c < m ? f * z.x : 0.f, r < m && c + 1 < m ? f * z.y : 0.f);
    }
    if (mx != 0.f) atomicOr(a.counters, LK_BIT_NOCONVERGE);
  } while (false);
  // the last CTA to leave clears the barrier for the next launch
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(a.sync + 1, 1u) == gridDim.x - 1) {
      a.sync[0] = 0u;
      a.sync[1] = 0u;
      a.sync[2] = 0u;
      __threadfence();
    }
  }
}

constexpr int NF_VALS = 4;             // values per lane in flight
// Xa = xbar + X' wbar + P, P = X' T; mean and spread, warp per state row. Where P's mean is
// taken out (*keep zero), what xbar's rounding has left in the anomalies, which P passes on, is
// added back. The common part is a pair of floats, so that a member is rounded once.
__global__ void __launch_bounds__(LK_WARP_CTA)
    ns_finish_kernel(const LkInst *__restrict__ insts, int mpt, const float *__restrict__ P,
                     const float *__restrict__ Xp, const float *__restrict__ xm,
                     const float *__restrict__ wh, const float *__restrict__ wl,
                     const unsigned *__restrict__ keep,
                     float *__restrict__ mean, float *__restrict__ spread,
                     int *__restrict__ counters) {
  lk_pdl_wait();
  const LkInst &I = insts[0];
  const long long r = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, m = I.m;
  if (r >= 2LL * I.n_pts) return;
  float *x = static_cast<float *>(I.X) + r * m;
  const bool kept = *keep != 0;
  float pm = 0.f, xr = 0.f;
  Df xw = df(0.f);
  for (int j0 = lane; j0 < m; j0 += 32 * NF_VALS) {  // (loads in flight together)
    float p[NF_VALS], xp[NF_VALS];
    Df w[NF_VALS];
#pragma unroll
    for (int u = 0; u < NF_VALS; ++u) {
      const int j = j0 + 32 * u;
      p[u] = j < m ? P[r * mpt + j] : 0.f;
      xp[u] = j < m ? Xp[r * mpt + j] : 0.f;
      w[u] = j < m ? Df{wh[j], wl[j]} : df(0.f);
    }
#pragma unroll
    for (int u = 0; u < NF_VALS; ++u) {
      pm += p[u];
      xr += xp[u];
      xw = df_add(xw, df_mul(df(xp[u]), w[u]));
    }
  }
  xw = df_warp_sum(xw);
  if (kept) {
    pm = 0.f;
  } else {
    pm = lk_warp_sum(pm) / float(m);
    xw = df_add(xw, df(lk_warp_sum(xr) / float(m)));
  }
  const Df base = df_add(df(xm[r]), xw);
  float sum = 0.f;
#pragma unroll 4
  for (int j = lane; j < m; j += 32) {
    const float xa = base.h + (base.l + (P[r * mpt + j] - pm));
    x[j] = xa;
    sum += xa;
  }
  const float mu = lk_warp_sum(sum) / float(m);
  float sq = 0.f;
  for (int j = lane; j < m; j += 32) {
    const float d = x[j] - mu;
    sq = fmaf(d, d, sq);
  }
  const float sp = sqrtf(lk_warp_sum(sq) / float(m - 1));
  if (lane == 0) {
    if (mean) mean[r] = mu;
    if (spread) spread[r] = sp;
    if (!isfinite(mu) || !isfinite(sp)) atomicOr(&counters[0], LK_BIT_NONFINITE);
  }
}

}  // namespace

int lk_ns_tile() { return NS_TILE; }

// Workspace (one allocation, zeroed once): A64, c64, w64, part (FP64); the
// iteration's eight matrices, T and its transpose (FP32 [mpt][mpt]); r, v (FP32
// [mpt]); Xp and the product (FP32 [n_pad][mpt]), xm [n_pad]; the barrier words.
// (The FP32 part starts 256-byte aligned: the products load float4.)
static size_t ns_fp64_bytes(int mpt) {
  return (((size_t)mpt * mpt * 8 + 2 * (size_t)mpt * 8 + 1024 * 8) + 255) & ~size_t(255);
}

size_t lk_ns_workspace_bytes(int mpt, long long n_pad) {
  const size_t f = 10 * (size_t)mpt * mpt + 2 * (size_t)mpt + 2 * (size_t)n_pad * mpt +
                   (size_t)n_pad;
  return ns_fp64_bytes(mpt) + f * 4 + 64 * sizeof(unsigned) + 1024;
}

cudaError_t lk_ns_setup() {
  return lk_raise_smem(ns_root_kernel, NR_SMEM * sizeof(float));
}

cudaError_t lk_launch_ns_global(letkf_ctx *h, const double *gpart, const double *cpart,
                                int kchunks, int mpt, int sms, void *ws, void *mean,
                                void *spread) {
  const LkInst &I = h->inst[0];
  const size_t nn = (size_t)mpt * mpt;
  NsArgs a;
  a.insts = h->d_inst;
  a.gpart = gpart;
  a.cpart = cpart;
  a.kchunks = kchunks;
  a.mpt = mpt;
  a.n_pad = ((2LL * I.n_pts + NS_TILE - 1) / NS_TILE) * NS_TILE;
  unsigned char *b = static_cast<unsigned char *>(ws);
  a.A64 = reinterpret_cast<double *>(b);
  a.c64 = a.A64 + nn;
  a.w64 = a.c64 + mpt;
  a.part = a.w64 + mpt;
  a.mat = reinterpret_cast<float *>(b + ns_fp64_bytes(mpt));
  a.T = a.mat + 8 * nn;
  a.TT = a.T + nn;
  a.rv = a.TT + nn;
  a.vv = a.rv + mpt;
  a.Xp = a.vv + mpt;
  float *Pr = a.Xp + (size_t)a.n_pad * mpt;
  a.xm = Pr + (size_t)a.n_pad * mpt;
  a.sync = reinterpret_cast<unsigned *>(a.xm + a.n_pad);
  a.counters = h->counters;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(sms < 1024 ? sms : 1024));
  cfg.blockDim = dim3(NR_THREADS);
  cfg.dynamicSmemBytes = NR_SMEM * sizeof(float);
  cfg.stream = h->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, ns_root_kernel, a);
  if (e == cudaSuccess)
    e = lk_launch_pdl(ns_gemm_kernel, dim3(mpt / NS_TILE, (unsigned)(a.n_pad / NS_TILE)),
                      NS_THREADS, 0, h->stream, mpt, (const float *)a.Xp, mpt,
                      (const float *)a.T, mpt, Pr, mpt);
  const unsigned fb = (unsigned)((2LL * I.n_pts * 32 + LK_WARP_CTA - 1) / LK_WARP_CTA);
  if (e == cudaSuccess)
    e = lk_launch_pdl(ns_finish_kernel, fb, LK_WARP_CTA, 0, h->stream,
                      (const LkInst *)h->d_inst, mpt, (const float *)Pr, (const float *)a.Xp,
                      (const float *)a.xm, (const float *)a.rv, (const float *)a.vv,
                      (const unsigned *)(a.sync + 3),
                      static_cast<float *>(mean), static_cast<float *>(spread), h->counters);
  return e;
}
