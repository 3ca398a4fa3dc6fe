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
//   apply    T = wbar 1^T + sqrt((m-1) / s_A) Z, Xa = xbar + X' T over all
//            state rows, mean and spread
//
// Scaled steps: the singular values x = sqrt(eig(Z Y)) start in [x_0, 1] with
// x_0 = sqrt(alpha / s_A), alpha = (m-1)/rho the smallest eigenvalue A can have.
// A step maps x -> (3 mu x - (mu x)^3) / 2; mu^2 = 3 / (1 + x_0 + x_0^2) makes
// both ends of the interval equal, so that the lower one grows by up to
// 1.5 sqrt(3) = 2.6 per step instead of 1.5, and the next interval is known
// without looking at the matrices (Chen & Chow's and Higham's scaled iterations).
// From x_0 = 0.003 (the prior draw's kappa of 1e5) ten steps reach 1 - 1e-5
// where the unscaled iteration took 26; a loop's kappa of 50 takes six.
//
// Everything between the Gram and the apply is one cooperative kernel: a grid
// barrier (about 1 us) per dependent stage instead of a launch, and the
// number of iterations is the device's own. The products run in 32 x 32 tiles of
// 512 threads, eight groups of 64 splitting the K dimension. (Forming only the upper triangle
// of these products of commuting symmetric matrices and mirroring it would
// halve the flops, but it breaks the coupling of the iteration: in FP32 at the
// prior draw's kappa ~ 1.5e5, m = 200, the symmetrised iteration overflows
// after 20 steps where the full one converges.)
#include <math.h>

#include "letkf_device.cuh"

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
// transposed), is multiplied.
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
  float2 acc[4][2];
#pragma unroll
  for (int j = 0; j < 4; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
  load(0);
  for (int k0 = 0; k0 < K; k0 += NS_KT) {
    store();
    __syncthreads();
    if (k0 + NS_KT < K) load(k0 + NS_KT);
#pragma unroll 8
    for (int k = 0; k < NS_KT; ++k)
      tile4x4(acc, *reinterpret_cast<const float4 *>(&As[k][tr * 4]),
              *reinterpret_cast<const float4 *>(&Bs[k][tc * 4]));
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
constexpr int NR_THREADS = 512, NR_TILE = 32, NR_KT = 16, NR_SPLIT = 8, NR_LD = NR_TILE + 4;
constexpr int NR_MAX_ITERS = 24, NR_REFINE = 4;
constexpr unsigned NR_SPIN = 1u << 21;       // polls of a grid barrier (about a second)

struct NsArgs {
  const LkInst *insts;
  const double *gpart, *cpart;
  int kchunks, mpt;
  long long n_pad;
  double *A64, *c64, *w64, *part, *scale;    // part [grid]: sums of squares
  float *Y, *Z, *T, *U, *rv, *vv, *Xp, *xm;
  unsigned *sync;                            // [0] arrivals, [1] departures, [2] abort,
                                             // [4 ..] per refinement: max |r| (float bits)
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

// Output tile (row0, col0) of A B, n x n: this thread's two outputs, row tid / 16,
// columns 2 (tid % 16). Group q of 64 threads takes the 16-deep slices q, q + 8, ...;
// the groups' partial tiles are added in group order through shared memory.
// The operands were written by other CTAs during this launch: L2 loads only.
__device__ __forceinline__ float2 ns_tile(int n, const float *A, const float *B, int row0,
                                          int col0, float *smem) {
  const int tid = threadIdx.x, q = tid >> 6, lt = tid & 63, lane = tid & 31;
  float(*as)[NR_LD] = reinterpret_cast<float(*)[NR_LD]>(smem + q * 2 * NR_KT * NR_LD);
  float(*bs)[NR_LD] = as + NR_KT;
  // thread tiles 8 x 8 of 4 x 4; a warp 8 x 4 of them
  const int tr = lane & 7, tc = (lt >> 5) * 4 + (lane >> 3);
  const int ar = lt >> 2, ak = (lt & 3) * 4, bk = lt >> 3, bc = (lt & 7) * 4;
  float4 ra[2], rb[2];
  auto load = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      ra[j] = __ldcg(reinterpret_cast<const float4 *>(A + (size_t)(row0 + ar + 16 * j) * n + k0 + ak));
      rb[j] = __ldcg(reinterpret_cast<const float4 *>(B + (size_t)(k0 + bk + 8 * j) * n + col0 + bc));
    }
  };
  float2 acc[4][2];
#pragma unroll
  for (int j = 0; j < 4; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
  const int nk = n / NR_KT, steps = (nk + NR_SPLIT - 1) / NR_SPLIT;
  load(q * NR_KT);                                   // n >= 128: every group has a slice
  for (int s = 0; s < steps; ++s) {
    const int kt = q + NR_SPLIT * s;
    const bool valid = kt < nk;
    if (valid) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int r = ar + 16 * j;
        as[ak + 0][r] = ra[j].x;
        as[ak + 1][r] = ra[j].y;
        as[ak + 2][r] = ra[j].z;
        as[ak + 3][r] = ra[j].w;
        *reinterpret_cast<float4 *>(&bs[bk + 8 * j][bc]) = rb[j];
      }
    }
    __syncthreads();
    if (kt + NR_SPLIT < nk) load((kt + NR_SPLIT) * NR_KT);
    if (valid) {
#pragma unroll
      for (int k = 0; k < NR_KT; ++k)
        tile4x4(acc, *reinterpret_cast<const float4 *>(&as[k][tr * 4]),
                *reinterpret_cast<const float4 *>(&bs[k][tc * 4]));
    }
    __syncthreads();
  }
  float(*ps)[NR_LD] = reinterpret_cast<float(*)[NR_LD]>(smem + q * NR_TILE * NR_LD);
#pragma unroll
  for (int i = 0; i < 4; ++i)
    *reinterpret_cast<float4 *>(&ps[tr * 4 + i][tc * 4]) =
        i & 1 ? make_float4(acc[0][i >> 1].y, acc[1][i >> 1].y, acc[2][i >> 1].y, acc[3][i >> 1].y)
              : make_float4(acc[0][i >> 1].x, acc[1][i >> 1].x, acc[2][i >> 1].x, acc[3][i >> 1].x);
  __syncthreads();
  float2 t = make_float2(0.f, 0.f);
#pragma unroll
  for (int g = 0; g < NR_SPLIT; ++g) {
    const float2 u = *reinterpret_cast<const float2 *>(smem + g * NR_TILE * NR_LD +
                                                       (tid >> 4) * NR_LD + 2 * (tid & 15));
    t = __fadd2_rn(t, u);
  }
  __syncthreads();                                   // the tile's memory is free again
  return t;
}

__global__ void __launch_bounds__(NR_THREADS, 1) ns_root_kernel(NsArgs a) {
  __shared__ __align__(16) float smem[2 * NR_SPLIT * NR_KT * NR_LD];
  __shared__ double red[NR_THREADS / 32];
  __shared__ unsigned flag;
  const LkInst &I = a.insts[0];
  const int n = a.mpt, m = I.m, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gw = blockIdx.x * (NR_THREADS / 32) + warp, nw = gridDim.x * (NR_THREADS / 32);
  const int nt = n / NR_TILE;
  unsigned target = 0;
  bool live = true;
  do {
    // ---- A (FP64) from the Gram's partial sums of its upper triangle, c, |A|_F ----
    double sq = 0.0;
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
      for (int j = i + tid; j < n; j += NR_THREADS) {
        double s = 0.0;
        for (int k = 0; k < a.kchunks; ++k) s += a.gpart[((size_t)k * n + i) * n + j];
        // (m-1)/rho on the diagonal, the padding included: the padding's
        // eigenvalues then sit with the smallest real ones
        if (i == j) s += I.alpha;
        a.A64[(size_t)i * n + j] = s;
        if (j > i) a.A64[(size_t)j * n + i] = s;
        sq = fma(i == j ? s : 2.0 * s, s, sq);
      }
      if (tid == 0) {
        double c = 0.0;
        for (int k = 0; k < a.kchunks; ++k) c += a.cpart[(size_t)k * n + i];
        a.c64[i] = c;
        a.w64[i] = 0.0;
        a.rv[i] = (float)c;
      }
    }
    sq = lk_warp_sum(sq);
    if (lane == 0) red[warp] = sq;
    if (blockIdx.x == 0 && tid < NR_REFINE) a.sync[4 + tid] = 0u;
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
    for (long long e = (long long)blockIdx.x * NR_THREADS + tid; e < (long long)n * n;
         e += (long long)gridDim.x * NR_THREADS) {
      a.Y[e] = (float)(__ldcg(a.A64 + e) * inv);
      a.Z[e] = e / n == e % n ? 1.f : 0.f;
    }
    if (!(live = grid_sync(a, target, &flag))) break;
    // ---- Newton-Schulz; x: the lower end of the interval ----
    float *Y = a.Y, *Z = a.Z, *T = a.T, *U = a.U;
    float x = (float)sqrt(I.alpha * inv);
    int it = 0;
    for (; x < 1.f - 1e-5f && it < NR_MAX_ITERS; ++it) {
      const float mu2 = 3.f / (1.f + x + x * x), mu = sqrtf(mu2);
      const float ca = 1.5f * mu, cb = 0.5f * mu * mu2;
      for (int t = blockIdx.x; t < nt * nt; t += gridDim.x) {
        const int row0 = t / nt * NR_TILE, col0 = t % nt * NR_TILE;
        const float2 p = ns_tile(n, Z, Y, row0, col0, smem);
        const int r = row0 + (tid >> 4), c = col0 + 2 * (tid & 15);
        *reinterpret_cast<float2 *>(T + (size_t)r * n + c) =
            make_float2((r == c ? ca : 0.f) - cb * p.x, (r == c + 1 ? ca : 0.f) - cb * p.y);
      }
      if (!(live = grid_sync(a, target, &flag))) break;
      // U = Y T; Z' = T Z into the old Y's place needs Y read out: a fourth buffer
      float *V = a.Xp + a.n_pad * n;                 // [n][n], the product's place
      for (int t = blockIdx.x; t < 2 * nt * nt; t += gridDim.x) {
        const bool second = t >= nt * nt;
        const int tt = second ? t - nt * nt : t;
        const int row0 = tt / nt * NR_TILE, col0 = tt % nt * NR_TILE;
        const float2 p = second ? ns_tile(n, T, Z, row0, col0, smem)
                                : ns_tile(n, Y, T, row0, col0, smem);
        const int r = row0 + (tid >> 4), c = col0 + 2 * (tid & 15);
        *reinterpret_cast<float2 *>((second ? (it & 1 ? a.Z : V) : (it & 1 ? a.Y : U)) +
                                    (size_t)r * n + c) = p;
      }
      if (!(live = grid_sync(a, target, &flag))) break;
      Y = it & 1 ? a.Y : U;
      Z = it & 1 ? a.Z : V;
      const float y = mu * x;
      x = fminf(1.f, 0.5f * y * (3.f - y * y));
    }
    if (!live) break;
    // ---- wbar = A^-1 c by refinement with A^-1 ~ Z Z / s_A; done when the residual
    // bounds the relative error of wbar by 1e-9 ----
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
                        1e-9f * (float)(I.alpha * inv) * __uint_as_float(__ldcg(a.sync + 4)))
        break;
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
        if (lane == 0) a.w64[i] = __ldcg(a.w64 + i) + (double)s * inv;
      }
      if (!(live = grid_sync(a, target, &flag))) break;
    }
    if (!live) break;
    // ---- T = wbar 1^T + sqrt((m-1) / s_A) Z on the m x m block, zero elsewhere; the
    // iteration failed if Z Y strays from I by more than 1e-3 ----
    const float f = (float)sqrt((m - 1) * inv);
    float mx = 0.f;
    for (int t = blockIdx.x; t < nt * nt; t += gridDim.x) {
      const int row0 = t / nt * NR_TILE, col0 = t % nt * NR_TILE;
      const float2 p = ns_tile(n, Z, Y, row0, col0, smem);
      const int r = row0 + (tid >> 4), c = col0 + 2 * (tid & 15);
      const float e0 = fabsf(p.x - (r == c ? 1.f : 0.f)), e1 = fabsf(p.y - (r == c + 1 ? 1.f : 0.f));
      if (!(e0 <= 1e-3f) || !(e1 <= 1e-3f)) mx = 1.f;
      const float2 z = __ldcg(reinterpret_cast<const float2 *>(Z + (size_t)r * n + c));
      const float w = (float)__ldcg(a.w64 + r);
      *reinterpret_cast<float2 *>(T + (size_t)r * n + c) =
          make_float2(r < m && c < m ? fmaf(f, z.x, w) : 0.f,
                      r < m && c + 1 < m ? fmaf(f, z.y, w) : 0.f);
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

// Xa = xbar + (X' T), mean and spread, warp per state row.
__global__ void __launch_bounds__(LK_WARP_CTA)
    ns_finish_kernel(const LkInst *__restrict__ insts, int mpt, const float *__restrict__ P,
                     const float *__restrict__ xm, float *__restrict__ mean,
                     float *__restrict__ spread, int *__restrict__ counters) {
  lk_pdl_wait();
  const LkInst &I = insts[0];
  const long long r = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, m = I.m;
  if (r >= 2LL * I.n_pts) return;
  float *x = static_cast<float *>(I.X) + r * m;
  float sum = 0.f;
  for (int j = lane; j < m; j += 32) {
    const float xa = xm[r] + P[r * mpt + j];
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

// Workspace (one allocation, zeroed once): A64, c64, w64, part (FP64); Y, Z, T, U
// (FP32 [mpt][mpt]); r, v (FP32 [mpt]); Xp (FP32 [n_pad][mpt]), then the product of
// the same shape, which the iteration uses as its fifth matrix before; xm [n_pad];
// the barrier words. (The FP32 part starts 256-byte aligned: the products load float4.)
static size_t ns_fp64_bytes(int mpt) {
  return (((size_t)mpt * mpt * 8 + 2 * (size_t)mpt * 8 + 1024 * 8) + 255) & ~size_t(255);
}

static size_t ns_prod_rows(int mpt, long long n_pad) {
  return n_pad > mpt ? (size_t)n_pad : (size_t)mpt;
}

size_t lk_ns_workspace_bytes(int mpt, long long n_pad) {
  const size_t f = 4 * (size_t)mpt * mpt + 2 * (size_t)mpt + (size_t)n_pad * mpt +
                   ns_prod_rows(mpt, n_pad) * mpt + (size_t)n_pad;
  return ns_fp64_bytes(mpt) + f * 4 + 64 * sizeof(unsigned) + 1024;
}

cudaError_t lk_launch_ns_global(letkf_ctx *h, const double *gpart, const double *cpart,
                                int kchunks, int mpt, int sms, void *ws, void *mean,
                                void *spread) {
  const LkInst &I = h->inst[0];
  NsArgs a;
  a.insts = h->d_inst;
  a.gpart = gpart;
  a.cpart = cpart;
  a.kchunks = kchunks;
  a.mpt = mpt;
  a.n_pad = ((2LL * I.n_pts + NS_TILE - 1) / NS_TILE) * NS_TILE;
  unsigned char *b = static_cast<unsigned char *>(ws);
  a.A64 = reinterpret_cast<double *>(b);
  a.c64 = a.A64 + (size_t)mpt * mpt;
  a.w64 = a.c64 + mpt;
  a.part = a.w64 + mpt;
  a.Y = reinterpret_cast<float *>(b + ns_fp64_bytes(mpt));
  a.Z = a.Y + (size_t)mpt * mpt;
  a.T = a.Z + (size_t)mpt * mpt;
  a.U = a.T + (size_t)mpt * mpt;
  a.rv = a.U + (size_t)mpt * mpt;
  a.vv = a.rv + mpt;
  a.Xp = a.vv + mpt;
  float *Pr = a.Xp + (size_t)a.n_pad * mpt;
  a.xm = Pr + ns_prod_rows(mpt, a.n_pad) * mpt;
  a.sync = reinterpret_cast<unsigned *>(a.xm + a.n_pad);
  a.counters = h->counters;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(sms < 1024 ? sms : 1024));
  cfg.blockDim = dim3(NR_THREADS);
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
                      (const LkInst *)h->d_inst, mpt, (const float *)Pr, (const float *)a.xm,
                      static_cast<float *>(mean), static_cast<float *>(spread), h->counters);
  return e;
}
