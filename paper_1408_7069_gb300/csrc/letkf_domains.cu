// Local analysis on multi-actuator domains (Section 4.1-4.2) and the
// differential-piston least squares (Section 4.4).
//
// The node grid is split by a P x P partition (block b of a side covers nodes
// [floor(b N / P), floor((b + 1) N / P)), N = nsub + 1); the valid nodes of a
// block form a local domain of n_d = 2 x nodes state rows. Its observation
// region is the union of its nodes' w x w windows, both slopes of every valid
// subaperture, weighted by R^-1 = diag(tau / sigma2), tau = Gaspari-Cohn of the
// distance from the subaperture centre to the domain's node box (0 inside).
//
// One CTA per domain, 4 MPD threads, MPD = m padded to a multiple of 8
// (identity on the padding):
//   gather  S = diag(sqrt(tau/sigma2)) Yb_region (p_d x MPD), s = sqrt(tau/sigma2) d,
//           the domain's anomaly rows X' (n_d x MPD), into shared memory
//   Gram    A = (m-1)/rho I + S^T S, c = S^T s
//   EVD     one-sided Jacobi on the columns of B = A: MPD/2 groups of 8 lanes,
//           group g holds columns 2g and 2g+1, lane l of it rows l, l+8, ...;
//           the MPD rounds of a sweep follow the odd-even transposition order
//           (even round: own pair; odd round: the pair straddling two groups,
//           the last group swapping), columns moving between groups through
//           shared memory after every round. Converged columns are lambda q.
//   apply   G = X' Q, z = Lambda^-1 Q^T c, Xa_r = xbar_r + sum_c G_rc (z_c +
//           sqrt((m-1)/lambda_c) Q_jc) for every row r of the domain
// A partition of 1 (one domain over the whole grid, the global ETKF of
// Section 3.1.1 when the window covers the pupil) runs as the multi-kernel
// pipeline below instead, for any number of slopes and nodes.
// Then the piston kernels: per domain and state row the constant that
// minimises the squared jumps of the mean increment across border edges
// (4-neighbour nodes in different domains), c = K b with b the per-domain
// edge sums and K the Laplacian's constrained pseudo-inverse (zero
// node-weighted mean per connected group of domains), precomputed on the host
// in FP64; every member of the domain's rows moves by c.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "letkf_device.cuh"

struct LkDom {
  int n_dom = 0, max_nodes = 0, max_obs = 0, rpl = 0, piston = 0;
  int *node_off = nullptr, *node_ids = nullptr;   // CSR: domain -> point ids
  int *obs_off = nullptr, *obs_slot = nullptr;    // CSR: domain -> grid slot (cell * 2 + slope)
  float *obs_w = nullptr;                         // tau / sigma2 of each observed slope
  int *node_dom = nullptr;                        // [n_pts]
  int2 *edges = nullptr;                          // [E] (i, j) point ids, dom(i) != dom(j)
  int *dedge_off = nullptr, *dedge = nullptr;     // per domain: incident edges, +(e+1) / -(e+1)
  float *K = nullptr;                             // [D][D] piston projection
  float *bsum = nullptr;                          // [D][2] per-domain edge sums
  int *sweep = nullptr;                           // [D] nonzero: left to the eigensolve
  int series = 0, splits = 1;                     // the series form fits; CTAs per domain
  float *delta = nullptr;                         // [n_pts][2] mean increments
  std::vector<double> tau;                        // host: tau of each observed slope
  // one domain covering the grid (partition 1): the global ETKF pipeline
  int global = 0, kchunks = 0, mpt = 0, sms = 1;
  void *ns_ws = nullptr;                          // Newton-Schulz workspace (global, m > 64)
  double *gpart = nullptr;                        // [kchunks][MPD][MPD] Gram partial sums
  double *cpart = nullptr;                        // [kchunks][MPD]
  float *T = nullptr;                             // [m][m] transform wbar 1^T + W
};

namespace {

constexpr int DM_GROUP = 8;      // lanes per column pair

__device__ __forceinline__ float group8_sum(float v) {
  v += __shfl_xor_sync(FULL, v, 4);
  v += __shfl_xor_sync(FULL, v, 2);
  v += __shfl_xor_sync(FULL, v, 1);
  return v;
}

struct DomArgs {
  const int *node_off, *node_ids, *obs_off, *obs_slot;
  const float *obs_w;
  float *mean, *spread, *delta;
  int *counters;
  const int *sweep;      // domains to take (NULL: all)
  float tol, stop, kappa_thr;
  int max_sweeps, max_obs, max_rows;
};

// Shared-memory layout (floats): S / Q region, s, c, z, sroot, the column
// exchange [2][G][MPD] and its norms [2][G] (G = X'Q reuses the exchange after
// the sweeps when it fits, so that two CTAs share an SM), X' [rows][MPD],
// xbar [rows], 4 reduction slots.
struct DomLayout {
  int ld, sq, sv, cv, zv, sr, xb, xn, xd, gm, xm, red, total;
};
__host__ __device__ inline DomLayout dom_layout(int mpd, int max_obs, int max_rows) {
  DomLayout L;
  L.ld = mpd + 1;
  const int srows = max_obs > mpd ? max_obs : mpd;
  L.sq = 0;
  L.sv = L.sq + srows * L.ld;
  L.cv = L.sv + max_obs;
  L.zv = L.cv + mpd;
  L.sr = L.zv + mpd;
  L.xb = L.sr + mpd;
  L.xn = L.xb + 2 * (mpd / 2) * mpd;
  L.xd = L.xn + 2 * (mpd / 2);
  L.xm = L.xd + max_rows * mpd;
  L.red = L.xm + max_rows;
  L.total = L.red + 4;
  if (max_rows <= mpd) {
    L.gm = L.xb;                       // [rows][MPD] <= [2][MPD/2][MPD]
  } else {
    L.gm = L.total;
    L.total += max_rows * mpd;
  }
  return L;
}

// One round on the group's pair (P, Q): rotate (or, for the idle slot of an
// odd round, swap) with the rotation that makes the two columns orthogonal,
// from the tracked squared norms and the group-reduced dot product. Returns
// bit 0: rotated, bit 1: rotated with a cosine above the stop cosine.
template <int RPL>
__device__ __forceinline__ int dom_round(float (&P)[RPL], float (&Q)[RPL], float &nP, float &nQ,
                                         float tol2, float stop2, bool idle) {
  float part = 0.f;
#pragma unroll
  for (int i = 0; i < RPL; ++i) part = fmaf(P[i], Q[i], part);
  const float dot = group8_sum(part);
  const float x = nQ - nP, y = 2.f * dot;
  const float rh = rsqrtf(fmaxf(fmaf(x, x, y * y), 1e-37f));
  const float c2 = fmaf(0.5f * fabsf(x), rh, 0.5f);
  const float rc = rsqrtf(c2);
  const float cr = c2 * rc;
  const float sr = (x >= 0.f ? y : -y) * (0.5f * rh) * rc;
  const float t = sr * rc;
  const float dd = dot * dot, nn = nP * nQ;
  const bool rot = !idle && dd > tol2 * nn;
  const float c = rot ? cr : (idle ? 0.f : 1.f);
  const float s = rot ? sr : (idle ? 1.f : 0.f);
  const float nP2 = rot ? fmaf(-t, dot, nP) : (idle ? nQ : nP);
  const float nQ2 = rot ? fmaf(t, dot, nQ) : (idle ? nP : nQ);
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const float p = P[i], q = Q[i];
    P[i] = fmaf(c, p, -s * q);
    Q[i] = fmaf(c, q, s * p);
  }
  nP = nP2;
  nQ = nQ2;
  return (rot ? 1 : 0) | ((rot && dd > stop2 * nn) ? 2 : 0);
}

// Column transfer between groups: every group publishes V (its rows) and n,
// then takes those of group `src`. Double-buffered, one barrier.
template <int RPL>
__device__ __forceinline__ void dom_xfer(float (&V)[RPL], float &n, float *xb, float *xn, int &buf,
                                         int g, int l, int src) {
  constexpr int MPD = 8 * RPL;
  float *b = xb + (size_t)buf * (MPD / 2) * MPD;
  float *bn = xn + buf * (MPD / 2);
#pragma unroll
  for (int i = 0; i < RPL; ++i) b[g * MPD + l + 8 * i] = V[i];
  if (l == 0) bn[g] = n;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < RPL; ++i) V[i] = b[src * MPD + l + 8 * i];
  n = bn[src];
  buf ^= 1;
}

template <int RPL>
__global__ void __launch_bounds__(32 * RPL)
    domain_kernel(const LkInst *__restrict__ insts, DomArgs a) {
  constexpr int MPD = 8 * RPL, G = MPD / 2, NT = 4 * MPD;
  extern __shared__ __align__(16) float dsm[];
  lk_pdl_wait();
  const LkInst &I = insts[0];
  const int m = I.m, tid = threadIdx.x;
  const int dom = blockIdx.x;
  if (a.sweep && !a.sweep[dom]) return;
  const int o0 = a.obs_off[dom], np = a.obs_off[dom + 1] - o0;
  const int n0 = a.node_off[dom], nd = 2 * (a.node_off[dom + 1] - n0);
  const DomLayout Ly = dom_layout(MPD, a.max_obs, a.max_rows);
  const int LD = Ly.ld;
  float *Sq = dsm + Ly.sq, *sv = dsm + Ly.sv, *cv = dsm + Ly.cv, *zv = dsm + Ly.zv;
  float *srt = dsm + Ly.sr, *xb = dsm + Ly.xb, *xn = dsm + Ly.xn, *Xd = dsm + Ly.xd;
  float *Gm = dsm + Ly.gm, *xm = dsm + Ly.xm, *red = dsm + Ly.red;
  const float *Ybp = static_cast<const float *>(I.Ybp);
  const float *dp = static_cast<const float *>(I.dp);
  float *X = static_cast<float *>(I.X);

  // ---- gather: S, s, the anomaly rows; tr(S^T S) for kappa_hat ----
  if (tid == 0) red[0] = 0.f;
  __syncthreads();
  float tr = 0.f;
  for (int e = tid; e < np * MPD; e += NT) {
    const int k = e / MPD, i = e - k * MPD;
    const int slot = a.obs_slot[o0 + k];
    const float sw = sqrtf(a.obs_w[o0 + k]);
    const float v = i < m ? sw * Ybp[(size_t)slot * m + i] : 0.f;
    Sq[k * LD + i] = v;
    tr = fmaf(v, v, tr);
  }
  for (int k = tid; k < np; k += NT) sv[k] = sqrtf(a.obs_w[o0 + k]) * dp[a.obs_slot[o0 + k]];
  for (int e = tid; e < nd * MPD; e += NT) {
    const int r = e / MPD, j = e - r * MPD;
    const int pid = a.node_ids[n0 + (r >> 1)];
    Xd[r * MPD + j] = j < m ? X[((size_t)pid * 2 + (r & 1)) * m + j] : 0.f;
  }
  tr = lk_warp_sum(tr);
  if ((tid & 31) == 0) atomicAdd(&red[0], tr);
  __syncthreads();
  const float inv_m = 1.f / float(m);
  for (int r = tid >> 5; r < nd; r += NT / 32) {   // warp per row: mean, anomalies
    float s = 0.f;
    for (int j = tid & 31; j < m; j += 32) s += Xd[r * MPD + j];
    s = lk_warp_sum(s) * inv_m;
    for (int j = tid & 31; j < m; j += 32) Xd[r * MPD + j] -= s;
    if ((tid & 31) == 0) xm[r] = s;
  }
  const float alpha = float(I.alpha);
  if (tid == 0 && a.kappa_thr > 0.f && 1.f + red[0] / alpha > a.kappa_thr)
    atomicAdd(&a.counters[1], 1);
  __syncthreads();

  // ---- Gram in the Jacobi layout, and c = S^T s ----
  const int g = tid >> 3, l = tid & 7;
  const int cP = 2 * g, cQ = 2 * g + 1;
  float P[RPL], Q[RPL];
#pragma unroll
  for (int i = 0; i < RPL; ++i) P[i] = Q[i] = 0.f;
  for (int k = 0; k < np; ++k) {
    const float *row = Sq + k * LD;
    const float sp = row[cP], sq = row[cQ];
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      const float sr = row[l + 8 * i];
      P[i] = fmaf(sr, sp, P[i]);
      Q[i] = fmaf(sr, sq, Q[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const int r = l + 8 * i;
    if (r == cP) P[i] += cP < m ? alpha : 1.f;
    if (r == cQ) Q[i] += cQ < m ? alpha : 1.f;
  }
  if (tid < MPD) {
    float s = 0.f;
    for (int k = 0; k < np; ++k) s = fmaf(Sq[k * LD + tid], sv[k], s);
    cv[tid] = s;
  }

  // ---- Jacobi sweeps ----
  const float tol2 = a.tol * a.tol, stop2 = a.stop * a.stop;
  int buf = 0, sweeps = 0;
  bool conv = false;
  for (int sweep = 0; sweep < a.max_sweeps; ++sweep) {
    float pp = 0.f, qq = 0.f;
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      pp = fmaf(P[i], P[i], pp);
      qq = fmaf(Q[i], Q[i], qq);
    }
    float nP = group8_sum(pp), nQ = group8_sum(qq);
    int flags = 0;
    for (int r = 0; r < G; ++r) {
      flags |= dom_round<RPL>(P, Q, nP, nQ, tol2, stop2, false);
      dom_xfer<RPL>(Q, nQ, xb, xn, buf, g, l, g + 1 < G ? g + 1 : 0);
      flags |= dom_round<RPL>(P, Q, nP, nQ, tol2, stop2, g == G - 1);
      dom_xfer<RPL>(P, nP, xb, xn, buf, g, l, g > 0 ? g - 1 : G - 1);
    }
    sweeps = sweep + 1;
    if (!__syncthreads_or(flags & 2)) {
      conv = true;
      break;
    }
  }
  if (tid == 0) {
    atomicMax(&a.counters[2], sweeps);
    atomicAdd(&a.counters[3], sweeps);
    if (!conv) atomicOr(&a.counters[0], LK_BIT_NOCONVERGE);
  }

  // ---- eigenpairs: lambda = |b|, q = b / lambda, into Q (aliases S) ----
  float pp = 0.f, qq = 0.f;
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    pp = fmaf(P[i], P[i], pp);
    qq = fmaf(Q[i], Q[i], qq);
  }
  const float lP = sqrtf(group8_sum(pp)), lQ = sqrtf(group8_sum(qq));
  __syncthreads();                                  // every read of S is done
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    Sq[(l + 8 * i) * LD + cP] = P[i] / lP;
    Sq[(l + 8 * i) * LD + cQ] = Q[i] / lQ;
  }
  if (l == 0) {
    zv[cP] = lP;
    zv[cQ] = lQ;
  }
  __syncthreads();
  if (tid < MPD) {                                  // z = Lambda^-1 Q^T c, sqrt((m-1)/lambda)
    const float lam = zv[tid];
    float u = 0.f;
    for (int r = 0; r < MPD; ++r) u = fmaf(Sq[r * LD + tid], cv[r], u);
    srt[tid] = sqrtf(float(m - 1) / lam);
    zv[tid] = u / lam;
  }
  for (int e = tid; e < nd * MPD; e += NT) {        // G = X' Q
    const int r = e / MPD, c = e - r * MPD;
    float s = 0.f;
    for (int j = 0; j < MPD; ++j) s = fmaf(Xd[r * MPD + j], Sq[j * LD + c], s);
    Gm[r * MPD + c] = s;
  }
  __syncthreads();

  // ---- apply: a warp per row ----
  const int lane = tid & 31;
  for (int r = tid >> 5; r < nd; r += NT / 32) {
    const int pid = a.node_ids[n0 + (r >> 1)], comp = r & 1;
    float wb = 0.f;                                 // X'_r wbar: the mean increment
    for (int c = lane; c < MPD; c += 32) wb = fmaf(Gm[r * MPD + c], zv[c], wb);
    wb = lk_warp_sum(wb);
    float sum = 0.f, sq = 0.f;
    float *xrow = X + ((size_t)pid * 2 + comp) * m;
    for (int j = lane; j < m; j += 32) {
      float q = 0.f;
      for (int c = 0; c < MPD; ++c) q = fmaf(Gm[r * MPD + c] * srt[c], Sq[j * LD + c], q);
      const float xa = xm[r] + wb + q;
      xrow[j] = xa;
      sum += xa;
    }
    const float mu = lk_warp_sum(sum) * inv_m;
    for (int j = lane; j < m; j += 32) {
      const float dv = xrow[j] - mu;
      sq = fmaf(dv, dv, sq);
    }
    const float sp = sqrtf(lk_warp_sum(sq) / float(m - 1));
    if (lane == 0) {
      if (a.mean) a.mean[(size_t)pid * 2 + comp] = mu;
      if (a.spread) a.spread[(size_t)pid * 2 + comp] = sp;
      a.delta[(size_t)pid * 2 + comp] = mu - xm[r];
      if (!isfinite(mu) || !isfinite(sp)) atomicOr(&a.counters[0], LK_BIT_NONFINITE);
    }
  }
}

// ---------------------------------------------------------------------------
// The same update by Chebyshev series, without the eigensolve (direct_apply in
// letkf_pair.cu describes the series): with the domain's n_d anomaly rows as
// a block T_0, a term is
//   T_k+1 = 2 T_k X - T_k-1, X = 2 G / (alpha ratio) - I:
// a small matrix product per term, summed with the coefficients of A^-1/2 and of
// A^-1 (whose rows' products with C d are the rows' X'_r wbar). A converged loop's
// ratio of about 4-7 (m = 101, 128 slopes) takes 18-21 terms of 0.35 M FMAs, where
// the eigensolve's eight sweeps take 14 M in rounds that each wait on two CTA
// barriers. Domains above LK_CHEB_MAXD are left to domain_kernel (their `sweep`
// flag).
//
// A CTA per domain, or per part of a domain's rows when the domains are too few
// to fill the GPU (every part forms the same G). Products in 4 x 4 register
// tiles, eight packed FMAs per two 16-byte shared-memory loads. A 16-byte load
// of a warp costs 2 clocks per eight different addresses (measured), so a warp's
// tiles are 8 row groups x 4 column groups (4 x 8 for at most 16 rows): 4
// clocks of loads against 4.3 of FMAs per column of the product and SM. T_k-1 and T_k
// stay in shared memory ([column][row], double-buffered), G in full.
// At most 16 rows leave half of the warps: there the two halves take half of the
// product's columns each and add up through shared memory.
// ---------------------------------------------------------------------------
constexpr int DS_ROWS = 32;      // rows per pass: 8 row groups

struct DomSeriesLayout {
  int g, part, sv, ow, slot, ids, xm, cv, red, total;   // offsets in 4-byte words
};
__host__ __device__ inline DomSeriesLayout dom_series_layout(int mpd, int max_obs, int max_rows) {
  DomSeriesLayout L;
  const int s = max_obs * mpd, t = 2 * mpd * DS_ROWS;
  L.g = s > t ? s : t;                     // S, then the two buffers of T, then the sums
  L.part = L.g + mpd * mpd;                // half products [warps][4][32][4], then X'_r wbar's parts
  L.cv = L.part + (mpd + 31) / 32 * 512;
  L.xm = L.cv + mpd;
  L.sv = L.xm + DS_ROWS;
  L.ow = L.sv + max_obs;
  L.slot = L.ow + max_obs;
  L.ids = L.slot + max_obs;
  L.red = L.ids + max_rows / 2;
  L.total = L.red + 32;
  return L;
}

template <int RPL>
struct DomSeries {
  static constexpr int MPD = 8 * RPL, CG = MPD / 4;
  static constexpr int CB = (CG + 3) / 4;                 // column blocks of 4 groups
  static constexpr int NW = CB < 2 ? 2 : (CB + 1) / 2 * 2;   // warps: 8 for MPD = 104
  static constexpr int NT = 32 * NW;
};

// acc += rows (4 floats at x of each of n columns, stride xs float4) times the 4
// columns at y (stride ys float4).
__device__ __forceinline__ void tile_product(float2 (&acc)[4][2], const float4 *x, int xs,
                                             const float4 *y, int ys, int n) {
#pragma unroll 4
  for (int q = 0; q < n; ++q) {
    const float4 a = x[q * xs], b = y[q * ys];
    const float bj[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 bb = make_float2(bj[j], bj[j]);
      acc[j][0] = __ffma2_rn(make_float2(a.x, a.y), bb, acc[j][0]);
      acc[j][1] = __ffma2_rn(make_float2(a.z, a.w), bb, acc[j][1]);
    }
  }
}

template <int RPL>
__global__ void __launch_bounds__(DomSeries<RPL>::NT, 2)
    domain_series_kernel(const LkInst *__restrict__ insts, DomArgs a, int *__restrict__ sweep,
                         const float2 *__restrict__ cheb) {
  using C = DomSeries<RPL>;
  constexpr int MPD = C::MPD, NT = C::NT, NW = C::NW, CG = C::CG, RS = DS_ROWS / 4;
  constexpr int VQ = (MPD + 31) / 32;
  extern __shared__ __align__(16) float dsm[];
  lk_pdl_wait();
  const LkInst &I = insts[0];
  const int m = I.m, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int dom = blockIdx.x, splits = gridDim.y;
  const int o0 = a.obs_off[dom], np = a.obs_off[dom + 1] - o0;
  const int n0 = a.node_off[dom], nn = a.node_off[dom + 1] - n0, nd = 2 * nn;
  const DomSeriesLayout Ly = dom_series_layout(MPD, a.max_obs, a.max_rows);
  float *S = dsm, *T = dsm, *G = dsm + Ly.g, *part = dsm + Ly.part, *sv = dsm + Ly.sv;
  float *ow = dsm + Ly.ow, *xm = dsm + Ly.xm, *cv = dsm + Ly.cv, *red = dsm + Ly.red;
  int *slot = reinterpret_cast<int *>(dsm + Ly.slot), *ids = reinterpret_cast<int *>(dsm + Ly.ids);
  const float *Ybp = static_cast<const float *>(I.Ybp);
  const float *dp = static_cast<const float *>(I.dp);
  float *X = static_cast<float *>(I.X);
  const float alpha = float(I.alpha);

  // ---- S = diag(sqrt(tau/sigma2)) Yb of the region and s: tables, then a warp per slope ----
  for (int k = tid; k < np; k += NT) {
    slot[k] = a.obs_slot[o0 + k];
    ow[k] = sqrtf(a.obs_w[o0 + k]);
  }
  for (int k = tid; k < nn; k += NT) ids[k] = a.node_ids[n0 + k];
  __syncthreads();
#pragma unroll 2
  for (int k = warp; k < np; k += NW) {
    const float *row = Ybp + (size_t)slot[k] * m;
    float v[VQ];
#pragma unroll
    for (int q = 0; q < VQ; ++q) v[q] = lane + 32 * q < m ? row[lane + 32 * q] : 0.f;
#pragma unroll
    for (int q = 0; q < VQ; ++q)
      if (lane + 32 * q < MPD) S[k * MPD + lane + 32 * q] = ow[k] * v[q];
  }
  for (int k = tid; k < np; k += NT) sv[k] = ow[k] * dp[slot[k]];
  __syncthreads();
  // ---- G = S^T S: the 4 x 4 tiles that touch the lower triangle, in blocks of 8 row
  // groups x 4 column groups per warp (a last block of fewer row groups takes
  // more column groups); the others by symmetry. c = S^T s, |G|_F^2, tr G. ----
  float fro = 0.f, tr = 0.f;
  constexpr int RBF = CG / 8, REM = CG % 8;          // full row blocks, row groups left
  constexpr int RL = REM ? (REM <= 2 ? 2 : 4) : 8, CL = 32 / RL;
  constexpr int FULL_TASKS = RBF * (RBF + 1);        // block rb: column blocks 0 .. 2 rb + 1
  constexpr int REM_TASKS = REM ? ((CG + CL - 1) / CL) * ((REM + RL - 1) / RL) : 0;
  for (int task = warp; task < FULL_TASKS + REM_TASKS; task += NW) {
    int ti, tj;
    if (task < FULL_TASKS) {
      int rb = 0, cb = task;
      while (cb > 2 * rb + 1) {
        cb -= 2 * rb + 2;
        ++rb;
      }
      ti = 8 * rb + (lane & 7);
      tj = 4 * cb + (lane >> 3);
    } else {
      constexpr int CBR = (CG + CL - 1) / CL;
      const int q = task - FULL_TASKS;
      ti = 8 * RBF + RL * (q / CBR) + lane % RL;
      tj = CL * (q % CBR) + lane / RL;
    }
    if (ti >= CG || tj > ti) continue;
    float2 acc[4][2];
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
    tile_product(acc, reinterpret_cast<const float4 *>(S) + ti, CG,
                 reinterpret_cast<const float4 *>(S) + tj, CG, np);
    const float w2 = ti == tj ? 1.f : 2.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float v[4] = {acc[j][0].x, acc[j][0].y, acc[j][1].x, acc[j][1].y};
      reinterpret_cast<float4 *>(G + (4 * tj + j) * MPD)[ti] =
          make_float4(v[0], v[1], v[2], v[3]);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        fro = fmaf(w2 * v[i], v[i], fro);
        if (ti == tj && i == j) tr += v[i];
      }
    }
    if (ti != tj) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        reinterpret_cast<float4 *>(G + (4 * ti + i) * MPD)[tj] =
            i & 1 ? make_float4(acc[0][i >> 1].y, acc[1][i >> 1].y, acc[2][i >> 1].y, acc[3][i >> 1].y)
                  : make_float4(acc[0][i >> 1].x, acc[1][i >> 1].x, acc[2][i >> 1].x, acc[3][i >> 1].x);
    }
  }
  for (int i = tid; i < MPD; i += NT) {
    float c0 = 0.f, c1 = 0.f;
    int k = 0;
#pragma unroll 4
    for (; k + 1 < np; k += 2) {
      c0 = fmaf(S[k * MPD + i], sv[k], c0);
      c1 = fmaf(S[(k + 1) * MPD + i], sv[k + 1], c1);
    }
    if (k < np) c0 = fmaf(S[k * MPD + i], sv[k], c0);
    cv[i] = c0 + c1;
  }
  fro = lk_warp_sum(fro);
  tr = lk_warp_sum(tr);
  if (lane == 0) {
    red[warp] = fro;
    red[16 + warp] = tr;
  }
  __syncthreads();
  fro = tr = 0.f;
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    fro += red[k];
    tr += red[16 + k];
  }
  const float ratio = sqrtf(fro) / alpha;
  const bool ok = ratio <= LK_CHEB_MAXD;             // (not with a NaN)
  if (tid == 0 && blockIdx.y == 0) {
    sweep[dom] = !ok;
    if (ok) {
      atomicMax(&a.counters[2], 1);
      atomicAdd(&a.counters[3], 1);
      if (a.kappa_thr > 0.f && 1.f + tr / alpha > a.kappa_thr) atomicAdd(&a.counters[1], 1);
    }
  }
  if (!ok) return;
  const float2 *co = cheb + (size_t)lk_cheb_class(ratio) * LK_CHEB_LD32;
  const float2 head = __ldg(co++);
  const float scale = head.x / alpha;
  const int deg = (int)head.y;
  const float inv_m = 1.f / float(m), rt = sqrtf(float(m - 1) / alpha), ia = 1.f / alpha;
  const int per = (nd + splits - 1) / splits;
  const int rbeg = blockIdx.y * per, rend = rbeg + per < nd ? rbeg + per : nd;

  for (int r0 = rbeg; r0 < rend; r0 += DS_ROWS) {
    const int nr = rend - r0 < DS_ROWS ? rend - r0 : DS_ROWS;   // rows of this pass
    __syncthreads();
    // ---- T_0: the anomaly rows (a warp per row), zero rows up to 32 ----
    for (int r = warp; r < DS_ROWS; r += NW) {
      float v[VQ], sum = 0.f;
      const float *x = r < nr ? X + ((size_t)ids[(r0 + r) >> 1] * 2 + ((r0 + r) & 1)) * m : nullptr;
#pragma unroll
      for (int q = 0; q < VQ; ++q) {
        v[q] = x && lane + 32 * q < m ? x[lane + 32 * q] : 0.f;
        sum += v[q];
      }
      const float mu = lk_warp_sum(sum) * inv_m;
#pragma unroll
      for (int q = 0; q < VQ; ++q) {
        const int j = lane + 32 * q;
        if (j < MPD) T[j * DS_ROWS + r] = j < m ? v[q] - mu : 0.f;
      }
      if (lane == 0) xm[r] = mu;
    }
    __syncthreads();
    // ---- the series on this thread's tile: rows 4 rg + i, columns 4 cg + j. At most
    // 16 rows: warps of 4 x 8 tiles, the second half of them on the second half
    // of the product's columns ----
    const bool narrow = nr <= 16 && NW >= 4;
    constexpr int HW = (CG + 7) / 8;                 // warps of 4 x 8 tiles
    const int half = narrow ? warp / HW : 0;
    const int rg = narrow ? lane & 3 : lane & 7;
    const int cg = narrow ? 8 * (warp - half * HW) + (lane >> 2) : 4 * warp + (lane >> 3);
    const bool two = narrow && 2 * HW <= NW;
    const bool work = cg < CG && half < (two ? 2 : 1);
    const int qn = two ? MPD / 2 : MPD, q0 = half * qn;
    float2 u[4][2], v[4][2];
    float f = scale, e = 1.f, o = 0.f;
    float2 c = __ldg(co);
    for (int k = 0; k <= deg; ++k) {
      float4 *cur = reinterpret_cast<float4 *>(T + (k & 1) * MPD * DS_ROWS);
      float4 *nxt = reinterpret_cast<float4 *>(T + ((k + 1) & 1) * MPD * DS_ROWS);
      const float2 cn = k < deg ? __ldg(co + k + 1) : c;   // in flight during the product
      float2 acc[4][2];
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
      if (work && k < deg) {
        tile_product(acc, cur + q0 * RS + rg, RS, reinterpret_cast<const float4 *>(G) + q0 * CG + cg,
                     CG, qn);
        if (half == 1) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            reinterpret_cast<float4 *>(part)[((warp - HW) * 4 + j) * 32 + lane] =
                make_float4(acc[j][0].x, acc[j][0].y, acc[j][1].x, acc[j][1].y);
        }
      }
      if (two) __syncthreads();
      if (work && half == 0) {
        const float2 ca = make_float2(c.x, c.x), cb = make_float2(c.y, c.y);
        const float2 ff = make_float2(f, f), ee = make_float2(-e, -e), oo = make_float2(-o, -o);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 t4 = cur[(4 * cg + j) * RS + rg];
          const float2 t0 = make_float2(t4.x, t4.y), t1 = make_float2(t4.z, t4.w);
          if (k == 0) {
            u[j][0] = __fmul2_rn(ca, t0);
            u[j][1] = __fmul2_rn(ca, t1);
            v[j][0] = __fmul2_rn(cb, t0);
            v[j][1] = __fmul2_rn(cb, t1);
          } else {
            u[j][0] = __ffma2_rn(ca, t0, u[j][0]);
            u[j][1] = __ffma2_rn(ca, t1, u[j][1]);
            v[j][0] = __ffma2_rn(cb, t0, v[j][0]);
            v[j][1] = __ffma2_rn(cb, t1, v[j][1]);
          }
          if (k < deg) {
            // T_k+1 = f T_k G - e T_k - o T_k-1 (f, e, o = scale, 1, 0, then 2 scale, 2, 1)
            if (two) {
              const float4 h = reinterpret_cast<const float4 *>(part)[(warp * 4 + j) * 32 + lane];
              acc[j][0] = __fadd2_rn(acc[j][0], make_float2(h.x, h.y));
              acc[j][1] = __fadd2_rn(acc[j][1], make_float2(h.z, h.w));
            }
            float4 p4 = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k) p4 = nxt[(4 * cg + j) * RS + rg];
            const float2 w0 = __ffma2_rn(ff, acc[j][0], __ffma2_rn(ee, t0,
                                         __fmul2_rn(oo, make_float2(p4.x, p4.y))));
            const float2 w1 = __ffma2_rn(ff, acc[j][1], __ffma2_rn(ee, t1,
                                         __fmul2_rn(oo, make_float2(p4.z, p4.w))));
            nxt[(4 * cg + j) * RS + rg] = make_float4(w0.x, w0.y, w1.x, w1.y);
          }
        }
      }
      c = cn;
      f = 2.f * scale;
      e = 2.f;
      o = 1.f;
      __syncthreads();
    }
    // ---- the sums of A^-1/2 row-major in T's place; the rows' parts of X'_r wbar ----
    if (work && half == 0) {
      const float4 c4 = reinterpret_cast<const float4 *>(cv)[cg];
      float4 pw;
      float *pp = reinterpret_cast<float *>(&pw);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float s0 = i & 1 ? v[0][i >> 1].y : v[0][i >> 1].x;
        const float s1 = i & 1 ? v[1][i >> 1].y : v[1][i >> 1].x;
        const float s2 = i & 1 ? v[2][i >> 1].y : v[2][i >> 1].x;
        const float s3 = i & 1 ? v[3][i >> 1].y : v[3][i >> 1].x;
        pp[i] = fmaf(s0, c4.x, s1 * c4.y) + fmaf(s2, c4.z, s3 * c4.w);
        reinterpret_cast<float4 *>(T + (size_t)(4 * rg + i) * MPD)[cg] =
            i & 1 ? make_float4(u[0][i >> 1].y, u[1][i >> 1].y, u[2][i >> 1].y, u[3][i >> 1].y)
                  : make_float4(u[0][i >> 1].x, u[1][i >> 1].x, u[2][i >> 1].x, u[3][i >> 1].x);
      }
      reinterpret_cast<float4 *>(part)[cg * RS + rg] = pw;
    }
    __syncthreads();
    // ---- apply, a warp per row: Xa_r = xbar_r + X'_r wbar + sqrt((m-1)/alpha) u_r ----
    for (int r = warp; r < nr; r += NW) {
      const int pid = ids[(r0 + r) >> 1], comp = (r0 + r) & 1;
      float *x = X + ((size_t)pid * 2 + comp) * m;
      const float mu0 = xm[r];
      const float w = lk_warp_sum(lane < CG ? part[lane * DS_ROWS + r] : 0.f) * ia;
      float xa[VQ], sum = 0.f;
#pragma unroll
      for (int q = 0; q < VQ; ++q) {
        const int j = lane + 32 * q;
        xa[q] = 0.f;
        if (j < m) {
          xa[q] = mu0 + w + rt * T[(size_t)r * MPD + j];
          x[j] = xa[q];
        }
        sum += xa[q];
      }
      const float mu = lk_warp_sum(sum) * inv_m;
      float sq = 0.f;
#pragma unroll
      for (int q = 0; q < VQ; ++q) {
        const float d = lane + 32 * q < m ? xa[q] - mu : 0.f;
        sq = fmaf(d, d, sq);
      }
      const float sp = sqrtf(lk_warp_sum(sq) / float(m - 1));
      if (lane == 0) {
        if (a.mean) a.mean[(size_t)pid * 2 + comp] = mu;
        if (a.spread) a.spread[(size_t)pid * 2 + comp] = sp;
        a.delta[(size_t)pid * 2 + comp] = mu - mu0;
        if (!isfinite(mu) || !isfinite(sp)) atomicOr(&a.counters[0], LK_BIT_NONFINITE);
      }
    }
  }
}

// b_d = sum over the border edges of domain d of (delta_other - delta_own) for
// both state rows: a warp per domain, its incident edges over the lanes.
__global__ void __launch_bounds__(LK_WARP_CTA)
    piston_sum_kernel(int n_dom, const int2 *__restrict__ edges, const int *__restrict__ dedge_off,
                      const int *__restrict__ dedge, const float *__restrict__ delta,
                      float *__restrict__ bsum) {
  lk_pdl_wait();
  lk_pdl_trigger();
  const int d = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (d >= n_dom) return;
  float b0 = 0.f, b1 = 0.f;
  for (int q = dedge_off[d] + lane; q < dedge_off[d + 1]; q += 32) {
    const int se = dedge[q];
    const int2 ed = edges[(se > 0 ? se : -se) - 1];
    const int own = se > 0 ? ed.x : ed.y, oth = se > 0 ? ed.y : ed.x;
    b0 += delta[2 * oth] - delta[2 * own];
    b1 += delta[2 * oth + 1] - delta[2 * own + 1];
  }
  b0 = lk_warp_sum(b0);
  b1 = lk_warp_sum(b1);
  if (lane == 0) {
    bsum[2 * d] = b0;
    bsum[2 * d + 1] = b1;
  }
}

// c_d = (K b)_d, then every member of the domain's rows moves by it (and so does
// the analysis mean): a CTA per domain, so that the product's n_dom^2 terms are
// read by as many CTAs as there are rows (one CTA for all took 17 us at 75
// domains and 53 us at 373), and a warp per node whose values are in flight
// while the product forms.
constexpr int PA_WARPS = 16, PA_VALS = 4;            // nodes at a time; values per lane and row
__global__ void __launch_bounds__(PA_WARPS * 32)
    piston_apply_kernel(const LkInst *__restrict__ insts, int n_dom,
                        const int *__restrict__ node_off, const int *__restrict__ node_ids,
                        const float *__restrict__ K, const float *__restrict__ bsum,
                        float *__restrict__ mean) {
  __shared__ float part[2][PA_WARPS];
  lk_pdl_wait();
  const LkInst &I = insts[0];
  const int d = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, m = I.m;
  const int q0 = node_off[d], q1 = node_off[d + 1];
  float c0 = 0.f, c1 = 0.f;
  for (int e = threadIdx.x; e < n_dom; e += PA_WARPS * 32) {
    const float k = K[(size_t)d * n_dom + e];
    const float2 b = reinterpret_cast<const float2 *>(bsum)[e];
    c0 = fmaf(k, b.x, c0);
    c1 = fmaf(k, b.y, c1);
  }
  c0 = lk_warp_sum(c0);
  c1 = lk_warp_sum(c1);
  if (lane == 0) {
    part[0][warp] = c0;
    part[1][warp] = c1;
  }
  int node = q0 + warp < q1 ? node_ids[q0 + warp] : -1;
  float v0[PA_VALS], v1[PA_VALS];                    // m <= 128: all of the row
  auto load = [&]() {
    const float *x = static_cast<const float *>(I.X) + (size_t)node * 2 * m;
#pragma unroll
    for (int q = 0; q < PA_VALS; ++q) {
      const bool in = node >= 0 && lane + 32 * q < m;
      v0[q] = in ? x[lane + 32 * q] : 0.f;
      v1[q] = in ? x[m + lane + 32 * q] : 0.f;
    }
  };
  load();
  __syncthreads();
  c0 = c1 = 0.f;
#pragma unroll
  for (int w = 0; w < PA_WARPS; ++w) {
    c0 += part[0][w];
    c1 += part[1][w];
  }
  for (int q = q0 + warp; node >= 0;) {
    float *x = static_cast<float *>(I.X) + (size_t)node * 2 * m;
#pragma unroll
    for (int k = 0; k < PA_VALS; ++k)
      if (lane + 32 * k < m) {
        x[lane + 32 * k] = v0[k] + c0;
        x[m + lane + 32 * k] = v1[k] + c1;
      }
    if (lane < 2 && mean) mean[2 * node + lane] += lane ? c1 : c0;
    q += PA_WARPS;
    node = q < q1 ? node_ids[q] : -1;
    load();
  }
}

// ---------------------------------------------------------------------------
// One domain covering the grid (partition 1): the global ETKF (Section 3.1.1)
// for any number of slopes and nodes, as three kernels:
//   gram    partial sums of A = S^T S and c = S^T s over parts of the slopes, one
//           CTA per (upper-triangle 32 x 32 tile of A, part): every term
//           w_k y_ka y_kb (w = tau / sigma2, y the grid's FP32 values) summed as
//           an unevaluated float pair: about 1e-12 relative to the sum of |terms|,
//           on the FP32 pipe, against FP64 FMAs at 1/75 of its rate. Six
//           operations a term (gl_add_anchored) instead of the seventeen of
//           two-products and two-sums: m = 626, 1624 slopes 183 -> 62 us
//   solve   one CTA: A = (m-1)/rho I + the partials (FP64), its FP32 rounding
//           diagonalised by the domain kernel's Jacobi (A = Q Lambda Q^T), then
//           wbar = A^-1 c by mixed-precision iterative refinement (residual
//           c - A wbar in FP64, correction Q Lambda^-1 Q^T r in FP32: the error
//           contracts by about kappa eps32 per step, so a few steps reach the
//           FP64 solution although kappa_hat reaches 1e4-1e5 for the whole
//           pupil), and T = wbar 1^T + Q ((m-1) Lambda^-1)^(1/2) Q^T
//   apply   a CTA per 16 state rows: Xa_r = xbar_r + X'_r T, mean, spread
// ---------------------------------------------------------------------------
constexpr int GL_TILE = 32, GL_KC = 64, GL_REFINE = 4;

// hi + lo += w a b: the product a b as two floats (FMA two-product), each times w
// (again two-product for the high part), added to the pair by Knuth's two-sum.
// The _rn intrinsics keep the compiler from contracting the steps.
__device__ __forceinline__ void gl_add_wab(float &hi, float &lo, float w, float a, float b) {
  const float ph = __fmul_rn(a, b);
  const float pl = fmaf(a, b, -ph);
  const float qh = __fmul_rn(w, ph);
  const float ql = fmaf(w, ph, -qh);
  const float t = fmaf(w, pl, ql);
  const float s = __fadd_rn(hi, qh);
  const float bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(qh, bb));
  hi = s;
  lo = __fadd_rn(lo, __fadd_rn(e, t));
}

// hi + lo += (ah + al) b, with q = the product's multiple of ulp(sigma): sigma a
// constant 1.5 2^M with the sum of all |q| of a chunk below 2^M, so that hi sums
// the q exactly and lo the rests, each rest one FMA (the extraction of Rump, Ogita
// and Oishi's accurate summation): six operations, two outputs each.
__device__ __forceinline__ void gl_add_anchored(float2 &hi, float2 &lo, float2 ah, float2 al,
                                                float2 b, float2 sg, float2 msg) {
  const float2 q = __fadd2_rn(__ffma2_rn(ah, b, sg), msg);
  const float2 mq = make_float2(-q.x, -q.y);
  const float2 r = __ffma2_rn(al, b, __ffma2_rn(ah, b, mq));
  hi = __fadd2_rn(hi, q);
  lo = __fadd2_rn(lo, r);
}

// Blocks: (upper-triangle tile of A, part of the slopes); a part is a run of
// chunks of GL_KC slopes, each summed with its own anchor and then added to
// the running pairs by two-sums.
__global__ void __launch_bounds__(256)
    global_gram_kernel(const LkInst *__restrict__ insts, const int *__restrict__ obs_slot,
                       const float *__restrict__ obs_w, int np, int mpt,
                       double *__restrict__ gpart, double *__restrict__ cpart) {
  constexpr int LD = GL_TILE + 2;
  __shared__ __align__(16) float sh[GL_KC][LD], sl[GL_KC][LD], sj[GL_KC][LD];
  __shared__ float sw[GL_KC], sd[GL_KC], mxi[8], mxj[8];
  lk_pdl_wait();
  const LkInst &I = insts[0];
  const int m = I.m, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float *Ybp = static_cast<const float *>(I.Ybp);
  const float *dp = static_cast<const float *>(I.dp);
  // upper-triangle tile (ti <= tj) from blockIdx.x
  const int nt = mpt / GL_TILE;
  int ti = 0, tj = blockIdx.x;
  while (tj >= nt - ti) {
    tj -= nt - ti;
    ++ti;
  }
  tj += ti;
  const int chunks = (np + GL_KC - 1) / GL_KC;
  const int per = (chunks + gridDim.y - 1) / gridDim.y;
  const int c0 = blockIdx.y * per, c1 = c0 + per < chunks ? c0 + per : chunks;
  const int a0 = (threadIdx.x / 16) * 2, b0 = (threadIdx.x % 16) * 2;
  float2 H[2], L[2];
  H[0] = H[1] = L[0] = L[1] = make_float2(0.f, 0.f);
  float ch = 0.f, cl = 0.f;
  for (int kc = c0; kc < c1; ++kc) {
    const int k0 = kc * GL_KC, kn = np - k0 < GL_KC ? np - k0 : GL_KC;
    __syncthreads();
    float ma = 0.f, mb = 0.f;
    for (int k = warp; k < GL_KC; k += 8) {          // a warp per slope, a lane per column
      float x = 0.f, y = 0.f, w = 0.f;
      if (k < kn) {
        const int slot = obs_slot[k0 + k];
        const int ri = ti * GL_TILE + lane, rj = tj * GL_TILE + lane;
        w = obs_w[k0 + k];
        if (ri < m) x = Ybp[(size_t)slot * m + ri];
        if (rj < m) y = Ybp[(size_t)slot * m + rj];
        if (lane == 0) sd[k] = dp[slot];
      } else if (lane == 0) {
        sd[k] = 0.f;
      }
      const float p = __fmul_rn(w, x);               // w x as a pair
      sh[k][lane] = p;
      sl[k][lane] = fmaf(w, x, -p);
      sj[k][lane] = y;
      if (lane == 0) sw[k] = w;
      ma = fmaxf(ma, fabsf(p));
      mb = fmaxf(mb, fabsf(y));
    }
    for (int o = 16; o > 0; o >>= 1) {
      ma = fmaxf(ma, __shfl_xor_sync(FULL, ma, o));
      mb = fmaxf(mb, __shfl_xor_sync(FULL, mb, o));
    }
    if (lane == 0) {
      mxi[warp] = ma;
      mxj[warp] = mb;
    }
    __syncthreads();
    ma = mxi[0];
    mb = mxj[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) {
      ma = fmaxf(ma, mxi[w]);
      mb = fmaxf(mb, mxj[w]);
    }
    // |q| < 2^(ilogb ma + ilogb mb + 2), GL_KC = 64 of them
    int M = -100;
    if (ma > 0.f && mb > 0.f) {
      // (an infinite slope has INT_MAX for an exponent: 127 takes its place in the sum)
      M = ilogbf(fminf(ma, 0x1p127f)) + ilogbf(fminf(mb, 0x1p127f)) + 9;
      M = M < -100 ? -100 : M;
    }
    const float s = scalbnf(1.5f, M);                // infinite where a product is: NaN follows
    const float2 sg = make_float2(s, s), msg = make_float2(-s, -s);
    float2 hi[2], lo[2];
    hi[0] = hi[1] = lo[0] = lo[1] = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int k = 0; k < GL_KC; ++k) {
      const float2 x = *reinterpret_cast<const float2 *>(&sh[k][a0]);
      const float2 xl = *reinterpret_cast<const float2 *>(&sl[k][a0]);
      const float2 y = *reinterpret_cast<const float2 *>(&sj[k][b0]);
      gl_add_anchored(hi[0], lo[0], make_float2(x.x, x.x), make_float2(xl.x, xl.x), y, sg, msg);
      gl_add_anchored(hi[1], lo[1], make_float2(x.y, x.y), make_float2(xl.y, xl.y), y, sg, msg);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {                    // (H, L) += (hi, lo), Knuth's two-sum
      const float2 t = __fadd2_rn(H[i], hi[i]);
      const float2 mH = make_float2(-H[i].x, -H[i].y);
      const float2 bb = __fadd2_rn(t, mH);
      const float2 d = __fadd2_rn(t, make_float2(-bb.x, -bb.y));
      const float2 e = __fadd2_rn(__fadd2_rn(H[i], make_float2(-d.x, -d.y)),
                                  __fadd2_rn(hi[i], make_float2(-bb.x, -bb.y)));
      H[i] = t;
      L[i] = __fadd2_rn(L[i], __fadd2_rn(e, lo[i]));
    }
    if (ti == tj && threadIdx.x < GL_TILE)
      for (int k = 0; k < GL_KC; ++k)                // w x d, x = the column's own slope
        gl_add_wab(ch, cl, sw[k], sj[k][threadIdx.x], sd[k]);
  }
  double *out = gpart + (size_t)blockIdx.y * mpt * mpt;
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    double *o = out + (size_t)(ti * GL_TILE + a0 + x) * mpt + tj * GL_TILE + b0;
    o[0] = (double)H[x].x + (double)L[x].x;
    o[1] = (double)H[x].y + (double)L[x].y;
  }
  if (ti == tj && threadIdx.x < GL_TILE)
    cpart[(size_t)blockIdx.y * mpt + ti * GL_TILE + threadIdx.x] = (double)ch + (double)cl;
}

// Shared memory of the solve kernel: A (FP64, [MPD][MPD+1]), c, wbar, r (FP64),
// then one float region used first as the Jacobi's column exchange and then
// for Q ([MPD][MPD+1]), and lambda, t, sroot.
template <int RPL>
__host__ __device__ constexpr size_t gsolve_qfloats() {
  constexpr size_t MPD = 8 * RPL, q = MPD * (MPD + 1), x = 2 * (MPD / 2) * MPD + 2 * (MPD / 2);
  return q > x ? q : x;
}
template <int RPL>
size_t global_solve_smem() {
  constexpr int MPD = 8 * RPL;
  return sizeof(double) * ((size_t)MPD * (MPD + 1) + 3 * MPD) +
         sizeof(float) * (gsolve_qfloats<RPL>() + 3 * MPD);
}

template <int RPL>
__global__ void __launch_bounds__(32 * RPL)
    global_solve_kernel(const LkInst *__restrict__ insts, const double *__restrict__ gpart,
                        const double *__restrict__ cpart, int kchunks, int mpt,
                        float *__restrict__ T, float tol, float stop, int max_sweeps,
                        int *__restrict__ counters) {
  constexpr int MPD = 8 * RPL, G = MPD / 2, NT = 4 * MPD, LD = MPD + 1;
  extern __shared__ __align__(16) double gsm[];
  lk_pdl_wait();
  const LkInst &I = insts[0];
  const int m = I.m, tid = threadIdx.x;
  double *A = gsm;                              // [MPD][LD] FP64
  double *c64 = A + MPD * LD, *w64 = c64 + MPD, *r64 = w64 + MPD;
  float *Qs = reinterpret_cast<float *>(r64 + MPD);   // [MPD][LD], after the sweeps
  float *xb = Qs, *xn = xb + 2 * G * MPD;             // exchange, during the sweeps
  float *lam = Qs + gsolve_qfloats<RPL>(), *tv = lam + MPD, *sr = tv + MPD;
  const double alpha = I.alpha;
  // ---- A and c from the partial sums: element (i, j) of the upper triangle
  // was summed in tile (min / 32, max / 32) at (min, max) ----
  for (int e = tid; e < MPD * MPD; e += NT) {
    const int i = e / MPD, j = e - i * MPD;
    const int a = i <= j ? i : j, b = i <= j ? j : i;
    double s = 0.0;
    for (int k = 0; k < kchunks; ++k) s += gpart[((size_t)k * mpt + a) * mpt + b];
    if (i == j) s += i < m ? alpha : 1.0;
    A[i * LD + j] = s;
  }
  if (tid < MPD) {
    double s = 0.0;
    for (int k = 0; k < kchunks; ++k) s += cpart[(size_t)k * mpt + tid];
    c64[tid] = s;
    w64[tid] = 0.0;
  }
  __syncthreads();
  // ---- FP32 Jacobi on the rounded A (the domain kernel's layout and rounds) ----
  const int g = tid >> 3, l = tid & 7;
  float P[RPL], Q[RPL];
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    P[i] = (float)A[(l + 8 * i) * LD + 2 * g];
    Q[i] = (float)A[(l + 8 * i) * LD + 2 * g + 1];
  }
  const float tol2 = tol * tol, stop2 = stop * stop;
  int buf = 0, sweeps = 0;
  bool conv = false;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    float pp = 0.f, qq = 0.f;
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      pp = fmaf(P[i], P[i], pp);
      qq = fmaf(Q[i], Q[i], qq);
    }
    float nP = group8_sum(pp), nQ = group8_sum(qq);
    int flags = 0;
    for (int r = 0; r < G; ++r) {
      flags |= dom_round<RPL>(P, Q, nP, nQ, tol2, stop2, false);
      dom_xfer<RPL>(Q, nQ, xb, xn, buf, g, l, g + 1 < G ? g + 1 : 0);
      flags |= dom_round<RPL>(P, Q, nP, nQ, tol2, stop2, g == G - 1);
      dom_xfer<RPL>(P, nP, xb, xn, buf, g, l, g > 0 ? g - 1 : G - 1);
    }
    sweeps = sweep + 1;
    if (!__syncthreads_or(flags & 2)) {
      conv = true;
      break;
    }
  }
  if (tid == 0) {
    atomicMax(&counters[2], sweeps);
    atomicAdd(&counters[3], sweeps);
    if (!conv) atomicOr(&counters[0], LK_BIT_NOCONVERGE);
  }
  float pp = 0.f, qq = 0.f;
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    pp = fmaf(P[i], P[i], pp);
    qq = fmaf(Q[i], Q[i], qq);
  }
  const float lP = sqrtf(group8_sum(pp)), lQ = sqrtf(group8_sum(qq));
  __syncthreads();                              // the exchange region becomes Q
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    Qs[(l + 8 * i) * LD + 2 * g] = P[i] / lP;
    Qs[(l + 8 * i) * LD + 2 * g + 1] = Q[i] / lQ;
  }
  if (l == 0) {
    lam[2 * g] = lP;
    lam[2 * g + 1] = lQ;
  }
  __syncthreads();
  if (tid < MPD) sr[tid] = sqrtf(float(m - 1) / lam[tid]);
  // ---- wbar = A^-1 c by iterative refinement ----
  for (int it = 0; it < GL_REFINE; ++it) {
    if (tid < MPD) {                              // r = c - A w (FP64)
      double s = c64[tid];
      for (int j = 0; j < MPD; ++j) s = fma(-A[tid * LD + j], w64[j], s);
      r64[tid] = s;
    }
    __syncthreads();
    if (tid < MPD) {                              // t = Lambda^-1 Q^T r
      float s = 0.f;
      for (int j = 0; j < MPD; ++j) s = fmaf(Qs[j * LD + tid], (float)r64[j], s);
      tv[tid] = s / lam[tid];
    }
    __syncthreads();
    if (tid < MPD) {                              // w += Q t
      float s = 0.f;
      for (int c = 0; c < MPD; ++c) s = fmaf(Qs[tid * LD + c], tv[c], s);
      w64[tid] += (double)s;
    }
    __syncthreads();
  }
  // ---- T = wbar 1^T + Q diag(sroot) Q^T ----
  for (int e = tid; e < m * m; e += NT) {
    const int i = e / m, j = e - i * m;
    float s = 0.f;
    for (int c = 0; c < MPD; ++c) s = fmaf(Qs[i * LD + c] * sr[c], Qs[j * LD + c], s);
    T[e] = (float)w64[i] + s;
  }
}

// Xa_r = xbar_r + X'_r T for 16 state rows per CTA (rows = node-major, 2 per node).
__global__ void __launch_bounds__(256)
    global_apply_kernel(const LkInst *__restrict__ insts, const float *__restrict__ T,
                        float *__restrict__ mean, float *__restrict__ spread,
                        int *__restrict__ counters) {
  extern __shared__ __align__(16) float asm_[];
  lk_pdl_wait();
  const LkInst &I = insts[0];
  const int m = I.m, tid = threadIdx.x;
  float *Ts = asm_;                               // [m][m]
  float *xr = Ts + m * m;                         // [16][m]
  for (int e = tid; e < m * m; e += blockDim.x) Ts[e] = T[e];
  const long long r0 = (long long)blockIdx.x * 16, nrows = 2LL * I.n_pts;
  float *X = static_cast<float *>(I.X);
  for (int e = tid; e < 16 * m; e += blockDim.x) {
    const long long r = r0 + e / m;
    xr[e] = r < nrows ? X[r * m + e % m] : 0.f;
  }
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31;
  const float inv_m = 1.f / float(m);
  for (int q = warp; q < 16; q += 8) {
    const long long r = r0 + q;
    if (r >= nrows) break;
    float s = 0.f;
    for (int j = lane; j < m; j += 32) s += xr[q * m + j];
    const float xbar = lk_warp_sum(s) * inv_m;
    float sum = 0.f;
    for (int j = lane; j < m; j += 32) {
      float acc = 0.f;
      for (int i = 0; i < m; ++i) acc = fmaf(xr[q * m + i] - xbar, Ts[i * m + j], acc);
      const float xa = xbar + acc;
      X[r * m + j] = xa;
      sum += xa;
    }
    const float mu = lk_warp_sum(sum) * inv_m;
    float sq = 0.f;
    for (int j = lane; j < m; j += 32) {
      const float dv = X[r * m + j] - mu;
      sq = fmaf(dv, dv, sq);
    }
    const float sp = sqrtf(lk_warp_sum(sq) / float(m - 1));
    if (lane == 0) {
      if (mean) mean[r] = mu;
      if (spread) spread[r] = sp;
      if (!isfinite(mu) || !isfinite(sp)) atomicOr(&counters[0], LK_BIT_NONFINITE);
    }
  }
}

constexpr int gl_mpt(int mpd) { return ((mpd + GL_TILE - 1) / GL_TILE) * GL_TILE; }

template <int RPL>
cudaError_t launch_global_rpl(letkf_ctx *h, void *mean, void *spread) {
  const LkDom &D = *h->dom;
  const LkInst &I = h->inst[0];
  constexpr int MPT = gl_mpt(8 * RPL), NT = MPT / GL_TILE;
  cudaError_t e = lk_launch_pdl(global_gram_kernel, dim3(NT * (NT + 1) / 2, D.kchunks), 256, 0,
                                h->stream, h->d_inst, (const int *)D.obs_slot,
                                (const float *)D.obs_w, D.max_obs, MPT, D.gpart, D.cpart);
  if (e != cudaSuccess) return e;
  e = lk_launch_pdl(global_solve_kernel<RPL>, 1, 32 * RPL, global_solve_smem<RPL>(), h->stream,
                    h->d_inst, (const double *)D.gpart, (const double *)D.cpart, D.kchunks, MPT,
                    D.T, (float)h->tol32, (float)(h->stop32 > h->tol32 ? h->stop32 : h->tol32),
                    h->max_sweeps, h->counters);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (unsigned)((2LL * I.n_pts + 15) / 16);
  return lk_launch_pdl(global_apply_kernel, blocks, 256,
                       sizeof(float) * ((size_t)I.m * I.m + 16 * (size_t)I.m), h->stream,
                       h->d_inst, (const float *)D.T, static_cast<float *>(mean),
                       static_cast<float *>(spread), h->counters);
}

template <int RPL>
cudaError_t setup_global_rpl(const LkDom &D, int m) {
  cudaError_t e = lk_raise_smem(global_solve_kernel<RPL>, global_solve_smem<RPL>());
  if (e == cudaSuccess)
    e = lk_raise_smem(global_apply_kernel, sizeof(float) * ((size_t)m * m + 16 * (size_t)m));
  (void)D;
  return e;
}

template <int RPL>
cudaError_t launch_rpl(letkf_ctx *h, DomArgs a) {
  const LkDom &D = *h->dom;
  if (D.series && h->cheb32) {
    const size_t b = sizeof(float) *
                     (size_t)dom_series_layout(8 * RPL, D.max_obs, 2 * D.max_nodes).total;
    const cudaError_t e =
        lk_launch_pdl(domain_series_kernel<RPL>, dim3(D.n_dom, D.splits), DomSeries<RPL>::NT, b,
                      h->stream, h->d_inst, a, D.sweep, (const float2 *)h->cheb32);
    if (e != cudaSuccess) return e;
    a.sweep = D.sweep;                 // the others, if any
  }
  const size_t smem = (size_t)dom_layout(8 * RPL, D.max_obs, 2 * D.max_nodes).total * sizeof(float);
  return lk_launch_pdl(domain_kernel<RPL>, (unsigned)D.n_dom, 32 * RPL, smem, h->stream,
                       h->d_inst, a);
}

template <int RPL>
cudaError_t setup_rpl(const LkDom &D) {
  const size_t smem = (size_t)dom_layout(8 * RPL, D.max_obs, 2 * D.max_nodes).total * sizeof(float);
  const cudaError_t e = lk_raise_smem(domain_kernel<RPL>, smem);
  if (e != cudaSuccess || !D.series) return e;
  const size_t b = sizeof(float) *
                   (size_t)dom_series_layout(8 * RPL, D.max_obs, 2 * D.max_nodes).total;
  return lk_raise_smem(domain_series_kernel<RPL>, b);
}

// Rows per lane of the Jacobi layout (MPD = 8 RPL columns); 0: wider than the
// one-CTA layout takes (the global ETKF's Newton-Schulz path, letkf_global.cu).
int rpl_of(int m) {
  return m <= 16 ? 2 : m <= 32 ? 4 : m <= 64 ? 8 : m <= 104 ? 13 : m <= 128 ? 16 : 0;
}

template <typename T>
cudaError_t dup(T **dst, const std::vector<T> &src) {
  *dst = nullptr;
  if (src.empty()) return cudaSuccess;
  cudaError_t e = cudaMalloc((void **)dst, src.size() * sizeof(T));
  if (e == cudaSuccess) e = cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice);
  return e;
}

// Cholesky solve of the SPD system M X = B in place (n x n, B n x k), FP64.
bool chol_solve(std::vector<double> &M, int n, std::vector<double> &B, int k) {
  for (int j = 0; j < n; ++j) {
    double s = M[(size_t)j * n + j];
    for (int q = 0; q < j; ++q) s -= M[(size_t)j * n + q] * M[(size_t)j * n + q];
    if (!(s > 0)) return false;
    const double d = sqrt(s);
    M[(size_t)j * n + j] = d;
    for (int i = j + 1; i < n; ++i) {
      double t = M[(size_t)i * n + j];
      for (int q = 0; q < j; ++q) t -= M[(size_t)i * n + q] * M[(size_t)j * n + q];
      M[(size_t)i * n + j] = t / d;
    }
  }
  for (int c = 0; c < k; ++c) {
    for (int i = 0; i < n; ++i) {                 // L y = b
      double t = B[(size_t)i * k + c];
      for (int q = 0; q < i; ++q) t -= M[(size_t)i * n + q] * B[(size_t)q * k + c];
      B[(size_t)i * k + c] = t / M[(size_t)i * n + i];
    }
    for (int i = n - 1; i >= 0; --i) {            // L^T x = y
      double t = B[(size_t)i * k + c];
      for (int q = i + 1; q < n; ++q) t -= M[(size_t)q * n + i] * B[(size_t)q * k + c];
      B[(size_t)i * k + c] = t / M[(size_t)i * n + i];
    }
  }
  return true;
}

}  // namespace

// Domain tables of a single-instance handle (cfg.partition > 0); the per-node
// geometry (nodes, subapertures, grid) is already in h->inst[0].
letkf_status lk_domains_build(letkf_ctx *h, const letkf_config &c, const std::vector<int> &pid,
                              const std::vector<int2> &pts, const std::vector<int2> &saps,
                              std::string &err) {
  const LkInst &I = h->inst[0];
  const int nsub = c.nsub, nn = nsub + 1, P = c.partition, w = c.window, hw = w / 2;
  LkDom *D = new (std::nothrow) LkDom();
  if (!D) return LETKF_ERR_NOMEM;
  h->dom = D;
  D->piston = c.piston != 0;
  std::vector<int> sid((size_t)nsub * nsub, -1);
  for (size_t k = 0; k < saps.size(); ++k) sid[(size_t)saps[k].x * nsub + saps[k].y] = (int)k;
  std::vector<int> bb(P + 1);
  for (int b = 0; b <= P; ++b) bb[b] = (int)(((long long)b * nn) / P);
  const double cl = c.loc_len > 0 ? c.loc_len : w / 4.0;
  std::vector<int> node_off{0}, node_ids, obs_off{0}, obs_slot, node_dom(pts.size(), -1);
  std::vector<char> mark((size_t)nsub * nsub, 0);
  for (int bi = 0; bi < P; ++bi)
    for (int bj = 0; bj < P; ++bj) {
      std::vector<int> ids;
      for (int i = bb[bi]; i < bb[bi + 1]; ++i)
        for (int j = bb[bj]; j < bb[bj + 1]; ++j)
          if (pid[(size_t)i * nn + j] >= 0) ids.push_back(pid[(size_t)i * nn + j]);
      if (ids.empty()) continue;
      int i0 = nn, i1 = -1, j0 = nn, j1 = -1;
      for (int q : ids) {
        i0 = std::min(i0, pts[q].x);
        i1 = std::max(i1, pts[q].x);
        j0 = std::min(j0, pts[q].y);
        j1 = std::max(j1, pts[q].y);
        node_dom[q] = (int)node_off.size() - 1;
        node_ids.push_back(q);
      }
      node_off.push_back((int)node_ids.size());
      // union of the nodes' windows, row-major over the subaperture grid
      std::vector<int> region;
      for (int q : ids)
        for (int s = pts[q].x - hw; s < pts[q].x - hw + w; ++s)
          for (int t = pts[q].y - hw; t < pts[q].y - hw + w; ++t)
            if (s >= 0 && s < nsub && t >= 0 && t < nsub && sid[(size_t)s * nsub + t] >= 0 &&
                !mark[(size_t)s * nsub + t]) {
              mark[(size_t)s * nsub + t] = 1;
              region.push_back(s * nsub + t);
            }
      std::sort(region.begin(), region.end());
      for (int st : region) {
        const int s = st / nsub, t = st % nsub;
        mark[(size_t)st] = 0;
        double tau = 1.0;
        if (c.taper == 1) {
          const double dx = std::max({i0 - (s + 0.5), 0.0, (s + 0.5) - i1});
          const double dy = std::max({j0 - (t + 0.5), 0.0, (t + 0.5) - j1});
          tau = lk_gaspari_cohn(hypot(dx, dy) / cl);
        }
        const long long cell = (long long)(s + I.h) * I.gs_cols + (t + I.h);
        obs_slot.push_back((int)(cell * 2));
        obs_slot.push_back((int)(cell * 2 + 1));
        D->tau.push_back(tau);
        D->tau.push_back(tau);
      }
      obs_off.push_back((int)obs_slot.size());
      D->max_obs = std::max(D->max_obs, (int)region.size() * 2);
      D->max_nodes = std::max(D->max_nodes, (int)ids.size());
    }
  D->n_dom = (int)node_off.size() - 1;
  // the global ETKF of more than 64 members takes the Newton-Schulz path
  // (m = 101: 0.59 ms against 0.72 ms for the one-CTA Jacobi, measured)
  D->rpl = (P == 1 && c.m > 64) ? 0 : rpl_of(c.m);
  D->global = P == 1;
  if (D->rpl == 0 && !D->global) {
    err = "local domains of more than one take m <= 128";
    return LETKF_ERR_ARG;
  }
  const int mpd = D->rpl ? 8 * D->rpl : ((c.m + 63) / 64) * 64;
  const size_t smem = (size_t)dom_layout(mpd, D->max_obs, 2 * D->max_nodes).total * sizeof(float);
  int dev_smem = 0;
  cudaDeviceGetAttribute(&dev_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device);
  if (!D->global && smem > (size_t)dev_smem) {
    err = "local domains too large for one CTA's shared memory (fewer nodes per domain, a "
          "smaller window or fewer members)";
    return LETKF_ERR_ARG;
  }
  // The series form, where its shared memory fits too. Systems of so few domains
  // that half the SMs would idle give each domain's rows to two or more CTAs (at
  // least 8 rows each): the products, most of the work, split, the Gram repeats.
  int sms = 1;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device);
  if (!D->global) {
    D->splits = std::max(1, std::min({sms / std::max(1, D->n_dom), 2 * D->max_nodes / 8, 4}));
    const size_t b = sizeof(float) *
                     (size_t)dom_series_layout(mpd, D->max_obs, 2 * D->max_nodes).total;
    D->series = b <= (size_t)dev_smem;
  }
  // border edges and their incidence per domain
  std::vector<int2> edges;
  for (size_t q = 0; q < pts.size(); ++q) {
    const int i = pts[q].x, j = pts[q].y;
    const int nb[2] = {i + 1 < nn ? pid[(size_t)(i + 1) * nn + j] : -1,
                       j + 1 < nn ? pid[(size_t)i * nn + j + 1] : -1};
    for (int o : nb)
      if (o >= 0 && node_dom[o] != node_dom[q]) edges.push_back(make_int2((int)q, o));
  }
  const int Dn = D->n_dom;
  std::vector<std::vector<int>> inc(Dn);
  for (size_t e = 0; e < edges.size(); ++e) {
    inc[node_dom[edges[e].x]].push_back((int)e + 1);
    inc[node_dom[edges[e].y]].push_back(-((int)e + 1));
  }
  std::vector<int> dedge_off{0}, dedge;
  for (auto &v : inc) {
    dedge.insert(dedge.end(), v.begin(), v.end());
    dedge_off.push_back((int)dedge.size());
  }
  // K = (I - sum_comp 1_c w_c^T) L^+, L^+ = M^-1 - sum_comp u_c u_c^T with
  // M = L + sum_comp u_c u_c^T (u_c: normalised indicator of a connected group)
  std::vector<double> Lm((size_t)Dn * Dn, 0.0);
  for (const int2 &ed : edges) {
    const int a = node_dom[ed.x], b = node_dom[ed.y];
    Lm[(size_t)a * Dn + a] += 1;
    Lm[(size_t)b * Dn + b] += 1;
    Lm[(size_t)a * Dn + b] -= 1;
    Lm[(size_t)b * Dn + a] -= 1;
  }
  std::vector<int> comp(Dn, -1);
  int ncomp = 0;
  for (int s = 0; s < Dn; ++s) {
    if (comp[s] >= 0) continue;
    std::vector<int> stack{s};
    comp[s] = ncomp;
    while (!stack.empty()) {
      const int u = stack.back();
      stack.pop_back();
      for (int v = 0; v < Dn; ++v)
        if (comp[v] < 0 && Lm[(size_t)u * Dn + v] != 0.0) {
          comp[v] = ncomp;
          stack.push_back(v);
        }
    }
    ++ncomp;
  }
  std::vector<double> csize(ncomp, 0.0), cnodes(ncomp, 0.0);
  for (int d = 0; d < Dn; ++d) {
    csize[comp[d]] += 1;
    cnodes[comp[d]] += node_off[d + 1] - node_off[d];
  }
  std::vector<double> M = Lm;
  for (int a = 0; a < Dn; ++a)
    for (int b = 0; b < Dn; ++b)
      if (comp[a] == comp[b]) M[(size_t)a * Dn + b] += 1.0 / csize[comp[a]];
  std::vector<double> Lp((size_t)Dn * Dn, 0.0);
  for (int d = 0; d < Dn; ++d) Lp[(size_t)d * Dn + d] = 1.0;
  if (!chol_solve(M, Dn, Lp, Dn)) {
    err = "piston system is not positive definite";
    return LETKF_ERR_ARG;
  }
  for (int a = 0; a < Dn; ++a)
    for (int b = 0; b < Dn; ++b)
      if (comp[a] == comp[b]) Lp[(size_t)a * Dn + b] -= 1.0 / csize[comp[a]];
  // weighted centring per group: K = Lp - 1_c (w_c^T Lp)
  std::vector<double> wrow((size_t)ncomp * Dn, 0.0);
  for (int d = 0; d < Dn; ++d) {
    const double wd = (node_off[d + 1] - node_off[d]) / cnodes[comp[d]];
    for (int b = 0; b < Dn; ++b) wrow[(size_t)comp[d] * Dn + b] += wd * Lp[(size_t)d * Dn + b];
  }
  std::vector<float> K((size_t)Dn * Dn);
  for (int a = 0; a < Dn; ++a)
    for (int b = 0; b < Dn; ++b)
      K[(size_t)a * Dn + b] = (float)(Lp[(size_t)a * Dn + b] - wrow[(size_t)comp[a] * Dn + b]);
  std::vector<float> wv(D->tau.size());
  for (size_t q = 0; q < wv.size(); ++q) wv[q] = (float)(D->tau[q] / c.sigma2);
  cudaError_t e = dup(&D->node_off, node_off);
  if (e == cudaSuccess) e = dup(&D->node_ids, node_ids);
  if (e == cudaSuccess) e = dup(&D->obs_off, obs_off);
  if (e == cudaSuccess) e = dup(&D->obs_slot, obs_slot);
  if (e == cudaSuccess) e = dup(&D->obs_w, wv);
  if (e == cudaSuccess) e = dup(&D->node_dom, node_dom);
  if (e == cudaSuccess && !edges.empty()) e = dup(&D->edges, edges);
  if (e == cudaSuccess) e = dup(&D->dedge_off, dedge_off);
  if (e == cudaSuccess && !dedge.empty()) e = dup(&D->dedge, dedge);
  if (e == cudaSuccess) e = dup(&D->K, K);
  if (e == cudaSuccess) e = cudaMalloc((void **)&D->delta, pts.size() * 2 * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc((void **)&D->bsum, (size_t)Dn * 2 * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc((void **)&D->sweep, (size_t)Dn * sizeof(int));
  if (e == cudaSuccess && D->global) {
    const int mpt = D->rpl ? gl_mpt(mpd) : mpd;
    D->mpt = mpt;
    // parts of the slopes: about four CTAs per SM over the tiles, at least two chunks each
    const int tiles = (mpt / GL_TILE) * (mpt / GL_TILE + 1) / 2;
    D->kchunks = std::max(1, std::min((D->max_obs + 2 * GL_KC - 1) / (2 * GL_KC), (4 * sms + tiles - 1) / tiles));
    D->sms = sms;
    e = cudaMalloc((void **)&D->gpart, (size_t)D->kchunks * mpt * mpt * sizeof(double));
    if (e == cudaSuccess) e = cudaMemset(D->gpart, 0, (size_t)D->kchunks * mpt * mpt * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void **)&D->cpart, (size_t)D->kchunks * mpt * sizeof(double));
    if (e == cudaSuccess) e = cudaMemset(D->cpart, 0, (size_t)D->kchunks * mpt * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void **)&D->T, (size_t)c.m * c.m * sizeof(float));
    if (e == cudaSuccess && D->rpl == 0) {
      const long long n_pad = ((2LL * (long long)pts.size() + lk_ns_tile() - 1) / lk_ns_tile()) *
                              lk_ns_tile();
      e = cudaMalloc(&D->ns_ws, lk_ns_workspace_bytes(mpt, n_pad));
      if (e == cudaSuccess) e = cudaMemset(D->ns_ws, 0, lk_ns_workspace_bytes(mpt, n_pad));
      if (e == cudaSuccess) e = lk_ns_setup();
    } else if (e == cudaSuccess) {
      switch (D->rpl) {
        case 2: e = setup_global_rpl<2>(*D, c.m); break;
        case 4: e = setup_global_rpl<4>(*D, c.m); break;
        case 8: e = setup_global_rpl<8>(*D, c.m); break;
        case 13: e = setup_global_rpl<13>(*D, c.m); break;
        default: e = setup_global_rpl<16>(*D, c.m); break;
      }
    }
  } else if (e == cudaSuccess) {
    switch (D->rpl) {
      case 2: e = setup_rpl<2>(*D); break;
      case 4: e = setup_rpl<4>(*D); break;
      case 8: e = setup_rpl<8>(*D); break;
      case 13: e = setup_rpl<13>(*D); break;
      default: e = setup_rpl<16>(*D); break;
    }
  }
  if (e != cudaSuccess) {
    err = cudaGetErrorString(e);
    return LETKF_ERR_CUDA;
  }
  return LETKF_OK;
}

// New sigma2 / taper half-support: the domain weights tau / sigma2 again.
letkf_status lk_domains_set_params(letkf_ctx *h, const letkf_config &c, const std::vector<int> &pid,
                                   const std::vector<int2> &pts, const std::vector<int2> &saps,
                                   std::string &err) {
  lk_domains_release(h);
  return lk_domains_build(h, c, pid, pts, saps, err);
}

void lk_domains_release(letkf_ctx *h) {
  LkDom *D = h->dom;
  if (!D) return;
  void *bufs[] = {D->node_off, D->node_ids, D->obs_off, D->obs_slot, D->obs_w, D->node_dom,
                  D->edges,    D->dedge_off, D->dedge,   D->K,        D->delta, D->bsum, D->sweep,
                  D->gpart,    D->cpart,     D->T,       D->ns_ws};
  for (void *p : bufs)
    if (p) cudaFree(p);
  delete D;
  h->dom = nullptr;
}

int lk_domain_count(const letkf_ctx *h) { return h->dom ? h->dom->n_dom : 0; }

int lk_domain_of_nodes(const letkf_ctx *h, int *node_dom_host) {
  if (!h->dom) return 0;
  return cudaMemcpy(node_dom_host, h->dom->node_dom, h->inst[0].n_pts * sizeof(int),
                    cudaMemcpyDeviceToHost) == cudaSuccess;
}

int lk_domain_obs_counts(const letkf_ctx *h, int *obs_host) {
  if (!h->dom) return 0;
  std::vector<int> off(h->dom->n_dom + 1);
  if (cudaMemcpy(off.data(), h->dom->obs_off, off.size() * sizeof(int), cudaMemcpyDeviceToHost) !=
      cudaSuccess)
    return 0;
  for (int d = 0; d < h->dom->n_dom; ++d) obs_host[d] = off[d + 1] - off[d];
  return 1;
}

// Analysis of every domain, then (with the piston correction) the piston
// constants and their application.
cudaError_t lk_launch_domains(letkf_ctx *h, void *mean, void *spread) {
  const LkDom &D = *h->dom;
  if (D.global && D.rpl == 0) {
    const int nt = D.mpt / GL_TILE;
    cudaError_t e = lk_launch_pdl(global_gram_kernel, dim3(nt * (nt + 1) / 2, D.kchunks), 256, 0,
                                  h->stream, h->d_inst, (const int *)D.obs_slot,
                                  (const float *)D.obs_w, D.max_obs, D.mpt, D.gpart, D.cpart);
    if (e != cudaSuccess) return e;
    return lk_launch_ns_global(h, D.gpart, D.cpart, D.kchunks, D.mpt, D.sms, D.ns_ws, mean,
                               spread);
  }
  if (D.global) {
    switch (D.rpl) {
      case 2: return launch_global_rpl<2>(h, mean, spread);
      case 4: return launch_global_rpl<4>(h, mean, spread);
      case 8: return launch_global_rpl<8>(h, mean, spread);
      case 13: return launch_global_rpl<13>(h, mean, spread);
      default: return launch_global_rpl<16>(h, mean, spread);
    }
  }
  DomArgs a;
  a.node_off = D.node_off;
  a.node_ids = D.node_ids;
  a.obs_off = D.obs_off;
  a.obs_slot = D.obs_slot;
  a.obs_w = D.obs_w;
  a.mean = static_cast<float *>(mean);
  a.spread = static_cast<float *>(spread);
  a.delta = D.delta;
  a.counters = h->counters;
  a.sweep = nullptr;
  a.tol = (float)h->tol32;
  a.stop = (float)(h->stop32 > h->tol32 ? h->stop32 : h->tol32);
  a.kappa_thr = h->fp64_kappa > 0 ? (float)h->fp64_kappa : 0.f;
  a.max_sweeps = h->max_sweeps;
  a.max_obs = D.max_obs;
  a.max_rows = 2 * D.max_nodes;
  cudaError_t e;
  switch (D.rpl) {
    case 2: e = launch_rpl<2>(h, a); break;
    case 4: e = launch_rpl<4>(h, a); break;
    case 8: e = launch_rpl<8>(h, a); break;
    case 13: e = launch_rpl<13>(h, a); break;
    default: e = launch_rpl<16>(h, a); break;
  }
  if (e != cudaSuccess || !D.piston || D.n_dom < 2) return e;
  e = lk_launch_pdl(piston_sum_kernel, (unsigned)((D.n_dom * 32 + LK_WARP_CTA - 1) / LK_WARP_CTA),
                    LK_WARP_CTA, 0, h->stream, D.n_dom, (const int2 *)D.edges,
                    (const int *)D.dedge_off, (const int *)D.dedge, (const float *)D.delta, D.bsum);
  if (e != cudaSuccess) return e;
  return lk_launch_pdl(piston_apply_kernel, (unsigned)D.n_dom, PA_WARPS * 32, 0, h->stream,
                       h->d_inst, D.n_dom, (const int *)D.node_off, (const int *)D.node_ids,
                       (const float *)D.K, (const float *)D.bsum, static_cast<float *>(mean));
}
