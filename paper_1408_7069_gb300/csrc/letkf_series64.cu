// FP64 node problems by Chebyshev series (FP64 handles): the analysis of
// Section 4.2 and its adjoint without an eigensolve.
//
// The analysis applies A^-1/2 and A^-1, A = alpha I + G, to the node's two
// anomaly rows only (see direct_apply in letkf_pair.cu): Chebyshev series in
// X = 2 G / (alpha ratio) - I of a degree that the ratio |G|_F / alpha fixes.
// GB300 issues one warp-wide FP64 instruction per 64 clocks and SM
// sub-partition, so the count of those is what bounds a node: a running loop's
// node (m = 24, ratio about 3) takes 35 products of the two vectors with G,
// 2 m^2 FMAs each, where the eigensolve's Newton-Schulz steps and sweeps took
// about fifteen times as many. Nodes with a ratio above LK_CHEB_MAX64 are
// queued for the eigensolve of letkf_node64.cu.
//
// One CTA per node, MPD = m padded to 8, 16, 24 or 32 columns: thread
// (row, vector, segment) holds a segment of L columns of its row of G in
// registers and multiplies it by that segment of its vector; the KS segments
// of a row are adjacent lanes and add by shuffles. The vectors' next terms go
// through shared memory, double-buffered: one barrier per product. Segment 0
// sums the series of A^-1/2, segment 1 that of A^-1, in one instruction.
// Measured on one GB300, eigensolve -> series: 8 x 8, m = 10, 16 frames 1971 ->
// 557 us; gradient of ten frames at 16 m, m = 24, 32.7 -> 7.2 ms; error against
// FP64 1.2e-12 -> 1.7e-13 in the gradient.
#include <math.h>

#include "letkf_device.cuh"

namespace {

template <int MPD>
struct S64 {
  static constexpr int KS = MPD <= 16 ? 4 : 2;        // segments per row
  static constexpr int L = MPD / KS;                  // columns per segment
  static constexpr int TS = L + 2;                    // stride of a segment of a vector
  static constexpr int NT = MPD * 2 * KS;             // threads: 64, 128, 96, 128
  static constexpr int VEC = 2 * KS * TS;             // doubles of a pair of vectors
  static constexpr int NTL = MPD / 4;                 // 4 x 4 tiles per side of the Gram
  static constexpr int TILES = NTL * (NTL + 1) / 2;   // its lower triangle
  static constexpr int GK = NT / TILES < 8 ? NT / TILES : 8;   // slope groups
  static constexpr int QC = 32;                       // slopes staged at a time
  static constexpr int LDY = MPD + 2;
  static constexpr int LDG = MPD + 1;
  static constexpr int STAGE = QC * LDY > GK * TILES * 16 ? QC * LDY : GK * TILES * 16;
  static constexpr int NW = NT / 32;
};

// Shared memory of one CTA, in doubles: staged slopes (then the Gram's partial
// sums), G, the term buffers, c = C d, the rows, innovations of the staged
// slopes, reduction slots; then the support list (weights, cells).
template <int MPD>
struct Smem64 {
  using C = S64<MPD>;
  double *Ys, *Gs, *tb, *cv, *xs, *ds, *red, *st;
  int *cell;
  static __host__ __device__ constexpr size_t fixed() {
    return (size_t)C::STAGE + MPD * C::LDG + 2 * C::VEC + MPD + 2 * MPD + C::QC + 16;
  }
  static __host__ __device__ size_t doubles(int w) {
    return fixed() + (size_t)w * w + ((size_t)w * w + 2) / 2;
  }
  __device__ Smem64(double *b, int w) {
    Ys = b;
    Gs = Ys + C::STAGE;
    tb = Gs + MPD * C::LDG;
    cv = tb + 2 * C::VEC;
    xs = cv + MPD;
    ds = xs + 2 * MPD;
    red = ds + C::QC;
    st = red + 16;
    cell = reinterpret_cast<int *>(st + w * w);
  }
};

// The cells of the node's window inside the taper's support: offsets ds * w + dt
// and square roots of tau / sigma2 (of 0 where rounding left tau below it at the
// edge of the support). Returns their number; one barrier.
__device__ __forceinline__ int support(const double *__restrict__ taper, int w, int *cell,
                                       double *st, double *red) {
  const int wc = w * w;
  if (threadIdx.x < 32) {
    int n = 0;
    for (int e0 = 0; e0 < wc; e0 += 32) {
      const int e = e0 + threadIdx.x;
      const double t = e < wc ? taper[e] : 0.0;
      const bool in = t != 0.0;
      const unsigned b = __ballot_sync(FULL, in);
      if (in) {
        const int q = n + __popc(b & ((1u << threadIdx.x) - 1u));
        cell[q] = e;
        st[q] = sqrt(fmax(t, 0.0));
      }
      n += __popc(b);
    }
    if (threadIdx.x == 0) reinterpret_cast<int *>(red)[0] = n;
  }
  __syncthreads();
  return reinterpret_cast<int *>(red)[0];
}

// Slopes q0 .. q0 + nq - 1 of the support list into Ys (times sqrt(tau / sigma2)
// with SCALE; zero on the padding) and their innovations into ds. No barrier.
template <int MPD, bool SCALE>
__device__ __forceinline__ void stage_slopes(const LkInst &I, int2 ij, const Smem64<MPD> &sm,
                                             int q0, int nq) {
  using C = S64<MPD>;
  const double *Ybp = static_cast<const double *>(I.Ybp);
  const double *dp = static_cast<const double *>(I.dp);
  const int m = I.m, w = I.w;
  for (int e = threadIdx.x; e < nq * MPD; e += C::NT) {
    const int q = e / MPD, i = e - q * MPD;
    const int k = (q0 + q) >> 1, cc = (q0 + q) & 1;
    const int ce = sm.cell[k], cs = ce / w;
    const size_t src = (size_t)(ij.x + cs) * I.gs_cols + (ij.y + ce - cs * w);
    const double v = i < m ? Ybp[(src * 2 + cc) * m + i] : 0.0;
    sm.Ys[q * C::LDY + i] = SCALE ? sm.st[k] * v : v;
    if (i == 0) sm.ds[q] = (SCALE ? sm.st[k] : 1.0) * dp[src * 2 + cc];
  }
}

// G = sum_j tau_j / sigma2 y_j y_j^T into sm.Gs and c = C d into sm.cv. The
// lower triangle in 4 x 4 tiles, GK groups of slopes in parallel, partial sums
// added in group order. Ends with a barrier.
template <int MPD>
__device__ __forceinline__ void gram64(const LkInst &I, int2 ij, const Smem64<MPD> &sm, int nsl) {
  using C = S64<MPD>;
  const int t = threadIdx.x;
  const int grp = t / C::TILES, tile = t - grp * C::TILES;
  int ti = 0, tj = tile;                             // tile (ti, tj), tj <= ti
  while (tj > ti) {
    ++ti;
    tj -= ti;
  }
  double acc[4][4] = {};
  const int row = t / (2 * C::KS), part = t - row * 2 * C::KS;
  double cs = 0.0;
  for (int q0 = 0; q0 < nsl; q0 += C::QC) {
    const int nq = nsl - q0 < C::QC ? nsl - q0 : C::QC;
    __syncthreads();
    stage_slopes<MPD, true>(I, ij, sm, q0, nq);
    __syncthreads();
    if (grp < C::GK)
      for (int q = grp; q < nq; q += C::GK) {
        const double2 *a2 = reinterpret_cast<const double2 *>(sm.Ys + q * C::LDY + 4 * ti);
        const double2 *b2 = reinterpret_cast<const double2 *>(sm.Ys + q * C::LDY + 4 * tj);
        const double2 a01 = a2[0], a23 = a2[1], b01 = b2[0], b23 = b2[1];
        const double a[4] = {a01.x, a01.y, a23.x, a23.y}, b[4] = {b01.x, b01.y, b23.x, b23.y};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
      }
    for (int q = part; q < nq; q += 2 * C::KS) cs = fma(sm.Ys[q * C::LDY + row], sm.ds[q], cs);
  }
#pragma unroll
  for (int o = C::KS; o > 0; o >>= 1) cs += __shfl_xor_sync(FULL, cs, o);
  __syncthreads();                                   // the staged slopes become partial sums
  if (part == 0) sm.cv[row] = cs;
  if (grp < C::GK) {
    double *p = sm.Ys + (size_t)(grp * C::TILES + tile) * 16;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) p[i * 4 + j] = acc[i][j];
  }
  __syncthreads();
  for (int e = t; e < C::TILES * 16; e += C::NT) {
    double s = 0.0;
#pragma unroll
    for (int g = 0; g < C::GK; ++g) s += sm.Ys[(size_t)g * C::TILES * 16 + e];
    const int tl = e >> 4;
    int a = 0, b = tl;
    while (b > a) {
      ++a;
      b -= a;
    }
    const int i = 4 * a + ((e >> 2) & 3), j = 4 * b + (e & 3);
    if (j <= i) {
      sm.Gs[i * C::LDG + j] = s;
      sm.Gs[j * C::LDG + i] = s;
    }
  }
  __syncthreads();
}

// Sum of v over the CTA, the same in every thread (warp sums added in warp
// order). Two barriers.
template <int NW, typename T>
__device__ __forceinline__ T cta_sum(T v, double *red) {
  T *r = reinterpret_cast<T *>(red);
  v = lk_warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) r[threadIdx.x >> 5] = v;
  __syncthreads();
  T s = r[0];
#pragma unroll
  for (int k = 1; k < NW; ++k) s += r[k];
  return s;
}

// This thread's segment of (G T)_row for its vector, summed over the row's
// segments. b: the term buffer of the current terms.
template <int MPD>
__device__ __forceinline__ double product(const double (&g)[S64<MPD>::L], const double *b, int vec,
                                          int seg) {
  using C = S64<MPD>;
  const double2 *p = reinterpret_cast<const double2 *>(b + (vec * C::KS + seg) * C::TS);
  double s0 = 0.0, s1 = 0.0;
#pragma unroll
  for (int j = 0; j < C::L / 2; ++j) {
    const double2 v = p[j];
    s0 = fma(g[2 * j], v.x, s0);
    s1 = fma(g[2 * j + 1], v.y, s1);
  }
  s0 += s1;
#pragma unroll
  for (int o = 1; o < C::KS; o <<= 1) s0 += __shfl_xor_sync(FULL, s0, o);
  return s0;
}

template <int MPD>
__device__ __forceinline__ int slot64(int vec, int row) {
  using C = S64<MPD>;
  return (vec * C::KS + row / C::L) * C::TS + row % C::L;
}

// The two rows of X at the node, their means, anomalies in the term buffer 0
// and (row, vector) of this thread. Ends with a barrier. xs keeps the anomalies.
template <int MPD>
__device__ __forceinline__ void rows64(const double *__restrict__ xrow, int m,
                                       const Smem64<MPD> &sm) {
  const int lane = threadIdx.x & 31, wv = threadIdx.x >> 5;
  if (wv < 2) {                                      // NT >= 64: two warps at least
    const double x = lane < m ? xrow[(size_t)wv * m + lane] : 0.0;
    const double mu = lk_warp_sum(x) / m;
    if (lane < MPD) {
      const double xa = lane < m ? x - mu : 0.0;
      sm.xs[wv * MPD + lane] = xa;
      sm.tb[slot64<MPD>(wv, lane)] = xa;
    }
    if (lane == 0) sm.red[8 + wv] = mu;
  }
  __syncthreads();
}

template <int MPD>
__global__ void __launch_bounds__(S64<MPD>::NT)
    series64_kernel(const LkInst *__restrict__ insts, const int2 *__restrict__ items,
                    double *__restrict__ mean, double *__restrict__ spread,
                    const double2 *__restrict__ cheb, int *__restrict__ counters,
                    int *__restrict__ queue, int2 *__restrict__ worklist) {
  using C = S64<MPD>;
  extern __shared__ __align__(16) double sm64[];
  lk_pdl_wait();
  const int2 it = items[blockIdx.x];
  const LkInst &I = insts[it.x];
  const int m = I.m, w = I.w;
  if (m > MPD || m <= MPD - 8) return;               // another width's node
  const Smem64<MPD> sm(sm64, w);
  const int pid = it.y;
  const int2 ij = I.pts[pid];
  const int nsl = 2 * support(static_cast<const double *>(I.taper), w, sm.cell, sm.st, sm.red);
  gram64<MPD>(I, ij, sm, nsl);
  const int t = threadIdx.x, seg = t % C::KS, vec = (t / C::KS) & 1, row = t / (2 * C::KS);
  double g[C::L];
  float f2 = 0.f;
#pragma unroll
  for (int j = 0; j < C::L; ++j) {
    g[j] = sm.Gs[row * C::LDG + seg * C::L + j];
    f2 = fmaf((float)g[j], (float)g[j], f2);
  }
  // both vectors' threads hold G: half the sum of squares is |G|_F^2
  const float ratio = sqrtf(0.5f * cta_sum<C::NW, float>(f2, sm.red)) / (float)I.alpha;
  if (!(ratio <= LK_CHEB_MAX64)) {                   // (a NaN too)
    if (t == 0) worklist[atomicAdd(queue, 1)] = make_int2(it.x, pid);
    return;
  }
  double *xrow = static_cast<double *>(I.X) + (size_t)pid * 2 * m;
  rows64<MPD>(xrow, m, sm);
  // ---- the series ----
  const double *co = reinterpret_cast<const double *>(cheb + (size_t)lk_cheb_class(ratio) * LK_CHEB_LD64);
  const double scale = co[0] / I.alpha;
  const int deg = (int)co[1];
  co += 2 + (seg & 1);
  double tp = 0.0, tc = sm.xs[vec * MPD + row];
  double acc = co[0] * tc;
  double f = scale, e = 1.0;
  const int sl = slot64<MPD>(vec, row);
  for (int k = 1; k <= deg; ++k) {
    const double ck = __ldg(co + 2 * k);
    const double gt = product<MPD>(g, sm.tb + ((k - 1) & 1) * C::VEC, vec, seg);
    const double tn = fma(f, gt, fma(-e, tc, -tp));  // T_k = 2 X T_k-1 - T_k-2
    tp = tc;
    tc = tn;
    acc = fma(ck, tc, acc);
    if (k == 1) {
      f = 2.0 * scale;
      e = 2.0;
    }
    if (seg == 0) sm.tb[(k & 1) * C::VEC + sl] = tc;
    __syncthreads();
  }
  // ---- X'_r wbar = (A^-1 x'_r) . C d, X'_r W, and the outputs ----
  const double ia = 1.0 / I.alpha;
  // (the lanes of the two vectors alternate every KS: each sums its own)
  double pr = seg == 1 ? acc * sm.cv[row] : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    if (o != C::KS) pr += __shfl_xor_sync(FULL, pr, o);
  if ((t & 31) == vec * C::KS) sm.red[2 * (t >> 5) + vec] = pr;
  __syncthreads();
  if (seg == 0) {
    double p = sm.red[vec];
#pragma unroll
    for (int k = 1; k < C::NW; ++k) p += sm.red[2 * k + vec];
    const double xa = sm.red[8 + vec] + p * ia + sqrt((m - 1) * ia) * acc;
    if (row < m) xrow[(size_t)vec * m + row] = xa;
    sm.xs[vec * MPD + row] = xa;
  }
  __syncthreads();
  const int lane = t & 31, wv = t >> 5;
  if (wv < 2) {
    const double xa = lane < m ? sm.xs[wv * MPD + lane] : 0.0;
    const double mu = lk_warp_sum(xa) / m;
    const double d = lane < m ? xa - mu : 0.0;
    const double sp = sqrt(lk_warp_sum(d * d) / (m - 1));
    if (lane == 0) {
      const long long r = 2 * (I.node_off + pid) + wv;
      if (mean) mean[r] = mu;
      if (spread) spread[r] = sp;
      if (!isfinite(mu) || !isfinite(sp)) atomicOr(&counters[0], LK_BIT_NONFINITE);
      if (wv == 0) {
        atomicMax(&counters[2], 1);
        atomicAdd(&counters[3], 1);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Adjoint of the node's analysis (reverse mode, Section 4.2 differentiated) by
// the same series. With x'_r the anomaly rows, g_r the adjoints of the analysis
// rows, s_r = g_r . 1:
//   wbar = A^-1 C d, b_bar = A^-1 (s_0 x'_0 + s_1 x'_1)             (series)
//   W g_r                                                            (series)
//   A_bar = -b_bar wbar^T + sqrt(m-1) sum_r D_r, D_r the adjoint of x'_r^T A^-1/2 g_r.
// For f = sum_k a_k T_k(X), the derivative of T_k in direction E is
//   sum_{j<k} (2 - [j = 0]) U_{k-1-j}(X) E T_j(X)
// (U: Chebyshev polynomials of the second kind), so D_r is a sum of outer products
//   D_r = sum_j (2 - [j = 0]) P_j (T_j g_r)^T, P_j = sum_{k>j} a_k U_{k-1-j}(X) x'_r,
// P_j being the vectors of Clenshaw's recurrence P_{j-1} = a_j x'_r + 2 X P_j - P_{j+1}.
// No eigenvalue differences appear, so equal eigenvalues need no care. The
// terms T_j g_r are kept in shared memory up to degree ADJ_KEEP (a running loop's
// 35 among them) and run backwards by their own recurrence beyond it.
// Then A_bar goes to the window's slopes as in adjoint_node_kernel.
// ---------------------------------------------------------------------------
constexpr int ADJ_KEEP = 64;

template <int MPD>
struct AdjSmem64 {
  using C = S64<MPD>;
  // after Smem64: the terms of g (or two buffers of them), later A_bar's symmetric
  // part and A_bar y of the staged slopes; terms of b and wbar_bar [2]; wbar,
  // b_bar; g; per-slope sums
  static constexpr int KEEP = (ADJ_KEEP + 1) * C::VEC;
  static constexpr int LATE = MPD * C::LDG + C::QC * C::LDY;
  static constexpr int TERMS = KEEP > LATE ? KEEP : LATE;
  static __host__ __device__ size_t doubles(int w) {
    return Smem64<MPD>::doubles(w) + 1 + TERMS + 2 * C::VEC + 4 * MPD + 2 * C::QC;
  }
};

template <int MPD>
__global__ void __launch_bounds__(S64<MPD>::NT)
    adjoint_series64_kernel(const LkInst *__restrict__ insts, LkAdjArgs a,
                            const double2 *__restrict__ cheb) {
  using C = S64<MPD>;
  using AS = AdjSmem64<MPD>;
  extern __shared__ __align__(16) double sm64[];
  const LkInst &I = insts[0];
  const int m = I.m, w = I.w, wc = w * w, pid = blockIdx.x;
  const Smem64<MPD> sm(sm64, w);
  double *terms = sm64 + ((Smem64<MPD>::doubles(w) + 1) & ~(size_t)1);
  double *sb = terms + AS::TERMS, *wb = sb + 2 * C::VEC, *gv = wb + 2 * MPD, *qs = gv + 2 * MPD;
  const int2 ij = I.pts[pid];
  const int nsl = 2 * support(static_cast<const double *>(I.taper), w, sm.cell, sm.st, sm.red);
  gram64<MPD>(I, ij, sm, nsl);
  const int t = threadIdx.x, seg = t % C::KS, vec = (t / C::KS) & 1, row = t / (2 * C::KS);
  const int lane = t & 31, wv = t >> 5;
  double g[C::L];
  float f2 = 0.f;
#pragma unroll
  for (int j = 0; j < C::L; ++j) {
    g[j] = sm.Gs[row * C::LDG + seg * C::L + j];
    f2 = fmaf((float)g[j], (float)g[j], f2);
  }
  const float ratio = sqrtf(0.5f * cta_sum<C::NW, float>(f2, sm.red)) / (float)I.alpha;
  if (!(ratio <= LK_CHEB_MAX64)) {
    if (t == 0) a.queue[atomicAdd(a.queue_len, 1)] = make_int2(0, pid);
    return;
  }
  rows64<MPD>(static_cast<const double *>(I.X) + (size_t)pid * 2 * m, m, sm);
  if (wv < 2) {                                      // g_r and s_r = g_r . 1
    const double x = lane < m ? a.lam_a[((size_t)pid * 2 + wv) * m + lane] : 0.0;
    const double s = lk_warp_sum(x);
    if (lane < MPD) {
      gv[wv * MPD + lane] = x;
      terms[slot64<MPD>(wv, lane)] = x;
    }
    if (lane == 0) {
      sm.red[10 + wv] = s;
      a.xbar_bar[(size_t)pid * 2 + wv] = s;
    }
  }
  __syncthreads();
  const double s0 = sm.red[10], s1 = sm.red[11];
  const int sl = slot64<MPD>(vec, row);
  const double x = sm.xs[vec * MPD + row];
  double yc = vec == 0 ? sm.cv[row] : s0 * sm.xs[row] + s1 * sm.xs[MPD + row];
  if (seg == 0) sb[sl] = yc;
  __syncthreads();
  // ---- series of g (A^-1/2) and of C d and wbar_bar (A^-1) ----
  const double *co = reinterpret_cast<const double *>(cheb + (size_t)lk_cheb_class(ratio) * LK_CHEB_LD64);
  const double scale = co[0] / I.alpha;
  const int deg = (int)co[1];
  const bool keep = deg <= ADJ_KEEP;
  co += 2;
  double tc = gv[vec * MPD + row], tp = 0.0, yp = 0.0;
  double ga = co[0] * tc, ya = co[1] * yc;
  double f = scale, e = 1.0;
  for (int k = 1; k <= deg; ++k) {
    const double ak = __ldg(co + 2 * k), bk = __ldg(co + 2 * k + 1);
    const double gt = product<MPD>(g, terms + (keep ? k - 1 : (k - 1) & 1) * C::VEC, vec, seg);
    const double gy = product<MPD>(g, sb + ((k - 1) & 1) * C::VEC, vec, seg);
    const double tn = fma(f, gt, fma(-e, tc, -tp)), yn = fma(f, gy, fma(-e, yc, -yp));
    tp = tc;
    tc = tn;
    yp = yc;
    yc = yn;
    ga = fma(ak, tc, ga);
    ya = fma(bk, yc, ya);
    if (k == 1) {
      f = 2.0 * scale;
      e = 2.0;
    }
    if (seg == 0) {
      terms[(keep ? k : k & 1) * C::VEC + sl] = tc;
      sb[(k & 1) * C::VEC + sl] = yc;
    }
    __syncthreads();
  }
  const double ia = 1.0 / I.alpha, rt = sqrt((m - 1) * ia);
  if (seg == 0) wb[vec * MPD + row] = ya * ia;       // wbar, then b_bar
  // ---- D_0 + D_1: Clenshaw's vectors of x' against the terms of g ----
  double acc[C::L];
#pragma unroll
  for (int j = 0; j < C::L; ++j) acc[j] = 0.0;
  double p = __ldg(co + 2 * deg) * x, pn = 0.0;      // P_{deg-1}, P_deg
  if (seg == 0) sm.tb[((deg - 1) & 1) * C::VEC + sl] = p;
  __syncthreads();
  if (seg == 0 && row < m)
    a.xp_bar[((size_t)pid * 2 + vec) * m + row] = fma(vec ? s1 : s0, wb[row], rt * ga);
  for (int j = deg - 1; j >= 0; --j) {
    // the terms' own recurrence run backwards holds T_{j+1} = tc, T_j = tp
    const double2 *q2 = reinterpret_cast<const double2 *>(
        terms + (keep ? j : j & 1) * C::VEC + (vec * C::KS + seg) * C::TS);
    const double pj = j ? 2.0 * p : p;
#pragma unroll
    for (int c = 0; c < C::L / 2; ++c) {
      const double2 q = q2[c];
      acc[2 * c] = fma(pj, q.x, acc[2 * c]);
      acc[2 * c + 1] = fma(pj, q.y, acc[2 * c + 1]);
    }
    if (j == 0) break;
    const double aj = __ldg(co + 2 * j);
    const double gp = product<MPD>(g, sm.tb + (j & 1) * C::VEC, vec, seg);
    const double pm = fma(2.0 * scale, gp, fma(-2.0, p, fma(aj, x, -pn)));
    pn = p;
    p = pm;
    if (!keep) {
      // T_{j-1} = 2 X T_j - T_{j+1} (T_0 = g needs no halving: j >= 1 here)
      const double gt = product<MPD>(g, terms + (j & 1) * C::VEC, vec, seg);
      const double tm = fma(2.0 * scale, gt, fma(-2.0, tp, -tc));
      tc = tp;
      tp = tm;
      if (seg == 0) terms[((j - 1) & 1) * C::VEC + sl] = tm;
    }
    if (seg == 0) sm.tb[((j - 1) & 1) * C::VEC + sl] = p;
    __syncthreads();
  }
  // ---- A_bar, its trace and its symmetric part ----
  const double cf = rt * scale;
  if (vec == 0) {
#pragma unroll
    for (int j = 0; j < C::L; ++j) sm.Gs[row * C::LDG + seg * C::L + j] = acc[j];
  }
  __syncthreads();
  double dg = 0.0;
  if (vec == 1) {
#pragma unroll
    for (int j = 0; j < C::L; ++j) {
      const int c = seg * C::L + j;
      const double v = fma(cf, sm.Gs[row * C::LDG + c] + acc[j], -wb[MPD + row] * wb[c]);
      sm.Gs[row * C::LDG + c] = v;
      if (c == row) dg = v;
    }
  }
  const double alpha_bar = cta_sum<C::NW, double>(dg, sm.red);
  double *As = terms, *ay = As + MPD * C::LDG;       // the terms are done with
  for (int q = t; q < MPD * MPD; q += C::NT) {
    const int i = q / MPD, c = q - i * MPD;
    As[i * C::LDG + c] = 0.5 * (sm.Gs[i * C::LDG + c] + sm.Gs[c * C::LDG + i]);
  }
  __syncthreads();
  // ---- window slopes: y_bar = 2 c A_bar y + c d b_bar, d_bar = c y . b_bar,
  // c_bar = y^T A_bar y + d y . b_bar. A warp per slope (lane = row) for A_bar y,
  // then a lane per slope for the sums over rows. Cells outside the support
  // keep the zeros the workspace was allocated with. ----
  double as[MPD];
#pragma unroll
  for (int i = 0; i < MPD; ++i) as[i] = lane < MPD ? As[lane * C::LDG + i] : 0.0;
  const double *bb = wb + MPD;
  const double *tap = static_cast<const double *>(I.taper);
  double *yb_out = a.ybw + (size_t)pid * wc * 2 * m;
  double *db_out = a.dbw + (size_t)pid * wc * 2;
  double gs2 = 0.0, gL = 0.0;
  for (int q0 = 0; q0 < nsl; q0 += C::QC) {
    const int nq = nsl - q0 < C::QC ? nsl - q0 : C::QC;
    __syncthreads();
    stage_slopes<MPD, false>(I, ij, sm, q0, nq);
    __syncthreads();
    for (int q = wv; q < nq; q += C::NW) {
      const double2 *y2 = reinterpret_cast<const double2 *>(sm.Ys + q * C::LDY);
      double v0 = 0.0, v1 = 0.0;
#pragma unroll
      for (int i = 0; i < MPD / 2; ++i) {
        const double2 y = y2[i];
        v0 = fma(as[2 * i], y.x, v0);
        v1 = fma(as[2 * i + 1], y.y, v1);
      }
      if (lane < MPD) ay[q * C::LDY + lane] = v0 + v1;
    }
    __syncthreads();
    if (wv < 2 && lane < nq) {
      double v = 0.0;
      if (wv == 0)
        for (int i = 0; i < MPD; ++i) v = fma(sm.Ys[lane * C::LDY + i], bb[i], v);
      else
        for (int i = 0; i < MPD; ++i)
          v = fma(sm.Ys[lane * C::LDY + i], ay[lane * C::LDY + i], v);
      qs[wv * C::QC + lane] = v;
    }
    __syncthreads();
    if (wv == 0 && lane < nq) {
      const int ce = sm.cell[(q0 + lane) >> 1], cc = (q0 + lane) & 1;
      const double cj = tap[ce], yb = qs[lane];
      const double cbar = fma(sm.ds[lane], yb, qs[C::QC + lane]);
      gs2 = fma(cbar, cj, gs2);
      gL = fma(cbar, a.dtap[ce], gL);
      db_out[ce * 2 + cc] = cj * yb;
    }
    for (int q = t; q < nq * MPD; q += C::NT) {
      const int k = q / MPD, i = q - k * MPD;
      if (i >= m) continue;
      const int ce = sm.cell[(q0 + k) >> 1], cc = (q0 + k) & 1;
      const double cj = tap[ce];
      yb_out[((size_t)ce * 2 + cc) * m + i] =
          fma(2.0 * cj, ay[k * C::LDY + i], cj * sm.ds[k] * bb[i]);
    }
  }
  if (wv == 0) {
    gs2 = lk_warp_sum(gs2);
    gL = lk_warp_sum(gL);
    if (lane == 0) {
      a.theta[(size_t)pid * 3 + 0] = alpha_bar * (-(m - 1) / (a.rho * a.rho));
      a.theta[(size_t)pid * 3 + 1] = -gs2 / a.sigma2;
      a.theta[(size_t)pid * 3 + 2] = gL;
    }
  }
}

template <int MPD>
cudaError_t launch_adj64(letkf_ctx *h, const LkAdjArgs &a) {
  const LkInst &I = h->inst[0];
  const size_t smem = AdjSmem64<MPD>::doubles(I.w) * sizeof(double);
  adjoint_series64_kernel<MPD><<<I.n_pts, S64<MPD>::NT, smem, h->stream>>>(
      h->d_inst, a, (const double2 *)h->cheb64);
  return cudaGetLastError();
}

template <int MPD>
cudaError_t launch_series64(letkf_ctx *h, int cls, void *mean, void *spread) {
  size_t need = 0;
  for (const LkInst &I : h->inst)
    if (I.m <= MPD && I.m > MPD - 8) {
      const size_t b = Smem64<MPD>::doubles(I.w) * sizeof(double);
      need = b > need ? b : need;
    }
  if (need == 0) return cudaSuccess;
  return lk_launch_pdl(series64_kernel<MPD>, (unsigned)h->n_pts_total, S64<MPD>::NT, need,
                       h->stream, h->d_inst, h->node_items, (double *)mean, (double *)spread,
                       (const double2 *)h->cheb64, h->counters, h->counters + 4 + cls,
                       h->worklist + (size_t)cls * h->n_pts_total);
}

template <int MPD>
cudaError_t setup_series64(int w) {
  cudaError_t e =
      cudaFuncSetAttribute(series64_kernel<MPD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(Smem64<MPD>::doubles(w) * sizeof(double)));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(adjoint_series64_kernel<MPD>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(AdjSmem64<MPD>::doubles(w) * sizeof(double)));
  return e;
}

}  // namespace

cudaError_t lk_launch_series64(letkf_ctx *h, int cls, void *mean, void *spread) {
  if (cls == 0) {
    cudaError_t e = launch_series64<8>(h, 0, mean, spread);
    return e == cudaSuccess ? launch_series64<16>(h, 0, mean, spread) : e;
  }
  cudaError_t e = launch_series64<24>(h, 1, mean, spread);
  return e == cudaSuccess ? launch_series64<32>(h, 1, mean, spread) : e;
}

cudaError_t lk_launch_adj_series64(letkf_ctx *h, const LkAdjArgs &a) {
  const int m = h->inst[0].m;
  return m <= 8 ? launch_adj64<8>(h, a)
                : m <= 16 ? launch_adj64<16>(h, a)
                          : m <= 24 ? launch_adj64<24>(h, a) : launch_adj64<32>(h, a);
}

cudaError_t lk_setup_series64(letkf_ctx *h) {
  int wmax = 1;
  for (const LkInst &I : h->inst) wmax = I.w > wmax ? I.w : wmax;
  cudaError_t e = setup_series64<8>(wmax);
  if (e == cudaSuccess) e = setup_series64<16>(wmax);
  if (e == cudaSuccess) e = setup_series64<24>(wmax);
  if (e == cudaSuccess) e = setup_series64<32>(wmax);
  return e;
}
