// FP64 node problems by Chebyshev series (FP64 handles): the analysis of
// Section 4.2 and its adjoint without an eigensolve.
//
// The analysis applies A^-1/2 and A^-1, A = alpha (I + G), G = sum_j tau_j / (sigma2
// alpha) y_j y_j^T, to the node's two anomaly rows only (see direct_apply in
// letkf_pair.cu): Chebyshev series in X = 2 G / ratio - I of a degree that the ratio
// |G|_F fixes. A running loop's node (m = 24, ratio about 3) takes 35 products of the
// two vectors with G, where the eigensolve's Newton-Schulz steps and sweeps took about
// fifteen times as many. Nodes with a ratio above LK_CHEB_MAX64 are queued for the
// eigensolve of letkf_node64.cu.
//
// GB300 issues one warp-wide FP64 instruction per 76 clocks and SM sub-partition, so
// everything that counts is done in pairs of floats (letkf_df.cuh), 48 bits, six times as
// fast; the condition of I + G, at most 1 + ratio, is small here. Values enter by their
// bits, scaled by powers of two to about 1: slopes by sqrt(tau / (sigma2 alpha)) and the
// innovations, rows and adjoints by their largest exponent, so the range is FP64's. Means
// and what is added to them stay FP64. About the second half of a series, whose
// coefficients are below 2^-27 (letkf_cheb.cu: last_in_pairs), runs in floats: its
// rounding is then below that of the pairs.
//
// One CTA per node, MPD = m padded to 8, 16, 24 or 32 columns: thread
// (row, vector, segment) holds a segment of L columns of its row of 2 X in
// registers and multiplies it by that segment of its vector; the KS segments
// of a row are adjacent lanes and add by shuffles. The vectors' next terms go
// through shared memory, double-buffered: one barrier per product. Segment 0
// sums the series of A^-1/2, segment 1 that of A^-1, in one instruction.
// Measured on one GB300: 8 x 8, m = 10, 16 frames: eigensolve 1971 us, series in FP64 557,
// in pairs 424, with the second half in floats 400; gradient of ten frames at 16 m,
// m = 24: 32.7, 7.2, 3.1, 2.45 ms (861 nodes: forward 116, 40, 33 us, adjoint 449, 161, 104,
// 45% of the issue slots used: bound by the products' chains at 12 to 15 warps per SM).
// Errors against FP64 of these two cases, eight seeds: the eigensolve's X 1e-15 to 5e-15 and
// gradient 8e-15 to 1.4e-12, now 9e-16 to 1e-14 and 2e-15 to 8e-14; over 16 drawn ones the
// geometric means are X 1.3e-15 and 5e-16, gradients 1.6e-14 and 1.1e-14.
#include <math.h>

#include "letkf_df.cuh"

namespace {

template <int MPD>
struct S64 {
  static constexpr int KS = MPD <= 16 ? 4 : 2;        // segments per row
  static constexpr int L = MPD / KS;                  // columns per segment
  static constexpr int TS = L + 2;                    // stride of a segment of a vector
  static constexpr int NT = MPD * 2 * KS;             // threads: 64, 128, 96, 128
  static constexpr int VEC = 2 * KS * TS;             // floats of one part of a pair of vectors
  static constexpr int NTL = MPD / 4;                 // 4 x 4 tiles per side of the Gram
  static constexpr int TILES = NTL * (NTL + 1) / 2;   // its lower triangle
  static constexpr int GK = NT / TILES < 8 ? NT / TILES : 8;   // slope groups
  static constexpr int QC = 32;                       // slopes staged at a time
  static constexpr int LDY = MPD + 4;
  static constexpr int LDG = MPD + 1;
  static constexpr int STAGE = QC * LDY > GK * TILES * 16 ? QC * LDY : GK * TILES * 16;
  static constexpr int NW = NT / 32;
};

// Shared memory of one CTA, in pairs: staged slopes (then the Gram's partial sums), high
// parts and low parts [STAGE] each; G; the term buffers [2][high, low][VEC]; c = C d / alpha;
// the rows; innovations of the staged slopes; reduction slots; then the support list
// (sqrt(tau / (sigma2 alpha)), cells).
template <int MPD>
struct Smem64 {
  using C = S64<MPD>;
  float *Yh, *Yl, *tb;
  float2 *Gs, *cv, *xs, *ds, *red, *st;
  int *cell;
  static __host__ __device__ constexpr size_t fixed() {
    return (size_t)C::STAGE + MPD * C::LDG + 2 * C::VEC + MPD + 2 * MPD + C::QC + 20;
  }
  static __host__ __device__ size_t doubles(int w) {
    return fixed() + (size_t)w * w + ((size_t)w * w + 2) / 2;
  }
  __device__ Smem64(double *b, int w) {
    Yh = reinterpret_cast<float *>(b);
    Yl = Yh + C::STAGE;
    Gs = reinterpret_cast<float2 *>(Yl + C::STAGE);
    tb = reinterpret_cast<float *>(Gs + MPD * C::LDG);
    cv = reinterpret_cast<float2 *>(tb + 4 * C::VEC);
    xs = cv + MPD;
    ds = xs + 2 * MPD;
    red = ds + C::QC;
    st = red + 20;
    cell = reinterpret_cast<int *>(st + w * w);
  }
  // red: [0, 8) sums, then doubles: [8, 10) the rows' means, [10, 12) sums of g; ints from
  // 12 on: slopes' number and exponent of the innovations, exponents of the rows
  __device__ double *red64() const { return reinterpret_cast<double *>(red); }
  __device__ int *redi() const { return reinterpret_cast<int *>(red + 12); }
};

__device__ __forceinline__ Df ld_df(const float2 &v) { return Df{v.x, v.y}; }
__device__ __forceinline__ float2 st_df(Df v) { return make_float2(v.h, v.l); }
// 2^e of any e (0 below the normal range)
__device__ __forceinline__ float pow2c(int e) { return e < -126 ? 0.f : pow2f(e > 127 ? 127 : e); }

// alpha = f 2^e and sqrt((m - 1) / alpha) = r 2^re
struct Alpha64 {
  Df ia, rt;                                         // 1 / alpha = ia 2^-e
  int e, re;
  __device__ Alpha64(double alpha, int m) {
    e = exponent64(alpha);
    ia = df_rcp(df_split(alpha, -e));
    const bool odd = e & 1;
    Df q = df_mul(ia, df(float(m - 1) * (odd ? 2.f : 1.f)));   // (m - 1) 2^odd / f
    rt = df_sqrt(q);
    re = -((e + (odd ? 1 : 0)) / 2);
  }
};

// The cells of the node's window inside the taper's support, by one warp: row and column (5
// bits each: windows are up to 31 wide) with the exponent of sqrt(tau / (sigma2 alpha)) above
// them, and that root's significand (0 where rounding left tau below it at the edge of the
// support). redi: their number, and the largest exponent of the innovations times the root.
constexpr int CELL_BITS = 10, CELL_EXP = 1 << 14;
__device__ __forceinline__ int cell_row(int c) { return (c >> 5) & 31; }
__device__ __forceinline__ int cell_col(int c) { return c & 31; }
constexpr int NO_EXP = -4000;                        // the exponent of nothing but zeros
template <int MPD>
__device__ __forceinline__ void support(const LkInst &I, int2 ij, const Smem64<MPD> &sm) {
  const double *__restrict__ taper = static_cast<const double *>(I.taper);
  const double2 *__restrict__ dp = static_cast<const double2 *>(I.dp);
  const int w = I.w, wc = w * w;
  const int ea = exponent64(I.alpha), lane = threadIdx.x & 31;
  const Df ia = df_rcp(df_split(I.alpha, -ea));
  int n = 0, ed = NO_EXP;
  constexpr int U = 3;                               // loads in flight
  for (int e0 = 0; e0 < wc; e0 += 32 * U) {
    double t[U];
    double2 d[U];
    int c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + 32 * u + lane, cs = e / w, ct = e - cs * w;
      c[u] = cs << 5 | ct;
      t[u] = e < wc ? taper[e] : 0.0;
      d[u] = e < wc ? dp[(size_t)(ij.x + cs) * I.gs_cols + ij.y + ct] : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool in = t[u] != 0.0;
      const unsigned b = __ballot_sync(FULL, in);
      if (in) {
        const int q = n + __popc(b & ((1u << lane) - 1u));
        const int et = exponent64(t[u]), x = et - ea, odd = x & 1;
        Df s = df(0.f);
        if (t[u] > 0.0) s = df_sqrt(df_mul(df_split(t[u], odd - et), ia));
        const int es = (x - odd) / 2;
        sm.cell[q] = (es + CELL_EXP) << CELL_BITS | c[u];
        sm.st[q] = st_df(s);
        const int em = max(exponent64(d[u].x), exponent64(d[u].y));
        if (em > -1022) ed = max(ed, em + es);
      }
      n += __popc(b);
    }
  }
  ed = __reduce_max_sync(FULL, ed);
  if (lane == 0) {
    sm.redi()[0] = n;
    sm.redi()[1] = ed;
  }
}

// Slopes q0 .. q0 + nq - 1 of the support list into Yh, Yl (zero on the padding): SCALE:
// times sqrt(tau / (sigma2 alpha)), and their innovations likewise, times 2^-ed, into ds;
// else times 2^ey, without the innovations. No barrier.
template <int MPD, bool SCALE>
__device__ __forceinline__ void stage_slopes(const LkInst &I, int2 ij, const Smem64<MPD> &sm,
                                             int q0, int nq, int ey) {
  using C = S64<MPD>;
  const double *__restrict__ Ybp = static_cast<const double *>(I.Ybp);
  const double *__restrict__ dp = static_cast<const double *>(I.dp);
  const int m = I.m;
#pragma unroll 4
  for (int e = threadIdx.x; e < nq * MPD; e += C::NT) {
    const int q = e / MPD, i = e - q * MPD;
    const int k = (q0 + q) >> 1, cc = (q0 + q) & 1;
    const int ce = sm.cell[k], es = (ce >> CELL_BITS) - CELL_EXP;
    const size_t src = (size_t)(ij.x + cell_row(ce)) * I.gs_cols + (ij.y + cell_col(ce));
    const double v = i < m ? Ybp[(src * 2 + cc) * m + i] : 0.0;
    Df z = df_split(v, SCALE ? es : ey);
    if (SCALE) z = df_mul(z, ld_df(sm.st[k]));
    sm.Yh[q * C::LDY + i] = z.h;
    sm.Yl[q * C::LDY + i] = z.l;
    if (SCALE && i == 0)
      sm.ds[q] = st_df(df_mul(df_split(dp[src * 2 + cc], es - ey), ld_df(sm.st[k])));
  }
}

// G into sm.Gs and c = C d / alpha, times 2^-ed, into sm.cv. The lower triangle in 4 x 4
// tiles, GK groups of slopes in parallel, partial sums added in group order. Ends with
// a barrier.
template <int MPD>
__device__ __forceinline__ void gram64(const LkInst &I, int2 ij, const Smem64<MPD> &sm, int nsl,
                                       int ed) {
  using C = S64<MPD>;
  const int t = threadIdx.x;
  const int grp = t / C::TILES, tile = t - grp * C::TILES;
  int ti = 0, tj = tile;                             // tile (ti, tj), tj <= ti
  while (tj > ti) {
    ++ti;
    tj -= ti;
  }
  float2 S[4][2], F[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) S[i][j] = F[i][j] = make_float2(0.f, 0.f);
  const int row = t / (2 * C::KS), part = t - row * 2 * C::KS;
  Df cs = df(0.f);
  for (int q0 = 0; q0 < nsl; q0 += C::QC) {
    const int nq = nsl - q0 < C::QC ? nsl - q0 : C::QC;
    __syncthreads();
    stage_slopes<MPD, true>(I, ij, sm, q0, nq, ed);
    __syncthreads();
    if (grp < C::GK)
      for (int q = grp; q < nq; q += C::GK) {
        const float4 ah = *reinterpret_cast<const float4 *>(sm.Yh + q * C::LDY + 4 * ti);
        const float4 al = *reinterpret_cast<const float4 *>(sm.Yl + q * C::LDY + 4 * ti);
        const float4 bh = *reinterpret_cast<const float4 *>(sm.Yh + q * C::LDY + 4 * tj);
        const float4 bl = *reinterpret_cast<const float4 *>(sm.Yl + q * C::LDY + 4 * tj);
        const float a[4] = {ah.x, ah.y, ah.z, ah.w}, e[4] = {al.x, al.y, al.z, al.w};
        const float2 b[2] = {make_float2(bh.x, bh.y), make_float2(bh.z, bh.w)};
        const float2 f[2] = {make_float2(bl.x, bl.y), make_float2(bl.z, bl.w)};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j)
            df_fma2(S[i][j], F[i][j], dup2(a[i]), dup2(-a[i]), dup2(e[i]), b[j], f[j]);
      }
    for (int q = part; q < nq; q += 2 * C::KS)
      cs = df_add(cs, df_mul(Df{sm.Yh[q * C::LDY + row], sm.Yl[q * C::LDY + row]}, ld_df(sm.ds[q])));
  }
#pragma unroll
  for (int o = C::KS; o > 0; o >>= 1) cs = df_add(cs, df_shfl_xor(cs, o));
  __syncthreads();                                   // the staged slopes become partial sums
  if (part == 0) sm.cv[row] = st_df(cs);
  if (grp < C::GK) {
    float4 *ph = reinterpret_cast<float4 *>(sm.Yh + (size_t)(grp * C::TILES + tile) * 16);
    float4 *pl = reinterpret_cast<float4 *>(sm.Yl + (size_t)(grp * C::TILES + tile) * 16);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const Df v0 = df_quick(S[i][0].x, F[i][0].x), v1 = df_quick(S[i][0].y, F[i][0].y);
      const Df v2 = df_quick(S[i][1].x, F[i][1].x), v3 = df_quick(S[i][1].y, F[i][1].y);
      ph[i] = make_float4(v0.h, v1.h, v2.h, v3.h);
      pl[i] = make_float4(v0.l, v1.l, v2.l, v3.l);
    }
  }
  __syncthreads();
  for (int e = t; e < C::TILES * 16; e += C::NT) {
    Df s = Df{sm.Yh[e], sm.Yl[e]};
#pragma unroll
    for (int g = 1; g < C::GK; ++g)
      s = df_add(s, Df{sm.Yh[g * C::TILES * 16 + e], sm.Yl[g * C::TILES * 16 + e]});
    const int tl = e >> 4;
    int a = 0, b = tl;
    while (b > a) {
      ++a;
      b -= a;
    }
    const int i = 4 * a + ((e >> 2) & 3), j = 4 * b + (e & 3);
    if (j <= i) {
      sm.Gs[i * C::LDG + j] = st_df(s);
      sm.Gs[j * C::LDG + i] = st_df(s);
    }
  }
  __syncthreads();
}

// Sum of v over the CTA, the same in every thread (warp sums added in warp
// order). Two barriers.
template <int NW>
__device__ __forceinline__ float cta_sum(float v, float2 *red) {
  float *r = reinterpret_cast<float *>(red);
  v = lk_warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) r[threadIdx.x >> 5] = v;
  __syncthreads();
  float s = r[0];
#pragma unroll
  for (int k = 1; k < NW; ++k) s += r[k];
  return s;
}

// This thread's segment of its row of 2 X (high and low parts).
template <int MPD>
struct Seg64 {
  float2 h[S64<MPD>::L / 2], l[S64<MPD>::L / 2];
};
template <int MPD>
__device__ __forceinline__ float seg_load(Seg64<MPD> &g, const Smem64<MPD> &sm, int row, int seg) {
  using C = S64<MPD>;
  float f2 = 0.f;
#pragma unroll
  for (int j = 0; j < C::L / 2; ++j) {
    const float2 a = sm.Gs[row * C::LDG + seg * C::L + 2 * j];
    const float2 b = sm.Gs[row * C::LDG + seg * C::L + 2 * j + 1];
    g.h[j] = make_float2(a.x, b.x);
    g.l[j] = make_float2(a.y, b.y);
    f2 = fmaf(a.x, a.x, fmaf(b.x, b.x, f2));
  }
  return f2;
}
// G to 2 (scale G - I)
template <int MPD>
__device__ __forceinline__ void seg_scale(Seg64<MPD> &g, Df scale, int row, int seg) {
  using C = S64<MPD>;
  const Df s = Df{2.f * scale.h, 2.f * scale.l};
#pragma unroll
  for (int j = 0; j < C::L / 2; ++j) {
    Df a = df_mul(s, Df{g.h[j].x, g.l[j].x}), b = df_mul(s, Df{g.h[j].y, g.l[j].y});
    if (seg * C::L + 2 * j == row) a = df_add(a, df(-2.f));
    if (seg * C::L + 2 * j + 1 == row) b = df_add(b, df(-2.f));
    g.h[j] = make_float2(a.h, b.h);
    g.l[j] = make_float2(a.l, b.l);
  }
}

// This thread's segment of (2 X T)_row for its vector, summed over the row's
// segments. b: the term buffer of the current terms.
template <int MPD>
__device__ __forceinline__ Df product(const Seg64<MPD> &g, const float *b, int vec, int seg) {
  using C = S64<MPD>;
  const float2 *ph = reinterpret_cast<const float2 *>(b + (vec * C::KS + seg) * C::TS);
  const float2 *pl = ph + C::VEC / 2;
  float2 S, F;
  {
    const float2 vh = ph[0], vl = pl[0];
    S = prod2(g.h[0], vh);
    F = __ffma2_rn(neg2(g.h[0]), vh, S);
    F = sub2(__ffma2_rn(g.h[0], vl, prod2(g.l[0], vh)), F);
  }
#pragma unroll
  for (int j = 1; j < C::L / 2; ++j) {
    const float2 vh = ph[j], vl = pl[j];
    df_fma2(S, F, vh, neg2(vh), vl, g.h[j], g.l[j]);
  }
  Df s = df_add(df_quick(S.x, F.x), df_quick(S.y, F.y));
#pragma unroll
  for (int o = 1; o < C::KS; o <<= 1) s = df_add(s, df_shfl_xor(s, o));
  return s;
}

// The same of the high parts alone.
template <int MPD>
__device__ __forceinline__ float product32(const Seg64<MPD> &g, const float *b, int vec, int seg) {
  using C = S64<MPD>;
  const float2 *ph = reinterpret_cast<const float2 *>(b + (vec * C::KS + seg) * C::TS);
  float2 S = make_float2(0.f, 0.f);
#pragma unroll
  for (int j = 0; j < C::L / 2; ++j) S = __ffma2_rn(g.h[j], ph[j], S);
  float s = S.x + S.y;
#pragma unroll
  for (int o = 1; o < C::KS; o <<= 1) s += __shfl_xor_sync(FULL, s, o);
  return s;
}

template <int MPD>
__device__ __forceinline__ int slot64(int vec, int row) {
  using C = S64<MPD>;
  return (vec * C::KS + row / C::L) * C::TS + row % C::L;
}
template <int MPD>
__device__ __forceinline__ void put64(float *buf, int slot, Df v) {
  buf[slot] = v.h;
  buf[S64<MPD>::VEC + slot] = v.l;
}

// Row r of X at the node, by one warp: its mean (red64[8 + r]), exponent (redi[2 + r]) and
// anomalies times 2^-exponent (xs and the term buffer 0).
template <int MPD>
__device__ __forceinline__ void row64(const double *__restrict__ xrow, int m, int r,
                                      const Smem64<MPD> &sm) {
  const int lane = threadIdx.x & 31;
  const double x = lane < m ? xrow[(size_t)r * m + lane] : 0.0;
  const double mu = lk_warp_sum(x) / m;
  const double xa = lane < m ? x - mu : 0.0;
  const int ex = __reduce_max_sync(FULL, exponent64(xa));
  const int sh = ex == -1022 ? NO_EXP : ex;
  if (lane < MPD) {
    const Df v = df_split(xa, -sh);
    sm.xs[r * MPD + lane] = st_df(v);
    put64<MPD>(sm.tb, slot64<MPD>(r, lane), v);
  }
  if (lane == 0) {
    sm.red64()[8 + r] = mu;
    sm.redi()[2 + r] = sh;
  }
}
// The warp that looks after row r while warp 0 lists the support (two warps at least).
template <int MPD>
__device__ __forceinline__ bool row_warp(int wv, int r) {
  return wv == (S64<MPD>::NW >= 3 ? 1 + r : 1);
}

template <int MPD>
// (24 warps per SM at 80 registers: m = 24, 861 nodes 33.8 us against 39.6 at the 124 that the
// compiler takes unbounded; 16 warps at 128 for 32 columns)
__global__ void __launch_bounds__(S64<MPD>::NT, (MPD <= 24 ? 768 : 512) / S64<MPD>::NT)
    series64_kernel(const LkInst *__restrict__ insts, const int2 *__restrict__ items,
                    double *__restrict__ mean, double *__restrict__ spread,
                    const float4 *__restrict__ cheb, int *__restrict__ counters,
                    int *__restrict__ queue, int2 *__restrict__ worklist,
                    const double *__restrict__ noise, unsigned char *__restrict__ left) {
  using C = S64<MPD>;
  extern __shared__ __align__(16) double sm64[];
  lk_pdl_wait();
  lk_pdl_trigger();
  const int2 it = items[blockIdx.x];
  const LkInst &I = insts[it.x];
  const int m = I.m, w = I.w;
  if (m > MPD || m <= MPD - 8) return;               // another width's node
  const Smem64<MPD> sm(sm64, w);
  const int pid = it.y;
  const int2 ij = I.pts[pid];
  const int t = threadIdx.x, seg = t % C::KS, vec = (t / C::KS) & 1, row = t / (2 * C::KS);
  const int lane = t & 31, wv = t >> 5;
  double *xrow = static_cast<double *>(I.X) + (size_t)pid * 2 * m;
  if (wv == 0) support<MPD>(I, ij, sm);
#pragma unroll
  for (int r = 0; r < 2; ++r)
    if (row_warp<MPD>(wv, r)) row64<MPD>(xrow, m, r, sm);
  __syncthreads();
  const int nsl = 2 * sm.redi()[0], ed = sm.redi()[1];
  gram64<MPD>(I, ij, sm, nsl, ed);
  Seg64<MPD> g;
  const float f2 = seg_load<MPD>(g, sm, row, seg);
  // both vectors' threads hold G: half the sum of squares is |G|_F^2
  const float ratio = sqrtf(0.5f * cta_sum<C::NW>(f2, sm.red));
  const bool ill = !(ratio <= LK_CHEB_MAX64);        // (a NaN too)
  if (left && t == 0) left[pid] = ill;               // (letkf_grad: one instance)
  if (ill) {
    if (t == 0) worklist[atomicAdd(queue, 1)] = make_int2(it.x, pid);
    return;
  }
  // ---- the series: terms up to `low` in pairs, then in floats ----
  const float4 *co = cheb + (size_t)lk_cheb_class(ratio) * LK_CHEB_LD64;
  const float4 c0 = co[0];
  const int deg = (int)c0.z, low = (int)c0.w;
  seg_scale<MPD>(g, Df{c0.x, c0.y}, row, seg);
  const float2 *ck = reinterpret_cast<const float2 *>(co + 1) + (seg & 1);
  Df tp = df(0.f), tc = ld_df(sm.xs[vec * MPD + row]);
  Df acc = df_mul(ld_df(__ldg(ck)), tc);
  const int sl = slot64<MPD>(vec, row);
  for (int k = 1; k <= low; ++k) {
    const Df c = ld_df(__ldg(ck + 2 * k));
    const Df gt = product<MPD>(g, sm.tb + ((k - 1) & 1) * 2 * C::VEC, vec, seg);
    // T_k = 2 X T_k-1 - T_k-2, T_1 = X T_0
    const Df tn = k == 1 ? Df{0.5f * gt.h, 0.5f * gt.l} : df_add(gt, df_neg(tp));
    if (seg == 0) put64<MPD>(sm.tb + (k & 1) * 2 * C::VEC, sl, tn);
    tp = tc;
    tc = tn;
    __syncthreads();
    acc = df_add(acc, df_mul(c, tc));
  }
  {
    float ah = 0.f, pf = tp.h, cf = tc.h;
    for (int k = low + 1; k <= deg; ++k) {
      const float c = __ldg(ck + 2 * k).x;
      const float tn = product32<MPD>(g, sm.tb + ((k - 1) & 1) * 2 * C::VEC, vec, seg) - pf;
      if (seg == 0) sm.tb[(k & 1) * 2 * C::VEC + sl] = tn;
      pf = cf;
      cf = tn;
      __syncthreads();
      ah = fmaf(c, tn, ah);
    }
    acc = df_add(acc, df(ah));
  }
  // ---- X'_r wbar = (A^-1 x'_r) . C d, X'_r W, and the outputs ----
  // (the lanes of the two vectors alternate every KS: each sums its own)
  Df pr = seg == 1 ? df_mul(acc, ld_df(sm.cv[row])) : df(0.f);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    if (o != C::KS) pr = df_add(pr, df_shfl_xor(pr, o));
  if ((t & 31) == vec * C::KS) sm.red[2 * (t >> 5) + vec] = st_df(pr);
  if (seg == 0) sm.xs[vec * MPD + row] = st_df(acc);
  __syncthreads();
  if (wv < 2) {                                      // a warp per row of X
    const Alpha64 al(I.alpha, m);
    Df p = ld_df(sm.red[wv]);
#pragma unroll
    for (int k = 1; k < C::NW; ++k) p = df_add(p, ld_df(sm.red[2 * k + wv]));
    const int ex = sm.redi()[2 + wv];
    const Df a = lane < m ? ld_df(sm.xs[wv * MPD + lane]) : df(0.f);
    const double y = sm.red64()[8 + wv] + df_to_double(p, ex + ed);
    double fc = 0.0;
    if (lane < m) {                                  // with noise, the forecast instead
      const double xa = y + df_to_double(df_mul(al.rt, a), ex + al.re);
      if (!noise) xrow[(size_t)wv * m + lane] = xa;
      if (noise && wv == 0) {
        xrow[m + lane] = xa;
        fc = lk_ar1<double>(I, noise, pid, lane, xa);
        xrow[lane] = fc;
      }
    }
    if (noise && wv == 0 && I.dm) {
      fc = lk_warp_sum(fc);
      if (lane == 0) static_cast<double *>(I.pmean)[pid] = fc / m;
    }
    // their mean and spread (|a| < 8: at most that of the anomalies, below 1 each)
    const Df rm = df_rcp(df((float)m));
    const Df am = df_mul(df_redux(a, 3), rm);
    const Df d = lane < m ? df_add(a, df_neg(am)) : df(0.f);
    const Df s2 = df_redux(df_mul(d, d), 6);
    Df s = df_mul(s2, df_rcp(df((float)(m - 1))));
    if (s.h > 0.f) s = df_sqrt(s);
    if (lane == 0) {
      const double mu = y + df_to_double(df_mul(al.rt, am), ex + al.re);
      double sp = df_to_double(df_mul(al.rt, s), ex + al.re);
      if (!isfinite(mu)) sp = mu - mu;               // (the integer sums have dropped a NaN)
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
  // after Smem64 (in pairs): the terms of g (or two buffers of them), later A_bar's
  // symmetric part and A_bar y of the staged slopes (high and low parts); terms of b and
  // wbar_bar [2]; wbar, b_bar; g; per-slope sums; per-slope factors
  static constexpr int KEEP = (ADJ_KEEP + 1) * C::VEC;
  static constexpr int LATE = MPD * C::LDG + C::QC * C::LDY;
  static constexpr int TERMS = ((KEEP > LATE ? KEEP : LATE) + 1) & ~1;
  static __host__ __device__ size_t doubles(int w) {
    return Smem64<MPD>::doubles(w) + 1 + TERMS + 2 * C::VEC + 4 * MPD + 2 * C::QC + 4 * C::QC;
  }
};

template <int MPD>
__global__ void __launch_bounds__(S64<MPD>::NT)
    adjoint_series64_kernel(const LkInst *__restrict__ insts, LkAdjArgs a,
                            const float4 *__restrict__ cheb) {
  using C = S64<MPD>;
  using AS = AdjSmem64<MPD>;
  extern __shared__ __align__(16) double sm64[];
  const LkInst &I = insts[0];
  const int m = I.m, w = I.w, wc = w * w, pid = blockIdx.x;
  const Smem64<MPD> sm(sm64, w);
  float *terms = reinterpret_cast<float *>(sm64 + ((Smem64<MPD>::doubles(w) + 1) & ~(size_t)1));
  float *sb = terms + 2 * AS::TERMS;
  float2 *wb = reinterpret_cast<float2 *>(sb + 4 * C::VEC), *gv = wb + 2 * MPD;
  float2 *qs = gv + 2 * MPD, *qc = qs + 2 * C::QC, *qd = qc + C::QC, *qf = qd + C::QC;
  int *qe = reinterpret_cast<int *>(qf + C::QC);
  const int2 ij = I.pts[pid];
  const int t = threadIdx.x, seg = t % C::KS, vec = (t / C::KS) & 1, row = t / (2 * C::KS);
  const int lane = t & 31, wv = t >> 5;
  int *ri = sm.redi();
  lk_pdl_trigger();                                  // adjoint_node_kernel runs beside this one
  if (a.left[pid]) return;                           // the eigensolve form's
  if (wv == 0) support<MPD>(I, ij, sm);
#pragma unroll
  for (int r = 0; r < 2; ++r)
    if (row_warp<MPD>(wv, r)) {
      row64<MPD>(static_cast<const double *>(I.X) + (size_t)pid * 2 * m, m, r, sm);
      // g_r and s_r = g_r . 1
      const double x = lane < m ? a.lam_a[((size_t)pid * 2 + r) * m + lane] : 0.0;
      const double s = lk_warp_sum(x);
      const int ex = __reduce_max_sync(FULL, exponent64(x)), sh = ex == -1022 ? NO_EXP : ex;
      if (lane < MPD) {
        const Df v = df_split(x, -sh);
        gv[r * MPD + lane] = st_df(v);
        put64<MPD>(terms, slot64<MPD>(r, lane), v);
      }
      if (lane == 0) {
        sm.red64()[10 + r] = s;
        ri[4 + r] = sh;
      }
    }
  __syncthreads();
  const int nsl = 2 * ri[0], ed = ri[1];
  gram64<MPD>(I, ij, sm, nsl, ed);
  Seg64<MPD> g;
  const float f2 = seg_load<MPD>(g, sm, row, seg);
  const float ratio = sqrtf(0.5f * cta_sum<C::NW>(f2, sm.red));
  if (t < 2) a.xbar_bar[(size_t)pid * 2 + t] = sm.red64()[10 + t];
  // s_0 x'_0 + s_1 x'_1 times 2^-eb
  const int ex0 = ri[2], ex1 = ri[3], eg0 = ri[4], eg1 = ri[5];
  const double s0 = sm.red64()[10], s1 = sm.red64()[11];
  const int es0 = s0 == 0.0 ? NO_EXP : exponent64(s0), es1 = s1 == 0.0 ? NO_EXP : exponent64(s1);
  const Df sd0 = df_split(s0, -es0), sd1 = df_split(s1, -es1);
  const int eb = max(es0 + ex0, es1 + ex1);
  const int sl = slot64<MPD>(vec, row);
  const Df x = ld_df(sm.xs[vec * MPD + row]);
  Df yc = ld_df(sm.cv[row]);
  if (vec) {
    const float f0 = pow2c(es0 + ex0 - eb), f1 = pow2c(es1 + ex1 - eb);
    const Df u = df_mul(Df{f0 * sd0.h, f0 * sd0.l}, ld_df(sm.xs[row]));
    yc = df_add(u, df_mul(Df{f1 * sd1.h, f1 * sd1.l}, ld_df(sm.xs[MPD + row])));
  }
  if (seg == 0) put64<MPD>(sb, sl, yc);
  __syncthreads();
  // ---- series of g (A^-1/2) and of C d and wbar_bar (A^-1) ----
  const float4 *co = cheb + (size_t)lk_cheb_class(ratio) * LK_CHEB_LD64;
  const float4 c0 = co[0];
  const Df scale = Df{c0.x, c0.y};
  const int deg = (int)c0.z;
  const bool keep = deg <= ADJ_KEEP;
  const int low = keep ? (int)c0.w : deg;            // (run backwards the terms stay pairs)
  seg_scale<MPD>(g, scale, row, seg);
  ++co;
  Df tc = ld_df(gv[vec * MPD + row]), tp = df(0.f), yp = df(0.f), ga, ya;
  {
    const float4 c = __ldg(co);
    ga = df_mul(Df{c.x, c.y}, tc);
    ya = df_mul(Df{c.z, c.w}, yc);
  }
  for (int k = 1; k <= low; ++k) {
    const float4 c = __ldg(co + k);
    const Df gt = product<MPD>(g, terms + (keep ? k - 1 : (k - 1) & 1) * 2 * C::VEC, vec, seg);
    const Df gy = product<MPD>(g, sb + ((k - 1) & 1) * 2 * C::VEC, vec, seg);
    const Df tn = k == 1 ? Df{0.5f * gt.h, 0.5f * gt.l} : df_add(gt, df_neg(tp));
    const Df yn = k == 1 ? Df{0.5f * gy.h, 0.5f * gy.l} : df_add(gy, df_neg(yp));
    tp = tc;
    tc = tn;
    yp = yc;
    yc = yn;
    if (seg == 0) {
      put64<MPD>(terms + (keep ? k : k & 1) * 2 * C::VEC, sl, tc);
      put64<MPD>(sb + (k & 1) * 2 * C::VEC, sl, yc);
    }
    __syncthreads();
    ga = df_add(ga, df_mul(Df{c.x, c.y}, tc));
    ya = df_add(ya, df_mul(Df{c.z, c.w}, yc));
  }
  {
    float gs = 0.f, ys = 0.f, tq = tp.h, tf = tc.h, yq = yp.h, yf = yc.h;
    for (int k = low + 1; k <= deg; ++k) {
      const float4 c = __ldg(co + k);
      const float tn = product32<MPD>(g, terms + (k - 1) * 2 * C::VEC, vec, seg) - tq;
      const float yn = product32<MPD>(g, sb + ((k - 1) & 1) * 2 * C::VEC, vec, seg) - yq;
      tq = tf;
      tf = tn;
      yq = yf;
      yf = yn;
      if (seg == 0) {
        terms[k * 2 * C::VEC + sl] = tn;
        sb[(k & 1) * 2 * C::VEC + sl] = yn;
      }
      __syncthreads();
      gs = fmaf(c.x, tn, gs);
      ys = fmaf(c.z, yn, ys);
    }
    ga = df_add(ga, df(gs));
    ya = df_add(ya, df(ys));
  }
  const Alpha64 al(I.alpha, m);
  // wbar times 2^-ed, then b_bar times 2^-ebb
  const int ebb = eb - al.e;
  if (seg == 0) wb[vec * MPD + row] = st_df(vec ? df_mul(ya, al.ia) : ya);
  // ---- D_0 + D_1: Clenshaw's vectors of x' against the terms of g ----
  float2 S[C::L / 2], F[C::L / 2];
#pragma unroll
  for (int j = 0; j < C::L / 2; ++j) S[j] = F[j] = make_float2(0.f, 0.f);
  // P_{deg-1} and P_deg; down to P_low in floats (with a zero low part in the buffer)
  Df p, pn = df(0.f);
  {
    const float4 c = __ldg(co + deg);
    p = df_mul(Df{c.x, c.y}, x);
    if (deg - 1 >= low) p.l = 0.f;
  }
  if (seg == 0) put64<MPD>(sm.tb + ((deg - 1) & 1) * 2 * C::VEC, sl, p);
  __syncthreads();
  if (seg == 0 && row < m) {
    const double u = df_to_double(df_mul(vec ? sd1 : sd0, ld_df(wb[row])), ed + (vec ? es1 : es0));
    a.xp_bar[((size_t)pid * 2 + vec) * m + row] =
        u + df_to_double(df_mul(al.rt, ga), al.re + (vec ? eg1 : eg0));
  }
  {
    float2 SF[C::L / 2];
#pragma unroll
    for (int c = 0; c < C::L / 2; ++c) SF[c] = make_float2(0.f, 0.f);
    for (int j = deg - 1; j >= low; --j) {           // (low >= 1)
      const float2 *qh = reinterpret_cast<const float2 *>(
          terms + j * 2 * C::VEC + (vec * C::KS + seg) * C::TS);
      const float2 ph = dup2(2.f * p.h);
#pragma unroll
      for (int c = 0; c < C::L / 2; ++c) SF[c] = __ffma2_rn(ph, qh[c], SF[c]);
      const float gp = product32<MPD>(g, sm.tb + (j & 1) * 2 * C::VEC, vec, seg);
      float pm = fmaf(__ldg(co + j).x, x.h, gp - pn.h), pl = 0.f;
      if (j == low) {                                // P_{low-1} in pairs again
        const float4 c = __ldg(co + j);
        const Df gd = product<MPD>(g, sm.tb + (j & 1) * 2 * C::VEC, vec, seg);
        const Df pd = df_add(df_add(gd, df_neg(pn)), df_mul(Df{c.x, c.y}, x));
        pm = pd.h;
        pl = pd.l;
      }
      pn = p;
      p = Df{pm, pl};
      if (seg == 0) put64<MPD>(sm.tb + ((j - 1) & 1) * 2 * C::VEC, sl, p);
      __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < C::L / 2; ++c) S[c] = SF[c];
  }
  for (int j = low - 1 < deg - 1 ? low - 1 : deg - 1; j >= 0; --j) {
    // the terms' own recurrence run backwards holds T_{j+1} = tc, T_j = tp
    const float2 *qh = reinterpret_cast<const float2 *>(
        terms + (keep ? j : j & 1) * 2 * C::VEC + (vec * C::KS + seg) * C::TS);
    const float2 *ql = qh + C::VEC / 2;
    const float fj = j ? 2.f : 1.f;
    const float2 ph = dup2(fj * p.h), np = dup2(-fj * p.h), pl = dup2(fj * p.l);
#pragma unroll
    for (int c = 0; c < C::L / 2; ++c) df_fma2(S[c], F[c], ph, np, pl, qh[c], ql[c]);
    if (j == 0) break;
    const float4 c = __ldg(co + j);
    const Df gp = product<MPD>(g, sm.tb + (j & 1) * 2 * C::VEC, vec, seg);
    const Df pm = df_add(df_add(gp, df_neg(pn)), df_mul(Df{c.x, c.y}, x));
    pn = p;
    p = pm;
    if (!keep) {
      // T_{j-1} = 2 X T_j - T_{j+1} (T_0 = g needs no halving: j >= 1 here)
      const Df gt = product<MPD>(g, terms + (j & 1) * 2 * C::VEC, vec, seg);
      const Df tm = df_add(gt, df_neg(tc));
      tc = tp;
      tp = tm;
      if (seg == 0) put64<MPD>(terms + ((j - 1) & 1) * 2 * C::VEC, sl, tm);
    }
    if (seg == 0) put64<MPD>(sm.tb + ((j - 1) & 1) * 2 * C::VEC, sl, p);
    __syncthreads();
  }
  // ---- A_bar = sqrt(m-1) alpha^-3/2 scale (D_0 + D_1) - b_bar wbar^T, times 2^-eA: the
  // exponents of the two D and of the outer product ----
  const int er = al.re - al.e, e0 = er + ex0 + eg0, e1 = er + ex1 + eg1, e2 = ebb + ed;
  const int eA = max(max(e0, e1), e2);
  const Df cf = df_mul(df_mul(al.rt, al.ia), scale);
  {
    const float fv = pow2c((vec ? e1 : e0) - eA);
    const Df cv = Df{fv * cf.h, fv * cf.l};
    const float fo = pow2c(e2 - eA);
    const Df br = vec ? ld_df(wb[MPD + row]) : df(0.f);
    Df v[C::L];
#pragma unroll
    for (int j = 0; j < C::L / 2; ++j) {
      v[2 * j] = df_mul(cv, df_quick(S[j].x, F[j].x));
      v[2 * j + 1] = df_mul(cv, df_quick(S[j].y, F[j].y));
    }
    if (vec == 0) {
#pragma unroll
      for (int j = 0; j < C::L; ++j) sm.Gs[row * C::LDG + seg * C::L + j] = st_df(v[j]);
    }
    __syncthreads();
    if (vec == 1) {
#pragma unroll
      for (int j = 0; j < C::L; ++j) {
        const int c = seg * C::L + j;
        const Df o = df_mul(Df{-fo * br.h, -fo * br.l}, ld_df(wb[c]));
        sm.Gs[row * C::LDG + c] =
            st_df(df_add(df_add(ld_df(sm.Gs[row * C::LDG + c]), v[j]), o));
      }
    }
  }
  __syncthreads();
  float2 *As = reinterpret_cast<float2 *>(terms);    // the terms are done with
  float *ayh = reinterpret_cast<float *>(As + MPD * C::LDG + (MPD * C::LDG & 1));
  float *ayl = ayh + C::QC * C::LDY;
  for (int q = t; q < MPD * MPD; q += C::NT) {
    const int i = q / MPD, c = q - i * MPD;
    const Df s = df_add(ld_df(sm.Gs[i * C::LDG + c]), ld_df(sm.Gs[c * C::LDG + i]));
    As[i * C::LDG + c] = make_float2(0.5f * s.h, 0.5f * s.l);
  }
  __syncthreads();
  // ---- window slopes: y_bar = 2 c A_bar y + c d b_bar, d_bar = c y . b_bar,
  // c_bar = y^T A_bar y + d y . b_bar. A warp per slope (lane = row) for A_bar y,
  // then a lane per slope for the sums over rows. Cells outside the support
  // keep the zeros the workspace was allocated with. y times 2^ey. ----
  const int ey = -((exponent64(a.sigma2) + al.e) / 2);
  float2 ah[MPD / 2], alo[MPD / 2];
#pragma unroll
  for (int i = 0; i < MPD / 2; ++i) {
    const float2 u = lane < MPD ? As[lane * C::LDG + 2 * i] : make_float2(0.f, 0.f);
    const float2 v = lane < MPD ? As[lane * C::LDG + 2 * i + 1] : make_float2(0.f, 0.f);
    ah[i] = make_float2(u.x, v.x);
    alo[i] = make_float2(u.y, v.y);
  }
  const Df alpha_bar =
      wv == 0 ? df_warp_sum(lane < MPD ? ld_df(As[lane * C::LDG + lane]) : df(0.f)) : df(0.f);
  const float2 *bb = wb + MPD;
  const double *tap = static_cast<const double *>(I.taper);
  const double *dp = static_cast<const double *>(I.dp);
  double *yb_out = a.ybw + (size_t)pid * wc * 2 * m;
  double *db_out = a.dbw + (size_t)pid * wc * 2;
  double gs2 = 0.0, gL = 0.0;
  for (int q0 = 0; q0 < nsl; q0 += C::QC) {
    const int nq = nsl - q0 < C::QC ? nsl - q0 : C::QC;
    __syncthreads();
    stage_slopes<MPD, false>(I, ij, sm, q0, nq, ey);
    double cj = 0.0, dj = 0.0;                       // the slope of warp 0's lane
    int ce = 0;
    if (wv == 0 && lane < nq) {
      const int c = sm.cell[(q0 + lane) >> 1];
      ce = cell_row(c) * w + cell_col(c);
      cj = tap[ce];
      dj = dp[((size_t)(ij.x + cell_row(c)) * I.gs_cols + (ij.y + cell_col(c))) * 2 + (lane & 1)];
      // y_bar = c 2^ec (2 (A_bar y) 2^(eA - ey) + d 2^el b_bar 2^ebb)
      const int ec = exponent64(cj), el = dj == 0.0 ? NO_EXP : exponent64(dj);
      const int ea = eA - ey + 1, eb2 = el + ebb, eo = max(ea, eb2);
      qc[lane] = st_df(df_split(cj, -ec));
      qd[lane] = st_df(df_split(dj, -el));
      qf[lane] = make_float2(pow2c(ea - eo), pow2c(eb2 - eo));
      qe[lane] = ec + eo;
    }
    __syncthreads();
    for (int q = wv; q < nq; q += C::NW) {
      const float4 *yh = reinterpret_cast<const float4 *>(sm.Yh + q * C::LDY);
      const float4 *yl = reinterpret_cast<const float4 *>(sm.Yl + q * C::LDY);
      float2 S0 = make_float2(0.f, 0.f), F0 = S0, S1 = S0, F1 = S0;
#pragma unroll
      for (int i = 0; i < MPD / 4; ++i) {
        const float4 u = yh[i], v = yl[i];
        const float2 u0 = make_float2(u.x, u.y), u1 = make_float2(u.z, u.w);
        df_fma2(S0, F0, u0, neg2(u0), make_float2(v.x, v.y), ah[2 * i], alo[2 * i]);
        df_fma2(S1, F1, u1, neg2(u1), make_float2(v.z, v.w), ah[2 * i + 1], alo[2 * i + 1]);
      }
      const Df s = df_add(df_add(df_quick(S0.x, F0.x), df_quick(S0.y, F0.y)),
                          df_add(df_quick(S1.x, F1.x), df_quick(S1.y, F1.y)));
      if (lane < MPD) {
        ayh[q * C::LDY + lane] = s.h;
        ayl[q * C::LDY + lane] = s.l;
      }
    }
    __syncthreads();
    if (wv < 2 && lane < nq) {
      Df v = df(0.f);
#pragma unroll 4
      for (int i = 0; i < MPD / 4; ++i) {
        const float4 u = reinterpret_cast<const float4 *>(sm.Yh + lane * C::LDY)[i];
        const float4 l = reinterpret_cast<const float4 *>(sm.Yl + lane * C::LDY)[i];
        Df o[4];
        if (wv == 0) {
#pragma unroll
          for (int c = 0; c < 4; ++c) o[c] = ld_df(bb[4 * i + c]);
        } else {
          const float4 h = reinterpret_cast<const float4 *>(ayh + lane * C::LDY)[i];
          const float4 k = reinterpret_cast<const float4 *>(ayl + lane * C::LDY)[i];
          o[0] = Df{h.x, k.x};
          o[1] = Df{h.y, k.y};
          o[2] = Df{h.z, k.z};
          o[3] = Df{h.w, k.w};
        }
        const Df p0 = df_add(df_mul(Df{u.x, l.x}, o[0]), df_mul(Df{u.y, l.y}, o[1]));
        const Df p1 = df_add(df_mul(Df{u.z, l.z}, o[2]), df_mul(Df{u.w, l.w}, o[3]));
        v = df_add(v, df_add(p0, p1));
      }
      qs[wv * C::QC + lane] = st_df(v);
    }
    __syncthreads();
    if (wv == 0 && lane < nq) {
      const double yb = df_to_double(ld_df(qs[lane]), ebb - ey);
      const double cbar = fma(dj, yb, df_to_double(ld_df(qs[C::QC + lane]), eA - 2 * ey));
      gs2 = fma(cbar, cj, gs2);
      gL = fma(cbar, a.dtap[ce], gL);
      db_out[ce * 2 + (lane & 1)] = cj * yb;
    }
    for (int q = t; q < nq * MPD; q += C::NT) {
      const int k = q / MPD, i = q - k * MPD;
      if (i >= m) continue;
      const int c = sm.cell[(q0 + k) >> 1], cell = cell_row(c) * w + cell_col(c);
      const float2 f = qf[k];
      const Df u = df_mul(Df{f.y * qd[k].x, f.y * qd[k].y}, ld_df(bb[i]));
      const Df v = df_add(Df{f.x * ayh[k * C::LDY + i], f.x * ayl[k * C::LDY + i]}, u);
      yb_out[((size_t)cell * 2 + ((q0 + k) & 1)) * m + i] =
          df_to_double(df_mul(ld_df(qc[k]), v), qe[k]);
    }
  }
  if (wv == 0) {
    gs2 = lk_warp_sum(gs2);
    gL = lk_warp_sum(gL);
    if (lane == 0) {
      a.theta[(size_t)pid * 3 + 0] = df_to_double(alpha_bar, eA) * (-(m - 1) / (a.rho * a.rho));
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
      h->d_inst, a, (const float4 *)h->cheb64);
  return cudaGetLastError();
}

template <int MPD>
cudaError_t launch_series64(letkf_ctx *h, int cls, void *mean, void *spread, const void *noise) {
  size_t need = 0;
  for (const LkInst &I : h->inst)
    if (I.m <= MPD && I.m > MPD - 8) {
      const size_t b = Smem64<MPD>::doubles(I.w) * sizeof(double);
      need = b > need ? b : need;
    }
  if (need == 0) return cudaSuccess;
  return lk_launch_pdl(series64_kernel<MPD>, (unsigned)h->n_pts_total, S64<MPD>::NT, need,
                       h->stream, h->d_inst, h->node_items, (double *)mean, (double *)spread,
                       (const float4 *)h->cheb64, h->counters, h->counters + 4 + cls,
                       h->worklist + (size_t)cls * h->n_pts_total, (const double *)noise, h->left64);
}

template <int MPD>
cudaError_t setup_series64(int w) {
  const cudaError_t e =
      lk_raise_smem(series64_kernel<MPD>, Smem64<MPD>::doubles(w) * sizeof(double));
  if (e != cudaSuccess) return e;
  return lk_raise_smem(adjoint_series64_kernel<MPD>, AdjSmem64<MPD>::doubles(w) * sizeof(double));
}

}  // namespace

cudaError_t lk_launch_series64(letkf_ctx *h, int cls, void *mean, void *spread, const LkCycle &cy) {
  if (cls == 0) {
    cudaError_t e = launch_series64<8>(h, 0, mean, spread, cy.noise);
    return e == cudaSuccess ? launch_series64<16>(h, 0, mean, spread, cy.noise) : e;
  }
  cudaError_t e = launch_series64<24>(h, 1, mean, spread, cy.noise);
  return e == cudaSuccess ? launch_series64<32>(h, 1, mean, spread, cy.noise) : e;
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
