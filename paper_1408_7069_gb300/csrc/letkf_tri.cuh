// Ill-conditioned node problems of FP32 handles (kappa_hat above fp64_kappa, up
// to LK_TRI_MAX): the analysis of Section 4.2 to about 48 bits by a
// tridiagonalisation, one warp per node, without an eigensolve.
//
// These nodes need A and what follows from it to far more than FP32 (the mean
// solve amplifies its rounding by kappa, 1e4-1e5 in the first frames), but GB300
// issues a warp-wide FP64 instruction once in 76 clocks and sub-partition (measured), so
// pairs of floats (hi + lo, FMA two-products and two-sums: 12 to 27 FP32
// operations for what FP64 does in one or two) are four times as fast. Per node:
//   Gram    G = sum_j tau_j/sigma2 y_j y_j^T exactly to about 2^-42 |G|: q = (a b +
//           sigma) - sigma takes a product's multiple of ulp(sigma), which sums
//           exactly, and the rest of it in one FMA (as the global Gram does)
//   reduce  Householder, lane = row of G, a step's column always in
//           register 0 (the rank-2 update writes its columns one place down):
//           T = Q^T G Q, and Q^T applied to the two anomaly rows and C d
//   solve   A^-1/2 b = sum_p w_p (A + s_p)^-1 b, the best rational approximation's
//           15 poles (lk_poles in letkf_cheb.cu; error 4e-9 to kappa 1e5, as far as nodes
//           come here; 7e-8 to 1e6): 15 poles x 2 rows, and A^-1 C d, are 31 shifted
//           tridiagonal systems, one per lane
//   apply   back through the reflectors, outputs
// About 48 k instructions per node of 32 members and 90 slopes. Bound by the FMA pipe, where a
// packed pair takes two issue slots, and by the chains of a step's sums (12 warps per SM;
// 58% of the issue slots used). Measured on one GB300, the analysis of the 80 x 80 system's
// first frame (5112 nodes, 32 members, kappa 1e4 to 5e4): FP64 sweeps 9.11 ms, this form
// 0.42 ms, of which this kernel 0.34; errors against FP64 equal.
#pragma once

#include "letkf_df.cuh"

namespace {

__device__ __forceinline__ void lk_cp_async4(float *dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src) : "memory");
}
__device__ __forceinline__ void lk_cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void lk_cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

constexpr int TRI_QC = 32;             // slopes staged at a time, two buffers

// Shared floats of a warp: two buffers of staged slopes [QC][MP], weights and innovations
// [QC] each, then Z of the solves (pairs [MP][32], system s of row i at s ^ i) and L (pairs
// [MP][16]: the two rows of a pole share it); the reflectors [MP][MP] (of step k the high
// parts, elements beyond k, in row k, the low parts in row MP-1-k from the other end: its
// elements up to MP-2-k, which that row's own high parts leave free); v and q of a step
// (hi and lo, MP each, zero beyond); d, e, b0, b1, bc, A^-1 C d and 1/h (pairs, MP each).
// From V on the taper's cells (16 bits each) stand until the Gram is done. 18.7 KB for 32
// members: three CTAs of four warps per SM.
template <int MP>
struct TriCfg {
  static constexpr int BUF = TRI_QC * (MP + 2), STAGE = 96 * MP;
  static_assert(STAGE >= 2 * BUF, "the staged slopes fit");
  static constexpr int V = STAGE, VB = V + MP * MP, D = VB + 4 * MP, RH = D + 12 * MP;
  static constexpr int TOTAL = RH + 2 * MP;
  static_assert(4 * (TOTAL - V) >= 2 * 31 * 31, "the cells of the largest window fit");
};

template <int MP>
struct TriState {
  float2 ah[MP / 2], al[MP / 2];       // the lane's row of G from the current column pair on
  Df b[3];                             // this lane's element of the two rows and of C d
};

// Steps k0 .. k0 + 7 of the reduction, columns held in LEN registers: column k in the
// first pair, whose place the next pair takes after every other step. EG: |G| < 2^EG;
// |b| < 8.
template <int MP, int LEN>
__device__ __forceinline__ void tri_steps(TriState<MP> &s, int k0, int m, int EG, float *ws) {
  using C = TriCfg<MP>;
  const int lane = threadIdx.x & 31;
  float *vh = ws + C::VB, *vl = vh + MP, *qh = vl + MP, *ql = qh + MP;
  float2 *dd = reinterpret_cast<float2 *>(ws + C::D), *ee = dd + MP;
  float2 *hh = reinterpret_cast<float2 *>(ws + C::RH);
  for (int k = k0; k < k0 + 8 && k < m; ++k) {
    const bool odd = k & 1;
    const Df x0 = Df{odd ? s.ah[0].y : s.ah[0].x, odd ? s.al[0].y : s.al[0].x};   // (lane, k)
    if (lane == k) dd[k] = make_float2(x0.h, x0.l);
    const Df x = lane > k && lane < m ? x0 : df(0.f);
    const Df x1 = df_shfl(x, k + 1 < 32 ? k + 1 : 31);
    const int E = warp_exponent(x.h);
    // below 2^-40 (G + alpha, alpha >= 0.01: nothing) there is nothing to annihilate
    if (k < m - 2 && E > -40) {                      // (the same in every lane)
      const Df sig = df_redux(df_mul(x, x), 2 * E);
      const Df sq = df_sqrt(sig);
      const int Ev = ((__float_as_int(sq.h) >> 23) - 126) + 1;     // |v| <= 2 sq < 2^Ev
      const Df al = x1.h >= 0.f ? df_neg(sq) : sq;
      const Df v = lane == k + 1 ? df_add(x, df_neg(al)) : x;
      const Df rh = df_rcp(df_add(sig, df_neg(df_mul(x1, al))));
      if (lane == 0) {
        ee[k] = make_float2(al.h, al.l);
        hh[k] = make_float2(rh.h, rh.l);
      }
      // columns of the held pairs at slots 0, 1, ...; zeros behind the last
      const int slot = lane >= (k & ~1) ? lane - (k & ~1) : lane - (k & ~1) + MP;
      if (lane < MP) {
        if (lane > k) {
          ws[C::V + k * MP + lane] = v.h;
          ws[C::V + (MP - 1 - k) * MP + MP - 1 - lane] = v.l;
        }
        vh[slot] = v.h;                              // (zero up to column k)
        vl[slot] = v.l;
      }
      __syncwarp();
      // p = G v / h
      float2 S = make_float2(0.f, 0.f), F = S;
#pragma unroll
      for (int j = 0; j < LEN / 2; ++j) {
        const float2 a = reinterpret_cast<const float2 *>(vh)[j];
        const float2 b = reinterpret_cast<const float2 *>(vl)[j];
        const float2 p = prod2(s.ah[j], a);
        float2 e;
        two_sum2(S, p, S, e);
        F = __fadd2_rn(F, e);
        F = __ffma2_rn(s.ah[j], b, F);
        F = __ffma2_rn(s.al[j], a, F);
        F = sub2(F, __ffma2_rn(s.ah[j], neg2(a), p));
      }
      const Df p = df_mul(df_add(df_quick(S.x, F.x), df_quick(S.y, F.y)), rh);
      // q = p - (v . p / 2h) v, b -= (v . b / h) v
      const Df t = df_redux(df_mul(v, p), EG + 1);
      Df tb[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) tb[r] = df_mul(df_redux(df_mul(v, s.b[r]), Ev + 3), rh);
      const Df q = df_add(p, df_neg(df_mul(df_mul(t, Df{0.5f * rh.h, 0.5f * rh.l}), v)));
#pragma unroll
      for (int r = 0; r < 3; ++r) s.b[r] = df_add(s.b[r], df_neg(df_mul(tb[r], v)));
      if (lane < MP) {
        qh[slot] = lane >= k ? q.h : 0.f;
        ql[slot] = lane >= k ? q.l : 0.f;
      }
      __syncwarp();
      // G -= v q^T + q v^T
      const float2 vih = dup2(v.h), nvh = dup2(-v.h), nvl = dup2(-v.l);
      const float2 qih = dup2(q.h), nqh = dup2(-q.h), nql = dup2(-q.l);
#pragma unroll
      for (int j = 0; j < LEN / 2; ++j) {
        const float2 vjh = reinterpret_cast<const float2 *>(vh)[j];
        const float2 vjl = reinterpret_cast<const float2 *>(vl)[j];
        const float2 qjh = reinterpret_cast<const float2 *>(qh)[j];
        const float2 qjl = reinterpret_cast<const float2 *>(ql)[j];
        const float2 p1 = prod2(vih, qjh), p2 = prod2(qih, vjh);
        float2 lo = __ffma2_rn(nvh, qjl, s.al[j]);
        lo = __ffma2_rn(nvl, qjh, lo);
        lo = __ffma2_rn(nqh, vjl, lo);
        lo = __ffma2_rn(nql, vjh, lo);
        lo = __fadd2_rn(lo, __ffma2_rn(nvh, qjh, p1));
        lo = __fadd2_rn(lo, __ffma2_rn(nqh, vjh, p2));
        float2 t1, e1, t2, e2;
        two_sum2(p1, p2, t1, e1);
        two_diff2(s.ah[j], t1, t2, e2);
        lo = __fadd2_rn(lo, sub2(e2, e1));
        // renormalised: where the pair cancels (windows with fewer slopes than members
        // leave a trailing block of rounding) the low part would outgrow the high one
        s.ah[j] = __fadd2_rn(t2, lo);
        s.al[j] = sub2(lo, sub2(s.ah[j], t2));
      }
    } else if (lane == 0) {                          // nothing to annihilate
      ee[k] = make_float2(x1.h, x1.l);
      hh[k] = make_float2(0.f, 0.f);
    }
    __syncwarp();
    if (odd) {                                       // two columns down
#pragma unroll
      for (int j = 0; j < LEN / 2; ++j) {
        const bool last = j + 1 == LEN / 2;
        s.ah[j] = last ? make_float2(0.f, 0.f) : s.ah[j + 1 < MP / 2 ? j + 1 : j];
        s.al[j] = last ? make_float2(0.f, 0.f) : s.al[j + 1 < MP / 2 ? j + 1 : j];
      }
    }
  }
}

// The node's analysis by one warp. ncell cells of the taper's support (row << 8 | column,
// from V on), poles: (s_p, w_p), EG: |G| < 2^EG.
template <int MP>
__device__ void tri_node(const LkInst &I, int pid, int ncell, int EG,
                         const double2 *__restrict__ poles, float *__restrict__ mean_out,
                         float *__restrict__ spread_out, int *__restrict__ counters, float *ws) {
  using C = TriCfg<MP>;
  const int lane = threadIdx.x & 31, m = I.m, nsl = 2 * ncell;
  const int2 ij = I.pts[pid];
  const float *Ybp = static_cast<const float *>(I.Ybp);
  const float *dp = static_cast<const float *>(I.dp);
  const float *taper = static_cast<const float *>(I.taper);
  const unsigned short *cell = reinterpret_cast<const unsigned short *>(ws + C::V);
  // ---- Gram, the next slopes on their way meanwhile ----
  auto stage = [&](int q0) {
    float *ys = ws + (q0 / TRI_QC & 1) * C::BUF;
    if (q0 + lane < nsl) {
      const int ce = cell[(q0 + lane) >> 1], cs = ce >> 8, cc = ce & 255;
      lk_cp_async4(&ys[TRI_QC * MP + lane], &taper[cs * I.w + cc]);
      lk_cp_async4(&ys[TRI_QC * (MP + 1) + lane],
                   &dp[((size_t)(ij.x + cs) * I.gs_cols + ij.y + cc) * 2 + (lane & 1)]);
    }
    const int nq = nsl - q0 < TRI_QC ? nsl - q0 : TRI_QC;
#pragma unroll 4
    for (int q = 0; q < nq; q += 2) {
      const int ce = cell[(q0 + q) >> 1];
      const float *src = Ybp + ((size_t)(ij.x + (ce >> 8)) * I.gs_cols + ij.y + (ce & 255)) * 2 * m;
      if (lane < m) {
        lk_cp_async4(&ys[q * MP + lane], &src[lane]);
        lk_cp_async4(&ys[(q + 1) * MP + lane], &src[m + lane]);
      }
    }
    lk_cp_async_commit();
  };
  if (lane >= m && lane < MP)
    for (int q = 0; q < TRI_QC; ++q) ws[q * MP + lane] = ws[C::BUF + q * MP + lane] = 0.f;
  stage(0);
  // anchor: the sums stay in [2^EG, 3 2^EG), their grid 2^(EG - 22)
  const float sg = pow2f(EG + 1);
  const float2 sg2 = dup2(sg);
  TriState<MP> s;
#pragma unroll
  for (int j = 0; j < MP / 2; ++j) {
    s.ah[j] = sg2;
    s.al[j] = make_float2(0.f, 0.f);
  }
  Df c = df(0.f);
  for (int q0 = 0; q0 < nsl; q0 += TRI_QC) {
    const int nq = nsl - q0 < TRI_QC ? nsl - q0 : TRI_QC;
    if (q0 + TRI_QC < nsl) {
      stage(q0 + TRI_QC);
      lk_cp_async_wait<1>();
    } else {
      lk_cp_async_wait<0>();
    }
    __syncwarp();
    const float *ys = ws + (q0 / TRI_QC & 1) * C::BUF;
    for (int q = 0; q < nq; ++q) {
      const float *yr = ys + q * MP;
      const float y = lane < MP ? yr[lane] : 0.f, tw = ys[TRI_QC * MP + q];
      const float th = __fmul_rn(tw, y), tl = fmaf(tw, y, -th), d = ys[TRI_QC * (MP + 1) + q];
      const float ch = __fmul_rn(th, d), t = __fadd_rn(c.h, ch), bb = __fsub_rn(t, c.h);
      c.l = __fadd_rn(c.l, __fadd_rn(__fsub_rn(c.h, __fsub_rn(t, bb)), __fsub_rn(ch, bb)));
      c.l = __fadd_rn(c.l, fmaf(tl, d, fmaf(th, d, -ch)));
      c.h = t;
      const float2 h2 = dup2(th), l2 = dup2(tl);
#pragma unroll
      for (int j = 0; j < MP / 2; ++j) {
        const float2 yj = reinterpret_cast<const float2 *>(yr)[j];
        const float2 a = __ffma2_rn(h2, yj, s.ah[j]);
        const float2 r = __ffma2_rn(h2, yj, sub2(s.ah[j], a));
        s.ah[j] = a;
        s.al[j] = __fadd2_rn(s.al[j], __ffma2_rn(l2, yj, r));
      }
    }
    __syncwarp();
    // the low parts back below the grid
#pragma unroll
    for (int j = 0; j < MP / 2; ++j) {
      const float2 a = __fadd2_rn(s.ah[j], s.al[j]);
      s.al[j] = __fadd2_rn(s.al[j], sub2(s.ah[j], a));
      s.ah[j] = a;
    }
  }
#pragma unroll
  for (int j = 0; j < MP / 2; ++j) {
    const float2 h = sub2(s.ah[j], sg2), a = __fadd2_rn(h, s.al[j]);
    s.al[j] = sub2(s.al[j], sub2(a, h));
    s.ah[j] = a;
  }
  // ---- the rows' means and anomalies, each scaled by a power of two to below 1 ----
  float *xrow = static_cast<float *>(I.X) + (size_t)pid * 2 * m;
  const Df rm = df_rcp(df((float)m));
  Df xb0 = df(lane < m ? xrow[lane] : 0.f), xb1 = df(lane < m ? xrow[m + lane] : 0.f);
  s.b[0] = xb0;
  s.b[1] = xb1;
  df_warp_sum2(xb0, xb1);
  xb0 = df_mul(xb0, rm);
  xb1 = df_mul(xb1, rm);
  s.b[0] = lane < m ? df_add(s.b[0], df_neg(xb0)) : df(0.f);
  s.b[1] = lane < m ? df_add(s.b[1], df_neg(xb1)) : df(0.f);
  s.b[2] = df_quick(c.h, c.l);
  int Eb[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    Eb[r] = warp_exponent(s.b[r].h);
    s.b[r] = Df{s.b[r].h * pow2f(-Eb[r]), s.b[r].l * pow2f(-Eb[r])};
  }
  // ---- T = Q^T G Q ----
  for (int i = lane; i < MP * MP + 4 * MP; i += 32) ws[C::V + i] = 0.f;
  __syncwarp();
  if constexpr (MP == 32) {
    tri_steps<MP, 32>(s, 0, m, EG, ws);
    tri_steps<MP, 24>(s, 8, m, EG, ws);
    tri_steps<MP, 16>(s, 16, m, EG, ws);
    tri_steps<MP, 8>(s, 24, m, EG, ws);
  } else {
    tri_steps<MP, 16>(s, 0, m, EG, ws);
    tri_steps<MP, 8>(s, 8, m, EG, ws);
  }
  float2 *dd = reinterpret_cast<float2 *>(ws + C::D), *ee = dd + MP, *bb = ee + MP, *xc = bb + 3 * MP;
  if (lane < MP)
#pragma unroll
    for (int r = 0; r < 3; ++r) bb[r * MP + lane] = make_float2(s.b[r].h, s.b[r].l);
  __syncwarp();
  // ---- (T + alpha + alpha s_p) x = b by L D L^T: lane 2 p + r: pole p, row r; lane 30:
  // A^-1 C d ----
  float2 *Zs = reinterpret_cast<float2 *>(ws), *Ls = Zs + 32 * MP;
  const double2 pw = lane < 30 ? poles[lane >> 1] : make_double2(0.0, 0.0);
  const Df sh = df_of(I.alpha * (1.0 + pw.x));
  const float2 *rhs = bb + (lane < 30 ? lane & 1 : 2) * MP;
  Df r = df(0.f), z = df(0.f);
  for (int i = 0; i < m; ++i) {
    const Df d = df_add(Df{dd[i].x, dd[i].y}, sh), b = Df{rhs[i].x, rhs[i].y};
    Df l = df(0.f), dl = d;
    if (i > 0) {
      const Df e = Df{ee[i - 1].x, ee[i - 1].y};
      l = df_mul(e, r);
      dl = df_add(d, df_neg(df_mul(e, l)));
      z = df_add(b, df_neg(df_mul(l, z)));
    } else {
      z = b;
    }
    r = df_rcp(dl);
    const Df zr = df_mul(z, r);
    if (!(lane & 1)) Ls[i * 16 + (lane >> 1)] = make_float2(l.h, l.l);
    Zs[i * 32 + (lane ^ i)] = make_float2(zr.h, zr.l);
  }
  __syncwarp();
  Df x = df(0.f), ln = df(0.f);
  const Df wt = df_of(pw.y * sqrt((double)I.alpha));
  for (int i = m - 1; i >= 0; --i) {
    const float2 zr = Zs[i * 32 + (lane ^ i)], l = Ls[i * 16 + (lane >> 1)];
    x = df_add(Df{zr.x, zr.y}, df_neg(df_mul(ln, x)));
    ln = Df{l.x, l.y};
    if (lane == 30) xc[i] = make_float2(x.h, x.l);
    const Df u = df_mul(wt, x);
    Zs[i * 32 + (lane ^ i)] = make_float2(u.h, u.l);
  }
  __syncwarp();
  // ---- X'_r wbar = b_r . A^-1 C d; the poles' sums, back through the reflectors ----
  Df w0 = df(0.f), w1 = df(0.f);
  if (lane < m) {
    const Df xv = Df{xc[lane].x, xc[lane].y};
    w0 = df_mul(s.b[0], xv);
    w1 = df_mul(s.b[1], xv);
  }
  df_warp_sum2(w0, w1);
  Df u0 = df(0.f), u1 = df(0.f);
  if (lane < m) {
#pragma unroll
    for (int p = 0; p < 15; ++p) {
      const float2 z0 = Zs[lane * 32 + ((2 * p) ^ lane)], z1 = Zs[lane * 32 + ((2 * p + 1) ^ lane)];
      u0 = df_add(u0, Df{z0.x, z0.y});
      u1 = df_add(u1, Df{z1.x, z1.y});
    }
  }
  const float2 *hh = reinterpret_cast<const float2 *>(ws + C::RH);
  for (int k = m - 3; k >= 0; --k) {
    const Df rh = Df{hh[k].x, hh[k].y};
    if (rh.h == 0.f) continue;                       // (the same in every lane)
    Df v = df(0.f);
    if (lane > k && lane < MP)
      v = Df{ws[C::V + k * MP + lane], ws[C::V + (MP - 1 - k) * MP + MP - 1 - lane]};
    // |v|^2 = 2 h < 2^(2 - e), e the exponent of 1 / h; |u| < 8
    const int Ev = ((2 - ((__float_as_int(rh.h) >> 23) - 127)) >> 1) + 1;
    const Df t0 = df_mul(df_redux(df_mul(v, u0), Ev + 3), rh);
    const Df t1 = df_mul(df_redux(df_mul(v, u1), Ev + 3), rh);
    u0 = df_add(u0, df_neg(df_mul(t0, v)));
    u1 = df_add(u1, df_neg(df_mul(t1, v)));
  }
  // ---- outputs ----
  const Df rt = df_sqrt(df(float(m - 1)));
  auto scaled = [](Df a, int e) { return Df{a.h * pow2f(e), a.l * pow2f(e)}; };
  const Df y0 = df_add(xb0, scaled(scaled(w0, Eb[0]), Eb[2]));
  const Df y1 = df_add(xb1, scaled(scaled(w1, Eb[1]), Eb[2]));
  const Df a0 = lane < m ? df_add(y0, scaled(df_mul(u0, rt), Eb[0])) : df(0.f);
  const Df a1 = lane < m ? df_add(y1, scaled(df_mul(u1, rt), Eb[1])) : df(0.f);
  if (lane < m) {
    xrow[lane] = a0.h;
    xrow[m + lane] = a1.h;
  }
  Df mu0 = a0, mu1 = a1;
  df_warp_sum2(mu0, mu1);
  mu0 = df_mul(mu0, rm);
  mu1 = df_mul(mu1, rm);
  const Df d0 = lane < m ? df_add(a0, df_neg(mu0)) : df(0.f);
  const Df d1 = lane < m ? df_add(a1, df_neg(mu1)) : df(0.f);
  Df s0 = df_mul(d0, d0), s1 = df_mul(d1, d1);
  df_warp_sum2(s0, s1);
  const float sp0 = sqrtf(s0.h / float(m - 1)), sp1 = sqrtf(s1.h / float(m - 1));
  if (lane == 0) {
    if (mean_out) {
      mean_out[0] = mu0.h;
      mean_out[1] = mu1.h;
    }
    if (spread_out) {
      spread_out[0] = sp0;
      spread_out[1] = sp1;
    }
    if (!isfinite(mu0.h) || !isfinite(mu1.h) || !isfinite(sp0) || !isfinite(sp1))
      atomicOr(&counters[0], LK_BIT_NONFINITE);
    atomicMax(&counters[2], 1);
    atomicAdd(&counters[3], 1);
  }
  __syncwarp();
}

}  // namespace
