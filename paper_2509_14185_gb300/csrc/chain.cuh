// The residual chain of one point, shared by the jet kernels (jet.cu: one warp per point,
// layers.cu: one thread per point and direction): dual numbers, field envelopes and the
// self-similar residuals on y-jets.  Paper references as in jet.cu.
#pragma once

#include <cmath>

#include "gn_internal.cuh"

namespace gn {
namespace {

struct Dl {
  double v, d;
};
__device__ __forceinline__ Dl operator+(Dl a, Dl b) { return {a.v + b.v, a.d + b.d}; }
__device__ __forceinline__ Dl operator-(Dl a, Dl b) { return {a.v - b.v, a.d - b.d}; }
__device__ __forceinline__ Dl operator-(Dl a) { return {-a.v, -a.d}; }
__device__ __forceinline__ Dl operator*(Dl a, Dl b) { return {a.v * b.v, fma(a.v, b.d, a.d * b.v)}; }
__device__ __forceinline__ Dl operator*(double s, Dl a) { return {s * a.v, s * a.d}; }
__device__ __forceinline__ Dl operator+(double s, Dl a) { return {s + a.v, a.d}; }
__device__ __forceinline__ Dl dconst(double v) { return {v, 0.0}; }
// u^e for a constant base u > 0 and a dual exponent e.
__device__ __forceinline__ Dl pow_cb(double u, Dl e) {
  const double lu = log(u);
  const double p = exp(e.v * lu);
  return {p, p * lu * e.d};
}

template <int EQ> struct Eq;
template <> struct Eq<GN_BURGERS> { static constexpr int D = 1, NF = 1, NE = 1; };
template <> struct Eq<GN_CCF> { static constexpr int D = 1, NF = 1, NE = 1; };
template <> struct Eq<GN_IPM> { static constexpr int D = 2, NF = 2, NE = 2; };
template <> struct Eq<GN_BOUSSINESQ> { static constexpr int D = 2, NF = 3, NE = 3; };

// Network-input jet components.  1D: (v, z, zz).  2D: (v, q, b, qq, qb, bb,
// qqq, qqb, qbb).  The reverse pass uses the first C_R of them.
template <int D> struct JT;
template <> struct JT<1> { static constexpr int CR = 2, CF = 3; };
template <> struct JT<2> { static constexpr int CR = 6, CF = 9; };

// Component reached by one more derivative along q (used for d/dlambda,
// since lambda enters the network only through q).
template <int D> __device__ __forceinline__ int q_shift(int c);
template <> __device__ __forceinline__ int q_shift<1>(int c) { return c + 1; }
template <> __device__ __forceinline__ int q_shift<2>(int c) {
  // v->q, q->qq, b->qb, qq->qqq, qb->qqb, bb->qbb
  const int m[6] = {1, 3, 4, 6, 7, 8};
  return m[c];
}

// y-jet of dual numbers: value, first derivatives, second derivatives
// (1D: h[0] = d11; 2D: h[0] = d11, h[1] = d12, h[2] = d22).
template <int D> struct YJ {
  Dl v;
  Dl g[D];
  Dl h[D == 1 ? 1 : 3];
};
template <int D> __device__ __forceinline__ int hix(int i, int j) { return D == 1 ? 0 : i + j; }

template <int D> __device__ __forceinline__ YJ<D> ymul(const YJ<D>& a, const YJ<D>& b) {
  YJ<D> c;
  c.v = a.v * b.v;
#pragma unroll
  for (int i = 0; i < D; i++) c.g[i] = a.g[i] * b.v + a.v * b.g[i];
#pragma unroll
  for (int i = 0; i < D; i++)
#pragma unroll
    for (int j = i; j < D; j++) {
      const int k = hix<D>(i, j);
      c.h[k] = a.h[k] * b.v + a.g[i] * b.g[j] + a.g[j] * b.g[i] + a.v * b.h[k];
    }
  return c;
}

// Envelope y1^m * u^e (u = 1 + |y|^2) as a y-jet; e is a dual number.
//   (u^e)_i = 2 e y_i u^e / u,  (u^e)_ij = 2 e u^e / u (delta_ij + 2 (e-1) y_i y_j / u).
template <int D> __device__ YJ<D> envelope(const double* y, double u, int m, Dl e) {
  const Dl W = pow_cb(u, e);
  const double iu = 1.0 / u;
  const Dl c1 = (2.0 * iu) * (e * W);  // 2 e W / u
  YJ<D> Wj;
  Wj.v = W;
#pragma unroll
  for (int i = 0; i < D; i++) Wj.g[i] = y[i] * c1;
  const Dl em1 = e + dconst(-1.0);
#pragma unroll
  for (int i = 0; i < D; i++)
#pragma unroll
    for (int j = i; j < D; j++) {
      const Dl inner = dconst(i == j ? 1.0 : 0.0) + (2.0 * y[i] * y[j] * iu) * em1;
      Wj.h[hix<D>(i, j)] = c1 * inner;
    }
  if (m == 0) return Wj;
  YJ<D> Y;
  const double y1 = y[0];
  Y.v = dconst(m == 1 ? y1 : y1 * y1);
#pragma unroll
  for (int i = 0; i < D; i++) Y.g[i] = dconst(0.0);
  Y.g[0] = dconst(m == 1 ? 1.0 : 2.0 * y1);
#pragma unroll
  for (int k = 0; k < (D == 1 ? 1 : 3); k++) Y.h[k] = dconst(0.0);
  Y.h[0] = dconst(m == 1 ? 0.0 : 2.0);
  return ymul<D>(Y, Wj);
}

// Exponential output map on one field's jet components a[0 .. CF) (value, q, (b,) the second
// orders, the q-direction third orders the lambda column needs): N = exp(a) by the chain rule,
// every component exp(a_v) times the complete Bell polynomial of the a-derivatives.
template <int D, int CF>
__device__ __forceinline__ void exp_jet(const double* a, double* N) {
  const double E = exp(a[0]);
  N[0] = E;
  if constexpr (D == 1) {
    N[1] = E * a[1];
    if constexpr (CF > 2) N[2] = E * (a[2] + a[1] * a[1]);
  } else {
    const double q = a[1], b = a[2];
    N[1] = E * q;
    N[2] = E * b;
    N[3] = E * (a[3] + q * q);
    N[4] = E * (a[4] + q * b);
    N[5] = E * (a[5] + b * b);
    if constexpr (CF > 6) {
      N[6] = E * (a[6] + 3.0 * q * a[3] + q * q * q);
      N[7] = E * (a[7] + b * a[3] + 2.0 * q * a[4] + q * q * b);
      N[8] = E * (a[8] + q * a[5] + 2.0 * b * a[4] + q * b * b);
    }
  }
}

// Its adjoint on the components the reverse pass carries (c < C_R): nb holds dN-bar on entry
// and the pre-activation adjoints a-bar_c = sum_k N-bar_k dN_k / da_c on exit.
template <int D>
__device__ __forceinline__ void exp_jet_adjoint(const double* a, double* nb) {
  const double E = exp(a[0]);
  if constexpr (D == 1) {
    const double a0 = nb[0] * E + nb[1] * (E * a[1]);
    nb[1] = nb[1] * E;
    nb[0] = a0;
  } else {
    const double q = a[1], b = a[2];
    const double N[6] = {E, E * q, E * b, E * (a[3] + q * q), E * (a[4] + q * b), E * (a[5] + b * b)};
    double s = 0.0;
#pragma unroll
    for (int c = 0; c < 6; c++) s = fma(nb[c], N[c], s);
    const double a1 = E * (nb[1] + 2.0 * q * nb[3] + b * nb[4]);
    const double a2 = E * (nb[2] + q * nb[4] + 2.0 * b * nb[5]);
    nb[0] = s;
    nb[1] = a1;
    nb[2] = a2;
    nb[3] *= E;
    nb[4] *= E;
    nb[5] *= E;
  }
}

// The field jets F_f = E_f N_f at one point, in dual numbers: nn holds the network-output jets
// (network-input components c < C_R), a = 1/(1 + lambda), q = u^(-a/2) and lamd the coordinates'
// lambda dependence along this lane's direction.
template <int EQ>
__device__ __forceinline__ void field_jets(const double* y, double u, Dl a, Dl q, Dl lamd, double beta,
                                           const Dl (&nn)[Eq<EQ>::NF][JT<Eq<EQ>::D>::CR],
                                           YJ<Eq<EQ>::D> (&F)[Eq<EQ>::NF]) {
  constexpr int D = Eq<EQ>::D, NF = Eq<EQ>::NF;
  // q jets: q_i = -a y_i q / u ; q_ij = -a q / u (delta_ij - (a+2) y_i y_j / u)
  const double iu = 1.0 / u;
  Dl qg[D], qh[D == 1 ? 1 : 3];
  const Dl aq_u = (-iu) * (a * q);
#pragma unroll
  for (int i = 0; i < D; i++) qg[i] = y[i] * aq_u;
#pragma unroll
  for (int i = 0; i < D; i++)
#pragma unroll
    for (int j = i; j < D; j++)
      qh[hix<D>(i, j)] = aq_u * (dconst(i == j ? 1.0 : 0.0) + (-y[i] * y[j] * iu) * (a + dconst(2.0)));
  // beta jets (2D): beta_1 = -y1 y2 u^-3/2, beta_2 = (1+y1^2) u^-3/2,
  // beta_11 = y2 (3 y1^2 - u) u^-5/2, beta_12 = y1 (3 y2^2 - u) u^-5/2,
  // beta_22 = -3 y2 (1 + y1^2) u^-5/2
  double bg[2] = {0.0, 0.0}, bh[3] = {0.0, 0.0, 0.0};
  if (D == 2) {
    const double s3 = iu / sqrt(u), s5 = s3 * iu;
    bg[0] = -y[0] * y[1] * s3;
    bg[1] = (1.0 + y[0] * y[0]) * s3;
    bh[0] = y[1] * (3.0 * y[0] * y[0] - u) * s5;
    bh[1] = y[0] * (3.0 * y[1] * y[1] - u) * s5;
    bh[2] = -3.0 * y[1] * (1.0 + y[0] * y[0]) * s5;
  }
  // fields F_f = E_f * N_f
#pragma unroll
  for (int f = 0; f < NF; f++) {
    YJ<D> N;
    N.v = nn[f][0];
    if (D == 1) {
      N.g[0] = nn[f][1] * qg[0];
      N.h[0] = dconst(0.0);  // not used by the 1D residuals
    } else {
#pragma unroll
      for (int i = 0; i < D; i++) N.g[i] = nn[f][1] * qg[i] + bg[i] * nn[f][2];
#pragma unroll
      for (int i = 0; i < D; i++)
#pragma unroll
        for (int j = i; j < D; j++) {
          const int k = hix<D>(i, j);
          N.h[k] = nn[f][3] * (qg[i] * qg[j]) + nn[f][4] * (bg[j] * qg[i] + bg[i] * qg[j]) +
                   (bg[i] * bg[j]) * nn[f][5] + nn[f][1] * qh[k] + bh[k] * nn[f][2];
        }
    }
    // exponent k_f(lambda) and prefactor (y1^m, extra power of u)
    Dl kf;
    int m;
    double e0;
    if (EQ == GN_BURGERS) { kf = lamd; m = 1; e0 = -0.5; }
    else if (EQ == GN_CCF) { kf = lamd; m = 2; e0 = -1.0; }
    else if (EQ == GN_IPM) {
      if (f == 0) { kf = lamd; m = 0; e0 = 0.0; }
      else { kf = dconst(1.0) + 2.0 * lamd; m = 1; e0 = -0.5; }
    } else {
      if (f == 0) { kf = dconst(-1.0); m = 1; e0 = -0.5; }
      else if (f == 1) { kf = lamd + dconst(-1.0); m = 0; e0 = 0.0; }
      else { kf = dconst(1.0) + 2.0 * lamd; m = 1; e0 = -0.5; }
    }
    const Dl e = dconst(e0) + 0.5 * (kf * a);
    F[f] = ymul<D>(envelope<D>(y, u, m, e), N);
  }
}

// The residuals of a point's rows (or the single value of a wall, node, norm, decay or bound row)
// from its field jets; sUv receives d R / d U of a CCF interior row.
template <int EQ>
__device__ __forceinline__ void residual_rows(const JetArgs& A, int kind, int64_t pt, const double* y, double u, Dl a,
                                              Dl lamd, const Dl (&nn)[Eq<EQ>::NF][JT<Eq<EQ>::D>::CR],
                                              YJ<Eq<EQ>::D> (&F)[Eq<EQ>::NF], Dl (&R)[Eq<EQ>::NE], double& sUv) {
  constexpr int D = Eq<EQ>::D, NF = Eq<EQ>::NF, NE = Eq<EQ>::NE;
  constexpr int NJ = 1 + D + (D == 1 ? 1 : 3);   // stage-1 values per field
  // stage 2: Phi = Phi_1 + eps Phi_2, Phi_1 a constant (its jets precomputed at this point)
  if (A.base && kind != KIND_NODE) {
    const double* b = A.base + pt * A.base_ld;
    const double ep = A.eps;
#pragma unroll
    for (int f = 0; f < NF; f++) {
      F[f].v = Dl{b[f * NJ] + ep * F[f].v.v, ep * F[f].v.d};
#pragma unroll
      for (int i = 0; i < D; i++) F[f].g[i] = Dl{b[f * NJ + 1 + i] + ep * F[f].g[i].v, ep * F[f].g[i].d};
#pragma unroll
      for (int k = 0; k < (D == 1 ? 1 : 3); k++)
        F[f].h[k] = Dl{b[f * NJ + 1 + D + k] + ep * F[f].h[k].v, ep * F[f].h[k].d};
    }
  }

  // residuals (or the single value of a wall/node/norm row)
  sUv = 0.0;
  const Dl opl = dconst(1.0) + lamd;
  if (kind == KIND_INTERIOR) {
    if (EQ == GN_BURGERS) {
      const YJ<D>& U = F[0];
      R[0] = (-1.0) * (lamd * U.v) + (y[0] * opl + U.v) * U.g[0];
    } else if (EQ == GN_CCF) {
      // U = sum_j K_ij g_j + D_i g(y_i); the K part's d/dlambda is added by
      // the Hilbert contraction (it carries the lambda column of J_g).
      const YJ<D> Eg = envelope<D>(y, u, 1, dconst(-1.0) + 0.5 * (lamd * a));
      Dl gi = Eg.v * nn[0][0];
      if (A.base) gi = Dl{A.base[pt * A.base_ld + NF * NJ] + A.eps * gi.v, A.eps * gi.d};
      const Dl Uv = dconst(A.ug[pt]) + A.dcoef[pt] * gi;
      const YJ<D>& T = F[0];
      R[0] = (-1.0) * (lamd * T.v) + (y[0] * opl + Uv) * T.g[0];
      sUv = T.g[0].v;
    } else if (EQ == GN_IPM) {
      const YJ<D>& P = F[0];
      const YJ<D>& S = F[1];
      const Dl V1 = y[0] * opl + S.g[1];
      const Dl V2 = y[D - 1] * opl + (-S.g[0]);
      R[0] = (-1.0) * (lamd * P.v) + V1 * P.g[0] + V2 * P.g[D - 1];
      R[NE > 1 ? 1 : 0] = S.h[0] + S.h[D == 1 ? 0 : 2] - P.g[0];
    } else {
      const YJ<D>& Om = F[0];
      const YJ<D>& Th = F[NF > 1 ? 1 : 0];
      const YJ<D>& S = F[NF - 1];
      const Dl V1 = y[0] * opl + S.g[D - 1];
      const Dl V2 = y[D - 1] * opl + (-S.g[0]);
      R[0] = Om.v + V1 * Om.g[0] + V2 * Om.g[D - 1] - Th.g[0];
      R[NE > 1 ? 1 : 0] = (dconst(1.0) - lamd) * Th.v + V1 * Th.g[0] + V2 * Th.g[D - 1];
      R[NE > 2 ? 2 : 0] = S.h[0] + S.h[D == 1 ? 0 : 2] + Om.v;
    }
  } else if (kind == KIND_WALL) {
    R[0] = F[NF - 1].v;
  } else if (kind == KIND_NORM || kind == KIND_INF || kind == KIND_RELU) {
    // normalisation: Phi_A0 or its d/dy1 minus the target; decay: Phi_A0 itself; bound:
    // relu(s (Phi_A0 - b)), zero (with a zero derivative) while the bound holds
    Dl val = F[0].v, dy1 = F[0].g[0];
#pragma unroll
    for (int f = 1; f < NF; f++)   // constant register indices only
      if (f == A.nfield) {
        val = F[f].v;
        dy1 = F[f].g[0];
      }
    R[0] = (kind == KIND_NORM && A.nderiv) ? dy1 : val;
    R[0].v -= A.c_norm;
    if (kind == KIND_RELU) {
      R[0] = (double)A.rsign * R[0];
      if (!(R[0].v > 0.0)) R[0] = Dl{0.0, 0.0};
    }
  } else {  // KIND_NODE (CCF): g = y/u * NN * q^{-lambda}
    const YJ<D> Eg = envelope<D>(y, u, 1, dconst(-1.0) + 0.5 * (lamd * a));
    R[0] = Eg.v * nn[0][0];
    if (A.base) R[0] = Dl{A.base[pt] + A.eps * R[0].v, A.eps * R[0].d};
  }

}

}  // namespace
}  // namespace gn
