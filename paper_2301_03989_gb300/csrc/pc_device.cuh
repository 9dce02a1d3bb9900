// Device helpers shared by the sweep kernels (pc_sweep.cu) and the adjoint
// kernels (pc_adjoint.cu): exactly rounded FP64 operations, NaN-propagating
// maxima, the ephemeris evaluation and the FP64 tensor-core MMA.
#pragma once

#include "pc_internal.h"

namespace pcx {
namespace {

__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dsub(double a, double b) { return __dsub_rn(a, b); }

// NaN-propagating maximum of non-negative values.
__device__ __forceinline__ double nanmax(double a, double b) { return (b > a || b != b) ? b : a; }
__device__ __forceinline__ float nanmaxf(float a, float b) { return (b > a || b != b) ? b : a; }

// Non-negative doubles / floats order like their bit patterns; NaN maps to the largest.
__device__ __forceinline__ unsigned long long err_bits(double e) {
  if (e != e) return 0x7FF8000000000000ULL;
  return (unsigned long long)__double_as_longlong(e);
}
__device__ __forceinline__ unsigned err_bits32(float e) {
  if (e != e) return 0x7FC00000u;
  return __float_as_uint(e);
}

// ---------------------------------------------------------------------------
// Ephemeris: the table's Chebyshev series r = sum_k c_k T_k(sigma) at the
// granule holding t.  T_0 = 1, T_1 = sigma, T_{k+1} = fma(2 sigma, T_k, -T_{k-1})
// are formed once per time and shared by every body and axis; each coordinate
// is then summed from the top degree down with one fused multiply-add per
// term.  This differs from Clenshaw's recurrence only in rounding: both agree
// to a few ulps of sum_k |c_k|.
// ---------------------------------------------------------------------------
struct EphemLoc {
  int g;
  double sig;
};

__device__ __forceinline__ EphemLoc ephem_locate(const Model &md, double t) {
  int g = (int)floor((t - md.t_begin) / md.granule);
  g = g < 0 ? 0 : (g > md.n_gr - 1 ? md.n_gr - 1 : g);
  const double tg = dadd(md.t_begin, dmul((double)g, md.granule));
  return {g, dsub(dmul(2.0, dsub(t, tg)) / md.granule, 1.0)};
}

constexpr int kEphemRegCoefs = 16;  // degrees up to 15 keep T_k in registers
constexpr int kEphemMaxCoefs = 64;  // degrees up to 63

// Calls out(b, r) for every body b in order with its position r[3].
template <class Out>
__device__ __forceinline__ void ephem_all(const Model &md, EphemLoc L, Out out);

// Same for the bodies b_lo <= b < b_hi.
template <class Out>
__device__ __forceinline__ void ephem_range(const Model &md, EphemLoc L, int b_lo, int b_hi, Out out) {
  Model sub = md;
  sub.coef = md.coef + (size_t)b_lo * md.n_gr * 3 * (md.deg + 1);
  sub.B = b_hi - b_lo;
  ephem_all(sub, L, [&](int b, const double r[3]) { out(b_lo + b, r); });
}

template <class Out>
__device__ __forceinline__ void ephem_all(const Model &md, EphemLoc L, Out out) {
  const int nc = md.deg + 1;
  const double s2 = 2.0 * L.sig;
  if (nc <= kEphemRegCoefs) {
    double T[kEphemRegCoefs];
    T[0] = 1.0;
    T[1] = L.sig;
#pragma unroll
    for (int k = 2; k < kEphemRegCoefs; k++) T[k] = fma(s2, T[k - 1], -T[k - 2]);
    for (int b = 0; b < md.B; b++) {
      const double *cf = md.coef + ((size_t)b * md.n_gr + L.g) * 3 * nc;
      double r[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int k = kEphemRegCoefs - 1; k >= 0; k--)
        if (k < nc)
#pragma unroll
          for (int ax = 0; ax < 3; ax++) r[ax] = fma(cf[ax * nc + k], T[k], r[ax]);
      out(b, r);
    }
  } else {
    double T[kEphemMaxCoefs];
    const int m = nc < kEphemMaxCoefs ? nc : kEphemMaxCoefs;
    T[0] = 1.0;
    T[1] = L.sig;
    for (int k = 2; k < m; k++) T[k] = fma(s2, T[k - 1], -T[k - 2]);
    for (int b = 0; b < md.B; b++) {
      const double *cf = md.coef + ((size_t)b * md.n_gr + L.g) * 3 * nc;
      double r[3] = {0.0, 0.0, 0.0};
      for (int k = m - 1; k >= 0; k--)
        for (int ax = 0; ax < 3; ax++) r[ax] = fma(cf[ax * nc + k], T[k], r[ax]);
      out(b, r);
    }
  }
}

// One body's position (same arithmetic as ephem_all).
__device__ __forceinline__ void ephem_body(const Model &md, EphemLoc L, int body, double r[3]) {
  Model one = md;
  one.coef = md.coef + (size_t)body * md.n_gr * 3 * (md.deg + 1);
  one.B = 1;
  ephem_all(one, L, [&](int, const double p[3]) {
    r[0] = p[0];
    r[1] = p[1];
    r[2] = p[2];
  });
}

// Body velocities: the time derivative of the table's series,
// (2 / granule) sum_{k>=1} c_k k U_{k-1}(sigma), with the Chebyshev
// polynomials of the second kind U_0 = 1, U_1 = 2 sigma, U_{k+1} = 2 sigma
// U_k - U_{k-1} formed once per time; out(b, v) for every body.
template <class Out>
__device__ __forceinline__ void ephem_vel_all(const Model &md, EphemLoc L, Out out) {
  const int nc = md.deg + 1;
  const int m = nc < kEphemMaxCoefs ? nc : kEphemMaxCoefs;
  double U[kEphemMaxCoefs];
  U[0] = 1.0;
  if (m > 1) U[1] = 2.0 * L.sig;
  for (int k = 2; k < m; k++) U[k] = fma(2.0 * L.sig, U[k - 1], -U[k - 2]);
  const double sc = 2.0 / md.granule;
  for (int b = 0; b < md.B; b++) {
    const double *cf = md.coef + ((size_t)b * md.n_gr + L.g) * 3 * nc;
    double v[3] = {0.0, 0.0, 0.0};
    for (int k = m - 1; k >= 1; k--)
      for (int ax = 0; ax < 3; ax++) v[ax] = fma(cf[ax * nc + k] * (double)k, U[k - 1], v[ax]);
    for (int ax = 0; ax < 3; ax++) v[ax] *= sc;
    out(b, v);
  }
}

// Einstein-Infeld-Hoffmann data of the bodies at one time, from their
// heliocentric positions rb and velocities vb [B][3] (the central body at the
// origin): X[7j + 0..2] the barycentric velocity V of body j (0 central, 1..B the
// table's), X[7j + 3..5] its Newtonian acceleration from the other bodies and
// X[7j + 6] = 2 V.V - (its Newtonian potential from them).  Each pair is formed
// once for both of its bodies.
__device__ __noinline__ void eih_bodies(const Model &md, const double *rb, const double *vb, double *X) {
  const int B = md.B, nb = B + 1;
  double msum = md.mu_c, vs[3] = {0.0, 0.0, 0.0};
  for (int b = 0; b < B; b++) {
    msum += md.mu[b];
    for (int q = 0; q < 3; q++) vs[q] -= md.mu[b] * vb[3 * b + q];
  }
  for (int q = 0; q < 3; q++) vs[q] /= msum;
  for (int j = 0; j < nb; j++) {
    double vv = 0.0;
    for (int q = 0; q < 3; q++) {
      const double v = (j ? vb[3 * (j - 1) + q] : 0.0) + vs[q];
      X[7 * j + q] = v;
      X[7 * j + 3 + q] = 0.0;
      vv = fma(v, v, vv);
    }
    X[7 * j + 6] = 2.0 * vv;
  }
  for (int j = 0; j < nb; j++) {
    const double mj = j ? md.mu[j - 1] : md.mu_c;
    for (int k = j + 1; k < nb; k++) {
      const double mk = md.mu[k - 1];
      double d[3];
      for (int q = 0; q < 3; q++) d[q] = rb[3 * (k - 1) + q] - (j ? rb[3 * (j - 1) + q] : 0.0);
      const double ir = rsqrt(fma(d[2], d[2], fma(d[1], d[1], d[0] * d[0])));
      const double i3 = ir * ir * ir;
      X[7 * j + 6] = fma(-mk, ir, X[7 * j + 6]);
      X[7 * k + 6] = fma(-mj, ir, X[7 * k + 6]);
      for (int q = 0; q < 3; q++) {
        X[7 * j + 3 + q] = fma(mk * i3, d[q], X[7 * j + 3 + q]);
        X[7 * k + 3 + q] = fma(-mj * i3, d[q], X[7 * k + 3 + q]);
      }
    }
  }
}

// Newtonian acceleration plus the 1/c^2 terms of the EIH equations for a massless
// particle at the heliocentric state (r, v) among the central body and the table's
// bodies (positions Eb[(3b + axis) * es], summed indirect term Ai[axis * es], EIH
// data Xb[f * es] as eih_bodies lays it out), velocities in the barycentric frame:
//   g - (indirect term) + [ (W.W - 4 phi) g
//     + sum_j k_j (S_j - 4 W.V_j - 3/2 (d_j.V_j)^2/r_j^2 + 1/2 d_j.A_j) d_j
//     + sum_j k_j (3 d_j.V_j - 4 d_j.W) (W - V_j) + 7/2 sum_j mu_j A_j / r_j ] / c^2,
// d_j = P_j - r, k_j = mu_j/r_j^3, g = sum_j k_j d_j, phi = sum_j mu_j/r_j,
// W = v + V_central, S_j = 2 V_j.V_j - Phi_j.  The terms common to all bodies come
// out of the sum, so one pass with one reciprocal square root and no division per
// body gives both parts (about 50 FP64 operations a body; as two passes with
// divisions, beside a Newtonian one, it was over 150).  NEWTON false: the 1/c^2
// part alone.
template <bool NEWTON>
__device__ __forceinline__ void eih_accel(const Model &md, const double *Eb, const double *Ai, const double *Xb,
                                          size_t es, const double r[3], const double v[3], double a[3]) {
  const int B = md.B;
  const double W[3] = {v[0] + Xb[0], v[1] + Xb[es], v[2] + Xb[2 * es]};
  double g[3] = {0.0, 0.0, 0.0}, h[3] = {0.0, 0.0, 0.0}, phi = 0.0, us = 0.0;
  for (int j = 0; j <= B; j++) {
    double d[3], V[3], A[3];
    for (int q = 0; q < 3; q++) {
      d[q] = (j ? Eb[(size_t)(3 * (j - 1) + q) * es] : 0.0) - r[q];
      V[q] = Xb[(size_t)(7 * j + q) * es];
      A[q] = Xb[(size_t)(7 * j + 3 + q) * es];
    }
    const double S = Xb[(size_t)(7 * j + 6) * es];
    const double ir = rsqrt(fma(d[2], d[2], fma(d[1], d[1], d[0] * d[0])));
    const double k1 = (j ? md.mu[j - 1] : md.mu_c) * ir, k3 = k1 * ir * ir;
    const double wv = fma(W[2], V[2], fma(W[1], V[1], W[0] * V[0]));
    const double dv = fma(d[2], V[2], fma(d[1], V[1], d[0] * V[0]));
    const double dw = fma(d[2], W[2], fma(d[1], W[1], d[0] * W[0]));
    const double da = fma(d[2], A[2], fma(d[1], A[1], d[0] * A[0]));
    const double nv = dv * ir;
    const double b = k3 * fma(0.5, da, fma(-1.5 * nv, nv, fma(-4.0, wv, S)));
    const double u = k3 * fma(3.0, dv, -4.0 * dw);
    const double ka = 3.5 * k1;
    phi += k1;
    us += u;
    for (int q = 0; q < 3; q++) {
      g[q] = fma(k3, d[q], g[q]);
      h[q] = fma(b, d[q], fma(-u, V[q], fma(ka, A[q], h[q])));
    }
  }
  const double ww = fma(W[2], W[2], fma(W[1], W[1], W[0] * W[0])), f = fma(-4.0, phi, ww);
  const double ic2 = 1.0 / (md.c_light * md.c_light);
  for (int q = 0; q < 3; q++) {
    const double rel = fma(f, g[q], fma(us, W[q], h[q]));
    a[q] = NEWTON ? fma(ic2, rel, md.indirect ? g[q] - Ai[(size_t)q * es] : g[q]) : ic2 * rel;
  }
}

// FP64 tensor-core MMA, mma.sync m16n8k4 .f64 (PTX ISA).  Fragment layouts,
// with g = lane/4 and t = lane%4:  A: a0 = A[g][t], a1 = A[g+8][t];
// B: b0 = B[t][g];  C/D: d0,d1 = C[g][2t..2t+1], d2,d3 = C[g+8][2t..2t+1].
__device__ __forceinline__ void dmma16x8x4(double (&d)[4], double a0, double a1, double b0) {
  asm volatile(
      "mma.sync.aligned.m16n8k4.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};\n"
      : "+d"(d[0]), "+d"(d[1]), "+d"(d[2]), "+d"(d[3])
      : "d"(a0), "d"(a1), "d"(b0));
}

}  // namespace
}  // namespace pcx
