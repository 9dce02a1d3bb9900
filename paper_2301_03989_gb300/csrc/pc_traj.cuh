// Per-trajectory device functions shared by the round kernels (pc_sweep.cu) and
// the resident kernel (pc_resident.cuh): Kepler's equation, the segment schedule,
// the outputs of a finished trajectory, the warm-start interpolation.  They work
// on a Ctl (structure of arrays, leading dimension s.ld) in global memory (the
// round kernels) or in shared memory (the resident kernel).
#pragma once

#include "pc_device.cuh"

namespace pcx {
namespace {

// ---------------------------------------------------------------------------
// Keplerian two-body propagation by dt (warm start).  Kepler's equation in the
// eccentric-anomaly increment X over dt,
//   F(X) = X - (e cos E0) sin X + (e sin E0)(1 - cos X) - n dt = 0,
// with e cos E0 = 1 - r0/a and e sin E0 = r0.v0/sqrt(mu a), is solved by
// Halley's method (third order: X <- X - 2 F F' / (2 F'^2 - F F'')), kept
// inside the bracket [n dt - 2, n dt + 2] by bisection, from the first-order
// root X = n dt a/r0 (clamped into the bracket).  Once a step is below 1e-6
// the cubic convergence puts the next error below 1e-17 and the iteration
// stops after applying it.  The Lagrange coefficients then map (r0, v0) to
// (r, v).  The quantities that depend only on the start state are formed once
// per segment (kepler_consts, when the segment is scheduled) and shared by all
// its nodes.  A start state that is not a bound ellipse, or an iteration that
// does not settle, gives no warm start.
// ---------------------------------------------------------------------------
constexpr int kKepConsts = kKeplerConsts;
// c[0] = 1/a (<= 0: not elliptic), c[1] = a, c[2] = e cos E0, c[3] = e sin E0,
// c[4] = n, c[5] = (r0.v0/sqrt(mu)) sqrt(a), c[6] = a/r0,
// c[7] = a (r0.v0)/mu, c[8] = r0 sqrt(a)/sqrt(mu), c[9] = -sqrt(mu) sqrt(a) / r0, c[10] = r0
__device__ void kepler_consts(double mu, const double x0[6], double c[kKepConsts]) {
  const double r0 = sqrt(x0[0] * x0[0] + x0[1] * x0[1] + x0[2] * x0[2]);
  const double vv = x0[3] * x0[3] + x0[4] * x0[4] + x0[5] * x0[5];
  const double rv = x0[0] * x0[3] + x0[1] * x0[4] + x0[2] * x0[5];
  const double inv_a = 2.0 / r0 - vv / mu;
  c[0] = inv_a;
  for (int k = 1; k < kKepConsts; k++) c[k] = 0.0;
  if (!(inv_a > 0.0)) return;
  const double a = 1.0 / inv_a;
  const double sqrt_a = sqrt(a);
  const double sqrt_mu = sqrt(mu);
  c[1] = a;
  c[2] = 1.0 - r0 * inv_a;
  c[3] = rv / (sqrt_mu * sqrt_a);
  c[4] = sqrt_mu * inv_a / sqrt_a;  // sqrt(mu / a^3)
  c[5] = rv / sqrt_mu * sqrt_a;
  c[6] = a / r0;
  c[7] = a * rv / mu;
  c[8] = r0 * sqrt_a / sqrt_mu;
  c[9] = -sqrt_mu * sqrt_a / r0;
  c[10] = r0;
}

// The iteration runs first in FP32 (same steps and bracket, to a step below
// 2e-6), which leaves the FP64 iteration one Halley step from that start in
// the usual case; the sine and cosine at the root then follow from those at
// the last iterate by the angle-addition formulas with the step's Taylor
// series (|step| <= 1e-5: the dropped terms are below 1e-32).  Only when the
// FP32 start is poor does the FP64 iteration take more steps.  An iterate
// with F = 0 is the root, and a Halley step onto the bracket's end is kept:
// at the root rounding can put the step exactly there, and bisecting from
// it would cost some thirty steps.
__device__ bool kepler_solve(const double c[kKepConsts], const double x0[6], double dt, double out[6]) {
  if (!(c[0] > 0.0)) return false;
  const double a = c[1], ecE = c[2], esE = c[3];
  const double M = c[4] * dt;
  double lo = M - 2.0, hi = M + 2.0;
  double X = fmin(fmax(M * c[6], lo + 0.5), hi - 0.5);
  {
    const float Mf = (float)M, ef = (float)ecE, sf = (float)esE;
    float lof = (float)lo, hif = (float)hi, Xf = (float)X;
    for (int it = 0; it < 32; it++) {
      float sXf, cXf;
      sincosf(Xf, &sXf, &cXf);
      const float F = Xf - ef * sXf + sf * (1.0f - cXf) - Mf;
      if (F == 0.0f) break;
      if (F > 0.0f) hif = Xf; else lof = Xf;
      const float d1 = 1.0f - ef * cXf + sf * sXf;
      const float d2 = ef * sXf + sf * cXf;
      float Xn = Xf - 2.0f * F * d1 / (2.0f * d1 * d1 - F * d2);
      if (!(Xn >= lof && Xn <= hif)) Xn = 0.5f * (lof + hif);
      const float step = fabsf(Xn - Xf);
      Xf = Xn;
      if (!(step > 2e-6f * (1.0f + fabsf(Xf)))) break;
    }
    if (isfinite(Xf)) X = fmin(fmax((double)Xf, lo), hi);
  }
  bool ok = false;
  double sX = 0.0, cX = 1.0, dl = 0.0;  // sine, cosine at the last evaluated iterate, step from it
  bool rotate = false;
  for (int it = 0; it < 64; it++) {
    sincos(X, &sX, &cX);
    const double F = X - ecE * sX + esE * (1.0 - cX) - M;
    if (F == 0.0) {
      ok = rotate = true;  // dl = 0: sX, cX are the root's
      dl = 0.0;
      break;
    }
    if (F > 0.0) hi = X; else lo = X;
    const double d1 = 1.0 - ecE * cX + esE * sX;
    const double d2 = ecE * sX + esE * cX;
    double Xn = X - 2.0 * F * d1 / (2.0 * d1 * d1 - F * d2);
    const bool halley = Xn >= lo && Xn <= hi;
    if (!halley) Xn = 0.5 * (lo + hi);
    dl = Xn - X;
    const double step = fabs(dl);
    X = Xn;
    if ((halley && step <= 1e-6 * (1.0 + fabs(X))) || step <= 1e-15 * (1.0 + fabs(X))) {
      ok = true;
      rotate = step <= 1e-5;
      break;
    }
  }
  if (!ok) return false;
  if (rotate) {
    // sin, cos at X = (previous iterate) + dl by angle addition
    const double d2 = dl * dl;
    const double sd = dl * (1.0 - d2 * (1.0 / 6.0) * (1.0 - d2 * 0.05));
    const double cd = 1.0 - d2 * 0.5 * (1.0 - d2 * (1.0 / 12.0));
    const double s1 = sX * cd + cX * sd, c1 = cX * cd - sX * sd;
    sX = s1;
    cX = c1;
  } else {
    sincos(X, &sX, &cX);
  }
  const double omc = 1.0 - cX;
  const double r = a + (c[10] - a) * cX + c[5] * sX;
  const double f = 1.0 - c[6] * omc;
  const double g = c[7] * omc + c[8] * sX;
  const double fd = c[9] / r * sX;
  const double gd = 1.0 - a / r * omc;
  for (int q = 0; q < 3; q++) {
    out[q] = f * x0[q] + g * x0[3 + q];
    out[3 + q] = fd * x0[q] + gd * x0[3 + q];
  }
  return true;
}

__device__ bool kepler_dt(double mu, const double x0[6], double dt, double out[6]) {
  double c[kKepConsts];
  kepler_consts(mu, x0, c);
  return kepler_solve(c, x0, dt, out);
}

// ---------------------------------------------------------------------------
// Segment schedule.  The arc [t0, tf] is measured in units u = hbase / 2^D; a
// segment at depth d starting at unit p spans 2^(D-d) units and is clipped to
// end exactly at tf.  Products and sums are rounded one at a time (no fused
// multiply-add) so every trajectory's segment bounds and node times are the
// exactly rounded values of these formulas.
// ---------------------------------------------------------------------------
struct SegmentBounds {
  double ta, tb;
  int last;
};
__device__ SegmentBounds segment_bounds(int D, double hbase, int depth, long long p, double t0, double tf, double sgn,
                                        double total) {
  const double u = scalbn(hbase, -D);
  const long long L = 1LL << (D - depth);
  SegmentBounds b;
  b.ta = dadd(t0, dmul(sgn, dmul((double)p, u)));
  b.last = dmul((double)(p + L), u) >= total;
  b.tb = b.last ? tf : dadd(t0, dmul(sgn, dmul((double)(p + L), u)));
  return b;
}
__device__ void schedule(const Sweep &s, const Ctl &c, int m) {
  const SegmentBounds b = segment_bounds(s.max_depth, c.hbase[m], c.depth[m], c.p[m], c.t0[m], c.tf[m], c.sgn[m],
                                         c.total[m]);
  const double ta = b.ta, tb = b.tb;
  c.ta[m] = ta;
  c.tb[m] = tb;
  if (s.warm) {
    double x0[6], kc[kKepConsts];
    for (int q = 0; q < 6; q++) x0[q] = c.x[q * s.ld + m];
    kepler_consts(s.mu_c, x0, kc);
    for (int q = 0; q < kKepConsts; q++) c.kc[q * s.ld + m] = kc[q];
  }
  c.w1[m] = dmul(0.5, dadd(tb, ta));
  c.w2[m] = dmul(0.5, dsub(tb, ta));
  c.last[m] = b.last;
  c.need_setup[m] = 1;
  c.seg_sweeps[m] = 0;
  c.nstall[m] = 0;
  c.ncorr[m] = 0;
  c.e_best[m] = __longlong_as_double(0x7FF0000000000000LL);  // +inf
  c.phase[m] = s.mixed ? PH_ITER32 : PH_ITER;
}

// Final outputs of a trajectory, written when it finishes.
__device__ __forceinline__ void write_outputs(const Sweep &s, const Ctl &c, int m) {
  const long long i = s.io_off + c.ic[m];
  for (int q = 0; q < 6; q++) s.xf[q * s.io_ld + i] = c.x[q * s.ld + m];
  if (s.status) s.status[i] = c.status[m];
  if (s.iters) s.iters[i] = c.sweeps[m];
  if (s.nseg) s.nseg[i] = c.nseg[m];
}

// Trajectory i of the call starts in slot m: its arc, its base segment length and
// its first segment.  Returns whether it has work to do; one that has none (a
// non-finite state, an arc outside the ephemeris table, a zero-length arc)
// writes its outputs at once, and *refused says whether it counts as stopped early.
__device__ bool init_trajectory(const Sweep &s, const Ctl &c, const Model &md, const double *__restrict__ x0, int m,
                                long long i, bool *refused) {
  const int ld = s.ld;
  double x[6];
  bool finite = true;
  for (int q = 0; q < 6; q++) {
    x[q] = x0[q * s.io_ld + s.io_off + i];
    c.x[q * ld + m] = x[q];
    finite = finite && isfinite(x[q]);
  }
  const double t0 = s.t0a ? s.t0a[s.io_off + i] : s.t0s;
  const double tf = s.tfa ? s.tfa[s.io_off + i] : s.tfs;
  const int segs = s.sega ? s.sega[s.io_off + i] : s.segments;
  const double total = fabs(dsub(tf, t0));
  c.t0[m] = t0;
  c.tf[m] = tf;
  c.total[m] = total;
  c.sgn[m] = (tf >= t0) ? 1.0 : -1.0;
  // an arc outside the ephemeris table, or a bad segment count, is refused
  bool arc_ok = isfinite(t0) && isfinite(tf) && segs >= 1;
  if (md.B > 0) {
    const double lo = md.t_begin, hi = dadd(md.t_begin, dmul(md.granule, (double)md.n_gr));
    arc_ok = arc_ok && fmin(t0, tf) >= lo && fmax(t0, tf) <= hi;
  }
  double h = total / (double)(segs >= 1 ? segs : 1);
  if (s.seg_mode == 1 && finite) {
    const double r0 = sqrt(dadd(dadd(dmul(x[0], x[0]), dmul(x[1], x[1])), dmul(x[2], x[2])));
    const double v2 = dadd(dadd(dmul(x[3], x[3]), dmul(x[4], x[4])), dmul(x[5], x[5]));
    const double alpha = dsub(2.0 / r0, v2 / md.mu_c);
    if (alpha > 0.0) {
      const double a = 1.0 / alpha;
      const double twopi = 6.283185307179586;  // 2 * M_PI rounded
      h = dmul(twopi, sqrt(dmul(dmul(a, a), a) / md.mu_c)) / (double)(segs >= 1 ? segs : 1);
    }
  }
  c.ic[m] = (int)i;
  c.hbase[m] = h;
  c.p[m] = 0;
  c.depth[m] = 0;
  c.status[m] = (finite ? 0 : PC_IC_NONFINITE) | (arc_ok ? 0 : PC_IC_OUT_OF_RANGE);
  c.sweeps[m] = 0;
  c.nseg[m] = 0;
  c.err[m] = 0ULL;
  c.err32[m] = 0u;
  c.need_setup[m] = 0;
  *refused = !finite || !arc_ok;
  if (!finite || !arc_ok || !(total > 0.0)) {
    c.phase[m] = PH_DONE;
    write_outputs(s, c, m);
    return false;
  }
  schedule(s, c, m);
  return true;
}

// Outcome of an FP64 sweep whose change is e: the oracle's rules in the oracle's
// order (blow-up, tolerance, stall, cap), before the resolution test.
__device__ int sweep_outcome(const Sweep &s, const Ctl &c, int m, double e) {
  c.sweeps[m] += 1;
  const int ss = ++c.seg_sweeps[m];
  if (!(e <= s.div_limit)) return SEG_FAIL_DIV;
  if (e < s.tol) return SEG_OK;
  if (e < c.e_best[m]) {
    c.e_best[m] = e;
    c.nstall[m] = 0;
  } else {
    c.nstall[m] += 1;
  }
  if (c.nstall[m] >= s.stall_sweeps && c.e_best[m] < s.stall_factor * s.tol) return SEG_STALLED;
  if (ss >= s.max_iters) return SEG_FAIL_CAP;
  return SEG_CONTINUE;
}

// Ends a segment attempt: accepted (stitch, advance, grow) or halved, and the
// trajectory's next segment scheduled.  Ylast points at component 0 of the last
// node of the attempt's iterate (components ys apart).  *tape_k is the
// segment's tape record when one is wanted (the caller copies the nodes), else -1.
enum : int { ADV_SEGMENT = 0, ADV_DONE = 1, ADV_STOPPED = 2 };
__device__ int end_attempt(const Sweep &s, const Ctl &c, int m, int out, const double *Ylast, size_t ys,
                           int *tape_k) {
  const int D = s.max_depth, ld = s.ld;
  *tape_k = -1;
  bool accept = (out == SEG_OK || out == SEG_STALLED);
  if (out == SEG_FAIL_TRUNC && c.depth[m] >= D) {
    accept = true;
    c.status[m] |= PC_IC_UNRESOLVED;
  }
  if (!accept) {
    c.depth[m] += 1;
    if (c.depth[m] > D) {
      c.status[m] |= (out == SEG_FAIL_DIV) ? PC_IC_NONFINITE : PC_IC_NOT_CONVERGED;
      c.phase[m] = PH_DONE;
      write_outputs(s, c, m);
      return ADV_STOPPED;
    }
    schedule(s, c, m);
    return ADV_SEGMENT;
  }
  if (out == SEG_STALLED) c.status[m] |= PC_IC_STALLED;
  const int k = c.nseg[m];
  if (s.ckpt && k < s.max_ckpt) {
    double *ck = s.ckpt + ((size_t)(s.io_off + c.ic[m]) * s.max_ckpt + k) * 7;
    ck[0] = c.ta[m];
    for (int q = 0; q < 6; q++) ck[1 + q] = c.x[q * ld + m];
  }
  if (s.tape && k < s.tape_seg) {
    double *rec = s.tape + ((size_t)(s.io_off + c.ic[m]) * s.tape_seg + k) * (size_t)tape_rec(s.n);
    rec[0] = c.ta[m];
    rec[1] = c.tb[m];
    *tape_k = k;
  }
  for (int q = 0; q < 6; q++) c.x[q * ld + m] = Ylast[(size_t)q * ys];
  c.nseg[m] = k + 1;
  c.p[m] += 1LL << (D - c.depth[m]);
  if (c.last[m]) {
    c.phase[m] = PH_DONE;
    write_outputs(s, c, m);
    return ADV_DONE;
  }
  if (c.depth[m] > 0) c.depth[m] -= 1;
  schedule(s, c, m);
  return ADV_SEGMENT;
}

// Indirect (frame) term of body b: the central body's own acceleration
// mu_b r_b/|r_b|^3, summed over bodies; it depends on the node time only.
__device__ __forceinline__ void add_indirect(const Model &md, int b, const double r[3], double ind[3]) {
  const double d2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
  const double rs = rsqrt(d2);
  const double k = md.mu[b] * rs * rs * rs;
  for (int ax = 0; ax < 3; ax++) ind[ax] = fma(k, r[ax], ind[ax]);
}

// The warm start of a segment is interpolated from 17 nodes when the segment
// spans at most 1.5 rad of mean anomaly (a degree-16 Chebyshev interpolant of
// the Kepler arc is then exact to rounding); longer segments, and arcs with
// no mean motion, are solved at every node.
constexpr double kInterpMaxAnomaly = 1.5;
__device__ __forceinline__ bool kepler_interpolated(const Sweep &s, const Ctl &c, int m) {
  return s.kep_stride > 0 && fabs(c.kc[4 * s.ld + m] * (c.tb[m] - c.ta[m])) <= kInterpMaxAnomaly &&
         c.kc[(size_t)0 * s.ld + m] > 0.0;
}

// Warm-start deviations at the 17 interpolation nodes: y17[k][q][e] (leading
// dimension ldk over entries e), FP32 pairs (hi, lo) of the solution minus the
// start state.
//
// The warm start at node j from the 17 solved nodes of entry e, interpolated in
// compensated FP32 arithmetic (each product split exactly by an FMA, each sum by
// Knuth's TwoSum, the remainders and the lo parts summed beside): about 1e-13 of
// the deviation, as an FP64 sum, at the cost of FP32 operations.  The FP32 phase
// relies on this accuracy: it treats the warm start as an exact Kepler arc.
// False when one of the 17 solves did not settle (NaN).
__device__ __forceinline__ bool warm_interpolate(const Sweep &s, const float2 *y17, int ldk, int j, int e,
                                                 const double x0[6], double y[6]) {
  float sh[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, sl[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  bool fin = true;
  const float *Lh = s.Lint + (size_t)j * kKepNodes;
  const float *Ll = s.Lint + ((size_t)s.n + j) * kKepNodes;
  for (int k = 1; k < kKepNodes; k++) {
    const float lh = Lh[k], ll = Ll[k];
#pragma unroll
    for (int q = 0; q < 6; q++) {
      const float2 dd = y17[((size_t)k * 6 + q) * ldk + e];
      const float dh = dd.x, dl = dd.y;
      fin = fin && isfinite(dh);
      const float pr = __fmul_rn(lh, dh);
      const float pe = __fmaf_rn(lh, dh, -pr);  // lh dh - pr, exactly
      const float sm = __fadd_rn(sh[q], pr);
      const float bv = __fsub_rn(sm, sh[q]);
      const float se = __fadd_rn(__fsub_rn(sh[q], __fsub_rn(sm, bv)), __fsub_rn(pr, bv));  // sh + pr - sm
      sh[q] = sm;
      sl[q] = __fadd_rn(sl[q], __fadd_rn(__fadd_rn(se, pe), __fmaf_rn(lh, dl, __fmul_rn(ll, dh))));
    }
  }
  if (fin)
    for (int q = 0; q < 6; q++) y[q] = x0[q] + ((double)sh[q] + (double)sl[q]);
  return fin;
}

// One of the 17 solves (node index k) of the segment in slot m: the deviation from the
// start state, d[6]; false where the iteration does not settle.  Node 0 is the start
// state.
__device__ __forceinline__ bool warm_deviation(const Sweep &s, const Ctl &c, const double *__restrict__ tau, int k,
                                               int m, double d[6]) {
  const int ld = s.ld, j = k * s.kep_stride;
  double x0[6], y[6];
  for (int q = 0; q < 6; q++) x0[q] = y[q] = c.x[q * ld + m];
  bool ok = true;
  if (j > 0) {
    double kc[kKepConsts];
    for (int q = 0; q < kKepConsts; q++) kc[q] = c.kc[q * ld + m];
    const double t = dadd(c.w1[m], dmul(c.w2[m], tau[j]));
    ok = kepler_solve(kc, x0, dsub(t, c.ta[m]), y);
  }
  for (int q = 0; q < 6; q++) d[q] = y[q] - x0[q];
  return ok;
}
// Stored for entry e as FP32 pairs (the rounds); NaN where the iteration does not settle.
__device__ __forceinline__ void warm_solve(const Sweep &s, const Ctl &c, const double *__restrict__ tau, int k, int m,
                                           float2 *y17, int ldk, int e) {
  double d[6];
  const bool ok = warm_deviation(s, c, tau, k, m, d);
  for (int q = 0; q < 6; q++) {
    const float hi = ok ? (float)d[q] : __int_as_float(0x7FC00000);
    y17[((size_t)k * 6 + q) * ldk + e] = make_float2(hi, ok ? (float)(d[q] - (double)hi) : hi);
  }
}

}  // namespace
}  // namespace pcx
