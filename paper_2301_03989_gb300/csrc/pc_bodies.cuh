// What the force at a node needs of the bodies at the node's time, in the form that
// tile_accel (pc_tile.cuh) and eih_accel (pc_device.cuh) read it.  Shared by the resident
// kernel (pc_resident.cuh), which forms it once per node of a segment, and by the force as
// an entry point of its own (pc_split.cu).
#pragma once

#include "pc_tile.cuh"
#include "pc_traj.cuh"

namespace pcx {
namespace {

// Body data at one time: positions [3B], summed indirect term [3] (NaN where it is not formed,
// see indirect_term), then the bodies' EIH data or (Newtonian force) the positions and minus
// the indirect term as float pairs.
__host__ __device__ inline size_t res_bodies(int B, bool eih) { return 3 * B + 3 + (eih ? eih_stride(B) : 3 * B + 3); }

// Positions of bodies b0 .. b1 - 1, in FP64 and as pairs.
constexpr int kBodyChunk = 3;  // bodies an ephemeris item evaluates: more items than threads even for one segment
__device__ __forceinline__ void body_positions(const Model &md, EphemLoc L, int b0, int b1, double *out) {
  float2 *pair = reinterpret_cast<float2 *>(out + 3 * md.B + 3);
  ephem_range(md, L, b0, b1, [&](int b, const double r[3]) {
    for (int ax = 0; ax < 3; ax++) {
      out[3 * b + ax] = r[ax];
      pair[3 * b + ax] = split_pair(r[ax]);
    }
  });
  if (b0 == 0 && !md.indirect)
    for (int ax = 0; ax < 3; ax++) {
      out[3 * md.B + ax] = 0.0;
      pair[3 * md.B + ax] = make_float2(0.0f, 0.0f);
    }
}
// The indirect term sum_b mu_b r_b/|r_b|^3 from the positions: minus it as a pair, summed in
// pairs (off by up to 3e-14 of itself), for the nodes where that is enough, and in FP64 for the
// others (tile_accel tells them apart).  The FP64 sum takes 12 FP64 operations a body.  Where
// c2, the square of the central attraction at the segment's start, says that hardly a node
// will want it (the term is below 2^-13 of the central one: heliocentric arcs inside Jupiter's
// orbit), NaN stands in its place and a node that does forms it: 2048 flybys among nine
// bodies 43.9 ms, with the FP64 sum for every node 46.2, with pairs alone 43.0.  No result
// depends on c2.
__device__ __forceinline__ void indirect_term(const Model &md, double *data, float c2) {
  float2 *pair = reinterpret_cast<float2 *>(data + 3 * md.B + 3);
  float sh[3] = {0.0f, 0.0f, 0.0f}, sl[3] = {0.0f, 0.0f, 0.0f};
  bool fits = true;  // the floats' range holds every body's term
  for (int b = 0; b < md.B; b++) {
    float h[3], l[3], Dh, kh, kl;
#pragma unroll
    for (int q = 0; q < 3; q++) {
      const float2 p = pair[3 * b + q];
      h[q] = __fadd_rn(p.x, p.y);
      l[q] = __fsub_rn(p.y, __fsub_rn(h[q], p.x));
    }
    pair_cube(h, l, md.mu2[b], Dh, kh, kl);
    fits = fits && (kh > 1e-30f || md.mu[b] == 0.0);
#pragma unroll
    for (int q = 0; q < 3; q++) {
      const float v = kh * h[q], w = __fmaf_rn(kl, h[q], __fmaf_rn(kh, l[q], __fmaf_rn(kh, h[q], -v)));
      float er;
      sh[q] = two_sum(sh[q], v, er);
      sl[q] += er + w;
    }
  }
  double3 sum = make_double3(__longlong_as_double(0x7FF8000000000000LL), 0.0, 0.0);
  if (!fits || !attraction_small(sh, c2, 67108864.0f)) sum = indirect_sum(md, data);
  const double s[3] = {sum.x, sum.y, sum.z};
#pragma unroll
  for (int q = 0; q < 3; q++) {
    data[3 * md.B + q] = s[q];
    pair[3 * md.B + q] = fits ? make_float2(-sh[q], -sl[q]) : split_pair(-s[q]);
  }
}
// Square of the central attraction at r.
__device__ __forceinline__ float central_square(const Model &md, const double r[3]) {
  const float x = trunc_float(r[0]), y = trunc_float(r[1]), z = trunc_float(r[2]);
  const float a = __fdividef(trunc_float(md.mu_c), x * x + y * y + z * z);
  return a * a;
}
// The data at one time by one thread; c2: see indirect_term (0: where they are used is not known).
template <bool EIH>
__device__ __forceinline__ void body_data(const Model &md, EphemLoc L, double *out, float c2 = 0.0f) {
  const int B = md.B;
  if (!EIH) {
    body_positions(md, L, 0, B, out);
    if (md.indirect) indirect_term(md, out, c2);
    return;
  }
  double rb[kMaxBodies * 3], vb[kMaxBodies * 3], X[7 * (kMaxBodies + 1)], ind[3] = {0.0, 0.0, 0.0};
  ephem_all(md, L, [&](int b, const double r[3]) {
    if (md.indirect) add_indirect(md, b, r, ind);
    for (int ax = 0; ax < 3; ax++) out[3 * b + ax] = rb[3 * b + ax] = r[ax];
  });
  ephem_vel_all(md, L, [&](int b, const double v[3]) {
    for (int ax = 0; ax < 3; ax++) vb[3 * b + ax] = v[ax];
  });
  eih_bodies(md, rb, vb, X);
  for (int ax = 0; ax < 3; ax++) out[3 * B + ax] = ind[ax];
  for (int f = 0; f < eih_stride(B); f++) out[3 * B + 3 + f] = X[f];
}

}  // namespace
}  // namespace pcx
