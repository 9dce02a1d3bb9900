// What the force at a node needs of the bodies at the node's time, in the form that
// tile_accel (pc_tile.cuh) and eih_accel (pc_device.cuh) read it.  Shared by the resident
// kernel (pc_resident.cuh), which forms it once per node of a segment, and by the force as
// an entry point of its own (pc_split.cu).
#pragma once

#include "pc_tile.cuh"
#include "pc_traj.cuh"

namespace pcx {
namespace {

// Body data at one time: positions [3B], summed indirect term [3], then the bodies' EIH
// data or (Newtonian force) the positions and minus the indirect term as float pairs.
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
// The indirect term sum_b mu_b r_b/|r_b|^3 from the position pairs, in pairs: it is below
// 2^-15 of a planetary node's central attraction, 48 bits of it are under that one's
// FP64 rounding.
__device__ __forceinline__ void indirect_pairs(const Model &md, double *data) {
  float2 *pair = reinterpret_cast<float2 *>(data + 3 * md.B + 3);
  float sh[3] = {0.0f, 0.0f, 0.0f}, sl[3] = {0.0f, 0.0f, 0.0f};
  for (int b = 0; b < md.B; b++) {
    float h[3], l[3], Dh, kh, kl;
#pragma unroll
    for (int q = 0; q < 3; q++) {
      const float2 p = pair[3 * b + q];
      h[q] = __fadd_rn(p.x, p.y);
      l[q] = __fsub_rn(p.y, __fsub_rn(h[q], p.x));
    }
    pair_cube(h, l, md.mu2[b], Dh, kh, kl);
#pragma unroll
    for (int q = 0; q < 3; q++) {
      const float v = kh * h[q], w = __fmaf_rn(kl, h[q], __fmaf_rn(kh, l[q], __fmaf_rn(kh, h[q], -v)));
      float er;
      sh[q] = two_sum(sh[q], v, er);
      sl[q] += er + w;
    }
  }
#pragma unroll
  for (int q = 0; q < 3; q++) {
    data[3 * md.B + q] = widen_float(sh[q]) + widen_float(sl[q]);
    pair[3 * md.B + q] = make_float2(-sh[q], -sl[q]);
  }
}
template <bool EIH>
__device__ __forceinline__ void body_data(const Model &md, EphemLoc L, double *out) {
  const int B = md.B;
  if (!EIH) {
    body_positions(md, L, 0, B, out);
    if (md.indirect) indirect_pairs(md, out);
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
