// One FP64 sweep of a tile of T trajectories by one CTA: force, operator product
// by exact digit products on the bf16 tensor cores, change.  Shared by the
// resident kernel (pc_resident.cuh) and the kernel-level product
// (pc_split.cu).
//
// The operator product.  GB300's FP64 pipe (DFMA and the .f64 mma shapes alike)
// runs at about 1 TFLOP/s, its bf16 tensor cores two orders of magnitude faster.
// Every operator row and every force column is cut into 7 signed 8-bit digits
// against its own largest exponent (split_digits7): K~ = sum_a d_a 2^-8a,
// F~ = sum_b e_b 2^-8b.  For each anti-diagonal a + b <= 8 (28 digit pairs) the
// tensor cores sum d_a e_b over the nodes in FP32 -- exactly, since every term
// and partial sum is an integer below 2^24 -- and the seven sums are combined in
// one 64-bit integer (a 62-bit fixed-point value), converted once to FP64 and
// scaled by the two exponents and omega2 in the fused multiply-add that adds x0.
// The pairs with a + b > 8 are below 2^-64 of the scale and dropped; the result's
// error is below that of an FP64 dot product.  The sums are exact, so a result
// does not depend on the tile it was computed in.
//
// What is multiplied is f = (v, a), not omega2 f: the scale costs nothing where
// the product is scaled anyway, and the velocity rows need no table of their own.
//
// FP64 operations bound a sweep (about 500 Gop/s against 75 T for FP32), so they
// are counted: 15 a node for the force (bodies far from the node in pairs of
// floats), per element one conversion, one multiply-add and one subtraction; exponents, digits and
// scales are integer work, the change is measured in FP32, and the resolution
// sums are formed only for a trajectory whose sweep would be accepted.
#pragma once

#include <cuda_bf16.h>

#include <type_traits>

#include "pc_device.cuh"

namespace pcx {
namespace {

// k extent of a digit row in shared memory: 16 per k-step plus 8 (304 bytes
// at 9 k-steps, so the 8 rows of an ldmatrix phase hit distinct banks)
__host__ __device__ inline int split_ksp(int n_ks) { return 16 * n_ks + 8; }
// digit rows of a product of NC components for T trajectories: row q*T + t holds
// component q of trajectory t, padded to tiles of 16, or of 8 for a single trajectory (what the padding rows hold only
// reaches result rows that nothing reads)
__host__ __device__ constexpr int tile_rows(int nc, int t) { return t == 1 ? 8 : (nc * t + 15) / 16 * 16; }
__host__ __device__ inline size_t tile_digit_bytes(int nc, int t, int n_ks) {
  return sizeof(__nv_bfloat16) * (size_t)kSplitDigits * tile_rows(nc, t) * split_ksp(n_ks);
}

struct SplitOp {
  const uint2 *kfrag;  // [n_nt][n_ks][7][32] B fragments of the operator digits
  const int *kexp;     // [N] largest biased exponent of each operator row
  int n_nt, n_ks;
};

// The trajectories of a tile, in shared memory.
template <int T>
struct TileShared {
  int col[T];          // column of slot t in the iterates, -1 when idle
  int fresh[T];        // first sweep on a segment: node 0's acceleration is not yet in A
  const double *eb[T]; // body data of its segment, [node][F] (see body_data)
  double w2[T];        // omega2 of its segment
  double x[6][T];      // state at the segment's start
  int colB[6 * T];     // largest biased exponent of each column (velocities, accelerations)
  int bad[T];          // an inf or NaN in one of the trajectory's columns
  unsigned emax[T];    // largest squared change (float bits, NaN the largest)
};

// Its arrays: iterates node-major, components and then columns (stride ld) inside;
// node 0 of both holds the segment's start state.
struct TileView {
  const double *Yc;    // [n][6][ld] iterate
  double *Yn;          // [n][6][ld] next iterate
  double *A;           // [n][3][T] accelerations, by slot
  size_t ld;
  int F;               // doubles per node of the body data
};

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const unsigned (&a)[4], uint2 b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

__device__ __forceinline__ void ldsm_x4(unsigned (&r)[4], const void *p) {
  const unsigned addr = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

// Conversions by integer operations (the FP64 pipe's own run at its rate), free of
// branches so that a thread's chains interleave: zero below the normal floats,
// infinite above them, NaN kept.
//
// A double as a float, truncated.
__device__ __forceinline__ float trunc_float(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ex = (hi >> 20) & 0x7ffu;
  unsigned m = (((hi & 0x7fffffffu) - (896u << 20)) << 3) | (lo >> 29);
  m = ex < 897u ? 0u : ex > 1150u ? (x != x ? 0x7fc00000u : 0x7f800000u) : m;
  return __uint_as_float((hi & 0x80000000u) | m);
}
// The same rounded to nearest even.
__device__ __forceinline__ float round_float(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned ex = (unsigned)(b >> 52) & 0x7ffu;
  const unsigned long long r = b + 0x0FFFFFFFULL + ((b >> 29) & 1ULL);
  unsigned m = ((((unsigned)(r >> 32) & 0x7fffffffu) - (896u << 20)) << 3) | ((unsigned)r >> 29);
  m = ex < 897u ? 0u : ex > 1150u ? (x != x ? 0x7fc00000u : 0x7f800000u) : m;
  return __uint_as_float(((unsigned)(b >> 32) & 0x80000000u) | m);
}
// A float as a double (zero for a subnormal, infinity and NaN not expected).
__device__ __forceinline__ double widen_float(float x) {
  const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
  return __hiloint2double((int)((u & 0x80000000u) | (m < 0x800000u ? 0u : (m >> 3) + (896u << 20))), (int)(u << 29));
}
// The same for a value known to be normal or to be negligible below 2^-126 (a zero
// or subnormal gives a value of about 2^-127).
__device__ __forceinline__ double bits_double(float x) {
  const unsigned u = __float_as_uint(x);
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}

// mu / d2^(3/2) from the FP32 reciprocal square root y of d2: with e = 1 - d2 y^2
// (|e| below 2^-21, formed by one FMA from the exact square), d2^(-3/2) =
// y^3 (1 + 3/2 e + 15/8 e^2 + ...), the quadratic term in FP32 (below 2^-41), the
// cubic one below 2^-62.  Six FP64 operations against about eight for
// mu rsqrt(d2)^3, and fewer roundings.  For d2 in inv_cube_range; mu_cube for any.
__device__ __forceinline__ bool inv_cube_range(double d2) {  // 2^-100 .. 2^100
  return (unsigned)(__double2hiint(d2) - (923 << 20)) < (unsigned)(200 << 20);
}
__device__ __forceinline__ double inv_cube(double mu, double d2) {
  const double y = bits_double(rsqrtf(trunc_float(d2)));
  const double y2 = y * y;
  const double e = fma(-d2, y2, 1.0);
  const float ef = trunc_float(e);
  const double m = mu * y * y2;
  return fma(m, fma(1.5, e, bits_double(fmaf(1.875f * ef, ef, 1e-30f))), m);
}

__device__ __forceinline__ double mu_cube(double mu, double d2) {
  if (inv_cube_range(d2)) return inv_cube(mu, d2);
  const double rs = rsqrt(d2);
  return mu * rs * rs * rs;
}

// A double as a pair of floats h + l (48 bits, truncated), by integer operations; zero
// below 2^-126 (l below 2^-74), infinite above the floats.
__device__ __forceinline__ float2 split_pair(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ex = (hi >> 20) & 0x7ffu, sign = hi & 0x80000000u;
  unsigned h = (((hi & 0x7fffffffu) - (896u << 20)) << 3) | (lo >> 29);
  h = ex < 897u ? 0u : ex > 1150u ? 0x7f800000u : h;
  const float l = __uint2float_rz(lo & 0x1fffffffu) * __uint_as_float(ex < 949u ? 0u : (ex - 948u) << 23);  // 2^(ex - 1075)
  return make_float2(__uint_as_float(sign | h), __uint_as_float(sign | __float_as_uint(l)));
}
// Sum and rounding error of two floats (Knuth).
__device__ __forceinline__ float two_sum(float a, float b, float &e) {
  const float s = __fadd_rn(a, b), v = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
  return s;
}
__device__ __forceinline__ float two_diff(float a, float b, float &e) { return two_sum(a, -b, e); }

// A difference of pairs, as a pair.
__device__ __forceinline__ void pair_diff(float2 a, float2 b, float &h, float &l) {
  float e;
  const float s = two_diff(a.x, b.x, e);
  e += a.y - b.y;
  h = __fadd_rn(s, e);
  l = __fsub_rn(e, __fsub_rn(h, s));
}
// mu / |d|^3 of a pair vector as a pair kh + kl, by the series of inv_cube; D: |d|^2.
__device__ __forceinline__ void pair_cube(const float dh[3], const float dl[3], float2 mu, float &Dh, float &kh,
                                          float &kl) {
  const float p0 = dh[0] * dh[0], p1 = dh[1] * dh[1], p2 = dh[2] * dh[2];
  float e1, e2;
  const float s1 = two_sum(p0, p1, e1), s2 = two_sum(s1, p2, e2);
  float e = (__fmaf_rn(dh[0], dh[0], -p0) + __fmaf_rn(dh[1], dh[1], -p1)) + __fmaf_rn(dh[2], dh[2], -p2);
  e = __fmaf_rn(2.0f * dh[0], dl[0], __fmaf_rn(2.0f * dh[1], dl[1], __fmaf_rn(2.0f * dh[2], dl[2], e))) + (e1 + e2);
  Dh = __fadd_rn(s2, e);
  const float Dl = __fsub_rn(e, __fsub_rn(Dh, s2));
  const float y = rsqrtf(Dh);
  const float yh = y * y, yl = __fmaf_rn(y, y, -yh);
  const float c = __fmaf_rn(-Dl, yh, __fmaf_rn(-Dh, yl, __fmaf_rn(-Dh, yh, 1.0f)));
  const float mh = mu.x * y, ml = __fmaf_rn(mu.y, y, __fmaf_rn(mu.x, y, -mh));
  kh = mh * yh;
  kl = __fmaf_rn(kh, c * __fmaf_rn(1.875f, c, 1.5f),
                 __fmaf_rn(mh, yl, __fmaf_rn(ml, yh, __fmaf_rn(mh, yh, -kh))));
}

// The indirect term in FP64 from the positions of a node's body data.
__device__ __noinline__ double3 indirect_sum(const Model &md, const double *Eb) {
  double s[3] = {0.0, 0.0, 0.0};
  for (int b = 0; b < md.B; b++) {
    const double *d = Eb + 3 * b;
    const double k = mu_cube(md.mu[b], fma(d[2], d[2], fma(d[1], d[1], d[0] * d[0])));
#pragma unroll
    for (int q = 0; q < 3; q++) s[q] = fma(k, d[q], s[q]);
  }
  return make_double3(s[0], s[1], s[2]);
}
// Whether the squared attraction of v, times `factor`, is at most c2, the central one's
// (false, too, when a range of the floats is left).
__device__ __forceinline__ bool attraction_small(const float v[3], float c2, float factor) {
  return (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]) * factor <= c2 && c2 > 1e-30f;
}

// Newtonian acceleration at r; Eb: the node's body data (positions, indirect term, both
// again as pairs of floats).
//
// The central term is formed in FP64.  A body is formed in pairs of floats, 48 bits, where
// mu/d is below 2^-11 of mu_c/r and its tidal coefficient mu/d^3 below 2^-8 of mu_c/r^3: its
// attraction is then below 2^-9.5 of the central one (2^-11 for a body farther away than the
// centre), and the pairs' error, about 2^-44 of the body's attraction and 2^-48 of its tidal
// pull over the node's own distance, below 2^-53 of the central term, its FP64 rounding.
// About 150 FP32 and integer operations take the place of 15 FP64 ones, of which the pipe
// does one for every 64 FP32 ones.  A nearer body (Venus within 1/11.7 of the solar distance)
// is formed in FP64, and so is the indirect term where it is above 2^-11 of the central term.
// Largest error over nodes from 0.3 to 40 AU and close to eight planets: 4.7e-16 of the sum of
// the terms' sizes, against 1.0e-15 of the FP64 formula with rsqrt.
__device__ __forceinline__ void tile_accel(const Model &md, const double *__restrict__ Eb, const double r[3],
                                           double a[3]) {
  const double r2 = fma(r[2], r[2], fma(r[1], r[1], r[0] * r[0]));
  const double kc = inv_cube(md.mu_c, r2);
  const bool range = inv_cube_range(r2);
  float sh[3] = {0.0f, 0.0f, 0.0f}, sl[3] = {0.0f, 0.0f, 0.0f};
  unsigned near = 0u;
  bool big = false;  // the indirect term in FP64
  if (md.B > 0) {
    const float2 *pair = reinterpret_cast<const float2 *>(Eb + 3 * md.B + 3);  // positions, then minus the indirect term
    const float kcf = trunc_float(kc), gcf = kcf * trunc_float(r2);
    float2 x[3];
#pragma unroll
    for (int q = 0; q < 3; q++) {
      x[q] = split_pair(r[q]);
      const float2 v = pair[3 * md.B + q];
      sh[q] = v.x;
      sl[q] = v.y;
    }
    big = !attraction_small(sh, kcf * gcf, 4194304.0f);
#pragma unroll
    for (int q = 0; q < 3; q++) {
      sh[q] = big ? 0.0f : sh[q];
      sl[q] = big ? 0.0f : sl[q];
    }
    // K bodies from b on: their terms side by side, added in order
    auto bodies = [&](int b, auto count) {
      constexpr int K = decltype(count)::value;
      float v[K][3], w[K][3];
#pragma unroll
      for (int k = 0; k < K; k++) {
        float dh[3], dl[3], Dh, kh, kl;
#pragma unroll
        for (int q = 0; q < 3; q++) pair_diff(x[q], pair[3 * (b + k) + q], dh[q], dl[q]);
        pair_cube(dh, dl, md.mu2[b + k], Dh, kh, kl);
        // (false, too, when a range of the floats is left)
        const bool far = kh * 256.0f <= kcf && kh * Dh * 2048.0f <= gcf && Dh > 1e-12f && kh > 1e-30f;
        near |= far ? 0u : 1u << (b + k);
#pragma unroll
        for (int q = 0; q < 3; q++) {
          v[k][q] = far ? kh * dh[q] : 0.0f;
          w[k][q] = far ? __fmaf_rn(kl, dh[q], __fmaf_rn(kh, dl[q], __fmaf_rn(kh, dh[q], -v[k][q]))) : 0.0f;
        }
      }
#pragma unroll
      for (int k = 0; k < K; k++)
#pragma unroll
        for (int q = 0; q < 3; q++) {
          float er;
          sh[q] = two_diff(sh[q], v[k][q], er);
          sl[q] += er - w[k][q];
        }
    };
    int b = 0;
    for (; b + 2 <= md.B; b += 2) bodies(b, std::integral_constant<int, 2>{});
    if (b < md.B) bodies(b, std::integral_constant<int, 1>{});
  }
#pragma unroll
  for (int q = 0; q < 3; q++) a[q] = fma(-kc, r[q], widen_float(sh[q]) + widen_float(sl[q]));
  // (one branch for what few nodes need, and its loop over the bodies in a function of its own:
  // as three branches it cost one trajectory 3 % more)
  if (!range || big || near != 0u) {
    if (!range) {
      const double rs = rsqrt(r2), k = md.mu_c * rs * rs * rs;
#pragma unroll
      for (int q = 0; q < 3; q++) a[q] = -k * r[q];
      near = md.B > 0 ? 0xffffffffu >> (32 - md.B) : 0u;
      big = md.B > 0;
    }
    if (big) {
      double3 s = make_double3(Eb[3 * md.B], Eb[3 * md.B + 1], Eb[3 * md.B + 2]);
      if (s.x != s.x) s = indirect_sum(md, Eb);
      a[0] -= s.x;
      a[1] -= s.y;
      a[2] -= s.z;
    }
    while (near) {
      const int b = __ffs(near) - 1;
      near &= near - 1u;
      const double d0 = r[0] - Eb[3 * b], d1 = r[1] - Eb[3 * b + 1], d2 = r[2] - Eb[3 * b + 2];
      const double kb = -mu_cube(md.mu[b], fma(d2, d2, fma(d1, d1, d0 * d0)));
      a[0] = fma(kb, d0, a[0]);
      a[1] = fma(kb, d1, a[1]);
      a[2] = fma(kb, d2, a[2]);
    }
  }
}

__device__ __forceinline__ int biased_exp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// Largest value of the lanes that share a slot (lanes t, t + T, ...).
template <int T>
__device__ __forceinline__ int slot_max(int v) {
#pragma unroll
  for (int o = 16; o >= T; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Accelerations of the tile's iterate into v.A and the columns' largest exponents
// into sh.colB (cleared before): the accelerations', and for a first-order sweep
// the velocities'.  A thread's slot is tid % T.  Node 0 does not move: its
// acceleration is formed once per segment, which leaves N = 2^k nodes for a power
// of two of threads.
template <int T, int TH, int ORDER, bool EIH>
__device__ __forceinline__ void tile_force(const Model &md, const TileView &v, TileShared<T> &sh, int n) {
  const int tid = threadIdx.x, t = tid % T, m = sh.col[t];
  int ea[3] = {0, 0, 0}, ev[3] = {0, 0, 0};
  if (m >= 0) {
    const double *eb = sh.eb[t];
    auto node = [&](int j) {
      const double *yp = v.Yc + (size_t)j * 6 * v.ld + m;
      double y[6], a[3];
#pragma unroll
      for (int q = 0; q < 6; q++) y[q] = (q < 3 || ORDER == 1 || EIH) ? yp[(size_t)q * v.ld] : 0.0;
      const double *ej = eb + (size_t)j * v.F;
      if (EIH) eih_accel<true>(md, ej, ej + 3 * md.B, ej + 3 * md.B + 3, 1, y, y + 3, a);
      else tile_accel(md, ej, y, a);
#pragma unroll
      for (int q = 0; q < 3; q++) {
        v.A[((size_t)j * 3 + q) * T + t] = a[q];
        ea[q] = max(ea[q], biased_exp(a[q]));
        if (ORDER == 1) ev[q] = max(ev[q], biased_exp(y[3 + q]));
      }
    };
    for (int j = 1 + tid / T; j < n; j += TH / T) node(j);
    if (tid < T) {
      if (sh.fresh[t]) {
        node(0);
      } else {
#pragma unroll
        for (int q = 0; q < 3; q++) {
          ea[q] = max(ea[q], biased_exp(v.A[(size_t)q * T + t]));
          if (ORDER == 1) ev[q] = max(ev[q], biased_exp(sh.x[3 + q][t]));
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 3; q++) {
    ea[q] = slot_max<T>(ea[q]);
    if (ORDER == 1) ev[q] = slot_max<T>(ev[q]);
    if ((tid & 31) < T) {
      atomicMax(&sh.colB[(3 + q) * T + t], ea[q]);
      if (ORDER == 1) atomicMax(&sh.colB[q * T + t], ev[q]);
    }
  }
}

// Value's fixed-point form against the column exponent Bc with 128 added to the
// six low digits: its bytes are then the digits of split_digits7 plus 128 (the
// top one a small signed integer).
__device__ __forceinline__ long long biased_digits(double v, int Bc) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int be = (int)((b >> 52) & 0x7ff);
  long long M = 0;
  if (be != 0 && be != 0x7ff) {
    const unsigned long long m = (b & ((1ULL << 52) - 1)) | (1ULL << 52);
    const int sh = Bc - be - 2;  // >= -2 since be <= Bc: M < 2^55
    if (sh <= 0) M = (long long)(m << (-sh));
    else if (sh < 63) M = (long long)((m + (1ULL << (sh - 1))) >> sh);
    if (b >> 63) M = -M;
  }
  return M + 0x0000808080808080LL;
}
// Digit a of a biased value as a float: the byte in the mantissa of 2^23, the
// bias taken off by an exact subtraction.
template <int A>
__device__ __forceinline__ float digit_float(long long M) {
  if (A == 0) return __uint_as_float(0x4B000100u + (unsigned)(int)(M >> 48)) - 8388864.0f;
  const unsigned w = (unsigned)(A >= 3 ? M : M >> 32);
  constexpr int byte = A >= 3 ? 6 - A : 2 - A;
  return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7540u + byte)) - 8388736.0f;
}

template <int T, int TH, int NC, class Src, class Place>
__device__ __forceinline__ void tile_split(const TileShared<T> &sh, const int *colB, int n, int n_ks, Src src,
                                           Place place);

// The tile's columns (component q of slot t at node k from src) as digit rows
// of bf16, two nodes per thread and step.  colB: the columns' exponents, q*T + t.
template <int T, int TH, int NC, class Src>
__device__ __forceinline__ void tile_split(const TileShared<T> &sh, const int *colB, __nv_bfloat16 *Gd, int n, int n_ks,
                                           Src src) {
  constexpr int R = tile_rows(NC, T);
  const int ksp = split_ksp(n_ks);
  tile_split<T, TH, NC>(sh, colB, n, n_ks, src, [&](int q, int t, int k, size_t &step) {
    step = (size_t)R * ksp / 2;
    return reinterpret_cast<unsigned *>(Gd + (size_t)(q * T + t) * ksp + k);
  });
}
// place(q, t, k, step): where digit 0 of component q of slot t at nodes k, k + 1 goes;
// the next digits lie step words apart.
template <int T, int TH, int NC, class Src, class Place>
__device__ __forceinline__ void tile_split(const TileShared<T> &sh, const int *colB, int n, int n_ks, Src src,
                                           Place place) {
  const int kp_n = 8 * n_ks;
  const int tid = threadIdx.x, t = tid % T, m = sh.col[t];
  auto put_pair = [&](int kp, int q) {
    const int k = 2 * kp, Bc = colB[q * T + t];
    const double a = (m >= 0 && k < n) ? src(q, t, m, k) : 0.0;
    const double b = (m >= 0 && k + 1 < n) ? src(q, t, m, k + 1) : 0.0;
    const long long Ma = biased_digits(a, Bc), Mb = biased_digits(b, Bc);
    size_t st;
    unsigned *o = place(q, t, k, st);
    auto put = [&](int d, float fa, float fb) {
      o[(size_t)d * st] = __byte_perm(__float_as_uint(fa), __float_as_uint(fb), 0x7632);
    };
    put(0, digit_float<0>(Ma), digit_float<0>(Mb));
    put(1, digit_float<1>(Ma), digit_float<1>(Mb));
    put(2, digit_float<2>(Ma), digit_float<2>(Mb));
    put(3, digit_float<3>(Ma), digit_float<3>(Mb));
    put(4, digit_float<4>(Ma), digit_float<4>(Mb));
    put(5, digit_float<5>(Ma), digit_float<5>(Mb));
    put(6, digit_float<6>(Ma), digit_float<6>(Mb));
  };
  if (T <= 2) {  // fewer pairs of nodes than threads: the components side by side
    int kp = tid / T, q = 0;
    for (;;) {
      while (kp >= kp_n && q < NC) {
        kp -= kp_n;
        q++;
      }
      if (q >= NC) break;
      put_pair(kp, q);
      kp += TH / T;
    }
  } else {
    for (int kp = tid / T; kp < kp_n; kp += TH / T)
#pragma unroll
      for (int q = 0; q < NC; q++) put_pair(kp, q);
  }
}

// w 2^e: by the exponent field when w and the result are normal.
__device__ __forceinline__ double scale_exp(double w, int e) {
  const int hi = __double2hiint(w), ex = (hi >> 20) & 0x7ff;
  if (ex > 0 && ex < 2047 && ex + e > 0 && ex + e < 2047) return __hiloint2double(hi + (e << 20), __double2loint(w));
  return ldexp(w, e);
}

// The seven exact sums of one element as an FP64 integer: sum_d S_d 2^(56 - 8d),
// rounded to 16 bits after the fourth sum's last.
__device__ __forceinline__ double combine_sums(const int S[kSplitDigits]) {
  const long long hi = S[0] * (1LL << 24) + S[1] * (1LL << 16) + S[2] * (1LL << 8) + S[3];
  const long long lo = S[4] * (1LL << 16) + S[5] * (1LL << 8) + S[6];
  return (double)(hi * (1LL << 16) + ((lo + 128) >> 8));
}

// out(t, j, q0, nq, value, e): components q0 .. q0 + nq - 1 of the product's rows
// for slot t at node j are value[i] 2^e[i].  With 8 or 16 slots a thread's
// accumulators hold every component of its slots (nq = NC), with fewer single
// ones.  A warp takes node tiles of 8 output nodes; the digits are the A operand
// (ldmatrix from shared memory), the operator digits the B operand (fragments laid
// out by the plan, 64-bit loads from L2, the next k-step's in flight during this
// one's products).
//
// A single slot's 6 (or 3) columns would fill a third of the 16 digit rows, so there the
// operator is the A operand (16 nodes; its two 8-node fragments are the four registers)
// and the columns the 8-wide B operand: half the products.
template <int TH, int NC, class Out>
__device__ __forceinline__ void tile_product_one(const SplitOp &op, int live, const int *colB,
                                                 const __nv_bfloat16 *Gd, int N, Out out) {
  const int ksp = split_ksp(op.n_ks);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  // ldmatrix: digits a and a + 1, both k halves of each
  const __nv_bfloat16 *Gl = Gd + ((size_t)(lane >> 4) * 8 + (lane & 7)) * ksp + ((lane >> 3) & 1) * 8;
  for (int mt = w; 2 * mt < op.n_nt; mt += TH / 32) {
    float acc[kSplitDigits][4];
#pragma unroll
    for (int dd = 0; dd < kSplitDigits; dd++)
#pragma unroll
      for (int i = 0; i < 4; i++) acc[dd][i] = 0.0f;
    const bool two = 2 * mt + 1 < op.n_nt;
    const size_t half = two ? (size_t)op.n_ks * kSplitDigits * 32 : 0;
    const uint2 *kf = op.kfrag + (size_t)2 * mt * op.n_ks * kSplitDigits * 32 + lane;
    uint2 n0[kSplitDigits], n1[kSplitDigits];
#pragma unroll
    for (int a = 0; a < kSplitDigits; a++) {
      n0[a] = __ldg(kf + a * 32);
      n1[a] = __ldg(kf + half + a * 32);
    }
    for (int ks = 0; ks < op.n_ks; ks++) {
      unsigned bf[kSplitDigits + 1][2];
#pragma unroll
      for (int b = 0; b < kSplitDigits; b += 2) {
        unsigned r[4];
        // the last one's second digit repeats the first
        ldsm_x4(r, (b + 1 < kSplitDigits || lane < 16 ? Gl : Gl - (size_t)8 * ksp) + (size_t)b * 8 * ksp + ks * 16);
        bf[b][0] = r[0];
        bf[b][1] = r[1];
        bf[b + 1][0] = r[2];
        bf[b + 1][1] = r[3];
      }
      unsigned af[kSplitDigits][4];
#pragma unroll
      for (int a = 0; a < kSplitDigits; a++) {
        af[a][0] = n0[a].x;
        af[a][1] = n1[a].x;
        af[a][2] = n0[a].y;
        af[a][3] = n1[a].y;
      }
      if (ks + 1 < op.n_ks)
#pragma unroll
        for (int a = 0; a < kSplitDigits; a++) {
          n0[a] = __ldg(kf + ((size_t)(ks + 1) * kSplitDigits + a) * 32);
          n1[a] = __ldg(kf + half + ((size_t)(ks + 1) * kSplitDigits + a) * 32);
        }
#pragma unroll
      for (int a = 0; a < kSplitDigits; a++)
#pragma unroll
        for (int b = 0; b < kSplitDigits - a; b++) mma_bf16_16816(acc[a + b], af[a], make_uint2(bf[b][0], bf[b][1]));
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const int r = mt * 16 + g + 8 * (i >> 1), q = 2 * t4 + (i & 1);
      if (r >= N || q >= NC || !live) continue;
      int S[kSplitDigits];
#pragma unroll
      for (int dd = 0; dd < kSplitDigits; dd++) S[dd] = __float2int_rn(acc[dd][i]);
      const double val[1] = {combine_sums(S)};
      const int ex[1] = {op.kexp[r] - 2042 - 56 + colB[q]};
      out(0, r + 1, q, val, ex);
    }
  }
}

template <int T, int TH, int NC, class Out>
__device__ __forceinline__ void tile_product(const SplitOp &op, const TileShared<T> &sh, const int *colB,
                                             const __nv_bfloat16 *Gd, int N, Out out) {
  if constexpr (T == 1) return tile_product_one<TH, NC>(op, sh.col[0] >= 0, colB, Gd, N, out);
  static_assert(NC * T <= 48, "at most three row tiles");
  constexpr int R = tile_rows(NC, T), MT = (R + 15) / 16;
  const int ksp = split_ksp(op.n_ks);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  const int arow = (lane & 7) + ((lane >> 3) & 1) * 8, acol = (lane >> 4) * 8;
  for (int nt = w; nt < op.n_nt; nt += TH / 32) {
    float acc[MT][kSplitDigits][4];
#pragma unroll
    for (int mt = 0; mt < MT; mt++)
#pragma unroll
      for (int dd = 0; dd < kSplitDigits; dd++)
#pragma unroll
        for (int i = 0; i < 4; i++) acc[mt][dd][i] = 0.0f;
    const uint2 *kf = op.kfrag + (size_t)nt * op.n_ks * kSplitDigits * 32 + lane;
    uint2 nx[kSplitDigits];
#pragma unroll
    for (int b = 0; b < kSplitDigits; b++) nx[b] = __ldg(kf + b * 32);
    for (int ks = 0; ks < op.n_ks; ks++) {
      uint2 bf[kSplitDigits];
#pragma unroll
      for (int b = 0; b < kSplitDigits; b++) bf[b] = nx[b];
      if (ks + 1 < op.n_ks)
#pragma unroll
        for (int b = 0; b < kSplitDigits; b++) nx[b] = __ldg(kf + ((size_t)(ks + 1) * kSplitDigits + b) * 32);
#pragma unroll
      for (int a = 0; a < kSplitDigits; a++) {
        unsigned af[MT][4];
#pragma unroll
        for (int mt = 0; mt < MT; mt++) ldsm_x4(af[mt], Gd + ((size_t)a * R + mt * 16 + arow) * ksp + ks * 16 + acol);
#pragma unroll
        for (int b = 0; b < kSplitDigits - a; b++)
#pragma unroll
          for (int mt = 0; mt < MT; mt++) mma_bf16_16816(acc[mt][a + b], af[mt], bf[b]);
      }
    }
    auto sums = [&](int mt, int i) {
      int S[kSplitDigits];
#pragma unroll
      for (int dd = 0; dd < kSplitDigits; dd++) S[dd] = __float2int_rn(acc[mt][dd][i]);
      return combine_sums(S);
    };
#pragma unroll
    for (int e = 0; e < 2; e++) {
      const int r = nt * 8 + 2 * t4 + e;
      if (r >= N) continue;
      const int kx = op.kexp[r] - 2042 - 56;
      if (T % 8 == 0) {
#pragma unroll
        for (int h = 0; h < T / 8; h++) {
          const int t = g + 8 * h;
          if (sh.col[t] < 0) continue;
          double val[NC];
          int ex[NC];
#pragma unroll
          for (int q = 0; q < NC; q++) {
            const int mt = (q * T + 8 * h) >> 4, i = (((q * T + 8 * h) >> 3) & 1) * 2 + e;  // compile-time
            val[q] = sums(mt, i);
            ex[q] = kx + colB[q * T + t];
          }
          out(t, r + 1, 0, val, ex);
        }
      } else {
#pragma unroll
        for (int mt = 0; mt < MT; mt++)
#pragma unroll
          for (int h = 0; h < 2; h++) {
            const int row = mt * 16 + g + 8 * h, q = row / T, t = row % T;
            if (q >= NC || sh.col[t] < 0) continue;
            const double val[1] = {sums(mt, 2 * h + e)};
            const int ex[1] = {kx + colB[row]};
            out(t, r + 1, q, val, ex);
          }
      }
    }
  }
}

// Squared change of half a state (new minus old, relative to the new one's norm).
// The decisions that use it need a few digits: FP32, the norm from truncated floats.
__device__ __forceinline__ float half_change(const double yn[3], const float d[3], int relative) {
  float s = 1.0f;
  if (relative) {
    const float a = trunc_float(yn[0]), b = trunc_float(yn[1]), c = trunc_float(yn[2]);
    const float nr = a * a + b * b + c * c;
    s = (nr > 0.0f && nr <= 3.0e38f) ? rsqrtf(nr) : 1.0f;
  }
  const float a = d[0] * s, b = d[1] * s, c = d[2] * s;
  return a * a + b * b + c * c;
}

// The whole sweep.  sh.col, fresh, eb, w2, x and cleared colB, bad, emax are in
// place and synchronised; on return (synchronised) v.Yn holds the next iterate and
// sh.emax the largest squared change of every slot.  mark(kind): the end of a phase,
// for the per-kernel times.
// A product through shared-memory digit rows and mma.sync (the other: TcProduct).
struct MmaProduct {
  static constexpr bool TC = false;
  const SplitOp &op;
  __nv_bfloat16 *Gd;
};

template <int T, int TH, int ORDER, bool EIH, class Product, class Mark>
__device__ __forceinline__ void tile_sweep(const Sweep &s, const Model &md, Product &pr, const TileView &v,
                                           TileShared<T> &sh, Mark mark) {
  constexpr bool TC = Product::TC;
  constexpr bool WHOLE = TC || T % 8 == 0;  // the epilogue sees whole half-states: the change is measured there
  const int tid = threadIdx.x, lane = tid & 31, n = s.n, N = s.N;
  tile_force<T, TH, ORDER, EIH>(md, v, sh, n);
  __syncthreads();
  mark(PC_KERNEL_FORCE);
  auto mark_bad = [&](int first, int rows) {
    for (int r = tid; r < rows; r += TH)
      if (sh.colB[first + r] == 0x7ff) sh.bad[r % T] = 1;
  };
  // largest squared change of the thread's slots in the epilogue: g + 8 h, or four (TC)
  constexpr int NE = TC ? 4 : WHOLE ? T / 8 : 1;
  float e2[NE];
#pragma unroll
  for (int h = 0; h < NE; h++) e2[h] = 0.0f;
  auto store = [&](int c0, auto nq, int t, int j, const double *val, const int *ex) {
    constexpr int NQ = decltype(nq)::value;
    const size_t o = ((size_t)j * 6 + c0) * v.ld + sh.col[t];
    double y[NQ];
#pragma unroll
    for (int q = 0; q < NQ; q++) {
      y[q] = sh.bad[t] ? __longlong_as_double(0x7FF8000000000000LL)
                       : fma(val[q], scale_exp(sh.w2[t], ex[q]), sh.x[c0 + q][t]);
      v.Yn[o + (size_t)q * v.ld] = y[q];
    }
    if (WHOLE) {
#pragma unroll
      for (int hf = 0; hf < NQ / 3; hf++) {
        float d[3];
#pragma unroll
        for (int q = 0; q < 3; q++) {
          d[q] = round_float(y[3 * hf + q] - v.Yc[o + (size_t)(3 * hf + q) * v.ld]);
        }
        const float c = half_change(y + 3 * hf, d, s.relative);
        const int h = t >> 3;
#pragma unroll
        for (int k = 0; k < T / 8; k++)
          if (k == h) e2[k % NE] = nanmaxf(e2[k % NE], c);
      }
    }
  };
  // four slots' half-states at once (TC): component c0 + q of slot t0 + u
  auto store4 = [&](int c0, const int *cb, int t0, int j, const double (&val)[3][4], int kx) {
    double y[3][4], o[3][4];
    const size_t at = ((size_t)j * 6 + c0) * v.ld + t0;
    const bool wide = v.ld == T;
#pragma unroll
    for (int q = 0; q < 3; q++) {
#pragma unroll
      for (int u = 0; u < 4; u += 2) {
        const double *yc = v.Yc + at + (size_t)q * v.ld + u;
        if (wide) {
          const double2 x = *reinterpret_cast<const double2 *>(yc);
          o[q][u] = x.x;
          o[q][u + 1] = x.y;
        } else {
          o[q][u] = sh.col[t0 + u] >= 0 ? yc[0] : 0.0;
          o[q][u + 1] = sh.col[t0 + u + 1] >= 0 ? yc[1] : 0.0;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; u++)
        y[q][u] = sh.bad[t0 + u] ? __longlong_as_double(0x7FF8000000000000LL)
                                 : fma(val[q][u], scale_exp(sh.w2[t0 + u], kx + cb[q * T + t0 + u]), sh.x[c0 + q][t0 + u]);
#pragma unroll
      for (int u = 0; u < 4; u += 2) {
        double *yn = v.Yn + at + (size_t)q * v.ld + u;
        if (wide) {
          *reinterpret_cast<double2 *>(yn) = make_double2(y[q][u], y[q][u + 1]);
        } else {
          if (sh.col[t0 + u] >= 0) yn[0] = y[q][u];
          if (sh.col[t0 + u + 1] >= 0) yn[1] = y[q][u + 1];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const double yu[3] = {y[0][u], y[1][u], y[2][u]};
      const float d[3] = {round_float(y[0][u] - o[0][u]), round_float(y[1][u] - o[1][u]),
                          round_float(y[2][u] - o[2][u])};
      const float c = half_change(yu, d, s.relative);
      if (sh.col[t0 + u] >= 0) e2[u % NE] = nanmaxf(e2[u % NE], c);
    }
  };
  using One = std::integral_constant<int, 1>;
  using Three = std::integral_constant<int, 3>;
  using Six = std::integral_constant<int, 6>;
  if (ORDER == 1) {
    mark_bad(0, 6 * T);
    auto src = [&](int q, int t, int m, int k) {
      return q < 3 ? v.Yc[((size_t)k * 6 + 3 + q) * v.ld + m] : v.A[((size_t)k * 3 + q - 3) * T + t];
    };
    if constexpr (TC) {
      pr.template split<T, TH, 6>(sh, sh.colB, n, src);
      __syncthreads();
      pr.template product<T, TH>(sh, sh.colB, N, [&](int t0, int j, int q0, const double (&val)[3][4], int kx) {
        store4(q0, sh.colB + q0 * T, t0, j, val, kx);
      });
    } else {
      tile_split<T, TH, 6>(sh, sh.colB, pr.Gd, n, pr.op.n_ks, src);
      __syncthreads();
      tile_product<T, TH, 6>(pr.op, sh, sh.colB, pr.Gd, N, [&](int t, int j, int q, const double *val, const int *ex) {
        if constexpr (WHOLE) store(0, Six{}, t, j, val, ex);
        else store(q, One{}, t, j, val, ex);
      });
    }
  } else {
    // velocities V' = v0 + omega2 K A(R) first, then positions R' = r0 + omega2 K V'
    mark_bad(3 * T, 3 * T);
    auto acc = [&](int q, int t, int, int k) { return v.A[((size_t)k * 3 + q) * T + t]; };
    if constexpr (TC) {
      pr.template split<T, TH, 3>(sh, sh.colB + 3 * T, n, acc);
      __syncthreads();
      pr.template product<T, TH>(sh, sh.colB + 3 * T, N, [&](int t0, int j, int, const double (&val)[3][4], int kx) {
        store4(3, sh.colB + 3 * T, t0, j, val, kx);
      });
    } else {
      tile_split<T, TH, 3>(sh, sh.colB + 3 * T, pr.Gd, n, pr.op.n_ks, acc);
      __syncthreads();
      tile_product<T, TH, 3>(pr.op, sh, sh.colB + 3 * T, pr.Gd, N,
                             [&](int t, int j, int q, const double *val, const int *ex) {
                               if constexpr (WHOLE) store(3, Three{}, t, j, val, ex);
                               else store(3 + q, One{}, t, j, val, ex);
                             });
    }
    __syncthreads();
    {
      const int t = tid % T, m = sh.col[t];
      int ev[3] = {0, 0, 0};
      if (m >= 0)
        for (int j = tid / T; j < n; j += TH / T)
#pragma unroll
          for (int q = 0; q < 3; q++) ev[q] = max(ev[q], biased_exp(v.Yn[((size_t)j * 6 + 3 + q) * v.ld + m]));
#pragma unroll
      for (int q = 0; q < 3; q++) {
        ev[q] = slot_max<T>(ev[q]);
        if (lane < T) atomicMax(&sh.colB[q * T + t], ev[q]);
      }
    }
    __syncthreads();
    mark_bad(0, 3 * T);
    auto vel = [&](int q, int, int m, int k) { return v.Yn[((size_t)k * 6 + 3 + q) * v.ld + m]; };
    if constexpr (TC) {
      pr.template split<T, TH, 3>(sh, sh.colB, n, vel);
      __syncthreads();
      pr.template product<T, TH>(sh, sh.colB, N, [&](int t0, int j, int, const double (&val)[3][4], int kx) {
        store4(0, sh.colB, t0, j, val, kx);
      });
    } else {
      tile_split<T, TH, 3>(sh, sh.colB, pr.Gd, n, pr.op.n_ks, vel);
      __syncthreads();
      tile_product<T, TH, 3>(pr.op, sh, sh.colB, pr.Gd, N, [&](int t, int j, int q, const double *val, const int *ex) {
        if constexpr (WHOLE) store(0, Three{}, t, j, val, ex);
        else store(q, One{}, t, j, val, ex);
      });
    }
  }
  if constexpr (TC) {
    const int h = tid >> 7, t0 = T == 16 ? 4 * h : 4 * (h & 1);
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const unsigned b = __reduce_max_sync(0xffffffffu, err_bits32(e2[u]));  // non-negative floats order like their bits
      if (lane == 0) atomicMax(&sh.emax[t0 + u], b);
    }
  } else if (WHOLE) {
#pragma unroll
    for (int h = 0; h < T / 8; h++) {
      float e = e2[h % NE];
      e = nanmaxf(e, __shfl_xor_sync(0xffffffffu, e, 1));
      e = nanmaxf(e, __shfl_xor_sync(0xffffffffu, e, 2));
      if ((lane & 3) == 0) atomicMax(&sh.emax[(lane >> 2) + 8 * h], err_bits32(e));
    }
  } else {
    __syncthreads();
    const int t = tid % T, m = sh.col[t];
    float e = 0.0f;
    if (m >= 0)
      for (int i = tid / T; i < 2 * N; i += TH / T) {  // (node, half of the state)
        const int hf = i >= N, j = 1 + i - (hf ? N : 0);
        const size_t o = ((size_t)j * 6 + 3 * hf) * v.ld + m;
        double y[3];
        float d[3];
#pragma unroll
        for (int q = 0; q < 3; q++) {
          y[q] = v.Yn[o + (size_t)q * v.ld];
          d[q] = round_float(y[q] - v.Yc[o + (size_t)q * v.ld]);
        }
        e = nanmaxf(e, half_change(y, d, s.relative));
      }
    const int b = slot_max<T>((int)err_bits32(e));  // non-negative floats order like their bits
    if (lane < T) atomicMax(&sh.emax[t], (unsigned)b);
  }
  __syncthreads();
  mark(PC_KERNEL_CONTRACT);
}

// Resolution test (Chebyshev tail of the force fit).  On the CGL nodes
// T_N(tau_j) = (-1)^(N+j) and T_{N-1}(tau_j) = (-1)^(N+j) tau_j, so the two
// top coefficients of the interpolant of g = omega2 f are
//   a_N = (1/N) sum''_j (-1)^(N+j) g_j,   a_{N-1} = (2/N) sum''_j (-1)^(N+j) tau_j g_j
// (sum'' halves the end terms).  The integrated error is about
// 2 |omega2| (|a_{N-1}| + |a_N|) per unit of f; position components are measured
// against max_j |r_j|, velocity ones against max_j |v_j| of the iterate the force
// was evaluated on (relative mode).  Formed only for the slots in `want` (bit t),
// from the accelerations and velocities the sweep used, in kTailParts node
// ranges added in order.  FP64 operations bound it: signs are integer work and the ends
// are halved apart, so a value costs an addition and a multiply-add (the two weights'
// products before cost one more: 53k cycles a tile of 16 slots at N = 128, now 34k),
// and eight groups of equal weight fill 512 threads twice.
constexpr int kTailParts = 8;
__host__ __device__ constexpr size_t tile_tail_doubles(int t) { return 14 * kTailParts * (size_t)t; }
template <int T, int TH>
__device__ __forceinline__ void tile_tail_sums(const Sweep &s, const TileView &v, const TileShared<T> &sh,
                                               const double *__restrict__ tau, unsigned want, double *part) {
  const int n = s.n, N = s.N, chunk = (n + kTailParts - 1) / kTailParts;
  const int t = threadIdx.x % T, m = sh.col[t];
  if (!((want >> t) & 1u)) return;
  for (int i = threadIdx.x / T; i < 8 * kTailParts; i += TH / T) {
    const int p = i / 8, g = i % 8;
    const int j0 = p * chunk, j1 = min(n, j0 + chunk);
    double a = 0.0, b = 0.0;
    if (g < 6) {
      const double *f = g < 3 ? v.Yc + (3 + g) * v.ld + m : v.A + (size_t)(g - 3) * T + t;
      const size_t st = g < 3 ? 6 * v.ld : (size_t)3 * T;
#pragma unroll 6
      for (int j = j0; j < j1; j++) {
        double x = f[(size_t)j * st];
        if (j == 0 || j == N) x *= 0.5;
        x = __hiloint2double(__double2hiint(x) ^ (((N + j) & 1) << 31), __double2loint(x));
        a += x;
        b = fma(tau[j], x, b);
      }
      part[((size_t)p * 14 + 2 * g) * T + t] = a;
      part[((size_t)p * 14 + 2 * g + 1) * T + t] = b;
    } else {  // largest |r|^2, |v|^2
      const double *y = v.Yc + (size_t)3 * (g - 6) * v.ld + m;
#pragma unroll 6
      for (int j = j0; j < j1; j++) {
        const double *yj = y + (size_t)j * 6 * v.ld;
        const double y0 = yj[0], y1 = yj[v.ld], y2 = yj[2 * v.ld];
        a = fmax(a, fma(y2, y2, fma(y1, y1, y0 * y0)));
      }
      part[((size_t)p * 14 + 6 + g) * T + t] = a;
    }
  }
}
// The parts of every value added (the last two: maxima) into the first range's place.
template <int T, int TH>
__device__ __forceinline__ void tile_tail_add(double *part) {
  for (int i = threadIdx.x; i < 14 * T; i += TH) {
    double v[kTailParts];
#pragma unroll
    for (int p = 0; p < kTailParts; p++) v[p] = part[(size_t)p * 14 * T + i];
    double a = v[0];
#pragma unroll
    for (int p = 1; p < kTailParts; p++) a = i < 12 * T ? a + v[p] : fmax(a, v[p]);
    part[i] = a;
  }
}
// The estimate of slot t from the sums.
template <int T>
__device__ double tile_tail(const Sweep &s, const TileShared<T> &sh, const double *part, int t) {
  const double invN = 1.0 / (double)s.N, w2 = fabs(sh.w2[t]);
  double er = 0.0, ev = 0.0;
  const double r2 = part[12 * T + t], v2 = part[13 * T + t];
#pragma unroll
  for (int g = 0; g < 6; g++) {
    const double tl = 2.0 * w2 * (fabs(2.0 * part[(2 * g + 1) * T + t] * invN) + fabs(part[2 * g * T + t] * invN));
    if (g < 3) er = nanmax(er, tl); else ev = nanmax(ev, tl);
  }
  if (s.relative) {
    if (r2 > 0.0) er /= sqrt(r2);
    if (v2 > 0.0) ev /= sqrt(v2);
  }
  return nanmax(er, ev);
}

}  // namespace
}  // namespace pcx
