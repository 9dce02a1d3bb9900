// FP32 solves of a tile of T trajectories by one CTA (mixed precision, an extension
// of the paper): sweeps on the deviation from the warm start of a new segment, or
// on the correction to an FP64 iterate, until every slot's change stops falling.
//
// NEW SEGMENT: the iterate is y = y_K + delta with y_K the FP64 warm start.  The
// Picard map gives delta' = rho + omega2 K (f(y_K + delta) - f_K), with f_K the
// two-body derivative of y_K and rho = x0 + omega2 K f_K - y_K the operator's
// residual on the Kepler arc (below the resolution tolerance on accepted
// segments; dropped here and restored by the FP64 sweeps that follow).  The
// central force deviation is formed without cancellation (Encke):
//   (mu_c/|r_K|^3) [F(q) (r_K + dr) - dr],  q = dr.(2 r_K + dr)/|r_K|^2,
//   F = 1 - (1+q)^(-3/2) = q s^2 (1 + s + s^2)/(1 + s),  s = (1+q)^(-1/2),
// plus the bodies' terms with r - r_b = (r_K - r_b) + dr, where r_K - r_b was
// formed in FP64 before rounding.  Its rounding error is relative to |delta|.
//
// CORRECTION: an FP64 sweep took the iterate Y to Y' = x0 + omega2 K G(Y) with
// residual R = Y' - Y (rounded to FP32).  The fixed point Y* satisfies Y* = Y + c
// with c = R + omega2 K [G(Y + c) - G(Y)], solved about the base Y = Y' - R (formed
// in FP64): the central and every body term as Encke differences, the velocity
// rows as omega2 c_v.  Then Y* = Y' + omega2 K [G(Y + c) - G(Y)].
//
// The product runs on the bf16 tensor cores: an FP32 value is exactly the sum of
// three bf16 (24 bits in pieces of 8), so K G is six products of pieces (the three
// dropped ones are below 2^-25 of a term), the leading one, the two next and the three
// last each in an FP32 accumulator of their own: 8 roundings at full scale at N = 128
// against 129 of a multiply-add chain.  Six bf16 products cost what three TF32 ones do and keep two bits more.
//
// A sweep is a handful of FP32 operations a node between two products, so the
// working set stays in the CTA: pieces, products and deviations in shared memory
// (where the FP64 sweep keeps its digits), the node records in scratch.  A thread
// takes two neighbouring nodes of its slot at a time (32-bit stores of the pieces and
// two independent chains of operations), or one when the CTA has a single slot.  Node 0 does not move, so its constant
// force row joins as a rank-one term and the product's k extent is the N nodes
// after it (8 k-steps at N = 128, not 9).
#pragma once

#include "pc_tile.cuh"

namespace pcx {
namespace {

constexpr float kSolveFloor = 2e-6f;
// A correction solve stops at a change below 2e-5 of the correction: the FP64
// sweep after it measures the change and decides convergence, so the floor only
// trades FP32 sweeps against FP64 ones.  On config 3, 2e-5 cuts 8 % of the FP32
// sweeps with the same FP64 sweeps as 2e-6; 1e-4 adds 2 % FP64 sweeps.
constexpr float kSolveCorrFloor = 2e-5f;
constexpr int kPieces = 3;

enum : int { SOLVE_NONE = 0, SOLVE_KEPLER = 1, SOLVE_CORR = 2 };
enum : int { SOLVE_RUN = 0, SOLVE_OK = 1, SOLVE_FAIL = 2 };

// Shared-memory areas: pieces [3][rows][kst] bf16, products [NC T][os] floats,
// deviations [groups of U nodes][6][T][U].
__host__ __device__ inline int solve_ks(int N) { return (N + 15) / 16; }
__host__ __device__ inline int solve_kst(int N) { return 16 * solve_ks(N) + 8; }
__host__ __device__ inline int solve_ostride(int N) { return (N + 31) / 32 * 32 + 8; }
// Nodes a thread takes at a time: one when a slot has threads to spare.
__host__ __device__ constexpr int solve_group(int T) { return T == 1 ? 1 : 2; }
__host__ __device__ inline size_t solve_smem(int nc, int T, int N) {
  return (size_t)kPieces * tile_rows(nc, T) * solve_kst(N) * sizeof(__nv_bfloat16) +
         sizeof(float) * ((size_t)nc * T * solve_ostride(N) + (size_t)(N + 1) / 2 * 12 * T);
}
// float4s of a node record, each a plane [n][T]: (r, mu_c/r^3), then (indirect term, 1/r^2)
// for a new segment or (position residual, 1/r^2) for a correction, then what the velocity
// half alone reads, (v, -) and (velocity residual, -), then (r - r_b, -) or
// (r - r_b, mu_b/|r - r_b|^3) per body.  A sweep reads all of them from L2 (33 KB a plane of
// 16 slots at N = 128); as many of the first two as the CTA's area holds stay in shared memory
// (65,536 mixed 233 -> 220 ms; a third one, in shared memory added for it, gained nothing).
__host__ __device__ constexpr int solve_record(int B) { return 4 + B; }

template <int T>
struct SolveShared {
  int mode[T], state[T], it[T], nst[T];
  float w2[T], ebest[T];
  unsigned emax[T], dmax[T];  // float bits (non-negative; a NaN change the largest)
  float a0[3][T];             // force row of node 0 (it does not move)
};

// Squared change and size of half a state and its force row are formed without
// IEEE divisions and square roots (reciprocal roots to 2 ulp, as in the force).
__device__ __forceinline__ float solve_encke(float q) {
  const float s = rsqrtf(1.0f + q);
  return __fdividef(q * s * s * (1.0f + s + s * s), 1.0f + s);
}

// omega2 times the force deviation at a node with deviation d; rec(f): its record.
template <class Rec>
__device__ __forceinline__ void solve_force(int mode, int B, const float *__restrict__ mu32, int indirect, float w2,
                                            const float d[3], Rec rec, float a[3]) {
  const float4 rk = rec(0);
  const float4 rr = rec(1);
  const float q = (d[0] * (2.0f * rk.x + d[0]) + d[1] * (2.0f * rk.y + d[1]) + d[2] * (2.0f * rk.z + d[2])) * rr.w;
  const float F = solve_encke(q);
  a[0] = rk.w * (F * (rk.x + d[0]) - d[0]);
  a[1] = rk.w * (F * (rk.y + d[1]) - d[1]);
  a[2] = rk.w * (F * (rk.z + d[2]) - d[2]);
  for (int b = 0; b < B; b++) {
    const float4 D = rec(4 + b);
    if (mode == SOLVE_KEPLER) {
      const float x = D.x + d[0], y = D.y + d[1], z = D.z + d[2];
      const float s = rsqrtf(x * x + y * y + z * z);
      const float k = __ldg(mu32 + b) * s * s * s;
      a[0] -= k * x;
      a[1] -= k * y;
      a[2] -= k * z;
    } else {
      const float ir = rsqrtf(D.x * D.x + D.y * D.y + D.z * D.z);
      const float Fb = solve_encke(
          (d[0] * (2.0f * D.x + d[0]) + d[1] * (2.0f * D.y + d[1]) + d[2] * (2.0f * D.z + d[2])) * ir * ir);
      a[0] += D.w * (Fb * (D.x + d[0]) - d[0]);
      a[1] += D.w * (Fb * (D.y + d[1]) - d[1]);
      a[2] += D.w * (Fb * (D.z + d[2]) - d[2]);
    }
  }
  if (mode == SOLVE_KEPLER && indirect) {
    a[0] -= rr.x;
    a[1] -= rr.y;
    a[2] -= rr.z;
  }
  for (int q3 = 0; q3 < 3; q3++) a[q3] *= w2;
}

// The three bf16 pieces (rounded to nearest, exact in sum) of U values at neighbouring k
// of a row.
template <int U>
__device__ __forceinline__ void put_pieces(__nv_bfloat16 *at, size_t piece, const float (&x)[U]) {
  if constexpr (U == 2) {
    const __nv_bfloat162 p0 = __floats2bfloat162_rn(x[0], x[1]);
    *reinterpret_cast<__nv_bfloat162 *>(at) = p0;
    const float x1 = x[0] - __low2float(p0), y1 = x[1] - __high2float(p0);
    const __nv_bfloat162 p1 = __floats2bfloat162_rn(x1, y1);
    *reinterpret_cast<__nv_bfloat162 *>(at + piece) = p1;
    *reinterpret_cast<__nv_bfloat162 *>(at + 2 * piece) =
        __floats2bfloat162_rn(x1 - __low2float(p1), y1 - __high2float(p1));
  } else {
    const __nv_bfloat16 p0 = __float2bfloat16_rn(x[0]);
    at[0] = p0;
    const float x1 = x[0] - __bfloat162float(p0);
    const __nv_bfloat16 p1 = __float2bfloat16_rn(x1);
    at[piece] = p1;
    at[2 * piece] = __float2bfloat16_rn(x1 - __bfloat162float(p1));
  }
}

// O[row][r] = sum_{k >= 1} K[r + 1][k] G[k][row] from the pieces of both.
//
// One slot: the operator as the A operand, as in tile_product_one.
template <int TH, int NC>
__device__ __forceinline__ void solve_product_one(const uint2 *__restrict__ kfrag, int n_nt, int n_ks, int ksp,
                                                  const __nv_bfloat16 *P, float *O, int os) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  const __nv_bfloat16 *Pl = P + ((size_t)(lane >> 4) * 8 + (lane & 7)) * ksp + ((lane >> 3) & 1) * 8;
  const __nv_bfloat16 *P2 = P + ((size_t)2 * 8 + (lane & 7)) * ksp + ((lane >> 3) & 1) * 8;
  for (int mt = w; 2 * mt < n_nt; mt += TH / 32) {
    float hi[4] = {0.0f, 0.0f, 0.0f, 0.0f}, lo[4] = {0.0f, 0.0f, 0.0f, 0.0f}, l2[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    const size_t half = 2 * mt + 1 < n_nt ? (size_t)n_ks * kPieces * 32 : 0;
    const uint2 *kf = kfrag + (size_t)2 * mt * n_ks * kPieces * 32 + lane;
    uint2 n0[kPieces], n1[kPieces];
#pragma unroll
    for (int a = 0; a < kPieces; a++) {
      n0[a] = __ldg(kf + a * 32);
      n1[a] = __ldg(kf + half + a * 32);
    }
    for (int ks = 0; ks < n_ks; ks++) {
      unsigned r01[4], r2[4], af[kPieces][4];
      ldsm_x4(r01, Pl + ks * 16);
      ldsm_x4(r2, P2 + ks * 16);
      const uint2 b0 = make_uint2(r01[0], r01[1]), b1 = make_uint2(r01[2], r01[3]), b2 = make_uint2(r2[0], r2[1]);
#pragma unroll
      for (int a = 0; a < kPieces; a++) {
        af[a][0] = n0[a].x;
        af[a][1] = n1[a].x;
        af[a][2] = n0[a].y;
        af[a][3] = n1[a].y;
      }
      if (ks + 1 < n_ks)
#pragma unroll
        for (int a = 0; a < kPieces; a++) {
          n0[a] = __ldg(kf + ((size_t)(ks + 1) * kPieces + a) * 32);
          n1[a] = __ldg(kf + half + ((size_t)(ks + 1) * kPieces + a) * 32);
        }
      mma_bf16_16816(l2, af[0], b2);
      mma_bf16_16816(hi, af[0], b0);
      mma_bf16_16816(lo, af[0], b1);
      mma_bf16_16816(l2, af[2], b0);
      mma_bf16_16816(lo, af[1], b0);
      mma_bf16_16816(l2, af[1], b1);
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const int r = mt * 16 + g + 8 * (i >> 1), q = 2 * t4 + (i & 1);
      if (q < NC && r < n_nt * 8) O[(size_t)q * os + r] = hi[i] + (lo[i] + l2[i]);
    }
  }
}

template <int T, int TH, int NC>
__device__ __forceinline__ void solve_product(const uint2 *__restrict__ kfrag, int n_nt, int n_ks, int ksp,
                                              const __nv_bfloat16 *P, float *O, int os) {
  if constexpr (T == 1) return solve_product_one<TH, NC>(kfrag, n_nt, n_ks, ksp, P, O, os);
  constexpr int R = tile_rows(NC, T), MT = (R + 15) / 16;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  const int arow = (lane & 7) + ((lane >> 3) & 1) * 8, acol = (lane >> 4) * 8;
  for (int nt = w; nt < n_nt; nt += TH / 32) {
    float hi[MT][4], lo[MT][4], l2[MT][4];
#pragma unroll
    for (int mt = 0; mt < MT; mt++)
#pragma unroll
      for (int i = 0; i < 4; i++) hi[mt][i] = lo[mt][i] = l2[mt][i] = 0.0f;
    const uint2 *kf = kfrag + (size_t)nt * n_ks * kPieces * 32 + lane;
    uint2 nx[kPieces];
#pragma unroll
    for (int b = 0; b < kPieces; b++) nx[b] = __ldg(kf + b * 32);
    for (int ks = 0; ks < n_ks; ks++) {
      uint2 bf[kPieces];
#pragma unroll
      for (int b = 0; b < kPieces; b++) bf[b] = nx[b];
      if (ks + 1 < n_ks)
#pragma unroll
        for (int b = 0; b < kPieces; b++) nx[b] = __ldg(kf + ((size_t)(ks + 1) * kPieces + b) * 32);
      unsigned af[kPieces][MT][4];
#pragma unroll
      for (int a = 0; a < kPieces; a++)
#pragma unroll
        for (int mt = 0; mt < MT; mt++) ldsm_x4(af[a][mt], P + ((size_t)a * R + mt * 16 + arow) * ksp + ks * 16 + acol);
#pragma unroll
      for (int mt = 0; mt < MT; mt++) {
        mma_bf16_16816(l2[mt], af[2][mt], bf[0]);
        mma_bf16_16816(hi[mt], af[0][mt], bf[0]);
        mma_bf16_16816(lo[mt], af[1][mt], bf[0]);
        mma_bf16_16816(l2[mt], af[0][mt], bf[2]);
        mma_bf16_16816(lo[mt], af[0][mt], bf[1]);
        mma_bf16_16816(l2[mt], af[1][mt], bf[1]);
      }
    }
#pragma unroll
    for (int mt = 0; mt < MT; mt++)
#pragma unroll
      for (int h = 0; h < 2; h++)
        if (mt * 16 + g + 8 * h < NC * T)
          *reinterpret_cast<float2 *>(O + (size_t)(mt * 16 + g + 8 * h) * os + nt * 8 + 2 * t4) =
              make_float2(hi[mt][2 * h] + (lo[mt][2 * h] + l2[mt][2 * h]),
                          hi[mt][2 * h + 1] + (lo[mt][2 * h + 1] + l2[mt][2 * h + 1]));
  }
}

struct SolveArgs {
  const uint2 *kfrag;   // [n_nt][solve_ks][3][32] B fragments of the operator's pieces, nodes 1..N
  const float *k0;      // [N] its column of node 0
  const float *mu32;    // [B]
  float4 *rec;          // [4 + B][n][T] node records
  float4 *near[2];      // where the first two planes are
  int B, indirect;
};

// Runs the solves of the slots with sv.mode != SOLVE_NONE (sv.mode, sv.w2 in place
// and synchronised, their records in sa.rec): on return (synchronised) sv.state
// says how each ended and sv.it its sweeps, and the returned deviations
// [group p][component][T][U], nodes U p + 1 .., hold the last product omega2 K [..].
template <int T, int TH, int ORDER>
__device__ __forceinline__ const float *tile_solve(const Sweep &s, const SolveArgs &sa, SolveShared<T> &sv,
                                                    unsigned char *sm) {
  constexpr int NC = ORDER == 1 ? 6 : 3, R = tile_rows(NC, T), AQ = ORDER == 1 ? 3 : 0;  // AQ: first acceleration row
  constexpr int U = solve_group(T);
  const int tid = threadIdx.x, lane = tid & 31, N = s.N, np = (N + U - 1) / U;
  const int n_ks = solve_ks(N), n_nt = (N + 7) / 8, kst = solve_kst(N), os = solve_ostride(N);
  const size_t piece = (size_t)R * kst;
  __nv_bfloat16 *P = reinterpret_cast<__nv_bfloat16 *>(sm);
  float *O = reinterpret_cast<float *>(sm + kPieces * piece * sizeof(__nv_bfloat16));
  float *dl = O + (size_t)NC * T * os;
  const int t = tid % T, mode = sv.mode[t];
  const float w2 = sv.w2[t];
  for (size_t i = tid; i < kPieces * piece / 2; i += TH) reinterpret_cast<unsigned *>(P)[i] = 0u;
  for (int i = tid; i < np * 6 * T * U; i += TH) dl[i] = 0.0f;
  if (tid < T) {
    sv.state[tid] = mode == SOLVE_NONE ? SOLVE_OK : SOLVE_RUN;
    sv.it[tid] = sv.nst[tid] = 0;
    sv.ebest[tid] = __int_as_float(0x7f800000);
    sv.emax[tid] = sv.dmax[tid] = 0u;
  }
  __syncthreads();
  auto record = [&](int j) {
    const size_t at = (size_t)j * T + t, plane = (size_t)s.n * T;
    return [&sa, at, plane](int f) { return f < 2 ? sa.near[f][at] : sa.rec[f * plane + at]; };
  };
  auto row = [&](int q, int p) { return P + (size_t)(q * T + t) * kst + U * p; };
  // residual of half a node (corrections)
  auto residual = [&](int j, int c0, float r[6]) {
    r[c0] = r[c0 + 1] = r[c0 + 2] = 0.0f;
    if (mode == SOLVE_CORR) {
      const float4 a = record(j)(c0 == 0 ? 1 : 3);
      r[c0] = a.x;
      r[c0 + 1] = a.y;
      r[c0 + 2] = a.z;
    }
  };
  // force rows of the group p at deviations d (and, first order, its velocity rows)
  auto put_force = [&](int p, const float d[U][6]) {
    float a[U][3];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int j = U * p + 1 + u;
      if (u == 0 || j <= N) {
        solve_force(mode, sa.B, sa.mu32, sa.indirect, w2, d[u], record(j), a[u]);
      } else {
        a[u][0] = a[u][1] = a[u][2] = 0.0f;
      }
    }
#pragma unroll
    for (int q = 0; q < 3; q++) {
      float x[U];
#pragma unroll
      for (int u = 0; u < U; u++) x[u] = a[u][q];
      put_pieces<U>(row(AQ + q, p), piece, x);
      if (ORDER == 1) {
#pragma unroll
        for (int u = 0; u < U; u++) x[u] = U * p + 1 + u <= N ? w2 * d[u][3 + q] : 0.0f;
        put_pieces<U>(row(q, p), piece, x);
      }
    }
  };
  if (mode != SOLVE_NONE) {
    const float z[U][6] = {};
    for (int p = tid / T; p < np; p += TH / T) put_force(p, z);
    if (tid < T) {
      float a[3];
      solve_force(mode, sa.B, sa.mu32, sa.indirect, w2, z[0], record(0), a);
#pragma unroll
      for (int q = 0; q < 3; q++) sv.a0[q][t] = a[q];
    }
  }
  // A correction's first force deviation is zero, and so is its product: when no
  // slot starts a new segment the first sweep goes without.
  bool zero = !__syncthreads_or(mode == SOLVE_KEPLER);
  const float a0[3] = {sv.a0[0][t], sv.a0[1][t], sv.a0[2][t]};
  for (;;) {
    float em = 0.0f, dm = 0.0f;  // squares
    const bool live = sv.state[t] == SOLVE_RUN, first = sv.it[t] == 0;
    // One half of the group's states (components c0 .. c0 + 2, product rows q0 ..): the
    // new product into dl, the new deviation (product and residual) in cn, its change
    // and size.  The first sweep starts at zero deviation.
    auto half = [&](int p, int c0, int q0, const float res[U][6], float acc[U][3], float cn[U][3]) {
      float d[U][3], k0[U];
#pragma unroll
      for (int u = 0; u < U; u++) k0[u] = c0 == 3 ? __ldg(sa.k0 + min(U * p + u, N - 1)) : 0.0f;
#pragma unroll
      for (int q = 0; q < 3; q++) {
        const float *o = O + (size_t)((q0 + q) * T + t) * os + U * p;
        float *dp = dl + (((size_t)p * 6 + c0 + q) * T + t) * U;
        float x[U], old[U];
        if constexpr (U == 2) {
          const float2 ov = zero ? make_float2(0.0f, 0.0f) : *reinterpret_cast<const float2 *>(o);
          const float2 dv = *reinterpret_cast<const float2 *>(dp);
          x[0] = ov.x;
          x[U - 1] = ov.y;
          old[0] = dv.x;
          old[U - 1] = dv.y;
        } else {
          x[0] = zero ? 0.0f : o[0];
          old[0] = dp[0];
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
          if (c0 == 3 && !zero) x[u] = fmaf(k0[u], a0[q], x[u]);
          acc[u][q] = x[u];
          cn[u][q] = res[u][c0 + q] + x[u];
          d[u][q] = first ? cn[u][q] : cn[u][q] - (res[u][c0 + q] + old[u]);
        }
        if constexpr (U == 2) *reinterpret_cast<float2 *>(dp) = make_float2(x[0], x[U - 1]);
        else dp[0] = x[0];
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        const int j = U * p + 1 + u;
        if (u > 0 && j > N) continue;
        float inv = 1.0f;
        if (s.relative) {
          const float4 b = record(j)(c0 == 0 ? 0 : 2);
          const float y0 = b.x + cn[u][0], y1 = b.y + cn[u][1], y2 = b.z + cn[u][2];
          const float yy = y0 * y0 + y1 * y1 + y2 * y2, ir = rsqrtf(yy);
          if (yy > 0.0f) inv = ir * ir;
        }
        em = nanmaxf(em, (d[u][0] * d[u][0] + d[u][1] * d[u][1] + d[u][2] * d[u][2]) * inv);
        dm = fmaxf(dm, (cn[u][0] * cn[u][0] + cn[u][1] * cn[u][1] + cn[u][2] * cn[u][2]) * inv);
      }
    };
    if (!zero) {
      solve_product<T, TH, NC>(sa.kfrag, n_nt, n_ks, kst, P, O, os);
      __syncthreads();
    }
    if (ORDER == 2) {
      if (live) {
        for (int p = tid / T; p < np; p += TH / T) {
          float res[U][6], acc[U][3], cn[U][3];
#pragma unroll
          for (int u = 0; u < U; u++) residual(min(U * p + 1 + u, N), 3, res[u]);
          half(p, 3, 0, res, acc, cn);
          // the position rows integrate the change of the sweep's velocities: delta_v
          // (new segment) or c_v - R_v (a correction: the residual of a second-order
          // sweep already holds R_v)
#pragma unroll
          for (int q = 0; q < 3; q++) {
            float x[U];
#pragma unroll
            for (int u = 0; u < U; u++) x[u] = U * p + 1 + u <= N ? w2 * acc[u][q] : 0.0f;
            put_pieces<U>(row(q, p), piece, x);
          }
        }
      }
      if (!zero) {
        __syncthreads();
        solve_product<T, TH, NC>(sa.kfrag, n_nt, n_ks, kst, P, O, os);
        __syncthreads();
      }
    }
    if (live) {
      for (int p = tid / T; p < np; p += TH / T) {
        float res[U][6], acc[U][3], cn[U][3], d[U][6];
#pragma unroll
        for (int hf = 0; hf < (ORDER == 1 ? 2 : 1); hf++) {
#pragma unroll
          for (int u = 0; u < U; u++) residual(min(U * p + 1 + u, N), 3 * hf, res[u]);
          half(p, 3 * hf, 3 * hf, res, acc, cn);
#pragma unroll
          for (int q = 0; q < 3; q++)
#pragma unroll
            for (int u = 0; u < U; u++) d[u][3 * hf + q] = cn[u][q];
        }
        put_force(p, d);
      }
    }
    {
      const int e = slot_max<T>((int)err_bits32(em)), d = slot_max<T>((int)err_bits32(dm));
      if (lane < T) {
        atomicMax(&sv.emax[t], (unsigned)e);
        atomicMax(&sv.dmax[t], (unsigned)d);
      }
    }
    __syncthreads();
    bool more = false;
    if (tid < T && live) {
      const float e = sqrtf(__uint_as_float(sv.emax[tid])), d = sqrtf(__uint_as_float(sv.dmax[tid]));
      const float eb = sv.ebest[tid];
      const int it = ++sv.it[tid];
      sv.emax[tid] = sv.dmax[tid] = 0u;
      if (!((double)e <= s.div_limit)) {
        sv.state[tid] = SOLVE_FAIL;
      } else {
        const int nst = e < 0.5f * eb ? 0 : sv.nst[tid] + 1;
        sv.nst[tid] = nst;
        sv.ebest[tid] = fminf(eb, e);
        if ((mode == SOLVE_KEPLER && (double)e < s.switch_tol) ||
            e < (mode == SOLVE_CORR ? kSolveCorrFloor : kSolveFloor) * d || nst >= 2 || it >= s.max_iters)
          sv.state[tid] = SOLVE_OK;
      }
      more = sv.state[tid] == SOLVE_RUN;
    }
    zero = false;
    if (!__syncthreads_or(more)) break;
  }
  return dl;
}

// Node records of the slots with a solve to run.  Kepler: about the warm start in Yc.
// Correction: about the iterate Yo = v.Yn that the last FP64 sweep started from, with
// its residual Yc - Yo.  Positions, differences and mu/r^3 are formed in float pairs
// (48 bits) and rounded to FP32; only the residual's cancellation needs FP64.
template <int T, int TH, bool EIH>
__device__ __forceinline__ void tile_records(const Model &md, const TileView &v, const TileShared<T> &sh,
                                             const SolveShared<T> &sv, const SolveArgs &sa, int n) {
  const int t = threadIdx.x % T, m = sh.col[t], mode = sv.mode[t], B = md.B;
  const size_t plane = (size_t)n * T;
  if (m < 0 || mode == SOLVE_NONE) return;
  const float2 muc = split_pair(md.mu_c);
  for (int j = threadIdx.x / T; j < n; j += TH / T) {
    const size_t at = (size_t)j * T + t;
    float4 *rec = sa.rec + at;
    const double *Ej = sh.eb[t] + (size_t)j * v.F;
    const float2 *pair = reinterpret_cast<const float2 *>(Ej + 3 * B + 3);
    const double *yb = (mode == SOLVE_CORR ? v.Yn : v.Yc) + (size_t)j * 6 * v.ld + m;
    float2 x[3];
    float h[3], l[3], vel[3];
#pragma unroll
    for (int q = 0; q < 3; q++) {
      x[q] = split_pair(yb[(size_t)q * v.ld]);
      h[q] = x[q].x + x[q].y;
      l[q] = x[q].y - (h[q] - x[q].x);
      vel[q] = round_float(yb[(size_t)(3 + q) * v.ld]);
    }
    float r2, kh, kl;
    pair_cube(h, l, muc, r2, kh, kl);
    sa.near[0][at] = make_float4(h[0], h[1], h[2], kh + kl);
    rec[2 * plane] = make_float4(vel[0], vel[1], vel[2], 0.0f);
    float r[6] = {};
    if (mode == SOLVE_CORR) {
      if (j > 0)
#pragma unroll
        for (int q = 0; q < 6; q++) r[q] = round_float(v.Yc[((size_t)j * 6 + q) * v.ld + m] - yb[(size_t)q * v.ld]);
      rec[3 * plane] = make_float4(r[3], r[4], r[5], 0.0f);
    } else {
#pragma unroll
      for (int q = 0; q < 3; q++) r[q] = EIH ? round_float(Ej[3 * B + q]) : -(pair[3 * B + q].x + pair[3 * B + q].y);
    }
    sa.near[1][at] = make_float4(r[0], r[1], r[2], __fdividef(1.0f, r2));
    for (int b = 0; b < B; b++) {
      float d[3];
#pragma unroll
      for (int q = 0; q < 3; q++) {
        const float2 p = EIH ? split_pair(Ej[3 * b + q]) : pair[3 * b + q];
        float e;
        const float s = two_diff(x[q].x, p.x, e);
        d[q] = s + (e + (x[q].y - p.y));
      }
      float k = 0.0f;
      if (mode == SOLVE_CORR) {
        const float ir = rsqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
        k = __ldg(sa.mu32 + b) * ir * ir * ir;
      }
      rec[(4 + b) * plane] = make_float4(d[0], d[1], d[2], k);
    }
  }
}

}  // namespace
}  // namespace pcx
