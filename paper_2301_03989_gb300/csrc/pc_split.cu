// The steps of the resident kernel's sweep as entry points of their own.
// pc_apply_operator: Y = 1 x0^T + K G over columns 0..n_ic-1 by the exact digit products of
// pc_tile.cuh (Section "Matrix form for vectorized and parallel computation", the operators
// collapsed into one (N+1)x(N+1) K).  pc_eval_dynamics: the force of tile_accel on the body
// data of pc_bodies.cuh.
#include <algorithm>

#include "pc_bodies.cuh"

namespace pcx {
namespace {

constexpr int kApplyT = 8, kApplyThreads = 128, kApplyCtas = 2;  // 48 digit rows, two CTAs an SM

__global__ void __launch_bounds__(kApplyThreads, kApplyCtas)
    k_apply_split(SplitOp op, const double *__restrict__ x0, const double *__restrict__ G, double *__restrict__ Y,
                  int n_ic, int ld, int N) {
  constexpr int T = kApplyT, TH = kApplyThreads;
  extern __shared__ __align__(16) unsigned char split_sm[];
  __shared__ TileShared<T> sh;
  __nv_bfloat16 *Gd = reinterpret_cast<__nv_bfloat16 *>(split_sm);
  const int tid = threadIdx.x, t = tid % T, n = N + 1;
  for (int e0 = blockIdx.x * T; e0 < n_ic; e0 += gridDim.x * T) {
    if (tid < T) {
      sh.col[tid] = e0 + tid < n_ic ? e0 + tid : -1;
      sh.bad[tid] = 0;
    }
    if (tid < 6 * T) sh.colB[tid] = 0;
    __syncthreads();
    const int m = sh.col[t];
    int ex[6] = {0, 0, 0, 0, 0, 0};
    if (m >= 0)
      for (int j = tid / T; j < n; j += TH / T)
#pragma unroll
        for (int q = 0; q < 6; q++) {
          ex[q] = max(ex[q], biased_exp(G[((size_t)j * 6 + q) * ld + m]));
          if (j == 0) Y[(size_t)q * ld + m] = x0[(size_t)q * ld + m];  // row 0 of K is zero
        }
#pragma unroll
    for (int q = 0; q < 6; q++) {
      ex[q] = slot_max<T>(ex[q]);
      if ((tid & 31) < T) atomicMax(&sh.colB[q * T + t], ex[q]);
    }
    __syncthreads();
    if (tid < 6 * T && sh.colB[tid] == 0x7ff) sh.bad[tid % T] = 1;
    tile_split<T, TH, 6>(sh, sh.colB, Gd, n, op.n_ks,
                         [&](int q, int, int c, int k) { return G[((size_t)k * 6 + q) * ld + c]; });
    __syncthreads();
    tile_product<T, TH, 6>(op, sh, sh.colB, Gd, N, [&](int u, int j, int, const double *val, const int *e) {
      const int c = sh.col[u];
#pragma unroll
      for (int q = 0; q < 6; q++)
        Y[((size_t)j * 6 + q) * ld + c] = sh.bad[u] ? __longlong_as_double(0x7FF8000000000000LL)
                                                    : fma(val[q], scale_exp(1.0, e[q]), x0[(size_t)q * ld + c]);
    });
    __syncthreads();  // shared memory is reused by the next tile
  }
}

// Dynamics at n points, a thread each; a thread's body data lie in shared memory (an odd
// number of doubles apart).  EIH: the relativistic terms are added to the Newtonian force
// (the sweeps form both in one pass of eih_accel).  Bound by FP64 latency and, with many
// bodies, by the ephemeris loads: 1,000,000 points 282 us with two bodies, 1,182 with nine
// (1,361 with blocks cut to 48 KB of shared memory).
template <bool EIH>
__global__ void k_eval_force(const Model md, long long n, int stride, const double *__restrict__ t,
                             const double *__restrict__ y, double *__restrict__ f) {
  extern __shared__ double bodies[];
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double *data = bodies + (size_t)threadIdx.x * stride;
  const EphemLoc L = ephem_locate(md, t[i]);
  double x[6], a[3];
  for (int q = 0; q < 6; q++) x[q] = y[(size_t)q * n + i];
  body_data<false>(md, L, data, central_square(md, x));
  tile_accel(md, data, x, a);
  if (EIH) {
    double vb[kMaxBodies * 3], X[7 * (kMaxBodies + 1)], rel[3];
    ephem_vel_all(md, L, [&](int b, const double v[3]) {
      for (int ax = 0; ax < 3; ax++) vb[3 * b + ax] = v[ax];
    });
    eih_bodies(md, data, vb, X);
    eih_accel<false>(md, data, data + 3 * md.B, X, 1, x, x + 3, rel);
    for (int q = 0; q < 3; q++) a[q] += rel[q];
  }
  for (int q = 0; q < 3; q++) {
    f[(size_t)q * n + i] = x[3 + q];
    f[(size_t)(3 + q) * n + i] = a[q];
  }
}

}  // namespace

bool split_supported(const pc_plan *p) { return p->d_Kdig != nullptr; }

cudaError_t launch_apply_split(const pc_plan *p, long long n_ic, int ld, const double *x0, const double *G, double *Y,
                               cudaStream_t st) {
  const size_t smem = tile_digit_bytes(6, kApplyT, p->split_ks);
  const cudaError_t e = allow_shared(k_apply_split);
  if (e != cudaSuccess) return e;
  const SplitOp op{reinterpret_cast<const uint2 *>(p->d_Kdig), p->d_Kexp, p->split_nt, p->split_ks};
  const long long tiles = (n_ic + kApplyT - 1) / kApplyT;
  const int sms = p->num_sms > 0 ? p->num_sms : 152;
  k_apply_split<<<(unsigned)std::min<long long>((long long)sms * kApplyCtas, tiles), kApplyThreads, smem, st>>>(
      op, x0, G, Y, (int)n_ic, ld, p->N);
  return cudaGetLastError();
}

cudaError_t launch_eval_force(const pc_plan *p, long long n, const double *t, const double *y, double *f,
                              cudaStream_t st) {
  auto kernel = p->model.c_light > 0.0 ? k_eval_force<true> : k_eval_force<false>;
  const cudaError_t e = allow_shared(kernel);
  if (e != cudaSuccess) return e;
  const int stride = (int)res_bodies(p->model.B, false) | 1;
  int threads = 128;  // 32 bodies: 201 doubles, 64 threads
  while (threads > 32 && sizeof(double) * stride * threads > 104 * 1024) threads /= 2;
  kernel<<<(unsigned)((n + threads - 1) / threads), threads, sizeof(double) * stride * threads, st>>>(p->model, n, stride,
                                                                                                      t, y, f);
  return cudaGetLastError();
}

}  // namespace pcx
