// The operator product as an entry point of its own (pc_apply_operator): Y = 1 x0^T + K G
// over columns 0..n_ic-1 by the exact digit products of pc_tile.cuh, the same product as
// the resident kernel's sweeps (Section "Matrix form for vectorized and parallel
// computation", the operators collapsed into one (N+1)x(N+1) K).
#include <algorithm>

#include "pc_tile.cuh"

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

}  // namespace pcx
