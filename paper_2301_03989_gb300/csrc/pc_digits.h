// Host side of the digit products: an FP64 matrix as mma fragments of its digits.
#pragma once

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "pc_internal.h"

namespace pcx {

// A device copy of v in *dst; *dst is written only when all of it succeeded, so that a later
// call does not take a part of it for the whole.
template <class U>
inline cudaError_t upload(U **dst, const std::vector<U> &v) {
  U *d = nullptr;
  cudaError_t e = cudaMalloc((void **)&d, sizeof(U) * v.size());
  if (e == cudaSuccess) e = cudaMemcpy(d, v.data(), sizeof(U) * v.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) *dst = d;
  else cudaFree(d);
  return e;
}

// Digits of an N x n matrix at(r, k) as bf16 mma B fragments [ceil(N/8)][ceil(n/16)]
// [7 digits][32 lanes] x 2 words (B[k][n] = row n, k; lane (g, t) holds k = 2t, 2t+1
// and 2t+8, 2t+9 of row g) and each row's largest biased exponent.  Returns the
// largest sum of an anti-diagonal's products for column digits of 128.
template <class At>
inline double digit_frags(int N, int n, At at, std::vector<int> &exps, std::vector<unsigned> &frag) {
  const int n_nt = (N + 7) / 8, n_ks = (n + 15) / 16;
  std::vector<int> dig((size_t)N * kSplitDigits * n_ks * 16, 0);
  exps.assign(N, 0);
  double most = 0.0;
  for (int r = 0; r < N; r++) {
    std::vector<double> row(n);
    int bmax = 0;
    for (int k = 0; k < n; k++) {
      row[k] = at(r, k);
      unsigned long long b;
      std::memcpy(&b, &row[k], sizeof(b));
      bmax = std::max(bmax, (int)((b >> 52) & 0x7ff));
    }
    exps[r] = bmax;
    double sum = 0.0;
    for (int k = 0; k < n; k++) {
      int d[kSplitDigits];
      split_digits7(row[k], bmax, d);
      for (int a = 0; a < kSplitDigits; a++) {
        dig[((size_t)r * kSplitDigits + a) * n_ks * 16 + k] = d[a];
        sum += 128.0 * std::abs(d[a]);
      }
    }
    most = std::max(most, sum);
  }
  auto bf16_bits = [](int v) -> unsigned {
    const float f = (float)v;  // |v| <= 128: exact, and so is its bf16 (the top 16 bits)
    unsigned u;
    std::memcpy(&u, &f, sizeof(u));
    return u >> 16;
  };
  auto digit = [&](int r, int a, int k) -> int {
    return (r < N && k < n) ? dig[((size_t)r * kSplitDigits + a) * n_ks * 16 + k] : 0;
  };
  frag.assign((size_t)n_nt * n_ks * kSplitDigits * 32 * 2, 0u);
  for (int nt = 0; nt < n_nt; nt++)
    for (int ks = 0; ks < n_ks; ks++)
      for (int a = 0; a < kSplitDigits; a++)
        for (int lane = 0; lane < 32; lane++) {
          const int g = lane >> 2, t = lane & 3, r = nt * 8 + g, k0 = ks * 16 + 2 * t;
          unsigned *f = frag.data() + ((((size_t)nt * n_ks + ks) * kSplitDigits + a) * 32 + lane) * 2;
          f[0] = bf16_bits(digit(r, a, k0)) | (bf16_bits(digit(r, a, k0 + 1)) << 16);
          f[1] = bf16_bits(digit(r, a, k0 + 8)) | (bf16_bits(digit(r, a, k0 + 9)) << 16);
        }
  return most;
}
// The same digits as tcgen05 operand tiles, [ceil(n/16) k-steps][7 digits][2 halves of 8
// k][16 groups of 8 rows][8 rows][8 k] bf16: rows 0..N-1 of 128, zero beyond.
template <class At>
inline std::vector<unsigned short> digit_tiles(int N, int n, At at) {
  const int n_ks = (n + 15) / 16;
  std::vector<unsigned short> tiles((size_t)n_ks * kSplitDigits * 2048, 0);
  for (int r = 0; r < N; r++) {
    std::vector<double> row(n);
    int bmax = 0;
    for (int k = 0; k < n; k++) {
      row[k] = at(r, k);
      unsigned long long b;
      std::memcpy(&b, &row[k], sizeof(b));
      bmax = std::max(bmax, (int)((b >> 52) & 0x7ff));
    }
    for (int k = 0; k < n; k++) {
      int d[kSplitDigits];
      split_digits7(row[k], bmax, d);
      for (int a = 0; a < kSplitDigits; a++) {
        const float f = (float)d[a];
        unsigned u;
        std::memcpy(&u, &f, sizeof(u));
        tiles[(((size_t)(k / 16) * kSplitDigits + a) * 2 + k / 8 % 2) * 1024 + (r / 8) * 64 + r % 8 * 8 + k % 8] =
            (unsigned short)(u >> 16);
      }
    }
  }
  return tiles;
}

}  // namespace pcx
