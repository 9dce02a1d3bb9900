// The operator product of a full tile on the 5th-generation tensor cores (tcgen05):
// 48 columns (16 trajectories x 3 components, or 8 x 6) of degree 65 to 128.
//
// D[node][d 48 + c] = sum_{a + b = d} sum_k K_a[node][k] F_b[k][c]: the digits of the
// columns stand side by side as the N extent of one operand, so operator digit a times
// columns' digits 0 .. 6 - a is one MMA (two where N = 48 (7 - a) passes 256) whose columns
// are the accumulators of the anti-diagonals a .. 6: nine MMAs a k-step for 28 digit
// pairs.  M = 128: the nodes 1..N, padded with zero rows.  The sums are the same exact
// integers as mma.sync's.
//
// The columns' digits lie in shared memory in the operand layout (8 x 8 core matrices of
// 128 contiguous bytes, no swizzle); the operator's 258 KB stream through a ring of three
// k-steps of 28 KB by bulk copies.  One thread issues the copies, another the MMAs: with
// a copy, a wait and a commit for every 4 KB tile the issuing thread took 1.4 thousand
// cycles a tile and the pass 90 thousand.  The ring's bytes are what hides the 1 us
// of a copy, so one CTA per SM takes all 48 columns.  The accumulators (336 of 512 TMEM
// columns) come back by tcgen05.ld, a thread per node and quarter of the columns.
// Every wait ends after a bounded number of polls and then raises the call's error flag.
#pragma once

#include "pc_tile.cuh"

namespace pcx {
namespace {

constexpr int kTcCols = 48;
constexpr int kTcRing = 3;                     // k-steps of the operator in flight
constexpr int kTcTile = 4096;                  // bytes of one digit of a k-step: 128 rows x 16 k
constexpr int kTcStage = kSplitDigits * kTcTile;
constexpr int kTcGroups = kSplitDigits * (kTcCols / 8);  // 8-row groups of the columns' digits
constexpr int kTcLbo = kTcGroups * 128;        // bytes between 8-k slices of the columns' digits
constexpr int kTcTmem = 512;
constexpr int kTcPolls = 1 << 18;

__host__ __device__ inline size_t tc_digit_bytes(int n_ks) { return (size_t)2 * n_ks * kTcLbo; }
__host__ __device__ inline size_t tc_smem(int n_ks) { return tc_digit_bytes(n_ks) + (size_t)kTcRing * kTcStage; }

struct TcShared {
  unsigned long long full[kTcRing], empty[kTcRing], done;
  unsigned tmem;
  int failed;
};
// Progress: k-steps asked for (the copying thread's count), products finished.
struct TcState {
  unsigned loaded = 0, passes = 0;
};
constexpr int kTcMmaThread = 0, kTcCopyThread = 32;

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_wait(unsigned long long *b, unsigned parity) {
  const unsigned a = smem_addr(b);
  for (int i = 0; i < kTcPolls; i++) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void async_proxy_fence() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// Set-up and release of the barriers and the tensor memory (all threads; synchronises).
__device__ __forceinline__ void tc_begin(TcShared &tc) {
  if (threadIdx.x == 0) {
    for (int i = 0; i < kTcRing; i++) {
      mbar_init(&tc.full[i], 1);
      mbar_init(&tc.empty[i], 1);
    }
    mbar_init(&tc.done, 1);
    tc.failed = 0;
    async_proxy_fence();
  }
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(&tc.tmem)),
                 "r"(kTcTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void tc_end(TcShared &tc) {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tc.tmem), "r"(kTcTmem) : "memory");
}

// Operand descriptor: no swizzle, K-major; lbo: bytes between the two 8-k slices, 128
// bytes between 8-row groups.
__device__ __forceinline__ unsigned long long tc_desc(unsigned addr, unsigned lbo) {
  return (unsigned long long)((addr & 0x3FFFFu) >> 4) | ((unsigned long long)(lbo >> 4) << 16) |
         ((unsigned long long)(128 >> 4) << 32) | (1ULL << 46);
}

// Place of digit b of column c at node k in the columns' operand, in bf16.
__device__ __forceinline__ size_t tc_place(int b, int c, int k) {
  return (size_t)(k >> 3) * (kTcLbo / 2) + (size_t)(b * (kTcCols / 8) + (c >> 3)) * 64 + (c & 7) * 8 + (k & 7);
}

// The copying thread: k-steps up to number `upto` of the call (they repeat with every
// pass, so the first of the next pass may be on their way before it starts).
__device__ __forceinline__ void tc_load(TcShared &tc, TcState &st, unsigned char *ring, const unsigned char *op,
                                        int n_ks, unsigned upto) {
  for (; st.loaded < upto && !tc.failed; st.loaded++) {
    const unsigned slot = st.loaded % kTcRing;
    if (st.loaded >= kTcRing && !mbar_wait(&tc.empty[slot], (st.loaded / kTcRing - 1) & 1)) {
      tc.failed = 1;
      return;
    }
    const unsigned bar = smem_addr(&tc.full[slot]);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(kTcStage) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     smem_addr(ring + (size_t)slot * kTcStage)),
                 "l"(op + (size_t)(st.loaded % n_ks) * kTcStage), "r"(kTcStage), "r"(bar)
                 : "memory");
  }
}
// Waits for the copies still in flight (the copying thread, before the CTA ends).
__device__ __forceinline__ void tc_drain(TcShared &tc, TcState &st, int n_ks) {
  for (unsigned u = st.passes * n_ks; u < st.loaded; u++) mbar_wait(&tc.full[u % kTcRing], (u / kTcRing) & 1);
}

// The product: out(t0, j, q0, val, kx) with val[3][4]: components q0 .. q0 + 2 of slots
// t0 .. t0 + 3 at node j.  The digits are in place; called by all threads after a barrier.
template <int T, int TH, class Out>
__device__ __forceinline__ void tc_product(TcShared &tc, TcState &st, const TileShared<T> &sh, const int *colB,
                                           const unsigned char *op, const int *kexp, int n_ks, int N,
                                           unsigned char *Gd, unsigned char *ring, bool prefetch, Out out) {
  static_assert(TH == 512 && (T == 16 || T == 8), "a thread per node and quarter of the columns");
  const unsigned first = st.passes * n_ks;
  if (threadIdx.x == kTcCopyThread) {
    tc_load(tc, st, ring, op, n_ks, first + n_ks + (prefetch ? kTcRing - 1 : 0));
  } else if (threadIdx.x == kTcMmaThread) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned long long dg = tc_desc(smem_addr(Gd), kTcLbo), dr = tc_desc(smem_addr(ring), 2048);
    const unsigned tmem = tc.tmem;
    for (int ks = 0; ks < n_ks; ks++) {
      const unsigned slot = (first + ks) % kTcRing;
      if (!mbar_wait(&tc.full[slot], ((first + ks) / kTcRing) & 1)) {
        tc.failed = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
      for (int a = 0; a < kSplitDigits; a++)
#pragma unroll
        for (int b = 0; b < kSplitDigits - a; b += 5) {  // columns' digits b .. (N <= 256)
          constexpr unsigned kKind = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);  // f32 += bf16 bf16, K-major
          const unsigned n = kTcCols * (kSplitDigits - a - b < 5 ? kSplitDigits - a - b : 5);
          asm volatile(
              "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
              "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem + kTcCols * (a + b)),
              "l"(dr + (slot * kTcStage + a * kTcTile) / 16), "l"(dg + (2 * ks * kTcLbo + b * (kTcCols / 8) * 128) / 16),
              "r"(kKind | ((n >> 3) << 17)), "r"(a > 0 ? 1u : (unsigned)ks)
              : "memory");
        }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                       smem_addr(&tc.empty[slot]))
                   : "memory");
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                     smem_addr(&tc.done))
                 : "memory");
  }
  __syncwarp();
  if (!mbar_wait(&tc.done, st.passes & 1)) tc.failed = 1;
  st.passes++;
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const int warp = threadIdx.x >> 5, h = warp >> 2, j = 1 + (warp & 3) * 32 + (threadIdx.x & 31);
  const unsigned lane0 = (unsigned)(warp & 3) * 32u << 16;
  const int t0 = T == 16 ? 4 * h : 4 * (h & 1), q0 = T == 16 ? 0 : 3 * (h >> 1);
  double val[3][4];
#pragma unroll
  for (int q = 0; q < 3; q++) {
    unsigned r[kSplitDigits][4];
#pragma unroll
    for (int d = 0; d < kSplitDigits; d++)
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n"
                   : "=r"(r[d][0]), "=r"(r[d][1]), "=r"(r[d][2]), "=r"(r[d][3])
                   : "r"(tc.tmem + lane0 + (unsigned)(d * kTcCols + (q0 + q) * T + t0)));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int u = 0; u < 4; u++) {
      int S[kSplitDigits];
#pragma unroll
      for (int d = 0; d < kSplitDigits; d++) S[d] = __float2int_rn(__uint_as_float(r[d][u]));
      val[q][u] = combine_sums(S);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  if (j <= N) {
    const int kx = kexp[j - 1] - 2042 - 56;
    out(t0, j, q0, val, kx);
  }
}

}  // namespace
}  // namespace pcx
