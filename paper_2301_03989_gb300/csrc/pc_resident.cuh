// The resident kernel: a whole propagation (PC_CONTRACT_SPLIT) in one launch.
//
// Trajectories never wait on each other, so nothing needs a grid-wide step.  A
// CTA owns T slots and keeps a trajectory in a slot from its first segment to its
// last: set-up of a new segment (ephemeris, Keplerian warm start), in mixed precision
// its FP32 solves (pc_tile32.cuh), FP64 sweeps (pc_tile.cuh), stop, resolution and
// schedule decisions; a slot whose trajectory ends takes the next one from a counter.  The control state lives in shared
// memory, the iterate, accelerations and body positions in shared memory when
// they fit or in scratch that stays in L2 (26 KB a slot at N = 128 and two bodies).
//
// Against one launch per step of a round over all trajectories (seven kernels, 40
// to 180 us a round however few trajectories there were) this takes out the
// launches, the host's look at the counters, the rounds a finished batch still
// ran, and every pass over HBM: one trajectory of 97 sweeps 5.4 -> 0.91 ms, 129 flybys
// 101 -> 7.9, 65,536 mixed 392 -> 211.  Two or more CTAs share an SM where registers allow,
// so that one's tensor-core product runs beside another's FP64 work.  What bounds it for
// full tiles is the FP64 pipe (45 % busy; force and epilogue, see pc_tile.cuh) and the
// latency of phases that follow one another (8 % of stalls wait for instructions, a
// quarter for L2), and for a few trajectories the chain of phases of one sweep.
#pragma once

#include <algorithm>

#include "pc_bodies.cuh"
#include "pc_tc.cuh"
#include "pc_tile32.cuh"

namespace pcx {
namespace {

// Scratch of one CTA in doubles: per slot two iterates, body positions and summed
// indirect term (EIH: the bodies' data), the 17 warm-start solves; accelerations
// and tail parts by slot of the tile.
__host__ __device__ inline size_t res_scratch(int n, int B, bool eih, bool mixed, int cols, int T) {
  return (size_t)cols * ((size_t)n * (12 + res_bodies(B, eih)) + (size_t)kKepNodes * 6) + (size_t)n * 3 * T +
         tile_tail_doubles(T) + (mixed ? (size_t)n * 2 * solve_record(B) * T + 2 : 0);
}
// Whether the iterates have a column for every slot of the tile, used or not: then the
// epilogue of a tcgen05 product has no case for fewer.  In mixed precision, whose kernel is
// short of registers, that is worth 3 % (65,536 trajectories 219.4 -> 213.4 ms, 4096 16.05
// -> 15.95); in FP64 it costs half a percent.
__host__ __device__ constexpr bool res_whole_rows(bool mixed, bool tc) { return mixed && tc; }
// Shared memory of a CTA before its scratch: the digits, or the FP32 solves' areas in their place.
template <int T, int ORDER>
__host__ __device__ inline size_t res_area(int N, int n_ks, bool mixed, bool tc) {
  const size_t d = tc ? tc_smem(n_ks) : tile_digit_bytes(ORDER == 1 ? 6 : 3, T, n_ks);
  const size_t f = mixed ? (solve_smem(ORDER == 1 ? 6 : 3, T, N) + 15) / 16 * 16 : 0;
  return d > f ? d : f;
}

// Body data of the base segments of a common arc (every trajectory's schedule unless
// a segment is halved), formed once per call with the schedule's own arithmetic:
// the ephemeris of a tile's slots was 2 to 4 % of a sweep-bound call at two bodies
// and a quarter of an EIH one.  Thread (segment, node).
template <bool EIH>
__global__ void k_base_segments(Sweep s, Model md, const double *__restrict__ tau, int F, int n_base, double *out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)n_base * s.n) return;
  const int k = (int)(i / s.n), j = (int)(i % s.n);
  const SegmentBounds b = segment_bounds(s.max_depth, fabs(dsub(s.tfs, s.t0s)) / (double)s.segments, 0,
                                         (long long)k << s.max_depth, s.t0s, s.tfs, s.tfs >= s.t0s ? 1.0 : -1.0,
                                         fabs(dsub(s.tfs, s.t0s)));
  const double w1 = dmul(0.5, dadd(b.tb, b.ta)), w2 = dmul(0.5, dsub(b.tb, b.ta));
  body_data<EIH>(md, ephem_locate(md, dadd(w1, dmul(w2, tau[j]))), out + (size_t)i * F);
}

// Control state of the tile's slots in shared memory, with leading dimension T.
template <int T>
struct ResCtl {
  double x[6 * T], t0[T], tf[T], total[T], sgn[T], hbase[T], ta[T], tb[T], w1[T], w2[T], e_best[T];
  double kc[kKeplerConsts * T];
  unsigned long long err[T];
  long long p[T];
  int depth[T], phase[T], status[T], sweeps[T], seg_sweeps[T], nstall[T], nseg[T], need_setup[T], last[T], ic[T];
  unsigned err32[T];
  int ncorr[T];
  __device__ Ctl view() {
    Ctl c{};
    c.x = x; c.t0 = t0; c.tf = tf; c.total = total; c.sgn = sgn; c.hbase = hbase;
    c.ta = ta; c.tb = tb; c.w1 = w1; c.w2 = w2; c.e_best = e_best; c.kc = kc;
    c.err = err; c.p = p; c.depth = depth; c.phase = phase; c.status = status; c.sweeps = sweeps;
    c.seg_sweeps = seg_sweeps; c.nstall = nstall; c.nseg = nseg; c.need_setup = need_setup; c.last = last;
    c.ic = ic; c.err32 = err32; c.ncorr = ncorr;
    return c;
  }
};

struct ResArgs {
  const double *x0;    // start states (planar, io_ld)
  const double *tau;   // [n]
  const unsigned char *tc_op;  // operator tiles for tcgen05
  const double *base;  // body data of the arc's base segments, [n_base][n][F], or nullptr
  int n_base;
  double *scratch;     // [CTAs][scratch_stride], or nullptr: scratch in shared memory
  size_t scratch_stride;
  int tpc;             // slots used per CTA, <= T
  int *queue;          // next trajectory to take, beyond the first gridDim * tpc
  int *done;           // [0] finished, [1] stopped early
  int *error;          // set when a bounded wait ran out
  int *rounds;         // most rounds (FP64 sweeps and FP32 solves) any trajectory took
  long long max_rounds;  // a trajectory stops after this many
  SplitOp warm;          // the warm start's interpolation weights from the 16 solved nodes
  const uint2 *kfrag32;  // operator pieces of the FP32 solves and its column of node 0
  const float *k0;
  const float *mu32;
  int prof;            // 1: cycles per kind of work to s.cnt64[2..]
};

// A product through tcgen05 (pc_tc.cuh).
struct TcProduct {
  static constexpr bool TC = true;
  TcShared &tc;
  TcState st;
  const unsigned char *op;  // operator tiles
  const int *kexp;
  int n_ks;
  unsigned char *Gd, *ring;
  bool prefetch;            // the ring survives between products
  template <int T, int TH, int NC, class Src>
  __device__ __forceinline__ void split(const TileShared<T> &sh, const int *colB, int n, Src src) {
    __nv_bfloat16 *g = reinterpret_cast<__nv_bfloat16 *>(Gd);
    tile_split<T, TH, NC>(sh, colB, n, n_ks, src, [&](int q, int t, int k, size_t &step) {
      step = kTcCols / 8 * 64 / 2;
      return reinterpret_cast<unsigned *>(g + tc_place(0, q * T + t, k));
    });
    async_proxy_fence();  // the MMAs read through the asynchronous proxy
  }
  template <int T, int TH, class Out>
  __device__ __forceinline__ void product(const TileShared<T> &sh, const int *colB, int N, Out out) {
    tc_product<T, TH>(tc, st, sh, colB, op, kexp, n_ks, N, Gd, ring, prefetch, out);
  }
};

template <int T, int TH, int CTAS, int ORDER, bool EIH, bool MIXED, bool TC>
__global__ void __launch_bounds__(TH, CTAS)
    k_resident(Sweep s, const Model md, const SplitOp op, const ResArgs ra) {
  extern __shared__ __align__(16) unsigned char res_sm[];
  __shared__ TileShared<T> sh;
  __shared__ ResCtl<T> rc;
  __shared__ int slot_new[T], ebuf[T], tape_seg[T], tape_ic[T];
  __shared__ int n_new, n_own, own_list[T], alive[T], rnd[T], interp[T];
  __shared__ unsigned want;
  __shared__ SolveShared<T> sv;
  __shared__ int any_interp;
  __shared__ TcShared tcs;
  __shared__ unsigned long long prof_cycles[PC_KERNEL_KINDS];
  const int tid = threadIdx.x, n = s.n, N = s.N, B = md.B, tpc = ra.tpc;
  const int ld = res_whole_rows(MIXED, TC) ? T : tpc;  // columns of the iterates
  constexpr int NC = ORDER == 1 ? 6 : 3;
  __nv_bfloat16 *Gd = reinterpret_cast<__nv_bfloat16 *>(res_sm);
  double *scr = ra.scratch ? ra.scratch + (size_t)blockIdx.x * ra.scratch_stride
                           : reinterpret_cast<double *>(res_sm + res_area<T, ORDER>(N, op.n_ks, MIXED, TC));
  // iterates with ld columns; tpc buffers of body data, [node][3B + 3 (+ EIH data)]
  double *Y[2] = {scr, scr + (size_t)n * 6 * ld};
  const int F = (int)res_bodies(B, EIH);
  double *E = Y[1] + (size_t)n * 6 * ld;
  double *y17 = E + (size_t)n * F * ld;
  double *A = y17 + (size_t)kKepNodes * 6 * ld;
  double *part = A + (size_t)n * 3 * T;
  // node records of the FP32 solves, on a 16-byte boundary of the scratch
  const size_t rec_at = (size_t)(part - scr) + tile_tail_doubles(T);
  float4 *rec = reinterpret_cast<float4 *>(scr + (rec_at + 1) / 2 * 2);
  const size_t solve_at = (solve_smem(NC, T, N) + 15) / 16 * 16, plane = (size_t)n * T;
  float4 *spare = reinterpret_cast<float4 *>(res_sm + solve_at);  // of the area, beside the solves' arrays
  const size_t spared = MIXED ? (res_area<T, ORDER>(N, op.n_ks, MIXED, TC) - solve_at) / (plane * sizeof(float4)) : 0;
  const SolveArgs sa{ra.kfrag32, ra.k0, ra.mu32, rec,
                     {spared > 0 ? spare : rec, spared > 1 ? spare + plane : rec + plane}, B, md.indirect};

  std::conditional_t<TC, TcProduct, MmaProduct> pr = [&] {
    if constexpr (TC) {
      tc_begin(tcs);
      // (in mixed precision the solves' areas lie over the ring: nothing stays in flight)
      return TcProduct{tcs, TcState{}, ra.tc_op, op.kexp, op.n_ks, res_sm, res_sm + tc_digit_bytes(op.n_ks), !MIXED};
    } else {
      return MmaProduct{op, Gd};
    }
  }();
  const Ctl c = rc.view();  // s.ld is its leading dimension, T

  auto take = [&](int t, long long i) {
    for (;;) {
      alive[t] = i < s.n_ic;
      rnd[t] = 0;
      if (!alive[t]) return;
      bool refused;
      if (init_trajectory(s, c, md, ra.x0, t, i, &refused)) return;
      atomicAdd(ra.done, 1);
      if (refused) atomicAdd(ra.done + 1, 1);
      i = (long long)gridDim.x * tpc + atomicAdd(ra.queue, 1);
    }
  };
  if (tid < T) {
    rc.need_setup[tid] = 0;
    ebuf[tid] = 0;
    if (tid < tpc) take(tid, (long long)tid * gridDim.x + blockIdx.x);
    else alive[tid] = 0;
  }
  if (tid < PC_KERNEL_KINDS) prof_cycles[tid] = 0ULL;
  long long prof_at = ra.prof ? clock64() : 0;
  auto mark = [&](int kind) {
    if (ra.prof && tid == 0) {
      const long long now = clock64();
      prof_cycles[kind] += (unsigned long long)(now - prof_at);
      prof_at = now;
    }
  };
  __syncthreads();

  // index of slot t's segment among the call's base segments, -1 when it is none
  auto base_of = [&](int t) -> int {
    if (!ra.base || rc.depth[t] != 0) return -1;
    const long long p = rc.p[t], k = p >> s.max_depth;
    return (k << s.max_depth) == p && k < ra.n_base ? (int)k : -1;
  };

  int cur = 0;
  unsigned long long swept = 0, swept32 = 0;
  for (;;) {
    if (!__syncthreads_or(tid < T && alive[tid])) break;
    if (TC && tcs.failed) break;
    // ---- new segments: which slots, and one owner per distinct node-time grid.
    // Slots with the same (w1, w2) have the same node times bit for bit and share
    // a buffer of body data; a buffer is free when no slot's segment uses it, and
    // there are as many as slots.  A base segment of a common arc has its body data
    // from the call's table.
    if (tid < 32) {
      const int t = tid < T ? tid : 0;
      const bool live = tid < T && alive[t];
      const bool need = live && rc.need_setup[t], own_data = need && base_of(t) < 0;
      const unsigned mask = __ballot_sync(0xffffffffu, need), dmask = __ballot_sync(0xffffffffu, own_data);
      const unsigned used = __reduce_or_sync(0xffffffffu, live && !need ? 1u << ebuf[t] : 0u);
      int own = tid;
      if (own_data) {
        for (int b = 0; b < tid; b++)
          if (((dmask >> b) & 1u) && __double_as_longlong(rc.w1[b]) == __double_as_longlong(rc.w1[tid]) &&
              __double_as_longlong(rc.w2[b]) == __double_as_longlong(rc.w2[tid])) {
            own = b;
            break;
          }
      }
      if (need) slot_new[__popc(mask & ((1u << tid) - 1u))] = tid;
      const unsigned om = __ballot_sync(0xffffffffu, own_data && own == tid);
      if (own_data && own == tid) {
        const int k = __popc(om & ((1u << tid) - 1u));
        own_list[k] = tid;
        ebuf[tid] = (int)__fns(~used, 0, k + 1);
      }
      __syncwarp();
      if (own_data && own != tid) ebuf[tid] = ebuf[own];
      const bool ki = need && s.warm && kepler_interpolated(s, c, tid);
      const unsigned im = __ballot_sync(0xffffffffu, ki);
      if (tid == 0) {
        n_new = __popc(mask);
        n_own = __popc(om);
        any_interp = im != 0;
      }
      if (tid < T) {
        sh.col[tid] = ki || (im == 0 && live) ? tid : -1;  // the interpolation's slots first
        interp[tid] = ki;
        sh.fresh[tid] = need;
        if (MIXED) {
          sv.mode[tid] = !live ? SOLVE_NONE : need ? SOLVE_KEPLER : rc.phase[tid] == PH_CORR32 ? SOLVE_CORR : SOLVE_NONE;
          sv.w2[tid] = (float)rc.w2[tid];
        }
        sh.eb[tid] = live && base_of(tid) >= 0 ? ra.base + (size_t)base_of(tid) * n * F : E + (size_t)ebuf[tid] * n * F;
        sh.w2[tid] = rc.w2[tid];
        sh.emax[tid] = 0u;
        sh.bad[tid] = 0;
        for (int q = 0; q < 6; q++) {
          sh.x[q][tid] = rc.x[q * T + tid];
          sh.colB[q * T + tid] = 0;
        }
      }
    }
    __syncthreads();
    if (n_new > 0) {
      // Kepler's equation at the 17 interpolation nodes of every new segment, the
      // ephemeris at the nodes of every distinct grid
      const int nk = s.warm && s.kep_stride > 0 ? n_new * (kKepNodes - 1) : 0;
      const int chunks = EIH ? 1 : (B + kBodyChunk - 1) / kBodyChunk, ne = n_own * n * chunks;
      for (int i = tid; i < nk + ne; i += TH) {
        if (i < nk) {
          const int m = slot_new[i % n_new];
          if (interp[m]) {
            const int k = 1 + i / n_new;
            double d[6];
            const bool ok = warm_deviation(s, c, ra.tau, k, m, d);
#pragma unroll
            for (int q = 0; q < 6; q++) {
              y17[((size_t)k * 6 + q) * ld + m] = d[q];
              atomicMax(&sh.colB[q * T + m], ok ? biased_exp(d[q]) : 0x7ff);
            }
          }
        } else {
          const int c = (i - nk) % chunks, k = (i - nk) / chunks, j = k / n_own, m = own_list[k % n_own];
          const EphemLoc L = ephem_locate(md, dadd(rc.w1[m], dmul(rc.w2[m], ra.tau[j])));
          double *out = E + ((size_t)ebuf[m] * n + j) * F;
          if (EIH) body_data<EIH>(md, L, out);
          else body_positions(md, L, c * kBodyChunk, min(B, (c + 1) * kBodyChunk), out);
        }
      }
      __syncthreads();
      // first iterate: the warm start, interpolated (the product of the weights with the
      // 16 solved deviations, by digits like a sweep's: exact to 2^-55 of the largest
      // deviation) or solved at every node
      if (any_interp) {
        if (tid < T && interp[tid]) {
          for (int q = 0; q < 6; q++)
            if (sh.colB[q * T + tid] == 0x7ff) sh.bad[tid] = 1;  // a solve did not settle: the segment starts cold
        }
        __syncthreads();
#pragma unroll
        for (int c0 = 0; c0 < 6; c0 += NC) {
          tile_split<T, TH, NC>(sh, sh.colB + c0 * T, Gd, kKepNodes - 1, 1, [&](int q, int, int m, int k) {
            return y17[((size_t)(k + 1) * 6 + c0 + q) * ld + m];
          });
          __syncthreads();
          tile_product<T, TH, NC>(ra.warm, sh, sh.colB + c0 * T, Gd, N,
                                  [&](int t, int j, int q0, const double *val, const int *ex) {
#pragma unroll
                                    for (int q = 0; q < (T % 8 == 0 ? NC : 1); q++) {
                                      const double x = sh.x[c0 + q0 + q][t];
                                      Y[cur][((size_t)j * 6 + c0 + q0 + q) * ld + t] =
                                          sh.bad[t] ? x : fma(val[q], scale_exp(1.0, ex[q]), x);
                                    }
                                  });
          __syncthreads();
        }
        if (tid < T) {
          sh.col[tid] = alive[tid] ? tid : -1;
          sh.bad[tid] = 0;
          for (int q = 0; q < 6; q++) sh.colB[q * T + tid] = 0;
        }
      }
      if (!EIH && md.indirect)
        for (int i = tid; i < n_own * n; i += TH) {
          const int m = own_list[i % n_own];
          const double r[3] = {rc.x[m], rc.x[T + m], rc.x[2 * T + m]};
          indirect_term(md, E + ((size_t)ebuf[m] * n + i / n_own) * F, central_square(md, r));
        }
      for (int i = tid; i < n_new * n; i += TH) {
        const int j = i / n_new, m = slot_new[i % n_new];
        if (j > 0 && interp[m]) continue;
        double x0[6], y[6];
        for (int q = 0; q < 6; q++) x0[q] = rc.x[q * T + m];
        bool ok = false;
        if (j > 0 && s.warm) {
          double kc[kKepConsts];
          for (int q = 0; q < kKepConsts; q++) kc[q] = rc.kc[q * T + m];
          ok = kepler_solve(kc, x0, dsub(dadd(rc.w1[m], dmul(rc.w2[m], ra.tau[j])), rc.ta[m]), y);
        }
        for (int q = 0; q < 6; q++) {
          const size_t o = ((size_t)j * 6 + q) * ld + m;
          Y[cur][o] = ok ? y[q] : x0[q];
          if (j == 0) Y[cur ^ 1][o] = x0[q];
        }
      }
      __syncthreads();
    }
    const TileView v{Y[cur], Y[cur ^ 1], A, (size_t)ld, F};
    mark(PC_KERNEL_SETUP);
    // ---- mixed precision: the FP32 solves of new segments and of corrections; their
    // results are added to the iterate
    if (MIXED && __syncthreads_or(tid < T && sv.mode[tid < T ? tid : 0] != SOLVE_NONE)) {
      tile_records<T, TH, EIH>(md, v, sh, sv, sa, n);
      __syncthreads();
      const float *dl = tile_solve<T, TH, ORDER>(s, sa, sv, res_sm);
      {
        const int t = tid % T, m = sh.col[t];
        if (m >= 0 && sv.mode[t] != SOLVE_NONE && sv.state[t] == SOLVE_OK)
          for (int j = 1 + tid / T; j <= N; j += TH / T) {
            constexpr int U = solve_group(T);
            const float *d = dl + ((size_t)((j - 1) / U) * 6 * T + t) * U + (j - 1) % U;
            double *y = Y[cur] + (size_t)j * 6 * ld + m;
#pragma unroll
            for (int q = 0; q < 6; q++) y[(size_t)q * ld] += widen_float(d[(size_t)q * T * U]);
          }
      }
      __syncthreads();
      if (tid < T && sv.mode[tid] != SOLVE_NONE) {
        const bool fail = sv.state[tid] == SOLVE_FAIL;
        rc.sweeps[tid] += sv.it[tid];
        swept32 += (unsigned long long)sv.it[tid];
        rnd[tid] += 1;
        if (sv.mode[tid] == SOLVE_CORR) {
          if (fail) rc.ncorr[tid] = s.max_corr;
          rc.phase[tid] = PH_ITER;
        } else if (fail) {
          sh.col[tid] = -1;  // the segment attempt is over: no FP64 sweep
        } else {
          rc.phase[tid] = PH_ITER;
        }
      }
      __syncthreads();
    }
    mark(PC_KERNEL_FP32);
    // ---- one FP64 sweep
    tile_sweep<T, TH, ORDER, EIH>(s, md, pr, v, sh, mark);
    // ---- stop decisions, resolution test, schedule
    int out = SEG_CONTINUE;
    if (tid < 32) {
      bool test = false;
      if (tid < T && alive[tid]) {
        rc.need_setup[tid] = 0;
        if (sh.col[tid] >= 0) {
          const double e = (double)sqrtf(__uint_as_float(sh.emax[tid]));
          swept++;
          rnd[tid] += 1;
          out = sweep_outcome(s, c, tid, e);
          test = (out == SEG_OK || out == SEG_STALLED) && s.trunc_tol > 0.0;
          // an unfinished segment with a small change: the correction in FP32 next
          if (MIXED && out == SEG_CONTINUE && s.refine && e < s.corr_hi && rc.ncorr[tid] < s.max_corr) {
            rc.phase[tid] = PH_CORR32;
            rc.ncorr[tid] += 1;
          }
        } else {
          out = SEG_FAIL_DIV;  // the FP32 solve blew up
        }
      }
      const unsigned w = __ballot_sync(0xffffffffu, test);
      if (tid == 0) want = w;
    }
    if (__syncthreads_or(out != SEG_CONTINUE)) {
      if (want) {
        tile_tail_sums<T, TH>(s, v, sh, ra.tau, want, part);
        __syncthreads();
        tile_tail_add<T, TH>(part);
        __syncthreads();
      }
      if (tid < T) {
        tape_seg[tid] = -1;
        if (out != SEG_CONTINUE) {
          if (((want >> tid) & 1u) && !(tile_tail<T>(s, sh, part, tid) <= s.trunc_tol)) out = SEG_FAIL_TRUNC;
          tape_ic[tid] = rc.ic[tid];
          const int adv = end_attempt(s, c, tid, out, v.Yn + (size_t)N * 6 * ld + tid, ld, &tape_seg[tid]);
          if (adv != ADV_SEGMENT) {
            atomicAdd(ra.done, 1);
            if (adv == ADV_STOPPED) atomicAdd(ra.done + 1, 1);
          }
        }
      }
      if (s.tape) {  // nodes of the accepted segments to the adjoint tape
        __syncthreads();
        for (int t = 0; t < tpc; t++) {
          if (tape_seg[t] < 0) continue;
          double *rec = s.tape + ((size_t)(s.io_off + tape_ic[t]) * s.tape_seg + tape_seg[t]) * (size_t)tape_rec(n) + 2;
          for (int i = tid; i < 6 * n; i += TH) rec[i] = v.Yn[(size_t)i * ld + t];
        }
      }
      if (tid < T && alive[tid] && rc.phase[tid] == PH_DONE) {
        atomicMax(ra.rounds, rnd[tid]);
        take(tid, (long long)gridDim.x * tpc + atomicAdd(ra.queue, 1));
      }
    }
    if (tid < T && alive[tid] && rnd[tid] >= ra.max_rounds) {  // the call's round cap
      rc.status[tid] |= PC_IC_NOT_CONVERGED;
      rc.phase[tid] = PH_DONE;
      write_outputs(s, c, tid);
      atomicAdd(ra.done, 1);
      atomicAdd(ra.done + 1, 1);
      atomicMax(ra.rounds, rnd[tid]);
      take(tid, (long long)gridDim.x * tpc + atomicAdd(ra.queue, 1));
    }
    mark(PC_KERNEL_CONTROL);
    cur ^= 1;
  }
  if constexpr (TC) {
    if (tid == kTcCopyThread) tc_drain(tcs, pr.st, op.n_ks);
    if (tid == 0 && tcs.failed) *ra.error = 1;  // a wait ran out: the call fails
    tc_end(tcs);
  }
  if (tid < 32) {
    for (int o = 16; o > 0; o >>= 1) {
      swept += __shfl_xor_sync(0xffffffffu, swept, o);
      swept32 += __shfl_xor_sync(0xffffffffu, swept32, o);
    }
    if (tid == 0) {
      atomicAdd(s.cnt64, swept);
      atomicAdd(s.cnt64 + 1, swept32);
      if (ra.prof)
        for (int k = 0; k < PC_KERNEL_KINDS; k++) atomicAdd(s.cnt64 + 2 + k, prof_cycles[k]);
    }
  }
}

// ---- launch shape -----------------------------------------------------------
// Base segments whose body data the call forms once: a common arc in equal
// segments, up to 64 MB of them.
inline int res_base_segments(const pc_plan *p, const Sweep &s) {
  if (s.seg_mode != 0 || s.t0a || s.sega || p->model.B == 0) return 0;
  const size_t each = sizeof(double) * res_bodies(p->model.B, p->model.c_light > 0.0) * (size_t)p->n;
  return each * (size_t)s.segments <= (size_t)64 << 20 ? s.segments : 0;
}

// A kernel shape: T slots a CTA, threads, CTAs per SM its registers allow.
template <int T_, int TH_, int CTAS_, bool TC_ = false>
struct ResKernel {
  static constexpr int T = T_, TH = TH_, CTAS = CTAS_;
  static constexpr bool TC = TC_;
};
struct ResShape {
  int tpc, grid, rounds;         // slots used per CTA, CTAs, trajectories a slot takes in turn
  size_t smem, scratch, stride;  // scratch: bytes of the device buffer (0: in shared memory)
};
// Static shared memory of an instance, from above (its scalars and the alignment between the
// parts in 256 bytes).  The compiler reports 6,784 bytes at 16 slots and 7,488 in mixed
// precision, where this gives 6,976 and 7,680.
template <int T>
constexpr size_t res_static(bool mixed) {
  return sizeof(TileShared<T>) + sizeof(ResCtl<T>) + sizeof(TcShared) + (mixed ? sizeof(SolveShared<T>) : 0) +
         8 * T * sizeof(int) + 256;
}
// Dynamic shared memory that lets `ctas` share an SM (228 KB, less the static part and
// the system's 1 KB each) and that one block may have beside its static part (227 KB in all).
template <int T>
constexpr size_t res_smem_limit(int ctas, bool mixed) {
  return std::min((size_t)(228 * 1024) / ctas - 6 * 1024, kBlockShared - res_static<T>(mixed));
}

template <class K, int ORDER>
ResShape res_shape(const pc_plan *p, long long n_ic) {
  ResShape r{};
  const long long sms = p->num_sms > 0 ? p->num_sms : 152;
  const bool mixed = p->opt.precision == PC_PREC_MIXED;
  r.smem = res_area<K::T, ORDER>(p->N, p->split_ks, mixed, K::TC);
  int per_sm = K::CTAS;
  while (per_sm > 1 && r.smem > res_smem_limit<K::T>(per_sm, mixed)) per_sm--;
  const long long ctas = sms * per_sm;
  r.rounds = (int)((n_ic + ctas * K::T - 1) / (ctas * K::T));
  // the fewest slots a CTA that need no further round, so that the last one is full
  r.tpc = (int)((n_ic + ctas * r.rounds - 1) / (ctas * r.rounds));
  r.grid = (int)std::min((n_ic + r.tpc - 1) / r.tpc, ctas);
  r.stride = res_scratch(p->n, p->model.B, p->model.c_light > 0.0, mixed,
                         res_whole_rows(mixed, K::TC) ? K::T : r.tpc, K::T);
  r.stride = (r.stride + 1) / 2 * 2;  // every CTA's scratch on a 16-byte boundary
  const size_t all = r.smem + r.stride * sizeof(double);
  if (all <= res_smem_limit<K::T>((int)((r.grid + sms - 1) / sms), mixed)) r.smem = all;
  else r.scratch = r.stride * sizeof(double) * (size_t)r.grid;
  return r;
}

template <class K, int ORDER, bool EIH, bool MIXED>
cudaError_t res_launch(const pc_plan *p, const Sweep &s, const double *x0, cudaStream_t st, size_t *scratch) {
  const Workspace &w = p->ws;
  const ResShape r = res_shape<K, ORDER>(p, s.n_ic);
  const int n_base = res_base_segments(p, s), F = (int)res_bodies(p->model.B, EIH);
  if (scratch) {  // only the bytes of device scratch the call needs (and the plan's operator tiles)
    if (K::TC) {
      const cudaError_t e = ensure_tc_operator(const_cast<pc_plan *>(p));
      if (e != cudaSuccess) return e;
    }
    *scratch = r.scratch + sizeof(double) * (size_t)F * (size_t)p->n * (size_t)n_base;
    return cudaSuccess;
  }
  auto kernel = k_resident<K::T, K::TH, K::CTAS, ORDER, EIH, MIXED, K::TC>;
  const cudaError_t e = allow_shared(kernel);
  if (e != cudaSuccess) return e;
  const SplitOp op{reinterpret_cast<const uint2 *>(p->d_Kdig), p->d_Kexp, p->split_nt, p->split_ks};
  ResArgs ra{};
  ra.x0 = x0;
  if (n_base > 0) {
    double *base = w.res_scratch + r.scratch / sizeof(double);
    ra.n_base = n_base;
    ra.base = base;
    const long long work = (long long)n_base * s.n;
    k_base_segments<EIH><<<(unsigned)((work + 63) / 64), 64, 0, st>>>(s, p->model, p->d_tau, F, n_base, base);
    p->acc_launches += 1;
  }
  ra.tc_op = reinterpret_cast<const unsigned char *>(p->d_Ktc);
  ra.tau = p->d_tau;
  ra.scratch = r.scratch ? w.res_scratch : nullptr;
  ra.scratch_stride = r.stride;
  ra.tpc = r.tpc;
  ra.queue = w.ints + 15;
  ra.done = w.ints;
  ra.rounds = w.ints + 16;
  ra.error = w.ints + 17;
  ra.max_rounds = p->opt.max_rounds > 0 ? p->opt.max_rounds : 10000000LL;
  ra.warm = SplitOp{reinterpret_cast<const uint2 *>(p->d_Ldig), p->d_Lexp, p->split_nt, 1};
  ra.kfrag32 = reinterpret_cast<const uint2 *>(p->d_Kpieces);
  ra.k0 = p->d_K32c0;
  ra.mu32 = p->d_mu32;
  ra.prof = p->prof_on;
  Sweep sc = s;
  sc.ld = K::T;  // the control state's leading dimension
  kernel<<<r.grid, K::TH, r.smem, st>>>(sc, p->model, op, ra);
  return cudaGetLastError();
}

// Which shape.  SOLO, ONE: one slot and 256 threads, one or two CTAs per SM -- the
// shortest chain of phases, for up to a trajectory an SM (with all of an SM's
// registers: 129 flybys 7.8 against 9.1 ms with half) or two.  SMALL1, SMALL: one slot,
// or the slots whose rows fill one tile of 16, in 128 threads and four or five CTAs
// (five slots of one: 5 to 25 % slower, the registers spill).  LARGE: two tiles of 16
// rows in 256 threads and two CTAs, which reads the operator half as often.  LARGETC: 48
// columns in 512 threads and one CTA, the product by tcgen05 (pc_tc.cuh), for degrees 65
// to 128 (16,384 second-order FP64 trajectories 78.7 against 97.6 ms, first-order 146
// against 163, 65,536 mixed 240 against 253, all as first measured; 77, 143 and 211 with
// the later steps).
//
// Trajectories that start their segments together (a common arc in equal segments)
// keep a tile's slots in step; then the shape is chosen by rounds of trajectories
// through the slots times a round's cost, a measured ratio (N = 128, 20,000
// trajectories: LARGE 89 against SMALL 98 ms mixed, 172 against 175 FP64; 2501 FP64
// trajectories, two rounds against three: SMALL 14.3 against LARGE 18.8 ms).
//
// With arcs or segment lengths of their own, slots fall out of step and idle while a
// neighbour's set-up or FP32 solve runs: one slot per CTA is faster (2048 mixed
// flybys 58 against 61 ms with two slots and 73 with four; 6000 uneven arcs 149
// against 157 and 165, as first measured) until there are so many trajectories that the rounds of
// single slots cost more.  The line at 4096, about seven turns of single slots, is where FP64
// flybys are equal (1300: 31.8 against 34.5 ms with two slots, 4096: 79.9 and 81.0, 5000: 96.5
// both, 12,000: 219 against 211).  It is not as sharp as that: uneven arcs of degree 64 are
// faster with two slots from 1300 on in mixed precision (4.2 against 3.2; 12,000: 37.9 against
// 29.2), of degree 128 about equal (28.2 and 27.5), and of degree 256 single slots stay faster
// (7.1 against 9.8; 12,000: 49.5 against 65.7).  Their lengths
// differ, so up to two rounds of ONE's faster sweeps come before SMALL1 (512 gradients 42
// against 47 ms; 1000 flybys 29 against 25).
//
// The EIH force is a long chain of FP64 operations a body: 256 threads, and the smaller
// tile while every trajectory has a slot in it (second order, 1000 trajectories: 8.5 ms against
// 15.9 in the larger one, half of whose lanes idle; 1216: 8.5 and 15.9, 1500, in two turns:
// 16.6 against 15.8.  First order: 700 trajectories 11.1 against 13.8, 1216: 14.7 and 13.8).
template <int ORDER, bool MIXED, class Solo, class One, class Small1, class Small, class Large, class LargeTc, class Eih>
cudaError_t res_choose(const pc_plan *p, const Sweep &s, const double *x0, cudaStream_t st, size_t *scratch) {
  const long long sms = p->num_sms > 0 ? p->num_sms : 152;
  const bool in_step = s.seg_mode == 0 && !s.t0a && !s.sega;
  const ResShape s1 = res_shape<Small1, ORDER>(p, s.n_ic), sm = res_shape<Small, ORDER>(p, s.n_ic),
                 lg = res_shape<Large, ORDER>(p, s.n_ic);
  auto cost = [](const ResShape &r, int T, double round) { return r.rounds * round * (0.8 + 0.2 * r.tpc / T); };
  if (p->model.c_light > 0.0) {
    if (s.n_ic <= sms * One::CTAS) return res_launch<One, ORDER, true, MIXED>(p, s, x0, st, scratch);
    if (res_shape<Eih, ORDER>(p, s.n_ic).rounds == 1) return res_launch<Eih, ORDER, true, MIXED>(p, s, x0, st, scratch);
    return res_launch<Large, ORDER, true, MIXED>(p, s, x0, st, scratch);
  }
  if (s.n_ic <= sms) return res_launch<Solo, ORDER, false, MIXED>(p, s, x0, st, scratch);
  if (s.n_ic <= sms * One::CTAS) return res_launch<One, ORDER, false, MIXED>(p, s, x0, st, scratch);
  if (!in_step) {
    if (s.n_ic <= 2 * sms * One::CTAS) return res_launch<One, ORDER, false, MIXED>(p, s, x0, st, scratch);
    if (s.n_ic <= 4096) return res_launch<Small1, ORDER, false, MIXED>(p, s, x0, st, scratch);
    return res_launch<Small, ORDER, false, MIXED>(p, s, x0, st, scratch);
  }
  const double c1 = cost(s1, Small1::T, 0.75), cs = cost(sm, Small::T, MIXED ? 1.35 : 1.25);
  double cl = cost(lg, Large::T, 1.0);
  const bool tc = p->N > 64 && p->N <= 128;  // one 128-row operand, at least half of it filled
  if (tc) cl = std::min(cl, cost(res_shape<LargeTc, ORDER>(p, s.n_ic), LargeTc::T, ORDER == 1 ? 0.9 : MIXED ? 0.95 : 0.8));
  if (c1 <= cs && c1 <= cl) return res_launch<Small1, ORDER, false, MIXED>(p, s, x0, st, scratch);
  if (cs < cl) return res_launch<Small, ORDER, false, MIXED>(p, s, x0, st, scratch);
  if (tc) return res_launch<LargeTc, ORDER, false, MIXED>(p, s, x0, st, scratch);
  return res_launch<Large, ORDER, false, MIXED>(p, s, x0, st, scratch);
}

}  // namespace
}  // namespace pcx
