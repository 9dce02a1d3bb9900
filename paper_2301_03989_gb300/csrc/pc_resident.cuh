// The resident kernel: a whole FP64 propagation (PC_CONTRACT_SPLIT) in one launch.
//
// Trajectories never wait on each other, so nothing needs a grid-wide step.  A
// CTA owns T slots and keeps a trajectory in a slot from its first segment to its
// last: set-up of a new segment (ephemeris, Keplerian warm start), sweeps
// (pc_tile.cuh), stop, resolution and schedule decisions; a slot whose trajectory
// ends takes the next one from a counter.  The control state lives in shared
// memory, the iterate, accelerations and body positions in shared memory when
// they fit or in scratch that stays in L2 (26 KB a slot at N = 128 and two bodies).
//
// Against one launch per step of a round over all trajectories (seven kernels, 40
// to 180 us a round however few trajectories there were) this takes out the
// launches, the host's look at the counters, the rounds a finished batch still
// ran, and every pass over HBM.  Two CTAs of 128 threads per SM: one's tensor-core
// product runs beside the other's FP64 work.  What bounds it is the FP64 pipe
// (force and epilogue, see pc_tile.cuh) for full tiles, and the chain of phases of
// one sweep for a few trajectories.
#pragma once

#include <algorithm>

#include "pc_tile.cuh"
#include "pc_traj.cuh"

namespace pcx {
namespace {

// Threads of a CTA and CTAs per SM by the slots' digit rows: 16 rows (a few
// trajectories, where the length of a sweep's chain of phases counts) 256 threads,
// more rows 128 threads and as many CTAs as their digits and registers leave.
__host__ __device__ constexpr int res_rows(int T, int order) { return tile_rows(order == 1 ? 6 : 3, T); }
__host__ __device__ constexpr int res_threads(int T, int order) { return res_rows(T, order) == 16 ? 256 : 128; }
__host__ __device__ constexpr int res_ctas(int T, int order) { return res_rows(T, order) == 32 ? 3 : 2; }
constexpr long long kResMaxSweeps = 10000000LL;  // of one CTA: the round cap of a call

// Scratch of one CTA in doubles: per slot two iterates, body positions and summed
// indirect term (EIH: the bodies' data), the 17 warm-start solves; accelerations
// and tail parts by slot of the tile.
__host__ __device__ inline size_t res_bodies(int B, bool eih) { return 3 * B + 3 + (eih ? eih_stride(B) : 0); }
__host__ __device__ inline size_t res_scratch(int n, int B, bool eih, int cols, int T) {
  return (size_t)cols * ((size_t)n * (12 + res_bodies(B, eih)) + (size_t)kKepNodes * 6) + (size_t)n * 3 * T +
         tile_tail_doubles(T);
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
  double *scratch;     // [CTAs][scratch_stride], or nullptr: scratch in shared memory
  size_t scratch_stride;
  int tpc;             // slots used per CTA, <= T
  int *queue;          // next trajectory to take, beyond the first gridDim * tpc
  int *done;           // [0] finished, [1] stopped early
  int *rounds;         // most sweeps any CTA ran
};

template <int T, int ORDER, bool EIH>
__global__ void __launch_bounds__(res_threads(T, ORDER), res_ctas(T, ORDER))
    k_resident(Sweep s, const Model md, const SplitOp op, const ResArgs ra) {
  extern __shared__ __align__(16) unsigned char res_sm[];
  __shared__ TileShared<T> sh;
  __shared__ ResCtl<T> rc;
  __shared__ int slot_new[T], ebuf[T], tape_seg[T], tape_ic[T];
  __shared__ int n_new, n_own, own_list[T];
  __shared__ unsigned want;
  const int tid = threadIdx.x, n = s.n, N = s.N, B = md.B, tpc = ra.tpc;
  constexpr int NC = ORDER == 1 ? 6 : 3, TH = res_threads(T, ORDER);
  __nv_bfloat16 *Gd = reinterpret_cast<__nv_bfloat16 *>(res_sm);
  const size_t digits = tile_digit_bytes(NC, T, op.n_ks);
  double *scr = ra.scratch ? ra.scratch + (size_t)blockIdx.x * ra.scratch_stride
                           : reinterpret_cast<double *>(res_sm + digits);
  // iterates with tpc columns; tpc buffers of body data, [node][3B + 3 (+ EIH data)]
  double *Y[2] = {scr, scr + (size_t)n * 6 * tpc};
  const int F = (int)res_bodies(B, EIH), xs = EIH ? eih_stride(B) : 0;
  double *E = Y[1] + (size_t)n * 6 * tpc;
  float2 *y17 = reinterpret_cast<float2 *>(E + (size_t)n * F * tpc);
  double *A = reinterpret_cast<double *>(y17 + (size_t)kKepNodes * 6 * tpc);
  double *part = A + (size_t)n * 3 * T;

  const Ctl c = rc.view();  // s.ld is its leading dimension, T

  // zero digit rows stay zero
  for (size_t i = tid; i < digits / 4; i += TH) reinterpret_cast<unsigned *>(res_sm)[i] = 0u;
  auto take = [&](int t, long long i) {
    for (;;) {
      if (i >= s.n_ic) {
        sh.col[t] = -1;
        return;
      }
      bool refused;
      if (init_trajectory(s, c, md, ra.x0, t, i, &refused)) {
        sh.col[t] = t;
        return;
      }
      atomicAdd(ra.done, 1);
      if (refused) atomicAdd(ra.done + 1, 1);
      i = (long long)gridDim.x * tpc + atomicAdd(ra.queue, 1);
    }
  };
  if (tid < T) {
    rc.need_setup[tid] = 0;
    ebuf[tid] = 0;
    if (tid < tpc) take(tid, (long long)tid * gridDim.x + blockIdx.x);
    else sh.col[tid] = -1;
  }
  __syncthreads();

  int cur = 0;
  unsigned long long swept = 0;
  for (long long it = 0;; it++) {
    if (!__syncthreads_or(tid < T && sh.col[tid] >= 0)) {
      if (tid == 0) atomicMax(ra.rounds, (int)it);
      break;
    }
    // ---- new segments: which slots, and one owner per distinct node-time grid.
    // Slots with the same (w1, w2) have the same node times bit for bit and share
    // a buffer of body data; a buffer is free when no slot's segment uses it, and
    // there are as many as slots.
    if (tid < 32) {
      const int t = tid < T ? tid : 0;
      const bool live = tid < T && sh.col[t] >= 0;
      const bool need = live && rc.need_setup[t];
      const unsigned mask = __ballot_sync(0xffffffffu, need);
      const unsigned used = __reduce_or_sync(0xffffffffu, live && !need ? 1u << ebuf[t] : 0u);
      int own = tid;
      if (need) {
        for (int b = 0; b < tid; b++)
          if (((mask >> b) & 1u) && __double_as_longlong(rc.w1[b]) == __double_as_longlong(rc.w1[tid]) &&
              __double_as_longlong(rc.w2[b]) == __double_as_longlong(rc.w2[tid])) {
            own = b;
            break;
          }
        slot_new[__popc(mask & ((1u << tid) - 1u))] = tid;
      }
      const unsigned om = __ballot_sync(0xffffffffu, need && own == tid);
      if (need && own == tid) {
        const int k = __popc(om & ((1u << tid) - 1u));
        own_list[k] = tid;
        ebuf[tid] = (int)__fns(~used, 0, k + 1);
      }
      __syncwarp();
      if (need && own != tid) ebuf[tid] = ebuf[own];
      if (tid == 0) {
        n_new = __popc(mask);
        n_own = __popc(om);
      }
      if (tid < T) {
        sh.fresh[tid] = need;
        sh.eoff[tid] = (unsigned)ebuf[tid] * (unsigned)(n * F);
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
      const int nk = s.warm && s.kep_stride > 0 ? n_new * kKepNodes : 0, ne = n_own * n;
      for (int i = tid; i < nk + ne; i += TH) {
        if (i < nk) {
          const int m = slot_new[i % n_new];
          if (kepler_interpolated(s, c, m)) warm_solve(s, c, ra.tau, i / n_new, m, y17, tpc, m);
        } else {
          const int j = (i - nk) / n_own, m = own_list[(i - nk) % n_own];
          const EphemLoc L = ephem_locate(md, dadd(rc.w1[m], dmul(rc.w2[m], ra.tau[j])));
          double *Ej = E + (size_t)ebuf[m] * n * F + (size_t)j * F;
          if (EIH) {
            double rb[kMaxBodies * 3], vb[kMaxBodies * 3], X[7 * (kMaxBodies + 1)];
            ephem_all(md, L, [&](int b, const double r[3]) {
              for (int ax = 0; ax < 3; ax++) rb[3 * b + ax] = r[ax];
            });
            ephem_vel_all(md, L, [&](int b, const double v[3]) {
              for (int ax = 0; ax < 3; ax++) vb[3 * b + ax] = v[ax];
            });
            eih_bodies(md, rb, vb, X);
            for (int f = 0; f < xs; f++) Ej[3 * B + 3 + f] = X[f];
          }
          double ind[3] = {0.0, 0.0, 0.0};
          ephem_all(md, L, [&](int b, const double r[3]) {
            if (md.indirect) add_indirect(md, b, r, ind);
            for (int ax = 0; ax < 3; ax++) Ej[b * 3 + ax] = r[ax];
          });
          for (int ax = 0; ax < 3; ax++) Ej[3 * B + ax] = ind[ax];
        }
      }
      __syncthreads();
      // first iterate: the warm start (interpolated, or solved at every node)
      for (int i = tid; i < n_new * n; i += TH) {
        const int j = i / n_new, m = slot_new[i % n_new];
        double x0[6], y[6];
        for (int q = 0; q < 6; q++) x0[q] = rc.x[q * T + m];
        bool ok = false;
        if (j > 0 && s.warm) {
          if (kepler_interpolated(s, c, m)) {
            ok = warm_interpolate(s, y17, tpc, j, m, x0, y);
          } else {
            double kc[kKepConsts];
            for (int q = 0; q < kKepConsts; q++) kc[q] = rc.kc[q * T + m];
            ok = kepler_solve(kc, x0, dsub(dadd(rc.w1[m], dmul(rc.w2[m], ra.tau[j])), rc.ta[m]), y);
          }
        }
        for (int q = 0; q < 6; q++) {
          const size_t o = ((size_t)j * 6 + q) * tpc + m;
          Y[cur][o] = ok ? y[q] : x0[q];
          if (j == 0) Y[cur ^ 1][o] = x0[q];
        }
      }
      __syncthreads();
    }
    // ---- one sweep of every live slot
    const TileView v{Y[cur], Y[cur ^ 1], A, E, E + 3 * B, E + 3 * B + 3, (size_t)tpc, (size_t)F, (size_t)F, (size_t)F, 1};
    tile_sweep<T, TH, ORDER, EIH>(s, md, op, v, sh, Gd, nullptr);
    // ---- stop decisions, resolution test, schedule
    int out = SEG_CONTINUE;
    if (tid < 32) {
      bool test = false;
      if (tid < T && sh.col[tid] >= 0) {
        rc.need_setup[tid] = 0;
        swept++;
        out = sweep_outcome(s, c, tid, sqrt((double)__uint_as_float(sh.emax[tid])));
        test = (out == SEG_OK || out == SEG_STALLED) && s.trunc_tol > 0.0;
      }
      const unsigned w = __ballot_sync(0xffffffffu, test);
      if (tid == 0) want = w;
    }
    if (__syncthreads_or(out != SEG_CONTINUE)) {
      if (want) {
        tile_tail_sums<T, TH>(s, v, sh, ra.tau, want, part);
        __syncthreads();
      }
      if (tid < T) {
        tape_seg[tid] = -1;
        if (out != SEG_CONTINUE) {
          if (((want >> tid) & 1u) && !(tile_tail<T>(s, sh, part, tid) <= s.trunc_tol)) out = SEG_FAIL_TRUNC;
          tape_ic[tid] = rc.ic[tid];
          const int adv = end_attempt(s, c, tid, out, v.Yn + (size_t)N * 6 * tpc + tid, tpc, &tape_seg[tid]);
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
          for (int i = tid; i < 6 * n; i += TH) rec[i] = v.Yn[(size_t)i * tpc + t];
        }
      }
      if (tid < T && sh.col[tid] >= 0 && rc.phase[tid] == PH_DONE)
        take(tid, (long long)gridDim.x * tpc + atomicAdd(ra.queue, 1));
    }
    cur ^= 1;
    if (it + 1 >= kResMaxSweeps && tid < T && sh.col[tid] >= 0) {
      // the call's round cap: the slot's trajectory, and every one it would have taken, stops here
      do {
        rc.status[tid] |= PC_IC_NOT_CONVERGED;
        write_outputs(s, c, tid);
        atomicAdd(ra.done, 1);
        atomicAdd(ra.done + 1, 1);
        take(tid, (long long)gridDim.x * tpc + atomicAdd(ra.queue, 1));
      } while (sh.col[tid] >= 0);
    }
  }
  if (tid < 32) {
    for (int o = 16; o > 0; o >>= 1) swept += __shfl_xor_sync(0xffffffffu, swept, o);
    if (tid == 0) atomicAdd(s.cnt64, swept);
  }
}

// ---- launch shape -----------------------------------------------------------
// Slots per CTA: as many as it takes to put every trajectory in a slot of one round
// of CTAs, up to the tile; more trajectories than that wait in the queue.
struct ResShape {
  int tile, tpc, grid;
  size_t smem, scratch, stride;  // scratch: bytes of the device buffer (0: in shared memory)
};
// Dynamic shared memory that lets `ctas` share an SM (228 KB, less the static part and
// the system's 1 KB each).
__host__ constexpr size_t res_smem_limit(int ctas) { return (228 * 1024) / ctas - 7 * 1024; }

// Shape with tiles of T, or tile 0 when larger tiles serve n_ic trajectories better.
template <int T, int ORDER>
ResShape res_shape(const pc_plan *p, long long n_ic, bool last) {
  ResShape r{};
  const long long sms = p->num_sms > 0 ? p->num_sms : 152;
  r.smem = tile_digit_bytes(ORDER == 1 ? 6 : 3, T, p->split_ks);
  int per_sm = res_ctas(T, ORDER);
  while (per_sm > 1 && r.smem > res_smem_limit(per_sm)) per_sm--;
  const long long slots = sms * per_sm;
  const long long want = (n_ic + slots - 1) / slots;
  if (want > T && !last) return r;
  r.tile = T;
  r.tpc = (int)std::min<long long>(want, T);
  r.grid = (int)std::min((n_ic + r.tpc - 1) / r.tpc, slots);
  r.stride = res_scratch(p->n, p->model.B, p->model.c_light > 0.0, r.tpc, T);
  const size_t all = r.smem + r.stride * sizeof(double);
  if (all <= res_smem_limit((int)((r.grid + sms - 1) / sms))) r.smem = all;
  else r.scratch = r.stride * sizeof(double) * (size_t)r.grid;
  return r;
}

template <int T, int ORDER, bool EIH>
cudaError_t res_launch(const pc_plan *p, const Sweep &s, const ResShape &r, const double *x0, cudaStream_t st) {
  const Workspace &w = p->ws;
  cudaError_t e = cudaFuncSetAttribute(k_resident<T, ORDER, EIH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)r.smem);
  if (e != cudaSuccess) return e;
  const SplitOp op{reinterpret_cast<const uint2 *>(p->d_Kdig), p->d_Kexp, p->split_nt, p->split_ks};
  const ResArgs ra{x0, p->d_tau, r.scratch ? w.res_scratch : nullptr, r.stride, r.tpc, w.ints + 15, w.ints, w.ints + 16};
  Sweep sc = s;
  sc.ld = T;  // the control state's leading dimension
  k_resident<T, ORDER, EIH><<<r.grid, res_threads(T, ORDER), r.smem, st>>>(sc, p->model, op, ra);
  return cudaGetLastError();
}

template <int T, int ORDER>
cudaError_t res_run(const pc_plan *p, const Sweep &s, const ResShape &r, const double *x0, cudaStream_t st) {
  return p->model.c_light > 0.0 ? res_launch<T, ORDER, true>(p, s, r, x0, st)
                                : res_launch<T, ORDER, false>(p, s, r, x0, st);
}

// With scratch != nullptr only the bytes of device scratch the call needs.
template <int ORDER, int T, int... More>
cudaError_t res_choose(const pc_plan *p, const Sweep &s, const double *x0, cudaStream_t st, size_t *scratch) {
  const ResShape r = res_shape<T, ORDER>(p, s.n_ic, sizeof...(More) == 0);
  if constexpr (sizeof...(More) > 0)
    if (!r.tile) return res_choose<ORDER, More...>(p, s, x0, st, scratch);
  if (scratch) {
    *scratch = r.scratch;
    return cudaSuccess;
  }
  return res_run<T, ORDER>(p, s, r, x0, st);
}

}  // namespace
}  // namespace pcx
