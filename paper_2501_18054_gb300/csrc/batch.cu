// Batched direct binary search: many independent runs in one launch.
//
// The paper notes that independent systems (one per optimisation frequency)
// are updated in parallel with no communication (section "Computational
// efficiency", Table 1 footnote 2); many random starts of DBS on one device
// are independent in the same way.  Here every run is one context (its own
// design region, possibly of a different size, its own W, state and trace),
// and one CTA advances one run at a time through the whole search: scoring,
// selection, the kept-flip update, the FP64 refresh and, on the mixed path,
// the flush of the delayed set, with only CTA-wide barriers.  (FP64 batches
// whose large runs are few go to clusters of four CTAs.)  All runs of a
// batch share one stream.  The runs wait in a queue, largest region first, and
// one CTA per SM takes the next run whenever it finishes one (an atomic
// counter): a large run then has its SM's FP64 pipe to itself, and the small
// runs fill the other SMs (longest-processing-time-first list scheduling).
//
// FIRST mode scores the visiting positions in chunks of blockDim starting at
// the current position and keeps the earliest improving one (the same
// sequential trajectory as scoring all remaining positions, with less
// speculative work when flips are kept often).
#include <cooperative_groups.h>
#include <algorithm>
#include <cstdio>
#include <memory>
#include <new>
#include <vector>

#include "delayed_search.cuh"
#include "rank1.cuh"

namespace pngf {
namespace {

constexpr int kBatchThreads = 256;

__device__ void cta_refresh(const SweepArgs& a, const ObjParams& op, c128* s_o, double* s_f) {
  __syncthreads();
  refresh_x(a, 0, a.n);
  __syncthreads();
  refresh_residual(a, 0, a.n);
  __syncthreads();
  refresh_correct(a, 0, a.n);
  __syncthreads();
  cta_ports(a, op, s_o, s_f);
}

__global__ void __launch_bounds__(kBatchThreads, 2) dbs_batch_kernel(const SweepArgs* __restrict__ runs, int n_runs,
                                                                      int* __restrict__ queue) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ c128 s_o[kMaxPorts];
  __shared__ double s_f;
  __shared__ ObjParams s_op;
  __shared__ Pivot s_pv;
  __shared__ float2 s_beta[kMaxDelay];
  __shared__ int s_k;
  __shared__ long long s_best;
  // tensor-core fold (tiles of 128 x 64): this CTA holds tc_tmem_cols(1) columns of tensor memory for all its runs
  __shared__ __align__(8) unsigned long long s_tc_bars[TC_NBAR];
  __shared__ unsigned s_tmem;
  const bool use_tc = n_runs > 0 && runs[0].tensor_fold;
  TcState tcs{};
  if (use_tc) tc_setup(tcs, s_tc_bars, &s_tmem, tc_tmem_cols(1));
  bool tc_failed = false;
  __shared__ int s_run;
  while (!tc_failed) {
    __syncthreads();  // every thread has read the previous s_run
    if (threadIdx.x == 0) s_run = atomicAdd(queue, 1);
    __syncthreads();
    const int run = s_run;
    if (run >= n_runs) break;
    const SweepArgs& a = runs[run];
    const int n = a.n;
    Control* ctl = a.ctl;
    __syncthreads();
    if (threadIdx.x == 0) {
      s_op = a.op;
      FOR_PORTS(p, a.n_o) s_o[p] = ctl->o[p];
      s_f = ctl->f;
    }
    __syncthreads();
    long long n_acc = 0, n_evals = 0, n_refresh = 0, n_flush = 0;
    int sweeps_done = 0, converged = 0, status = PNGF_OK;
    int since_refresh = ctl->since_refresh;
    int r = ctl->r_delay;
    int s = 0, t = 0, acc_in_sweep = 0;
    const long long E = (long long)n * (n + 1) / 2;
    c128* cs = reinterpret_cast<c128*>(dyn);  // FP64 path: the gathered column c, then alpha c
    c128* acs = cs + n;
    while (true) {
      const double f = s_f;
      const double thr = accept_threshold(s_op, f);
      // ---- score a chunk of positions (FIRST) or every pixel (BEST)
      long long best = LLONG_MAX;
      double g = -INFINITY;
      int pix = INT_MAX;
      c128 b_alpha = mk(0.0, 0.0), b_coef = b_alpha;
      if (a.mode == PNGF_FIRST_IMPROVEMENT) {
        const int q = t + threadIdx.x;
        if (q < n) {
          const int j = a.order ? a.order[(size_t)s * n + q] : q;
          double fn;
          c128 al, co;
          if ((unsigned)j < (unsigned)n && score_pixel(a, s_op, j, s_o, fn, nullptr, &al, &co) &&
              gain_of(s_op, fn, f) - thr > 0.0) {
            best = q;
            pix = j;
            b_alpha = al;
            b_coef = co;
          }
          if ((unsigned)j >= (unsigned)n) status = PNGF_EINVAL;
        }
        long long bmin = block_min_ll(best);
        if (bmin != LLONG_MAX && best == bmin) {
          s_k = pix;
          s_best = bmin;
          s_pv.k = pix;
          s_pv.alpha = b_alpha;
          s_pv.coef = b_coef;
          for (int p = 0; p < a.n_o; ++p) s_pv.Tk[p] = a.T[(size_t)p * a.ldt + pix];
        }
        if (threadIdx.x == 0 && bmin == LLONG_MAX) s_k = -1;
        __syncthreads();
        if (__syncthreads_or(status == PNGF_EINVAL)) {
          status = PNGF_EINVAL;
          break;
        }
        if (s_k < 0) {
          const int chunk_end = min(n, t + (int)blockDim.x);
          n_evals += chunk_end - t;
          t = chunk_end;
          if (t < n) continue;
          ++sweeps_done;
          if (acc_in_sweep == 0) { converged = 1; break; }
          ++s;
          if (s >= a.n_sweeps) break;
          t = 0;
          acc_in_sweep = 0;
          continue;
        }
        const int q_star = (int)s_best;
        n_evals += q_star - t + 1;
        t = q_star + 1;
      } else {
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
          double fn;
          c128 al, co;
          if (!score_pixel(a, s_op, j, s_o, fn, nullptr, &al, &co)) continue;
          double gg = gain_of(s_op, fn, f);
          if (better(gg, j, g, pix)) { g = gg; pix = j; b_alpha = al; b_coef = co; }
        }
        double gb = g;
        int pb2 = pix;
        block_best(gb, pb2);
        if (pb2 != INT_MAX && gb - thr > 0.0 && pix == pb2) {
          s_k = pix;
          s_pv.k = pix;
          s_pv.alpha = b_alpha;
          s_pv.coef = b_coef;
          for (int p = 0; p < a.n_o; ++p) s_pv.Tk[p] = a.T[(size_t)p * a.ldt + pix];
        }
        if (threadIdx.x == 0 && !(pb2 != INT_MAX && gb - thr > 0.0)) s_k = -1;
        __syncthreads();
        n_evals += n;
        ++sweeps_done;
        if (s_k < 0) { converged = 1; break; }
      }
      // ---- keep the flip of pixel k
      const int k = s_k;
      if (threadIdx.x == 0) {
        FOR_PORTS(p, a.n_o) s_o[p] = cfma(s_pv.coef, s_pv.Tk[p], s_o[p]);
        s_f = objective_of(s_op, s_o);
        if (n_acc < a.trace_cap) {
          if (a.trace) {
            int32_t* tr = a.trace + 4 * n_acc;
            tr[0] = a.mode == PNGF_FIRST_IMPROVEMENT ? s : (int)n_acc;
            tr[1] = a.mode == PNGF_FIRST_IMPROVEMENT ? t - 1 : 0;
            tr[2] = k;
            tr[3] = 0;
          }
          if (a.trace_f) a.trace_f[n_acc] = s_f;
        } else if (status == PNGF_OK) {
          status = PNGF_ECAPACITY;
        }
        if (a.mixed) a.xa[r] = s_pv.alpha;
      }
      ++n_acc;
      ++acc_in_sweep;
      if (!a.mixed) {
        // FP64: gather c = W[:,k] into shared memory, then the state and rank-1 updates
        for (int j = threadIdx.x; j < n; j += blockDim.x)
          cs[j] = (j >= k) ? a.W[(size_t)k * a.ldw + j] : a.W[(size_t)j * a.ldw + k];
        __syncthreads();
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
          c128 cj = cs[j];
          c128 aj = cmul(s_pv.alpha, cj);
          acs[j] = aj;
          a.diag[j] = cfma(aj, cj, a.diag[j]);
          a.e[j] = cfma(s_pv.coef, cj, a.e[j]);
          for (int p = 0; p < a.n_o; ++p) {
            c128* tp = a.T + (size_t)p * a.ldt + j;
            *tp = cfma(aj, s_pv.Tk[p], *tp);
          }
          if (j == k) {
            uint8_t nb = a.b[j] ^ 1;
            a.b[j] = nb;
            a.v[j] = nb ? a.dv[j] : mk(0.0, 0.0);
          }
        }
        __syncthreads();  // every alpha c_j formed
        rank1_upper_ac(a.W, n, a.ldw, acs, cs, 0, E);
        __syncthreads();
        ++since_refresh;
        if (a.refresh_k > 0 && since_refresh >= a.refresh_k) {
          since_refresh = 0;
          ++n_refresh;
          cta_refresh(a, s_op, s_o, &s_f);
        }
      } else {
        // mixed: beta, column assembly from the FP32 copy, FP64 state update
        for (int i = threadIdx.x; i < r; i += blockDim.x) {
          c128 al = a.xa[i];
          float2 x = a.X[(size_t)k * a.R + i];
          float ax = (float)al.x, ay = (float)al.y;
          s_beta[i] = make_float2(fmaf(ax, x.x, -ay * x.y), fmaf(ax, x.y, ay * x.x));
        }
        __syncthreads();
        mixed_accept_own(a, s_pv, s_beta, r, 0, n);
        ++r;
        ++since_refresh;
        if (r == a.R) {
          __syncthreads();
          if (use_tc) {
            tc_prepare(a, r, a.tcimgA, a.tcimgB, threadIdx.x, blockDim.x);
            __threadfence_block();
            __syncthreads();
            if (!tc_fold_tiles<1>(a, r, a.tcimgA, a.tcimgB, dyn, tcs, 0, 1)) {
              status = PNGF_ETIMEOUT;
              tc_failed = true;
              break;
            }
          } else {
            flush_tiles(a, r, reinterpret_cast<float*>(dyn), 0, 1);
          }
          __syncthreads();
          r = 0;
          ++n_flush;
          if (a.refresh_k > 0 && since_refresh >= a.refresh_k) {
            since_refresh = 0;
            ++n_refresh;
            cta_refresh(a, s_op, s_o, &s_f);
          }
        }
      }
      if (!isfinite(s_f)) {
        status = PNGF_ENUMERIC;
        break;
      }
      if (a.mode == PNGF_BEST_IMPROVEMENT && n_acc >= a.n_sweeps) break;
      if (a.mode == PNGF_FIRST_IMPROVEMENT && t >= n) {
        ++sweeps_done;
        ++s;
        if (s >= a.n_sweeps) break;
        t = 0;
        acc_in_sweep = 0;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      FOR_PORTS(p, a.n_o) ctl->o[p] = s_o[p];
      ctl->f = s_f;
      ctl->since_refresh = since_refresh;
      ctl->r_delay = r;
      ctl->n_acc_total += (int)n_acc;
      long long cnt[8] = {n_acc, n_evals, sweeps_done, converged, n_refresh, n_flush, status, 0};
      for (int q = 0; q < 8; ++q) ctl->counters[q] = cnt[q];
      if (a.counters)
        for (int q = 0; q < 8; ++q) a.counters[q] = cnt[q];
      if (status == PNGF_ENUMERIC || status == PNGF_EINVAL || status == PNGF_ETIMEOUT) latch_status(ctl, status);
    }
  }
  if (use_tc) tc_teardown(tcs, tc_failed);
}

// ---------------------------------------------------------------- FP64, FIRST mode
// The delayed search of delayed64.cuh with one CTA per run: only CTA-wide
// barriers, the folds on this SM's tensor core.  The visiting positions are
// scored kScoreChunk at a time from the current one (a scoring warp on each SM
// sub-partition; a flip is kept every few positions early in a search).
// Bound by the SM's FP64 pipe (the columns: r complex multiply-adds per pixel;
// the refreshes; the folds' sums in FP64: 81% busy at 1024 lossy-metal pixels) and the
// read-back of the folds.  76 such runs of ten sweeps take 377 ms, one kept flip 0.25
// ms (before: the triangle's rank-1 update on the FP64 pipe, 0.6 ms per kept flip).
constexpr int kScoreChunk = 128;

// the refresh of a whole run by one CTA; smem: the active-pixel list, then the
// staging of the correction (OZ_SMEM bytes)
__device__ void cta_refresh64(const SweepArgs& a, const ObjParams& op, c128* s_o, double* s_f, unsigned char* smem) {
  int* act = reinterpret_cast<int*>(smem);
  __syncthreads();
  refresh_x(a, 0, a.n);
  __syncthreads();
  const int m = refresh_residual(a, 0, a.n, act);
  for (int t = threadIdx.x; t < m; t += blockDim.x) a.actg[t] = act[t];
  const int t_end = count_below(act, m, a.n - 1);
  __syncthreads();
  correct_strips<false>(a, 0, a.n, a.actg, t_end, reinterpret_cast<float*>(smem), OZ_SMEM);
  __syncthreads();
  cta_ports(a, op, s_o, s_f);
}

__global__ void __launch_bounds__(OZ_THREADS, 1) dbs_batch_fp64_kernel(const SweepArgs* __restrict__ runs, int n_runs,
                                                                       int* __restrict__ queue) {
  extern __shared__ __align__(128) unsigned char b_smem[];
  constexpr int NW = OZ_THREADS / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ c128 s_o[kMaxPorts], s_alpha, s_coef, s_Tk[kMaxPorts];
  __shared__ double s_f;
  __shared__ ObjParams s_op;
  __shared__ c128 s_beta[kDelay64], s_al[kDelay64], s_invd[kDelay64];
  __shared__ int s_hist[kDelay64];
  __shared__ int s_best, s_k, s_bad, s_run;
  __shared__ __align__(8) unsigned long long s_bars[OZ_NBAR];
  __shared__ unsigned s_tmem;
  OzState oz;
  oz_setup(oz, s_bars, &s_tmem);
  bool oz_failed = false;
  while (!oz_failed) {
    __syncthreads();  // every thread has read the previous s_run
    if (tid == 0) s_run = atomicAdd(queue, 1);
    __syncthreads();
    const int run = s_run;
    if (run >= n_runs) break;
    const SweepArgs& a = runs[run];
    const int n = a.n, n_o = a.n_o;
    const size_t ldx = a.ldt;
    Control* ctl = a.ctl;
    if (tid == 0) {
      s_op = a.op;
      FOR_PORTS(p, n_o) s_o[p] = ctl->o[p];
      s_f = ctl->f;
      s_best = INT_MAX;
      s_bad = 0;
    }
    for (int q = tid; q < n; q += blockDim.x) a.last64[q] = -1;
    __syncthreads();
    long long n_acc = 0, n_evals = 0, n_refresh = 0;
    int sweeps_done = 0, converged = 0, status = PNGF_OK;
    int since_refresh = ctl->since_refresh;
    int s = 0, t = 0, acc_in_sweep = 0, r = 0;
    auto fold = [&]() -> bool {
      if (r == 0) return true;
      __syncthreads();
      bool ok = true;
      if (fold64_is_direct(r, n)) {
        fold64_direct(a.W, a.ldw, a.X64, ldx, s_al, s_invd, a.last64, nullptr, r, n, warp, NW);
        __syncthreads();
      } else {
        fold64_digits(a.X64, ldx, s_al, a.last64, r, n, a.oz, warp, NW);
        fold64_bases(a.W, a.ldw, a.X64, ldx, s_invd, s_hist, a.last64, nullptr, r, n, tid, blockDim.x);
        __syncthreads();
        ok = fold64_product(oz, b_smem, a.W, a.ldw, n, r, a.oz, 0, 1);
        if (const unsigned m = ok ? oz_listed(a.oz) : 0u) {
          fold64_redo(a.W, a.ldw, n, r, a.oz, m, warp, NW);
          __syncthreads();
        }
      }
      for (int q = tid; q < n; q += blockDim.x) {
        a.last64[q] = -1;
        a.diag[q] = a.W[(size_t)q * a.ldw + q];  // d is formed from the matrix's own diagonal
      }
      __syncthreads();
      r = 0;
      return ok;
    };
    while (true) {
      // ---- score a chunk of positions
      const int chunk_end = min(n, t + kScoreChunk);
      double fn = 0.0;
      c128 al = mk(0.0, 0.0), co = al, idv = al;
      int pos = INT_MAX, j = 0;
      if (tid < kScoreChunk) {
        const int q = t + tid;
        if (q < n) {
          const double f = s_f, thr = accept_threshold(s_op, f);
          j = a.order ? a.order[(size_t)s * n + q] : q;
          if ((unsigned)j >= (unsigned)n) s_bad = 1;
          else if (score_flip64(s_op, a.dv[j], a.b[j] != 0, a.diag[j], a.e[j],
                                [&](int p) { return a.T[(size_t)p * a.ldt + j]; }, s_o, fn, al, co, idv) &&
                   improves64(s_op, fn, f, thr))
            pos = q;
        }
        const int wmin = __reduce_min_sync(0xffffffffu, pos);
        if (lane == 0 && wmin != INT_MAX) atomicMin(&s_best, wmin);
      }
      __syncthreads();
      const int best = s_best;
      if (s_bad) {
        status = PNGF_EINVAL;
        break;
      }
      if (best == INT_MAX) {
        __syncthreads();  // every thread has read s_best and s_bad: the next chunk's scoring writes them
        n_evals += chunk_end - t;
        t = chunk_end;
        if (t < n) continue;
        ++sweeps_done;
        if (acc_in_sweep == 0) { converged = 1; break; }
        ++s;
        if (s >= a.n_sweeps) break;
        if (!fold()) { oz_failed = true; break; }
        t = 0;
        acc_in_sweep = 0;
        continue;
      }
      // ---- the kept flip; o and f exactly as the scorer formed them
      if (pos == best) {
        s_k = j;
        s_alpha = al;
        s_coef = co;
        s_al[r] = al;
        s_invd[r] = idv;
        s_hist[r] = j;
        s_f = fn;
        for (int p = 0; p < n_o; ++p) {
          const c128 tk = a.T[(size_t)p * a.ldt + j];
          s_Tk[p] = tk;
          s_o[p] = cfma(co, tk, s_o[p]);
        }
        if (n_acc < a.trace_cap) {
          if (a.trace) {
            int32_t* tr = a.trace + 4 * n_acc;
            tr[0] = s;
            tr[1] = best;
            tr[2] = j;
            tr[3] = 0;
          }
          if (a.trace_f) a.trace_f[n_acc] = fn;
        }
      }
      if (n_acc >= a.trace_cap && status == PNGF_OK) status = PNGF_ECAPACITY;
      n_evals += best - t + 1;
      t = best + 1;
      ++n_acc;
      ++acc_in_sweep;
      __syncthreads();
      const int k = s_k;
      if (tid == 0) s_best = INT_MAX;
      if (oz_exp(s_f) == 0x7ff) status = PNGF_ENUMERIC;
      const int lk = a.last64[k];
      for (int i = tid; i < r; i += blockDim.x)
        s_beta[i] = i > lk ? cmul(s_al[i], a.X64[(size_t)i * ldx + k]) : mk(0.0, 0.0);
      __syncthreads();
      // ---- the column and the state of every pixel (a warp per 32 pixels, so
      //      that an entry's chains, its column entry and its state stay on one lane)
      const c128 alpha = s_alpha, coef = s_coef;
      for (int q = tid; q < n; q += blockDim.x) {
        const int lj = a.last64[q];
        const c128 w = q == k ? a.diag[q] : delayed_base(a.W, a.ldw, k, q, lk, lj, s_invd, [&](int i, int p) {
          return a.X64[(size_t)i * ldx + p];
        });
        c128 ch[kChains64];
#pragma unroll
        for (int p = 0; p < kChains64; ++p) ch[p] = delayed_chain(s_beta, a.X64 + q, ldx, p, q == k ? r : lj, r);
        const c128 c = delayed_entry(w, ch, 1), ac = cmul(alpha, c), idk = s_invd[r];
        a.X64[(size_t)r * ldx + q] = c;
        // pixel k itself: y + alpha W_kk y = y / d
        a.diag[q] = q == k ? cmul(a.diag[q], idk) : cfma(ac, c, a.diag[q]);
        a.e[q] = q == k ? cmul(a.e[q], idk) : cfma(coef, c, a.e[q]);
#pragma unroll 1
        for (int p = 0; p < n_o; ++p) {
          c128* tp = a.T + (size_t)p * a.ldt + q;
          *tp = q == k ? cmul(*tp, idk) : cfma(ac, s_Tk[p], *tp);
        }
        if (q == k) {
          const uint8_t nb = a.b[q] ^ 1;
          a.b[q] = nb;
          a.v[q] = nb ? a.dv[q] : mk(0.0, 0.0);
          a.last64[q] = r;
        }
      }
      __syncthreads();
      ++r;
      ++since_refresh;
      const bool refresh = a.refresh_k > 0 && since_refresh >= a.refresh_k;
      if (r == kDelay64 || refresh || t >= n) {
        if (!fold()) { oz_failed = true; break; }
      }
      if (refresh) {
        since_refresh = 0;
        ++n_refresh;
        cta_refresh64(a, s_op, s_o, &s_f, b_smem);
      }
      if (status == PNGF_ENUMERIC) break;
      if (t >= n) {
        ++sweeps_done;
        ++s;
        if (s >= a.n_sweeps) break;
        t = 0;
        acc_in_sweep = 0;
      }
    }
    if (!oz_failed && !fold()) oz_failed = true;  // what a break left in the set
    if (oz_failed) status = PNGF_ETIMEOUT;
    __syncthreads();
    if (tid == 0) {
      FOR_PORTS(p, n_o) ctl->o[p] = s_o[p];
      ctl->f = s_f;
      ctl->since_refresh = since_refresh;
      ctl->n_acc_total += (int)n_acc;
      const long long cnt[8] = {n_acc, n_evals, sweeps_done, converged, n_refresh, 0, status, 0};
      for (int q = 0; q < 8; ++q) ctl->counters[q] = cnt[q];
      if (a.counters)
        for (int q = 0; q < 8; ++q) a.counters[q] = cnt[q];
      if (status == PNGF_ENUMERIC || status == PNGF_EINVAL || status == PNGF_ETIMEOUT) latch_status(ctl, status);
    }
  }
  oz_teardown(oz, oz_failed);
}

// ---------------------------------------------------------------- FP64, FIRST mode, few large runs
// Where the large runs are few: a cluster of kRunCtas CTAs advances one run at a
// time with the persistent search's own code (delayed_search.cuh; a run's result
// does not depend on how many CTAs share it).  One CTA per run leaves SMs idle
// while the large runs last, each bound by its SM's FP64 pipe and the latency of its
// chain of flips: four 1024-pixel runs of lossy metal take 313 ms on an SM each and
// 89 ms here, with the FP64 pipes of the four SMs 74% busy.
constexpr int kRunCtas = 4;

__global__ void __launch_bounds__(OZ_THREADS, 1) __cluster_dims__(kRunCtas, 1, 1)
    dbs_batch_cluster_kernel(const SweepArgs* __restrict__ runs, int n_runs, int* __restrict__ queue) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(128) unsigned char c_smem[];
  __shared__ __align__(8) unsigned long long s_bars[OZ_NBAR];
  __shared__ unsigned s_tmem;
  __shared__ int s_run, s_ok;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  OzState oz;
  oz_setup(oz, s_bars, &s_tmem);
  bool ok = true;
  while (ok) {
    if (rank == 0 && threadIdx.x == 0) s_run = atomicAdd(queue, 1);
    cluster.sync();
    const int run = *cluster.map_shared_rank(&s_run, 0);
    if (run < n_runs && rank == 0) {  // the run's barrier counter and words
      const SweepArgs& a = runs[run];
      if (threadIdx.x == 0) a.ctl->bar_count = 0;
      for (int q = threadIdx.x; q < 2 * kRunCtas * kWordStride; q += blockDim.x) a.slots[q] = 0;
    }
    cluster.sync();  // every CTA has the run's index, and the words are zero
    if (run >= n_runs) break;
    const bool mine = delayed_search<false, true>(runs[run], nullptr, nullptr, -1, kRunCtas, rank, c_smem, oz);
    if (threadIdx.x == 0) s_ok = mine;
    cluster.sync();  // after a timeout the whole cluster leaves
    for (int q = 0; q < kRunCtas; ++q) ok = ok && *cluster.map_shared_rank(&s_ok, q) != 0;
    cluster.sync();  // every CTA has read the others' words
  }
  oz_teardown(oz, !ok);
}

// The per-run argument table is written by the device from kernel parameters
// (chunks of the table passed by value), so that no host buffer has to outlive
// the call: a stream capture records the values themselves.
constexpr int kArgChunk = 30000 / (int)sizeof(SweepArgs);
struct ArgChunk {
  SweepArgs a[kArgChunk];
  int count;
};
static_assert(kArgChunk >= 1 && sizeof(ArgChunk) <= 32000, "kernel parameter space");

__global__ void write_args_kernel(const ArgChunk ch, SweepArgs* __restrict__ dst) {
  for (int i = threadIdx.x; i < ch.count; i += blockDim.x) dst[i] = ch.a[i];
}

}  // namespace

// the argument table, then the run queue's counter
static size_t batch_table_bytes(int n_runs) { return ((size_t)n_runs * sizeof(SweepArgs) + 255) / 256 * 256; }
size_t batch_workspace_bytes(int n_runs) { return batch_table_bytes(n_runs) + 256; }

// Clusters for a batch of n_runs, `large` of which have at least half the
// largest region's max_n pixels, or 0: one CTA per run.  Measured (ms, clusters
// against one CTA per run; n_d pixels, 4 / 38 / 76 equal runs of 10 sweeps, refresh
// every 64 kept flips):
//   1024: 89 / 157 / 241 against 313 / 370 / 377      100: 0.75 / 2.4 / 3.6 against 1.1 / 3.1 / 4.0
//    576: 20 / 39 / 64 against 59 / 80 / 82            64: 0.50 / 1.7 / 3.0 against 0.62 / 1.5 / 2.4
//    256: 2.7 / 6.9 / 11 against 6.4 / 12 / 13         16: 0.29 / 1.2 / 2.2 against 0.27 / 1.0 / 1.7
// so up to two rounds of clusters over the large runs, and from 96 pixels on.
// Every CTA holds a share of every run: at least one pixel, at most kOwn64.
static int batch_clusters(int n_runs, int large, int min_n, int max_n, int n_sm) {
  if (large * kRunCtas > 2 * n_sm || max_n < 96 || max_n > kRunCtas * kOwn64 || min_n < kRunCtas) return 0;
  return std::min(n_runs, n_sm / kRunCtas);
}

static pngf_status launch_batch_clusters(const void* runs, int n_runs, int* queue, int max_n, int max_o, int clusters,
                                         cudaStream_t stream) {
  if (cudaFuncSetAttribute(dbs_batch_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kDelayed64MaxSmem) != cudaSuccess)
    return PNGF_ECUDA;
  dbs_batch_cluster_kernel<<<clusters * kRunCtas, OZ_THREADS, delayed64_smem(max_o, own64_stride(max_n, kRunCtas)),
                             stream>>>(static_cast<const SweepArgs*>(runs), n_runs, queue);
  return cuda_status(cudaGetLastError());
}

pngf_status run_sweep_batch(pngf_ctx* const* ctxs, int n_runs, int n_sweeps, const int32_t* const* orders,
                            int32_t* const* traces, double* const* trace_f, int32_t trace_cap, int64_t* counters,
                            void* ws, size_t ws_bytes) {
  pngf_ctx* c0 = ctxs[0];
  SweepArgs* table = static_cast<SweepArgs*>(ws);
  int* queue = reinterpret_cast<int*>(static_cast<unsigned char*>(ws) + batch_table_bytes(n_runs));
  std::unique_ptr<ArgChunk> ch(new (std::nothrow) ArgChunk());
  if (!ch) return PNGF_ENOMEM;
  // queue order: largest region first (ties: the caller's order)
  std::vector<int> rank(n_runs);
  for (int r = 0; r < n_runs; ++r) rank[r] = r;
  std::stable_sort(rank.begin(), rank.end(), [&](int x, int y) { return ctxs[x]->cfg.n_d > ctxs[y]->cfg.n_d; });
  int max_n = 0;
  for (int r0 = 0; r0 < n_runs; r0 += kArgChunk) {
    ch->count = n_runs - r0 < kArgChunk ? n_runs - r0 : kArgChunk;
    for (int i = 0; i < ch->count; ++i) {
      const int r = rank[r0 + i];
      SweepArgs a = make_args(ctxs[r]);
      a.n_sweeps = n_sweeps;
      a.order = orders ? orders[r] : nullptr;
      a.trace = traces ? traces[r] : nullptr;
      a.trace_f = trace_f ? trace_f[r] : nullptr;
      a.trace_cap = trace_cap;
      a.counters = counters ? counters + 8 * (size_t)r : nullptr;
      ch->a[i] = a;
      if (a.n > max_n) max_n = a.n;
    }
    write_args_kernel<<<1, 128, 0, c0->stream>>>(*ch, table + r0);
    if (cudaGetLastError() != cudaSuccess) return PNGF_ECUDA;
  }
  const bool mixed = c0->cfg.precision == PNGF_MIXED;
  if (cudaMemsetAsync(queue, 0, sizeof(int), c0->stream) != cudaSuccess) return PNGF_ECUDA;
  int grid = c0->n_sm;  // one CTA per SM
  if (grid > n_runs) grid = n_runs;
  if (!mixed && c0->cfg.mode == PNGF_FIRST_IMPROVEMENT) {
    int max_o = 1, large = 0, min_n = max_n;
    for (int r = 0; r < n_runs; ++r) {
      large += 2 * ctxs[r]->cfg.n_d >= max_n;
      min_n = std::min(min_n, (int)ctxs[r]->cfg.n_d);
      max_o = std::max(max_o, (int)ctxs[r]->cfg.n_o);
    }
    const int clusters = batch_clusters(n_runs, large, min_n, max_n, c0->n_sm);
    if (clusters > 0)
      return launch_batch_clusters(ws, n_runs, queue, max_n, max_o, clusters, c0->stream);
    if (cudaFuncSetAttribute(dbs_batch_fp64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM) != cudaSuccess)
      return PNGF_ECUDA;
    dbs_batch_fp64_kernel<<<grid, OZ_THREADS, OZ_SMEM, c0->stream>>>(static_cast<const SweepArgs*>(ws), n_runs, queue);
    return cuda_status(cudaGetLastError());
  }
  size_t smem = mixed ? (kFlushSmem > (size_t)tc_fold_smem(1) ? kFlushSmem : (size_t)tc_fold_smem(1))
                      : 2 * (size_t)max_n * sizeof(c128);
  if (cudaFuncSetAttribute(dbs_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return PNGF_ECUDA;
  dbs_batch_kernel<<<grid, kBatchThreads, smem, c0->stream>>>(static_cast<const SweepArgs*>(ws), n_runs, queue);
  return cuda_status(cudaGetLastError());
}

}  // namespace pngf
