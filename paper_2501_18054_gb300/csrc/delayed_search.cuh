// The persistent search with delayed updates, for FP64 contexts in FIRST mode
// and for PEC contexts (searches in both modes and forced flips), see
// delayed64.cuh and pec.cu.
#pragma once

#include "delayed64.cuh"

namespace pngf {
namespace {

// One exchange per kept flip instead of grid barriers: every CTA publishes its
// earliest improving candidate as a record and one sequence-tagged word
// (position and pixel), every CTA waits for all words, reduces them itself and
// fetches the winner's record, W(k, own) and the coefficients beta in one round
// trip.  Words and records alternate between two buffers by round parity: a
// CTA runs at most one round ahead of the slowest reader.  The state of the own
// pixels lives in shared memory between refreshes.  Grid barriers remain
// around folds and refreshes.
//
// Bound by the latency of that chain, in us per kept flip at N_d = 1024 (lossy
// metal) on 64 CTAs: score 0.8, exchange 4.3, fetch 1.1, column 2.2, state 0.7,
// refresh 1.0, folds 3.1 (a fifth of their entries in FP64).  At N_d = 4096 (dielectric,
// 152 CTAs): 0.9, 4.7, 1.4, 2.6, 0.9, 5.2, 4.0.  Measured against the rank-1 kernel of
// sweep.cu: N_d = 4096 (10 sweeps) 75.3 -> 18.3 ms, N_d = 1024 23.2 -> 15.7 ms,
// N_d = 100 0.80 -> 0.53 ms.  16 pixels per CTA: a flip's column and state cost the
// same for 16 pixels as for one (a warp's FP64 instruction takes 64 cycles
// whatever its lanes), and fewer CTAs lengthen folds and refreshes more than
// they shorten the exchange (1024, before the folds summed anything in FP64: 12.8 us
// a flip on 48 CTAs or more, 13.7 on 32, 17.0 on 16).
constexpr int kOwn64 = 256;  // pixels per CTA, at most
// word = round sequence number << 32 | key, key = position << 15 | pixel (n_d <= 32768)
constexpr int kPixBits64 = 15;
constexpr unsigned kNoKey64 = ~0u;
constexpr int kWordStride = 16;  // 64-bit words between two CTAs' words (128 bytes)

struct Record64 {
  double f_new, gain;  // gain: BEST mode
  c128 alpha, coef, inv_d;
  c128 Tk[kMaxPorts];
};
static_assert((1 << kPixBits64) >= 32768, "pixel index");
static_assert(sizeof(Record64) <= kRecordBytes && sizeof(Record64) / 8 <= 32, "record slot, one word per lane");

__host__ __device__ constexpr int own64_stride(int n, int grid) { return ((n + grid - 1) / grid + 31) & ~31; }
// own state (T[n_o], diag, e, dv) after the fold's buffers
__host__ __device__ constexpr size_t delayed64_smem(int n_o, int oss) {
  return OZ_SMEM + (size_t)(n_o + 3) * oss * sizeof(c128);
}

static_assert(delayed64_smem(kMaxPorts, kOwn64) <= 216 * 1024, "own state");
constexpr size_t kDelayed64MaxSmem = 216 * 1024;  // with the static arrays below the 227 KB of a CTA

struct DelayedArgs {
  SweepArgs a;
  const int* forced;        // PEC: flips to apply in order (nullptr: a search)
  const int* forced_count;  //   and how many (device)
  int forced_one;           //   or one flip (>= 0)
};

// CTA `cta` of the P that run one search; the barrier counter and the words of
// the context are zero when the first of them starts.  Returns false after a
// timeout.  kBatch: a run of a batch (no active-pixel count, no phase cycles).
template <bool kPec, bool kBatch>
__device__ __forceinline__ bool delayed_search(const SweepArgs& a, const int* forced_list, const int* forced_count,
                                               int forced_one, int P, int cta, unsigned char* d_smem, OzState& oz) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = OZ_THREADS / 32;
  const int n = a.n, n_o = a.n_o;
  const int pb = (int)((long long)n * cta / P), pe = (int)((long long)n * (cta + 1) / P), own = pe - pb;
  Control* ctl = a.ctl;
  const unsigned long long spin_lim = spin_limit_of(ctl);
  const int OSS = own64_stride(n, P), OS = (own + 31) & ~31, nb = OS >> 5;
  c128* s_T = reinterpret_cast<c128*>(d_smem + OZ_SMEM);  // [n_o][OSS]
  c128* s_diag = s_T + n_o * OSS;
  c128* s_e = s_diag + OSS;
  c128* s_dv = s_e + OSS;
  // between folds their buffers hold what a flip passes between its steps and,
  // where they fit, the delayed columns of the own pixels
  c128* const s_part = reinterpret_cast<c128*>(d_smem);  // [kChains64][OSS] chain sums
  c128* const s_wk = s_part + kChains64 * OSS;           // what the column starts from
  c128* const s_c = s_wk + OSS;                          // the column
  c128* const s_ac = s_c + OSS;                          // alpha c
  c128* const Xn = s_ac + OSS;                           // [kDelay64][OS]
  const bool x_near = (size_t)(kChains64 + 3 + kDelay64) * OSS * sizeof(c128) <= (size_t)OZ_SMEM;
  const bool best_mode = kPec && a.mode == PNGF_BEST_IMPROVEMENT;
  const bool forced = kPec && (forced_list != nullptr || forced_one >= 0);
  const int n_forced = !forced ? 0 : forced_list ? *forced_count : 1;
  const size_t ldx = a.ldt;
  __shared__ int s_pos[kOwn64];
  __shared__ unsigned char s_b[kOwn64];
  __shared__ c128 s_beta[kDelay64], s_al[kDelay64], s_invd[kDelay64];
  __shared__ int s_hist[kDelay64], s_last[kOwn64];  // pixel of flip i; own pixels' last flips
  __shared__ c128 s_o[kMaxPorts];
  __shared__ double s_f;
  __shared__ c128 s_alpha, s_coef, s_Tk[kMaxPorts];
  __shared__ ObjParams s_op;
  __shared__ int s_best[2];                  // earliest improving position of the own pixels, by round parity
  __shared__ unsigned s_key[2];              // smallest key of the round
  __shared__ int s_fail;
  __syncthreads();  // every thread is done with an earlier search's arrays
  if (tid == 0) {
    s_op = a.op;
    FOR_PORTS(p, n_o) s_o[p] = ctl->o[p];
    s_f = ctl->f;
    s_fail = 0;
    s_best[0] = s_best[1] = INT_MAX;
    s_key[0] = s_key[1] = kNoKey64;
  }
  auto load_state = [&]() {
    for (int jl = tid; jl < own; jl += blockDim.x) {
      const int j = pb + jl;
      s_e[jl] = a.e[j];
      for (int p = 0; p < n_o; ++p) s_T[p * OSS + jl] = a.T[(size_t)p * a.ldt + j];
    }
  };
  auto store_state = [&](bool with_diag) {
    for (int jl = tid; jl < own; jl += blockDim.x) {
      const int j = pb + jl;
      a.e[j] = s_e[jl];
      if (with_diag) a.diag[j] = s_diag[jl];
      for (int p = 0; p < n_o; ++p) a.T[(size_t)p * a.ldt + j] = s_T[p * OSS + jl];
    }
  };
  for (int jl = tid; jl < own; jl += blockDim.x) {
    const int j = pb + jl;
    s_diag[jl] = a.diag[j];
    s_dv[jl] = kPec ? mk(0.0, 0.0) : a.dv[j];
    s_b[jl] = a.b[j];
    s_last[jl] = -1;
    a.last64[j] = -1;
    if (!a.order) s_pos[jl] = j;
  }
  load_state();
  long long n_acc = 0, n_evals = 0, n_refresh = 0, sum_active = 0;
  int sweeps_done = 0, converged = 0, status = PNGF_OK;
  const bool timer = !kBatch && cta == 0 && tid == 0;
  __shared__ long long ph[16];  // phase cycles, kept by the timer thread only
  if (timer)
    for (int q = 0; q < 16; ++q) ph[q] = 0;
  long long t_last = clock64(), t_begin = t_last;
  auto tick = [&](int phase) {
    if (timer) {
      const long long now = clock64();
      ph[phase] += now - t_last;
      t_last = now;
    }
  };
  int since_refresh = ctl->since_refresh;
  int s = 0, t = 0, acc_in_sweep = 0, r = 0;
  unsigned round = 0;
  bool failed = false;
  // positions of the own pixels in sweep sw; an entry outside [0, n) is rejected
  auto setup_sweep = [&](int sw) -> bool {
    if (!a.order || best_mode || forced) return true;
    for (int q = pb + tid; q < pe; q += blockDim.x) {
      const int px = a.order[(size_t)sw * n + q];
      if ((unsigned)px < (unsigned)n) a.pos_of[px] = q;
      else latch_status(ctl, PNGF_EINVAL);
    }
    if (!grid_sync(ctl, P)) return false;
    if (*reinterpret_cast<volatile int*>(&ctl->status) == PNGF_EINVAL) status = PNGF_EINVAL;
    for (int jl = tid; jl < own; jl += blockDim.x) s_pos[jl] = a.pos_of[pb + jl];
    __syncthreads();
    return true;
  };
  auto folded = [&]() {  // the set is empty
    r = 0;
    for (int jl = tid; jl < own; jl += blockDim.x) {
      s_last[jl] = -1;
      a.last64[pb + jl] = -1;
      s_diag[jl] = a.W[(size_t)(pb + jl) * a.ldw + pb + jl];  // d is formed from the matrix's own diagonal
    }
    __syncthreads();
  };
  // folds the delayed set into W
  auto fold = [&]() -> bool {
    if (r == 0) return true;
    if (!grid_sync(ctl, P)) return false;  // every CTA's part of the columns
    if (fold64_is_direct(r, n)) {
      fold64_direct(a.W, a.ldw, a.X64, ldx, s_al, s_invd, a.last64, kPec ? a.b : nullptr, r, n, warp * P + cta, P * NW);
      if (!grid_sync(ctl, P)) return false;
      folded();
      return true;
    }
    fold64_digits(a.X64, ldx, s_al, a.last64, r, n, a.oz, cta * NW + warp, P * NW);
    fold64_bases(a.W, a.ldw, a.X64, ldx, s_invd, s_hist, a.last64, kPec ? a.b : nullptr, r, n, cta * (int)blockDim.x + tid, P * (int)blockDim.x);
    if (!grid_sync(ctl, P)) return false;
    const bool ok = fold64_product(oz, d_smem, a.W, a.ldw, n, r, a.oz, cta, P);
    if (!ok && tid == 0) latch_status(ctl, PNGF_ETIMEOUT);
    if (!ok || !grid_sync(ctl, P)) return false;
    if (const unsigned m = oz_listed(a.oz)) {
      fold64_redo(a.W, a.ldw, n, r, a.oz, m, warp * P + cta, P * NW);
      if (!grid_sync(ctl, P)) return false;
    }
    folded();
    return true;
  };
  __syncthreads();
  if (!setup_sweep(0)) failed = true;
  while (!failed && status != PNGF_EINVAL) {
    const int par = (int)(round & 1);
    const unsigned seq = round + 1;
    unsigned long long* words = a.slots + (size_t)par * P * kWordStride;
    Record64* recs = reinterpret_cast<Record64*>(a.rec);  // stride kRecordBytes
    auto rec_at = [&](int q) {
      return reinterpret_cast<Record64*>(reinterpret_cast<unsigned char*>(recs) + ((size_t)par * P + q) * kRecordBytes);
    };
    // ---- score the own pixels still ahead in the sweep
    double fn = 0.0;
    c128 al = mk(0.0, 0.0), co = al, idv = al;
    int pos = INT_MAX;
    const double f_round = kPec ? s_f : 0.0;  // BEST mode decides by it after warp 0 may have moved on to the new s_f
    const int k_forced = !forced ? -1 : n_acc >= n_forced ? -1 : forced_list ? forced_list[n_acc] : forced_one;
    if (forced && (k_forced < 0 || k_forced >= n)) break;  // all done (the list holds pixels of the region)
    bool ok = false;
    if (tid < own) {
      const int q = forced ? (pb + tid == k_forced ? 0 : -1) : best_mode ? 0 : s_pos[tid];
      auto row = [&](int p) { return s_T[p * OSS + tid]; };
      if (q >= (forced || best_mode ? 0 : t)) {
        if (kPec) ok = score_pec(s_op, s_b[tid] != 0, s_diag[tid], s_e[tid], row, s_o, fn, al, co, idv);
        else ok = score_flip64(s_op, s_dv[tid], s_b[tid] != 0, s_diag[tid], s_e[tid], row, s_o, fn, al, co, idv);
        if (forced) {
          pos = ok ? 0 : 1;  // 1: the pivot is zero
        } else if (ok && !best_mode) {
          const double f = s_f;
          if (improves64(s_op, fn, f, accept_threshold(s_op, f))) pos = q;
        }
      }
    }
    double gain = 0.0;
    if (best_mode && !forced) {  // the CTA's largest gain, ties to the lowest pixel
      gain = ok ? gain_of(s_op, fn, s_f) : -INFINITY;
      double gb = gain;
      int pb2 = ok && !isnan(gain) ? pb + tid : INT_MAX;
      if (pb2 == INT_MAX) gb = -INFINITY;
      block_best(gb, pb2);
      if (pb2 == pb + tid) {
        pos = 0;
        s_best[par] = 0;
      }
    } else if (tid < OS) {
      const int wmin = __reduce_min_sync(0xffffffffu, pos);
      if (lane == 0 && wmin != INT_MAX) atomicMin(&s_best[par], wmin);
    }
    if (tid == 0) {  // next round's cells
      s_best[par ^ 1] = INT_MAX;
      s_key[par ^ 1] = kNoKey64;
    }
    __syncthreads();
    const int best = s_best[par];
    tick(0);
    if (best == INT_MAX ? tid == 0 : pos == best) {
      unsigned key = kNoKey64;
      if (best != INT_MAX) {
        Record64* rc = rec_at(cta);
        rc->f_new = fn;
        rc->gain = gain;
        rc->alpha = al;
        rc->coef = co;
        rc->inv_d = idv;
        for (int p = 0; p < n_o; ++p) rc->Tk[p] = s_T[p * OSS + tid];
        key = ((unsigned)best << kPixBits64) | (unsigned)(pb + tid);
      }
      fence_acq_rel_gpu();  // release: the record and the CTA's earlier columns before the word
      *reinterpret_cast<volatile unsigned long long*>(words + (size_t)cta * kWordStride) =
          ((unsigned long long)seq << 32) | key;
    }
    // ---- every CTA's word of this round; the smallest position wins
    unsigned my_key = kNoKey64;
    if (tid < ((P + 31) & ~31)) {
      unsigned key = kNoKey64;
      if (tid < P) {
        const volatile unsigned long long* w = words + (size_t)tid * kWordStride;
        unsigned long long it = 0;
        const unsigned long long t0 = global_ns();
        for (;;) {
          const unsigned long long v = *w;
          if ((unsigned)(v >> 32) == seq) {
            key = (unsigned)v;
            break;
          }
          if (++it > spin_lim || ((it & 63) == 0 && global_ns() - t0 > kWaitNs)) {
            s_fail = 1;
            latch_status(ctl, PNGF_ETIMEOUT);
            break;
          }
          if (it > 1024) __nanosleep(32);
        }
        fence_acq_rel_gpu();  // acquire: that CTA's record and columns
      }
      my_key = key;
      key = __reduce_min_sync(0xffffffffu, key);
      if (lane == 0) atomicMin(&s_key[par], key);
    }
    __syncthreads();
    ++round;
    if (s_fail) {
      failed = true;
      break;
    }
    unsigned key = s_key[par];
    if (best_mode && !forced) {
      // every CTA's candidate by its gain; the best is kept when it clears the threshold
      double gb = -INFINITY;
      int pix = INT_MAX;
      if (my_key != kNoKey64) {
        pix = (int)(my_key & ((1u << kPixBits64) - 1));
        gb = rec_at(tid)->gain;
      }
      block_best(gb, pix);
      key = pix != INT_MAX && improves64(s_op, rec_at((int)(((long long)(pix + 1) * P - 1) / n))->f_new, f_round,
                                         accept_threshold(s_op, f_round))
                ? (unsigned)pix
                : kNoKey64;
    }
    tick(1);
    if (forced && (key >> kPixBits64) == 1) {  // only a forced flip can meet a zero pivot
      status = PNGF_ESINGULAR;
      break;
    }
    if (key == kNoKey64 && best_mode) {
      n_evals += n;
      ++sweeps_done;
      converged = 1;
      break;
    }
    if (key == kNoKey64) {  // nothing improves in the rest of this sweep
      n_evals += n - t;
      ++sweeps_done;
      if (acc_in_sweep == 0) { converged = 1; break; }
      ++s;
      if (s >= a.n_sweeps) break;
      if (!fold()) { failed = true; break; }
      t = 0;
      acc_in_sweep = 0;
      if (!setup_sweep(s)) { failed = true; break; }
      __syncthreads();  // every thread has read this round's cells
      tick(6);
      continue;
    }
    const int pos_k = (int)(key >> kPixBits64), k = (int)(key & ((1u << kPixBits64) - 1));
    // ---- fetch: the winner's record (warp 0), beta_i = alpha_i x_i[k], W(k, own)
    const int own_warps0 = 4;
    // index of k's last flip in the set (from this CTA's own record of the
    // flips: the owner of k may already be entering this one)
    const unsigned h0 = __ballot_sync(0xffffffffu, lane < r && s_hist[lane] == k);
    const unsigned h1 = __ballot_sync(0xffffffffu, lane + 32 < r && s_hist[lane + 32] == k);
    const int lk = h1 ? 63 - __clz(h1) : h0 ? 31 - __clz(h0) : -1;
    if (warp == 0) {
      const double* rw = reinterpret_cast<const double*>(rec_at((int)(((long long)(k + 1) * P - 1) / n)));
      constexpr int oA = offsetof(Record64, alpha) / 8, oC = offsetof(Record64, coef) / 8, oD = offsetof(Record64, inv_d) / 8, oT = offsetof(Record64, Tk) / 8;
      const double wv = lane < (int)(sizeof(Record64) / 8) ? rw[lane] : 0.0;  // one word per lane
      auto word = [&](int i) { return __shfl_sync(0xffffffffu, wv, i); };
      const double fw = word(0);
      const c128 ra = mk(word(oA), word(oA + 1)), rco = mk(word(oC), word(oC + 1)), rd = mk(word(oD), word(oD + 1));
      c128 tk = mk(0.0, 0.0);
#pragma unroll
      for (int p = 0; p < kMaxPorts; ++p) {
        const c128 v = mk(word(oT + 2 * p), word(oT + 2 * p + 1));
        if (lane == p) tk = v;
      }
      if (lane < n_o) {
        s_Tk[lane] = tk;
        s_o[lane] = cfma(rco, tk, s_o[lane]);  // as the scorer formed it
      }
      if (lane == 0) {
        s_alpha = ra;
        s_coef = rco;
        s_f = fw;
        s_al[r] = ra;
        s_invd[r] = rd;
        s_hist[r] = k;
        if (cta == 0 && !forced) {
          if (n_acc < a.trace_cap) {
            if (a.trace) {
              int32_t* tr = a.trace + 4 * n_acc;
              tr[0] = best_mode ? (int)n_acc : s;
              tr[1] = pos_k;
              tr[2] = k;
              tr[3] = 0;
            }
            if (a.trace_f) a.trace_f[n_acc] = fw;
          }
        }
      }
    } else if (warp == 2 || warp == 3) {
      const int i = tid - 64;
      if (i < r) s_beta[i] = i > lk ? cmul(s_al[i], a.X64[(size_t)i * ldx + k]) : mk(0.0, 0.0);
    } else if (warp >= own_warps0) {
      for (int jl = tid - 32 * own_warps0; jl < own; jl += blockDim.x - 32 * own_warps0) {
        const int j = pb + jl;
        s_wk[jl] = j == k ? s_diag[jl] : delayed_base(a.W, a.ldw, k, j, lk, s_last[jl], s_invd,
                                                      [&](int i, int p) { return a.X64[(size_t)i * ldx + p]; });
      }
    }
    __syncthreads();
    tick(2);
    if (oz_exp(s_f) == 0x7ff) status = PNGF_ENUMERIC;
    if (n_acc >= a.trace_cap && status == PNGF_OK && !forced) status = PNGF_ECAPACITY;
    if (best_mode) {
      n_evals += n;
      ++sweeps_done;
    } else if (!forced) {
      n_evals += pos_k - t + 1;
      t = pos_k + 1;
    }
    ++acc_in_sweep;
    ++n_acc;
    // ---- the column: every chain of every own pixel on a lane of its own
    //      (W_kk itself is the maintained diagonal)
    for (int q = tid; q < kChains64 * own; q += blockDim.x) {
      const int part = q / own, jl = q - part * own, lj = pb + jl == k ? r : s_last[jl];
      s_part[part * OSS + jl] = x_near ? delayed_chain(s_beta, Xn + jl, OS, part, lj, r)
                                       : delayed_chain(s_beta, a.X64 + pb + jl, ldx, part, lj, r);
    }
    __syncthreads();
    if (tid < own) {
      const c128 c = delayed_entry(s_wk[tid], s_part + tid, OSS);
      s_c[tid] = c;
      s_ac[tid] = cmul(s_alpha, c);
      if (x_near) Xn[r * OS + tid] = c;
      a.X64[(size_t)r * ldx + pb + tid] = c;
      if (pb + tid == k) {
        const unsigned char nb2 = s_b[tid] ^ 1;
        s_b[tid] = nb2;
        a.b[k] = nb2;
        if (!kPec) a.v[k] = nb2 ? s_dv[tid] : mk(0.0, 0.0);
        s_last[tid] = r;
        a.last64[k] = r;
      }
    }
    __syncthreads();
    tick(3);
    // ---- the state: quantity q (0: diag, 1: e, 2 + p: row p of T) of 32 pixels per item
    for (int it = warp; it < nb * (2 + n_o); it += NW) {
      const int q = it % (2 + n_o), jl = it / (2 + n_o) * 32 + lane;
      if (jl < own) {
        c128* y = q == 0 ? s_diag + jl : q == 1 ? s_e + jl : s_T + (q - 2) * OSS + jl;
        if (pb + jl == k)  // y + alpha W_kk y = y / d; PEC: the diagonal becomes its reciprocal
          *y = kPec && q == 0 ? pec_unrotate(s_invd[r], s_b[jl] != 0) : cmul(*y, s_invd[r]);
        else *y = q == 0 ? cfma(s_ac[jl], s_c[jl], *y) : q == 1 ? cfma(s_coef, s_c[jl], *y) : cfma(s_ac[jl], s_Tk[q - 2], *y);
      }
    }
    __syncthreads();
    tick(4);
    ++r;
    ++since_refresh;
    const bool refresh = !kPec && a.refresh_k > 0 && since_refresh >= a.refresh_k;
    if (r == kDelay64 || refresh || t >= n) {
      if (!fold()) { failed = true; break; }
      tick(12);
    }
    if (!kPec && refresh) {
      since_refresh = 0;
      ++n_refresh;
      int* act = reinterpret_cast<int*>(d_smem);
      store_state(false);
      __syncthreads();
      refresh_x(a, pb, pe);
      if (!grid_sync(ctl, P)) { failed = true; break; }
      tick(8);
      const int m_act = refresh_residual(a, pb, pe, act);
      sum_active += m_act;
      if (cta == 0)  // for the correction, after the next barrier
        for (int q = tid; q < m_act; q += blockDim.x) a.actg[q] = act[q];
      const int t_end = count_below(act, m_act, pe - 1);
      if (!grid_sync(ctl, P)) { failed = true; break; }
      tick(9);
      correct_strips<false>(a, pb, pe, a.actg, t_end, reinterpret_cast<float*>(d_smem), OZ_SMEM);
      if (!grid_sync(ctl, P)) { failed = true; break; }
      tick(10);
      if (kBatch) {  // every CTA all of it: a run's results do not depend on who shares it
        load_state();
        cta_ports(a, s_op, s_o, &s_f);
      } else {
        ports_partial(a, pb, pe, cta);
        if (!grid_sync(ctl, P)) { failed = true; break; }
        load_state();
        ports_total(a, s_o, P);
        if (tid == 0) s_f = objective_of(s_op, s_o);
        __syncthreads();
      }
      tick(11);
    }
    if (status == PNGF_ENUMERIC) break;
    if (best_mode && !forced && n_acc >= a.n_sweeps) break;
    if (t >= n) {  // the sweep ended on a kept flip at its last position
      ++sweeps_done;
      ++s;
      if (s >= a.n_sweeps) break;
      t = 0;
      acc_in_sweep = 0;
      if (!setup_sweep(s)) { failed = true; break; }
    }
  }
  if (!failed && !fold()) failed = true;  // what a break left in the set
  __syncthreads();
  store_state(true);
  if (cta == 0 && tid == 0) {
    if (failed) status = PNGF_ETIMEOUT;
    FOR_PORTS(p, n_o) ctl->o[p] = s_o[p];
    ctl->f = s_f;
    if (!kPec) ctl->since_refresh = since_refresh;
    if (!forced) ctl->n_acc_total += (int)n_acc;
    const long long cnt[8] = {n_acc, n_evals, sweeps_done, converged, n_refresh, 0, status, kBatch ? 0 : sum_active};
    if (timer) ph[7] = clock64() - t_begin;
    for (int q = 0; q < 8 && !forced; ++q) ctl->counters[q] = cnt[q];
    for (int q = 0; q < 16 && !kBatch; ++q) ctl->phase_cycles[q] = ph[q];
    if (a.counters && !forced)
      for (int q = 0; q < 8; ++q) a.counters[q] = cnt[q];
    if (status != PNGF_OK && status != PNGF_ECAPACITY) latch_status(ctl, status);
  }
  return !failed;
}

template <bool kPec>
__global__ void __launch_bounds__(OZ_THREADS, 1) dbs_delayed_kernel(const __grid_constant__ DelayedArgs g) {
  extern __shared__ __align__(128) unsigned char d_smem[];
  __shared__ __align__(8) unsigned long long s_bars[OZ_NBAR];
  __shared__ unsigned s_tmem;
  hold_if_asked(g.a.ctl);
  OzState oz;
  oz_setup(oz, s_bars, &s_tmem);
  const bool ok = delayed_search<kPec, false>(g.a, g.forced, g.forced_count, g.forced_one, gridDim.x, blockIdx.x, d_smem, oz);
  oz_teardown(oz, !ok);
}

// CTAs of the delayed search, or 0 where it does not apply (FP64: BEST mode,
// whose state is checkpointed between single flips, and CTAs asked to hold more
// pixels than fit; PEC takes more CTAs than asked instead).  Refreshes every few
// kept flips each fold a small set first and run on fewer CTAs here: the rank-1
// kernel is the faster one (refresh_k = 1, 2, 4, 8, 16; ms here against there:
// N_d = 100 3.6, 2.0, 1.7, 1.15, 0.86 against 2.7, 1.8, 1.3, 1.07, 0.96; N_d = 1024
// 88, 47, 36, 23, 16 against 56, 36, 26, 21, 18; N_d = 4096, from 4: 102, 55, 31
// against 108, 84, 72).
int delayed64_grid(pngf_ctx* c) {
  const bool pec = c->cfg.precision == PNGF_PEC;
  if (!pec && c->cfg.mode != PNGF_FIRST_IMPROVEMENT) return 0;
  const int least_refresh = c->cfg.n_d < 2048 ? 12 : 4;
  if (!pec && c->cfg.refresh_k > 0 && c->cfg.refresh_k < least_refresh) return 0;
  int g = (c->cfg.n_d + 15) / 16;
  if (g > c->n_sm) g = c->n_sm;
  if (c->cfg.n_ctas > 0 && c->cfg.n_ctas < g) g = c->cfg.n_ctas;
  const int least = (c->cfg.n_d + kOwn64 - 1) / kOwn64;
  if (g < least) {
    if (!pec) return 0;
    g = least;
  }
  return g;
}

template <bool kPec>
pngf_status launch_delayed(pngf_ctx* c, const DelayedArgs& g, int grid) {
  const void* kernel = (const void*)dbs_delayed_kernel<kPec>;
  Control* ctl = g.a.ctl;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDelayed64MaxSmem) != cudaSuccess ||
      // the barrier words: a previous launch that timed out may have left them set
      cudaMemsetAsync(&ctl->bar_count, 0, 2 * sizeof(unsigned), c->stream) != cudaSuccess ||
      cudaMemsetAsync(g.a.slots, 0, (size_t)2 * grid * kWordStride * sizeof(unsigned long long), c->stream) != cudaSuccess)
    return PNGF_ECUDA;
  DelayedArgs args = g;
  void* params[] = {&args};
  return cuda_status(cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(OZ_THREADS), params,
                                                 delayed64_smem(c->cfg.n_o, own64_stride(c->cfg.n_d, grid)), c->stream));
}

}  // namespace
}  // namespace pngf
