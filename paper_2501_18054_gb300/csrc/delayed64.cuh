// FP64 search in sequential (FIRST) mode with a delayed maintained inverse,
// shared by the persistent search and the batch kernel:
//   W(current) = W + sum_{i<r} alpha_i x_i x_i^T,   x_i = column of W(current) at kept flip i.
// A kept flip of pixel k needs one column only,
//   c_j = W(k, j) + sum_{i<r} (alpha_i x_i[k]) x_i[j],
// which updates diag W, e and T and is appended to the delayed set; every
// kDelay64 flips (and before a refresh, at the end of a sweep and of a call) the
// set is folded into the upper triangle of W by one product on the tensor
// cores in FP64 accuracy (ozaki.cuh).  Per kept flip that is r complex
// multiply-adds per pixel instead of N_d / 2 on the FP64 pipe, which issues one
// warp instruction per 64 cycles on each SM sub-partition.
//
// Row and column k restart at a flip of k.  The flip divides them by d = 1 -
// delta W_kk, |d| from 10^3 (metal put in) to 10^-3 (taken out), and a sum W(k,
// j) + alpha W_kk W(k, j) would keep the rounding of the larger side: an error
// in a small W_kk counts |d|^2-fold once the pixel is flipped back.  So after a
// flip i of k, W(k, j) is x_i[j] / d_i with the flips after i added, and the
// entries of k in the delayed columns up to i are taken as zero.  last[j] is
// the index of pixel j's last flip in the set (-1: none).  (Lossy metal, 10
// sweeps at N_d = 1024, 12 starts, error of diag W against a refined solve: up
// to 2.9e-10 with rank-1 updates one by one, 4.5e-9 with plain sums, 2.2e-10 in
// this form.)
//
// Everything is the same arithmetic in the same order whatever the grid: the
// column sum runs in eight chains (i mod 8) added pairwise, the fold is exact
// up to one rounding per entry.  The set is empty between sweeps, so that a
// search resumed from a checkpoint is bit for bit the uninterrupted one.
#pragma once

#include "ozaki.cuh"

namespace pngf {
namespace {

constexpr int kDelay64 = OZ_KMAX;  // columns held; one exact accumulation of the fold
constexpr int kChains64 = 8;       // chains of the column sum

// Candidate flip of a pixel (Eq. 14): inv_d = 1 / d, d = 1 - delta W_kk, alpha =
// delta / d, coef = alpha e_k and the objective of o + coef T[:, k]; T(p) is row p of T at
// the pixel.  False for a singular candidate (|d| < 1e-14).  Ports of weight
// zero are left out: they add nothing to the objective.
template <class TRow>
__device__ __forceinline__ bool score_flip64(const ObjParams& op, c128 dv, bool on, c128 diag, c128 e, TRow T,
                                             const c128* o, double& f_new, c128& alpha, c128& coef, c128& inv_d) {
  const c128 delta = on ? mk(-dv.x, -dv.y) : dv;
  const c128 d = cfms(delta, diag, mk(1.0, 0.0));
  const double d2 = cabs2(d);
  if (__double_as_longlong(d2) < __double_as_longlong(1e-28)) return false;  // d2 >= 0 or NaN
  const double r = rcp_pos(d2);
  inv_d = mk(d.x * r, -d.y * r);
  alpha = cmul(delta, inv_d);
  coef = cmul(alpha, e);
  double f = 0.0;
#pragma unroll 1
  for (int p = 0; p < op.n_o; ++p) {
    if (op.w[p] == 0.0) continue;
    f += objective_term(op, p, cfma(coef, T(p), o[p]));
  }
  f_new = f;
  return true;
}

// The same for a perfect-conductor pixel (pec.cu): alpha = -1 / S_kk, and row k
// restarts from +-i / S_kk times the column (+: metal put in).
__device__ __forceinline__ c128 pec_rotate(c128 z, bool metal) {  // +i z or -i z
  return metal ? mk(-z.y, z.x) : mk(z.y, -z.x);
}
__device__ __forceinline__ c128 pec_unrotate(c128 z, bool metal) { return pec_rotate(z, !metal); }
template <class TRow>
__device__ __forceinline__ bool score_pec(const ObjParams& op, bool on, c128 diag, c128 e, TRow T, const c128* o,
                                          double& f_new, c128& alpha, c128& coef, c128& inv_d) {
  const double d2 = cabs2(diag);
  // a NaN of either sign is no zero pivot: a forced flip reports it as not finite
  if ((__double_as_longlong(d2) & 0x7fffffffffffffffll) < __double_as_longlong(1e-28)) return false;
  const double r = rcp_pos(d2);
  const c128 sg = mk(diag.x * r, -diag.y * r);
  alpha = mk(-sg.x, -sg.y);
  inv_d = pec_rotate(sg, !on);
  coef = cmul(alpha, e);
  double f = 0.0;
#pragma unroll 1
  for (int p = 0; p < op.n_o; ++p) {
    if (op.w[p] == 0.0) continue;
    f += objective_term(op, p, cfma(coef, T(p), o[p]));
  }
  f_new = f;
  return true;
}

// improvement beyond the threshold, by the sign of an FP64 difference
__device__ __forceinline__ bool improves64(const ObjParams& op, double f_new, double f, double thr) {
  return gain_of(op, f_new, f) - thr > 0.0;
}

// What W(k, j) starts from, j != k: the later of the two pixels' last flips (lk, lj),
// or the folded W where neither was flipped.  X(i, p): column i at pixel p.
template <class Col>
__device__ __forceinline__ c128 delayed_base(const c128* W, int ldw, int k, int j, int lk, int lj, const c128* inv_d,
                                             Col X) {
  if (lk < 0 && lj < 0) return j >= k ? W[(size_t)k * ldw + j] : W[(size_t)j * ldw + k];
  return lj > lk ? cmul(X(lj, k), inv_d[lj]) : cmul(X(lk, j), inv_d[lk]);
}
// one chain of the column sum: i = part, part + kChains64, ... in (lj, r) of beta_i X[i ld]
__device__ __forceinline__ c128 delayed_chain(const c128* beta, const c128* X, size_t ld, int part, int lj, int r) {
  c128 s = mk(0.0, 0.0);
  int i = part;
  if (i <= lj) i += (lj - i) / kChains64 * kChains64 + kChains64;
#pragma unroll 2
  for (; i < r; i += kChains64) s = cfma(beta[i], X[(size_t)i * ld], s);
  return s;
}
// base + the chains, added pairwise
__device__ __forceinline__ c128 delayed_entry(c128 base, const c128* s, int ld) {
  c128 t[kChains64];
#pragma unroll
  for (int q = 0; q < kChains64; ++q) t[q] = s[q * ld];
#pragma unroll
  for (int h = 1; h < kChains64; h *= 2)
#pragma unroll
    for (int q = 0; q < kChains64; q += 2 * h) t[q] = cadd(t[q], t[q + h]);
  return cadd(base, t[0]);
}

// ---------------------------------------------------------------- ports
// o = c_o + G_od (v .* e) over all pixels of a batch's run, by one CTA: the sum's order
// depends on the CTA's threads only, not on how many CTAs share the run
__device__ void cta_ports(const SweepArgs& a, const ObjParams& op, c128* s_o, double* s_f) {
  __shared__ c128 red[kMaxWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int p = 0; p < a.n_o; ++p) {
    c128 acc = mk(0.0, 0.0);
    for (int j = threadIdx.x; j < a.n; j += blockDim.x)
      acc = cfma(a.God[(size_t)p * a.n + j], cmul(a.v[j], a.e[j]), acc);
    for (int off = 16; off > 0; off >>= 1) {
      acc.x += __shfl_down_sync(0xffffffffu, acc.x, off);
      acc.y += __shfl_down_sync(0xffffffffu, acc.y, off);
    }
    __syncthreads();
    if (lane == 0) red[w] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      c128 sum = mk(0.0, 0.0);
      for (int q = 0; q < nw; ++q) sum = cadd(sum, red[q]);
      s_o[p] = cadd(a.co[p], sum);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) *s_f = objective_of(op, s_o);
  __syncthreads();
}

// ---------------------------------------------------------------- fold
// Operand images of the fold: A rows y_j = alpha 2^-h x_j, B rows 2^h x_j, where
// 2^h is about |alpha|^(1/2): both sides then carry the square root of their
// column's contribution to W, and the fixed point of a row is relative to its
// largest contribution.
// X[i ldx + j]: column i at pixel j; s_al: alpha_i; entries up to a pixel's last
// flip are zero.  Warps gw of nw.
__device__ __noinline__ void fold64_digits(const c128* X, size_t ldx, const c128* s_al, const int* last, int r, int n,
                                           const OzOperands& im, int gw, int nw) {
  const int nk = (r + OZ_KC - 1) / OZ_KC, qa = (n + OZ_M - 1) / OZ_M * (OZ_M / 4), qb = (n + OZ_N - 1) / OZ_N * (OZ_N / 4);
  auto half_scale = [&](int k) {  // the double 2^h
    const c128 al = s_al[k];
    const int ex = max(oz_exp(al.x), oz_exp(al.y));
    return ex == 0 || ex == 0x7ff ? 1.0 : __longlong_as_double((long long)(1023 + ((ex - 1023) >> 1)) << 52);
  };
  for (int q = gw; q < qa + qb; q += nw) {
    if (q < qa)
      oz_digitise_rows<OZ_M>(4 * q, r, nk, im.A, im.sqA, im.ea, im.na, im.fa, [&](int j, int k) {
        if (j >= n || k <= last[j]) return mk(0.0, 0.0);
        const double s = half_scale(k), is = __longlong_as_double((2046ll << 52) - __double_as_longlong(s));  // 1 / s
        const c128 al = s_al[k];
        return cmul(mk(al.x * is, al.y * is), X[(size_t)k * ldx + j]);
      });
    else
      oz_digitise_rows<OZ_N>(4 * (q - qa), r, nk, im.B, im.sqB, im.eb, im.nb, im.fb, [&](int j, int k) {
        if (j >= n || k <= last[j]) return mk(0.0, 0.0);
        const double s = half_scale(k);
        const c128 x = X[(size_t)k * ldx + j];
        return mk(x.x * s, x.y * s);
      });
  }
  if (gw == 0 && (threadIdx.x & 31) == 0) oz_list_clear(im);
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// the restarted rows and columns of W: x_i / d_i for the last flip i of every
// pixel in the set (hist[i]: the pixel flipped), threads gt of nt.  metal (PEC):
// the present design, whose restarted diagonal is the reciprocal pivot
__device__ __forceinline__ void fold64_bases(c128* W, int ldw, const c128* X, size_t ldx, const c128* inv_d,
                                             const int* hist, const int* last, const uint8_t* metal, int r, int n, int gt,
                                             int nt) {
  for (int q = gt; q < r * n; q += nt) {
    const int i = q / n, j = q - i * n, k = hist[i];
    if (last[k] != i || (j != k && last[j] > i)) continue;
    W[j >= k ? (size_t)k * ldw + j : (size_t)j * ldw + k] =
        metal && j == k ? pec_unrotate(inv_d[i], metal[k] != 0) : cmul(X[(size_t)i * ldx + j], inv_d[i]);
  }
}

// The fold of a small set, entry by entry in FP64, in place of all of the
// above: what W(i, j) starts from, then the flips after it.  Warps gw of nw, a row each
// at a time.  Takes r rank-1 updates on the FP64 pipe: 9 us each at N_d = 1024
// on 64 CTAs, against some 50 us of a product with its digits and barriers.  Such sets
// come from kept flips one call at a time and from refreshes every few flips
// (eight kept flips of a perfect-conductor region in a call each, N_d = 1024: 0.64
// -> 0.35 ms; 160 runs of 100 pixels refreshed every flip, a CTA each: 35 -> 28 ms, every
// fourth 13.5 -> 12.2).  The rule holds no grid: a result does not depend on it.
__device__ __forceinline__ bool fold64_is_direct(int r, int n) { return r <= 2 || (r <= 4 && r * n <= 1024); }
template <int R>  // an FP64 instruction that a predicate turns off takes its 64 cycles all the same
__device__ __noinline__ void fold64_direct_of(c128* W, int ldw, const c128* X, size_t ldx, const c128* s_al,
                                              const c128* inv_d, const int* last, const uint8_t* metal, int n, int gw,
                                              int nw) {
  for (int i = gw; i < n; i += nw) {
    const int li = last[i];
    c128 y[R];  // alpha x_i
#pragma unroll
    for (int q = 0; q < R; ++q) y[q] = cmul(s_al[q], X[(size_t)q * ldx + i]);
    c128* row = W + (size_t)i * ldw;
    for (int j = i + (threadIdx.x & 31); j < n; j += 32) {
      const int lj = last[j], m = max(li, lj);
      c128 w;
      if (m < 0) {
        w = row[j];
#pragma unroll
        for (int q = 0; q < R; ++q) w = cfma(y[q], X[(size_t)q * ldx + j], w);
      } else {
        w = metal && i == j ? pec_unrotate(inv_d[m], metal[i] != 0) : cmul(X[(size_t)m * ldx + (lj > li ? i : j)], inv_d[m]);
        for (int q = m + 1; q < R; ++q) w = cfma(cmul(s_al[q], X[(size_t)q * ldx + i]), X[(size_t)q * ldx + j], w);
      }
      row[j] = w;
    }
  }
}
__device__ __forceinline__ void fold64_direct(c128* W, int ldw, const c128* X, size_t ldx, const c128* s_al,
                                              const c128* inv_d, const int* last, const uint8_t* metal, int r, int n, int gw,
                                              int nw) {
  if (r == 1) fold64_direct_of<1>(W, ldw, X, ldx, s_al, inv_d, last, metal, n, gw, nw);
  else if (r == 2) fold64_direct_of<2>(W, ldw, X, ldx, s_al, inv_d, last, metal, n, gw, nw);
  else if (r == 3) fold64_direct_of<3>(W, ldw, X, ldx, s_al, inv_d, last, metal, n, gw, nw);
  else fold64_direct_of<4>(W, ldw, X, ldx, s_al, inv_d, last, metal, n, gw, nw);
}

// tiles of the upper triangle: row block I (128 rows) against the column
// blocks J >= 2 I (64 columns)
__device__ __forceinline__ int fold64_tiles(int n) {
  const int nI = (n + OZ_M - 1) / OZ_M, nJ = (n + OZ_N - 1) / OZ_N;
  return nI * nJ - nI * (nI - 1);
}
__device__ __forceinline__ c128* fold64_row(c128* W, int ldw, int n, int j, int J, int& cols) {
  cols = n - J * OZ_N;
  return j < n ? W + (size_t)j * ldw + J * OZ_N : nullptr;
}
__device__ __noinline__ bool fold64_product(OzState& oz, unsigned char* smem, c128* W, int ldw, int n, int r,
                                            const OzOperands& im, int t_begin, int t_step) {
  const int nI = (n + OZ_M - 1) / OZ_M, nJ = (n + OZ_N - 1) / OZ_N;
  return oz_tiles<1>(
      oz, smem, im, r, (float)r, fold64_tiles(n), t_begin, t_step,
      [&](long long t, int& I, int& J) {  // row block I starts at tile I nJ - I (I - 1)
        int lo = 0, hi = nI - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (mid * nJ - mid * (mid - 1) <= (int)t) lo = mid;
          else hi = mid - 1;
        }
        I = lo;
        J = 2 * lo + (int)t - (lo * nJ - lo * (lo - 1));
      },
      [&](int j, int J, int& cols) { return fold64_row(W, ldw, n, j, J, cols); });
}
// the m entries that the product left to FP64 (after a barrier), warps gw of nw
__device__ __noinline__ void fold64_redo(c128* W, int ldw, int n, int r, const OzOperands& im, unsigned m, int gw, int nw) {
  oz_redo<1>(im, m, r, gw, nw, [&](int j, int J, int& cols) { return fold64_row(W, ldw, n, j, J, cols); });
}

}  // namespace
}  // namespace pngf
