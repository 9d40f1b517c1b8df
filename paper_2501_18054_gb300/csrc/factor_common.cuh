// What both factorisations share: the panel with partial pivoting and the row
// interchanges, on a cooperative grid.
#pragma once

#include "fp64_fast.cuh"

namespace pngf {

struct FactorArgs {
  int n, n_o, ldw, ldt;
  const c128* G;
  const c128* God;
  const c128* cd;
  const c128* dv;
  const uint8_t* b_in;
  c128* LU;  // M_aa, m x m, leading dimension ldw
  c128* W;   // n x ldw, column n holds e
  c128* T;
  c128* v;
  uint8_t* b;
  c128* diag;
  c128* e;
  double* Gs;  // Re G + Im G
  int* act;    // the m pixels that are on, ascending, then the n - m others
  int* count;  // m
  const int* high;  // device: whether the contrast is high (contrast_kernel)
  OzOperands im;
  c128* cand;               // [2][P][NB] candidate pivot rows
  unsigned long long* key;  // [2][P] their keys; factor.cu: words, kPanelWord apart
  int* cand_row;            // [2][P]
  c128* drow;               // [2][NB] diagonal row of the column
  int* piv;                 // NB pivots of the panel
  c128* dinv;               // n reciprocals of the pivots
  int* perm;                // row i of the pivoted M_aa is row perm[i] of M_aa
  c128* binv;               // inverses of the BB x BB diagonal blocks: of L, then of U
  Control* ctl;
};

namespace {

constexpr int NB = 32;        // panel width

// |re| + |im| as an order-preserving key (NaN lowest: it is taken only where
// nothing else is left)
__device__ __forceinline__ unsigned long long pivot_key(c128 z) {
  const double a = cabs1(z);
  return isnan(a) ? 0ull : (unsigned long long)__double_as_longlong(a);
}

// ---------------------------------------------------------------- panel
// LU of rows [j0, m) x columns [j0, j0 + jb) with partial pivoting (|re| + |im|,
// ties -> lowest row).  CTA q holds its chunk of the rows in shared memory.
// Per column: every CTA publishes its candidate row (and the owner the
// diagonal row), one grid barrier, every CTA picks the winner, swaps what it
// owns and updates its rows, tracking the next column's candidate.  The rows
// travel with the candidates, so one exchange per column is enough: a grid
// barrier, or (kDivide = false) one word per CTA that every CTA waits for.
// kDivide: the largest pivot to the last bit and its reciprocal by FP64 division.
constexpr int kPanelWord = 16;  // 64-bit words between two CTAs' words
template <int WARPS, bool kDivide>
__device__ bool factor_panel(const FactorArgs& a, int m, int j0, int jb, c128* ps) {
  __shared__ unsigned long long s_key[WARPS];
  __shared__ int s_row[WARPS], s_q[WARPS], s_fail;
  __shared__ unsigned long long s_word;
  __shared__ c128 s_u[NB], s_d[NB];
  __shared__ c128 s_inv;
  __shared__ int s_p;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, P = gridDim.x, cta = blockIdx.x;
  const int rows = m - j0;
  const int rb = j0 + (int)((long long)rows * cta / P), re = j0 + (int)((long long)rows * (cta + 1) / P);
  const bool act_lane = lane < jb;
  if (tid == 0) s_fail = 0;
  unsigned long long bk = 0;
  int br = 0x7fffffff;
  for (int r = rb + warp; r < re; r += WARPS) {
    const c128 z = act_lane ? a.LU[(size_t)r * a.ldw + j0 + lane] : mk(0.0, 0.0);
    ps[(r - rb) * NB + lane] = z;
    if (lane == 0) {
      const unsigned long long k = pivot_key(z);
      if (br == 0x7fffffff || k > bk) { bk = k; br = r; }
    }
  }
  for (int jj = 0; jj < jb; ++jj) {
    const int col = j0 + jj, par = jj & 1;
    // ---- this CTA's candidate (held by lane jj of every warp)
    bk = __shfl_sync(0xffffffffu, bk, jj);
    br = __shfl_sync(0xffffffffu, br, jj);
    if (lane == 0) { s_key[warp] = bk; s_row[warp] = br; }
    __syncthreads();
    if (warp == 0) {
      unsigned long long k = lane < WARPS ? s_key[lane] : 0ull;
      int r = lane < WARPS ? s_row[lane] : 0x7fffffff;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long ok = __shfl_xor_sync(0xffffffffu, k, off);
        const int orr = __shfl_xor_sync(0xffffffffu, r, off);
        if (ok > k || (ok == k && orr < r)) { k = ok; r = orr; }
      }
      if (r != 0x7fffffff) a.cand[((size_t)par * P + cta) * NB + lane] = ps[(r - rb) * NB + lane];
      if (kDivide && lane == 0) {
        a.key[par * P + cta] = k;
        a.cand_row[par * P + cta] = r;
      }
      if (!kDivide) s_word = r == 0x7fffffff ? 0xffull : (k >> 32 << 32) | (unsigned)(r - rb);
    } else if (warp == 1 && col >= rb && col < re) {
      a.drow[par * NB + lane] = ps[(col - rb) * NB + lane];
    }
    if (!kDivide) {
      // one word per CTA instead of a barrier and a read of the keys: upper half
      // of the magnitude (a pivot within 2^-20 of the largest), column, row
      __syncthreads();
      unsigned long long* words = a.key + (size_t)par * P * kPanelWord;
      if (tid == 0) {
        fence_acq_rel_gpu();  // release: the candidate row and the diagonal row
        *reinterpret_cast<volatile unsigned long long*>(words + (size_t)cta * kPanelWord) =
            s_word | ((unsigned long long)(unsigned)(col + 1) << 8);
      }
      if (tid < ((P + 31) & ~31)) {
        unsigned k = 0;
        int r = 0x7fffffff;
        if (tid < P) {
          const volatile unsigned long long* w = words + (size_t)tid * kPanelWord;
          const unsigned long long lim = spin_limit_of(a.ctl), t0 = global_ns();
          for (unsigned long long it = 0;;) {
            const unsigned long long v = *w;
            if (((unsigned)v >> 8) == (unsigned)(col + 1)) {
              const int local = (int)(v & 0xff);
              k = (unsigned)(v >> 32);
              if (local != 0xff) r = j0 + (int)((long long)rows * tid / P) + local;
              break;
            }
            if (++it > lim || ((it & 63) == 0 && global_ns() - t0 > kWaitNs)) {
              s_fail = 1;
              latch_status(a.ctl, PNGF_ETIMEOUT);
              break;
            }
          }
          fence_acq_rel_gpu();  // acquire
        }
        const unsigned km = __reduce_max_sync(0xffffffffu, k);
        const int rm = __reduce_min_sync(0xffffffffu, k == km ? r : 0x7fffffff);
        const unsigned who = __ballot_sync(0xffffffffu, k == km && r == rm);
        if (lane == 0) {
          s_key[warp] = km;
          s_row[warp] = rm;
          s_q[warp] = 32 * warp + __ffs(who) - 1;
        }
      }
      __syncthreads();
      if (s_fail) return false;
    } else if (!grid_sync(a.ctl)) {
      return false;
    }
    // ---- the pivot, its row and its reciprocal (warp 0), the diagonal row (warp 1)
    if (warp == 0) {
      unsigned long long k = 0;
      int r = 0x7fffffff, q = -1;
      if (!kDivide) {
        if (lane < (P + 31) / 32) {
          k = s_key[lane];
          r = s_row[lane];
          q = s_q[lane];
        }
      } else {
        for (int c = lane; c < P; c += 32) {
          const unsigned long long ck = a.key[par * P + c];
          const int cr = a.cand_row[par * P + c];
          if (ck > k || (ck == k && cr < r)) { k = ck; r = cr; q = c; }
        }
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long ok = __shfl_xor_sync(0xffffffffu, k, off);
        const int orr = __shfl_xor_sync(0xffffffffu, r, off), oq = __shfl_xor_sync(0xffffffffu, q, off);
        if (ok > k || (ok == k && orr < r)) { k = ok; r = orr; q = oq; }
      }
      const bool singular = k == 0;  // an exactly zero (or NaN) column: keep the diagonal row
      const c128 u = singular ? a.drow[par * NB + lane] : a.cand[((size_t)par * P + q) * NB + lane];
      s_u[lane] = u;
      const c128 pv = mk(__shfl_sync(0xffffffffu, u.x, jj), __shfl_sync(0xffffffffu, u.y, jj));
      const c128 inv = kDivide ? cdiv(mk(1.0, 0.0), pv) : crecip(pv);
      if (lane == 0) {
        s_inv = inv;
        s_p = singular ? col : r;
        if (cta == 0) {
          a.piv[jj] = s_p;
          a.dinv[col] = inv;
          if (singular) latch_status(a.ctl, PNGF_ESINGULAR);
        }
      }
    } else if (warp == 1) {
      s_d[lane] = a.drow[par * NB + lane];
    }
    __syncthreads();
    const int p = s_p;
    if (warp == 0 && p != col && p >= rb && p < re) ps[(p - rb) * NB + lane] = s_d[lane];
    if (warp == 1 && col >= rb && col < re) ps[(col - rb) * NB + lane] = s_u[lane];
    __syncthreads();
    // ---- scale the column, update the rest of the panel (lane = column)
    const c128 inv = s_inv, u = s_u[lane];
    bk = 0;
    br = 0x7fffffff;
    for (int r = max(rb, col + 1) + warp; r < re; r += WARPS) {
      c128* row = ps + (r - rb) * NB;
      const c128 z = row[lane];
      const c128 l = cmul(row[jj], inv);
      __syncwarp();  // every lane has read row[jj]
      if (lane == jj) {
        row[lane] = l;
      } else if (lane > jj && act_lane) {
        const c128 nz = cfms(l, u, z);
        row[lane] = nz;
        if (lane == jj + 1) {
          const unsigned long long k = pivot_key(nz);
          if (br == 0x7fffffff || k > bk) { bk = k; br = r; }
        }
      }
      __syncwarp();
    }
    // lane jj + 1 holds the next candidate; the next iteration's shuffle takes it from there
    if (jj + 1 < jb) {
      bk = __shfl_sync(0xffffffffu, bk, jj + 1);
      br = __shfl_sync(0xffffffffu, br, jj + 1);
    }
  }
  __syncthreads();
  for (int r = rb + warp; r < re; r += WARPS)
    if (act_lane) a.LU[(size_t)r * a.ldw + j0 + lane] = ps[(r - rb) * NB + lane];
  return grid_sync(a.ctl);
}

// ---------------------------------------------------------------- interchanges
// Net effect of the panel's interchanges, formed by warp 0 of every CTA: the
// row top_src[i] moves to row j0 + i, and row ext_src[e] to the row
// ext_row[e] below the panel's block (e < n_ext <= NB).
struct Swaps {
  int top_src[NB], ext_row[NB], ext_src[NB], n_ext;
};

__device__ __forceinline__ void net_swaps(const FactorArgs& a, int j0, int jb, Swaps& sw) {
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  int top = j0 + lane, er = -1, es = -1, ne = 0;
  const int pl = lane < jb ? a.piv[lane] : -1;
  for (int jj = 0; jj < jb; ++jj) {
    const int p = __shfl_sync(0xffffffffu, pl, jj);
    const int tj = __shfl_sync(0xffffffffu, top, jj);
    if (p < j0 + jb) {
      const int tp = __shfl_sync(0xffffffffu, top, p - j0);
      if (lane == jj) top = tp;
      if (lane == p - j0) top = tj;
    } else {
      const unsigned hit = __ballot_sync(0xffffffffu, er == p);
      const int s = hit ? __ffs(hit) - 1 : ne++;
      if (!hit && lane == s) { er = p; es = p; }
      const int v = __shfl_sync(0xffffffffu, es, s);
      if (lane == jj) top = v;
      if (lane == s) es = tj;
    }
  }
  sw.top_src[lane] = top;
  sw.ext_row[lane] = er;
  sw.ext_src[lane] = es;
  if (lane == 0) sw.n_ext = ne;
}

__device__ __forceinline__ c128 shfl_c(c128 z, int src) {
  return mk(__shfl_sync(0xffffffffu, z.x, src), __shfl_sync(0xffffffffu, z.y, src));
}

// The panel's interchanges on the other columns of M and the row permutation,
// and L^-1 (Ls: the block, column-major) on the columns right of the panel: one
// warp per two columns, lane = row (a warp's FP64 instruction costs the same for
// one lane as for 32).  Warps gw of nw.
__device__ void swap_and_solve(const FactorArgs& a, const Swaps& sw, const c128* Ls, int m, int j0, int jb, int gw, int nw) {
  const int lane = threadIdx.x & 31, ldw = a.ldw, i1 = j0 + jb, rest = m - i1;
  const int ur = (rest + 1) / 2, ul = j0 / 2;
  const int ts = sw.top_src[lane], er = sw.ext_row[lane], es = sw.ext_src[lane];
  for (int u = gw; u < ur + ul; u += nw) {
    const bool left = u >= ur;
    const int c = left ? 2 * (u - ur) : i1 + 2 * u;
    const bool two = c + 1 < (left ? j0 : m);
    c128* base = a.LU + c;
    c128 x0 = mk(0.0, 0.0), x1 = x0, y0 = x0, y1 = x0;
    if (lane < jb) {
      const c128* p = base + (size_t)ts * ldw;
      x0 = p[0];
      if (two) x1 = p[1];
    }
    if (er >= 0) {
      const c128* p = base + (size_t)es * ldw;
      y0 = p[0];
      if (two) y1 = p[1];
    }
    __syncwarp();
    if (er >= 0) {
      c128* p = base + (size_t)er * ldw;
      p[0] = y0;
      if (two) p[1] = y1;
    }
    if (!left)
      for (int k = 0; k + 1 < jb; ++k) {
        const c128 l = Ls[k * NB + lane];  // zero for row <= k
        const c128 a0 = shfl_c(x0, k), a1 = shfl_c(x1, k);
        x0 = cfms(l, a0, x0);
        x1 = cfms(l, a1, x1);
      }
    if (lane < jb) {
      c128* p = base + (size_t)(j0 + lane) * ldw;
      p[0] = x0;
      if (two) p[1] = x1;
    }
  }
  if (gw == nw - 1) {  // the row permutation
    const int x = lane < jb ? a.perm[ts] : 0, y = er >= 0 ? a.perm[es] : 0;
    __syncwarp();
    if (lane < jb) a.perm[j0 + lane] = x;
    if (er >= 0) a.perm[er] = y;
  }
}

}  // namespace

// factor_pipe.cu
pngf_status factor_pipe(pngf_ctx* c, const FactorArgs& a);
}  // namespace pngf
