// Initial factorisation of the reduced system and formation of the maintained
// state (the inverse of the paper's initial system matrix C_0, section
// "Direct binary search optimization"; field form of Supplementary Note 4).
//
// M = I - G diag(v), v = dv .* b, differs from the identity only in the columns
// of the m pixels that are on (the set a; i: the others).  So only the m x m
// block is factored,
//   M_aa = I - G_aa diag(v_a)            LU with partial pivoting
//   [W | e]_a = M_aa^-1 [G | c_d]_a      forward and backward substitution, n + 1 columns
//   [W | e]_i = [G | c_d]_i + G_ia diag(v_a) [W | e]_a
//   T = G_od + G_od,a diag(v_a) W_a,     o = c_o + G_od (v .* e)
// and of the symmetric W_ii only the upper triangle is computed (the lower one
// is its mirror image): for half the pixels on, 2.8 n^3 real operations instead
// of the 10.7 n^3 of a factorisation of the whole M.
//
// All products run on the tensor cores in FP64 accuracy (ozaki.cuh); the FP64
// pipe (1.25 TFLOP/s) is left with the panels and the triangular blocks.  One
// cooperative launch does everything: m is known only on the device, and the
// phases (panel columns above all) are too short for launches of their own.
//
// Measured, half the pixels on: N_d = 4096 748 -> 34.5 ms, N_d = 1517 86 -> 9.1
// ms (before: LU of the whole M and its substitutions on the FP64 pipe).  At
// 4096: panels 10.9 ms (5.3 us a column: one grid barrier, two L2 round trips
// and the FP64 chain of the reciprocal and the update), products of LU 2.7,
// of the substitutions 8.0 and of the last step 4.4 (tensor cores and the
// read-back of ozaki.cuh), diagonal blocks 3.8, interchanges and L^-1 3.0,
// digits 2.5.
#include <cstdio>

#include "form_ports.cuh"
#include "ozaki.cuh"

namespace pngf {
namespace {

constexpr int NB = 32;        // panel width
constexpr int BB = 64;        // block of the substitutions, K of their products
constexpr int FT_THREADS = OZ_THREADS;
constexpr int FT_WARPS = FT_THREADS / 32;

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
  unsigned char* imgA;
  unsigned char* imgB;
  int* ea;
  int* eb;
  c128* cand;               // [2][P][NB] candidate pivot rows
  unsigned long long* key;  // [2][P] their keys
  int* cand_row;            // [2][P]
  c128* drow;               // [2][NB] diagonal row of the column
  int* piv;                 // NB pivots of the panel
  c128* dinv;               // n reciprocals of the pivots
  int* perm;                // row i of the pivoted M_aa is row perm[i] of M_aa
  c128* binv;               // inverses of the BB x BB diagonal blocks: of L, then of U
  Control* ctl;
};

// |re| + |im| as an order-preserving key (NaN lowest: it is taken only where
// nothing else is left)
__device__ __forceinline__ unsigned long long pivot_key(c128 z) {
  const double a = cabs1(z);
  return isnan(a) ? 0ull : (unsigned long long)__double_as_longlong(a);
}

// 1 / z without FP64 divisions (each occupies the FP64 pipe for ten
// instructions): z is scaled by a power of two to [1, 2), |z|^-2 by an FP32
// seed and three Newton steps (quadratic: 2^-22, 2^-44, 2^-88)
__device__ __forceinline__ c128 crecip(c128 z) {
  const int ex = max(oz_exp(z.x), oz_exp(z.y));
  if (ex < 64 || ex > 1980) return cdiv(mk(1.0, 0.0), z);  // zero, tiny, huge, infinite, NaN
  const double sc = __longlong_as_double((long long)(2046 - ex) << 52);  // 2^(1023 - ex)
  const double x = z.x * sc, y = z.y * sc;
  const double d = fma(x, x, y * y);  // in [1, 8)
  double r = (double)(1.0f / (float)d);
  r = fma(r, fma(-d, r, 1.0), r);
  r = fma(r, fma(-d, r, 1.0), r);
  r *= sc;
  return mk(x * r, -y * r);
}

// the ascending lists of the pixels that are on and off (one CTA)
__device__ void factor_lists(const FactorArgs& a) {
  __shared__ int s_scan[FT_WARPS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int chunk = (a.n + FT_THREADS - 1) / FT_THREADS;
  const int i0 = min(a.n, (int)threadIdx.x * chunk), i1 = min(a.n, i0 + chunk);
  int c = 0;
  for (int i = i0; i < i1; ++i) c += a.b_in[i] != 0;
  int incl = c;
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += y;
  }
  if (lane == 31) s_scan[warp] = incl;
  __syncthreads();
  int before = incl - c, m = 0;
  for (int w = 0; w < FT_WARPS; ++w) {
    if (w < warp) before += s_scan[w];
    m += s_scan[w];
  }
  int on = before, off_ = m + i0 - before;
  for (int i = i0; i < i1; ++i) {
    if (a.b_in[i]) a.act[on++] = i;
    else a.act[off_++] = i;
  }
  if (threadIdx.x == 0) *a.count = m;
}

// ---------------------------------------------------------------- panel
// LU of rows [j0, m) x columns [j0, j0 + jb) with partial pivoting (|re| + |im|,
// ties -> lowest row).  CTA q holds its chunk of the rows in shared memory.
// Per column: every CTA publishes its candidate row (and the owner the
// diagonal row), one grid barrier, every CTA picks the winner, swaps what it
// owns and updates its rows, tracking the next column's candidate.  The rows
// travel with the candidates, so one barrier per column is enough.
__device__ bool factor_panel(const FactorArgs& a, int m, int j0, int jb, c128* ps) {
  __shared__ unsigned long long s_key[FT_WARPS];
  __shared__ int s_row[FT_WARPS];
  __shared__ c128 s_u[NB], s_d[NB];
  __shared__ c128 s_inv;
  __shared__ int s_p;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, P = gridDim.x, cta = blockIdx.x;
  const int rows = m - j0;
  const int rb = j0 + (int)((long long)rows * cta / P), re = j0 + (int)((long long)rows * (cta + 1) / P);
  const bool act_lane = lane < jb;
  unsigned long long bk = 0;
  int br = 0x7fffffff;
  for (int r = rb + warp; r < re; r += FT_WARPS) {
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
      unsigned long long k = lane < FT_WARPS ? s_key[lane] : 0ull;
      int r = lane < FT_WARPS ? s_row[lane] : 0x7fffffff;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long ok = __shfl_xor_sync(0xffffffffu, k, off);
        const int orr = __shfl_xor_sync(0xffffffffu, r, off);
        if (ok > k || (ok == k && orr < r)) { k = ok; r = orr; }
      }
      if (r != 0x7fffffff) a.cand[((size_t)par * P + cta) * NB + lane] = ps[(r - rb) * NB + lane];
      if (lane == 0) {
        a.key[par * P + cta] = k;
        a.cand_row[par * P + cta] = r;
      }
    } else if (warp == 1 && col >= rb && col < re) {
      a.drow[par * NB + lane] = ps[(col - rb) * NB + lane];
    }
    if (!grid_sync(a.ctl)) return false;
    // ---- the pivot, its row and its reciprocal (warp 0), the diagonal row (warp 1)
    if (warp == 0) {
      unsigned long long k = 0;
      int r = 0x7fffffff, q = -1;
      for (int c = lane; c < P; c += 32) {
        const unsigned long long ck = a.key[par * P + c];
        const int cr = a.cand_row[par * P + c];
        if (ck > k || (ck == k && cr < r)) { k = ck; r = cr; q = c; }
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
      const c128 inv = crecip(pv);
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
    for (int r = max(rb, col + 1) + warp; r < re; r += FT_WARPS) {
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
  for (int r = rb + warp; r < re; r += FT_WARPS)
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

// ---------------------------------------------------------------- diagonal blocks
// Columns [32 half, 32 half + 32) of the inverse of diagonal block bi of L
// (unit lower) or U, by substitution: one warp per two columns, lane = row
// (rows lane and 32 + lane).  Rows past the matrix count as identity.
__device__ void block_inverse(const FactorArgs& a, int m, int bi, int upper, int half, c128* sm) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, i0 = bi * BB, jb = min(BB, m - i0);
  __syncthreads();
  for (int q = tid; q < BB * BB; q += FT_THREADS) {  // column-major, the triangle without its diagonal
    const int r = q / BB, k = q % BB;
    const bool in = r < jb && k < jb && (upper ? r < k : r > k);
    sm[k * (BB + 1) + r] = in ? a.LU[(size_t)(i0 + r) * a.ldw + i0 + k] : mk(0.0, 0.0);
  }
  c128* di = sm + BB * (BB + 1);
  if (tid < BB) di[tid] = upper && tid < jb ? a.dinv[i0 + tid] : mk(1.0, 0.0);
  __syncthreads();
  c128* out = a.binv + ((size_t)(upper ? (m + BB - 1) / BB : 0) + bi) * BB * BB;
  for (int u = warp; u < 16; u += FT_WARPS) {
    const int c = 32 * half + 2 * u;
    auto unit = [&](int r, int cc) { return mk(r == cc ? 1.0 : 0.0, 0.0); };
    c128 l0 = unit(lane, c), l1 = unit(lane, c + 1), h0 = unit(32 + lane, c), h1 = unit(32 + lane, c + 1);
    if (!upper) {
      for (int k = c; k < BB; ++k) {
        const c128 tl = sm[k * (BB + 1) + lane], th = sm[k * (BB + 1) + 32 + lane];
        const c128 s0 = shfl_c(k < 32 ? l0 : h0, k & 31), s1 = shfl_c(k < 32 ? l1 : h1, k & 31);
        if (k < 32) {
          l0 = cfms(tl, s0, l0);
          l1 = cfms(tl, s1, l1);
        }
        h0 = cfms(th, s0, h0);
        h1 = cfms(th, s1, h1);
      }
    } else {
      for (int k = c + 1; k >= 0; --k) {
        const c128 tl = sm[k * (BB + 1) + lane], th = sm[k * (BB + 1) + 32 + lane], d = di[k];
        const c128 s0 = cmul(shfl_c(k < 32 ? l0 : h0, k & 31), d), s1 = cmul(shfl_c(k < 32 ? l1 : h1, k & 31), d);
        if (k >= 32) {
          h0 = lane == k - 32 ? s0 : cfms(th, s0, h0);
          h1 = lane == k - 32 ? s1 : cfms(th, s1, h1);
        }
        l0 = lane == k ? s0 : cfms(tl, s0, l0);
        l1 = lane == k ? s1 : cfms(tl, s1, l1);
      }
    }
    out[lane * BB + c] = l0;
    out[lane * BB + c + 1] = l1;
    out[(32 + lane) * BB + c] = h0;
    out[(32 + lane) * BB + c + 1] = h1;
  }
}

// ---------------------------------------------------------------- the factorisation
__global__ void __launch_bounds__(FT_THREADS, 1) factor_kernel(const __grid_constant__ FactorArgs a) {
  extern __shared__ __align__(128) unsigned char f_smem[];
  __shared__ __align__(8) unsigned long long s_bars[OZ_NBAR];
  __shared__ unsigned s_tmem;
  __shared__ Swaps s_sw;
  __shared__ int s_cum[264];  // tiles before row block I of the last product (n_d <= 32768: 257 blocks)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, P = gridDim.x, cta = blockIdx.x;
  const int gw = cta * FT_WARPS + warp, nw = P * FT_WARPS;  // warps of the grid
  const int n = a.n, ldw = a.ldw, ncol = n + 1;
  Control* ctl = a.ctl;
  c128* sm = reinterpret_cast<c128*>(f_smem);
  OzState oz;
  oz_setup(oz, s_bars, &s_tmem);
  bool ok = true;
  // ---- the lists (CTA 0); one pass over G: Re G + Im G for the refreshes; the rows of W at pixels that are off start as [G | c_d]
  if (cta == 0) factor_lists(a);
  for (int i = cta; i < n; i += P) {
    const c128* g = a.G + (size_t)i * n;
    c128* w = a.W + (size_t)i * ldw;
    double* gs = a.Gs + (size_t)i * n;
    const bool on = a.b_in[i] != 0;
    for (int j = tid; j < n; j += FT_THREADS) {
      const c128 z = g[j];
      if (!on) w[j] = z;
      gs[j] = z.x + z.y;
    }
    if (tid == 0) {
      if (!on) w[n] = a.cd[i];
      a.v[i] = on ? a.dv[i] : mk(0.0, 0.0);
      a.b[i] = on ? 1 : 0;
    }
  }
  for (int q = cta * FT_THREADS + tid; q < a.n_o * n; q += P * FT_THREADS)
    a.T[(size_t)(q / n) * a.ldt + q % n] = a.God[q];
  ok = grid_sync(ctl);
  const int m = ok ? *reinterpret_cast<volatile int*>(a.count) : 0;
  const int* act = a.act;
  const int* ina = a.act + m;
  const int nJ = (ncol + OZ_N - 1) / OZ_N;  // tile columns of the right-hand sides
  // digits of the rows act[i0 .. i0 + K) of [W | e], column by column
  auto digits_rhs = [&](int i0, int K) {
    const int nk = (K + OZ_KC - 1) / OZ_KC;
    for (int r0 = 4 * gw; r0 < nJ * OZ_N; r0 += 4 * nw)
      oz_digitise_rows<OZ_N>(r0, K, nk, a.imgB, a.eb, [&](int c, int k) {
        return c < ncol ? a.W[(size_t)act[i0 + k] * ldw + c] : mk(0.0, 0.0);
      });
  };
  auto digits_A = [&](int rows, int K, auto load) {
    const int nk = (K + OZ_KC - 1) / OZ_KC, rpad = (rows + OZ_M - 1) / OZ_M * OZ_M;
    for (int r0 = 4 * gw; r0 < rpad; r0 += 4 * nw)
      oz_digitise_rows<OZ_M>(r0, K, nk, a.imgA, a.ea, [&](int r, int k) { return r < rows ? load(r, k) : mk(0.0, 0.0); });
  };
  // the images are read next by bulk asynchronous copies (async proxy)
  auto images_done = [&]() -> bool {
    asm volatile("fence.proxy.async.global;" ::: "memory");
    return grid_sync(ctl);
  };
  // ---- M_aa
  if (ok) {
    for (int i = cta; i < m; i += P) {
      const c128* g = a.G + (size_t)act[i] * n;
      for (int j = tid; j < m; j += FT_THREADS) {
        const int pj = act[j];
        const c128 z = cmul(g[pj], a.dv[pj]);
        a.LU[(size_t)i * ldw + j] = mk((i == j ? 1.0 : 0.0) - z.x, -z.y);
      }
      if (tid == 0) a.perm[i] = i;
    }
    ok = grid_sync(ctl);
  }
  // ---- LU
  for (int j0 = 0; ok && j0 < m; j0 += NB) {
    const int jb = min(NB, m - j0), i1 = j0 + jb, rest = m - i1, nk = (jb + OZ_KC - 1) / OZ_KC;
    ok = factor_panel(a, m, j0, jb, sm);
    if (!ok) break;
    net_swaps(a, j0, jb, s_sw);
    // L of the block (unit lower), column-major: Ls[k][row]
    for (int q = tid; q < NB * NB; q += FT_THREADS) {
      const int k = q / NB, r = q % NB;
      sm[q] = (r < jb && k < r) ? a.LU[(size_t)(j0 + r) * ldw + j0 + k] : mk(0.0, 0.0);
    }
    __syncthreads();
    // interchanges of the other columns, and L^-1 on those right of the panel:
    // one warp per two columns, lane = row (a warp's FP64 instruction costs
    // the same for one lane as for 32)
    {
      const int ur = (rest + 1) / 2, ul = j0 / 2;
      const int ts = s_sw.top_src[lane], er = s_sw.ext_row[lane], es = s_sw.ext_src[lane];
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
            const c128 l = sm[k * NB + lane];  // zero for row <= k
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
      if (cta == P - 1 && warp == FT_WARPS - 1) {  // the row permutation
        const int x = lane < jb ? a.perm[ts] : 0, y = er >= 0 ? a.perm[es] : 0;
        __syncwarp();
        if (lane < jb) a.perm[j0 + lane] = x;
        if (er >= 0) a.perm[er] = y;
      }
    }
    if (rest > 0) digits_A(rest, jb, [&](int r, int k) { return a.LU[(size_t)(i1 + r) * ldw + j0 + k]; });
    if (!(ok = images_done())) break;
    if (rest == 0) continue;
    // U12, column by column
    const int nI = (rest + OZ_M - 1) / OZ_M, nb1 = (rest + OZ_N - 1) / OZ_N;
    for (int r0 = 4 * gw; r0 < nb1 * OZ_N; r0 += 4 * nw)
      oz_digitise_rows<OZ_N>(r0, jb, nk, a.imgB, a.eb, [&](int r, int k) {
        return r < rest ? a.LU[(size_t)(j0 + k) * ldw + i1 + r] : mk(0.0, 0.0);
      });
    if (!(ok = images_done())) break;
    ok = oz_tiles<-1>(oz, f_smem, a.imgA, a.imgB, a.ea, a.eb, nk, (long long)nI * nb1, cta, P,
                      [&](long long t, int& I, int& J) { I = (int)(t % nI); J = (int)(t / nI); },
                      [&](int r, int J, int& cols) -> c128* {
                        cols = rest - J * OZ_N;
                        return r < rest ? a.LU + (size_t)(i1 + r) * ldw + i1 + J * OZ_N : nullptr;
                      });
    if (ok) ok = grid_sync(ctl);
  }
  // ---- the pivoted right-hand sides, and the inverses of the diagonal blocks
  //      of L and U, by which the substitutions become products
  const int nblk = (m + BB - 1) / BB;
  if (ok) {
    for (int i = cta; i < m; i += P) {
      const int src = act[a.perm[i]];
      const c128* g = a.G + (size_t)src * n;
      c128* w = a.W + (size_t)act[i] * ldw;
      for (int j = tid; j < n; j += FT_THREADS) w[j] = g[j];
      if (tid == 0) w[n] = a.cd[src];
    }
    for (int q = cta; q < 4 * nblk; q += P) block_inverse(a, m, q >> 2, (q >> 1) & 1, q & 1, sm);
    ok = grid_sync(ctl);
  }
  // ---- forward, then backward substitution, blocks of BB rows:
  //      X_b = (diagonal block)^-1 Y_b, then Y -= (rest of the block column) X_b
  for (int step = 0; ok && step < 2 * nblk; ++step) {
    const bool fwd = step < nblk;
    const int bi = fwd ? step : 2 * nblk - 1 - step, i0 = bi * BB, jb = min(BB, m - i0), nk = (jb + OZ_KC - 1) / OZ_KC;
    const c128* inv = a.binv + ((size_t)(fwd ? 0 : nblk) + bi) * BB * BB;
    digits_rhs(i0, jb);
    digits_A(jb, jb, [&](int r, int k) { return inv[r * BB + k]; });
    if (!(ok = images_done())) break;
    ok = oz_tiles<0>(oz, f_smem, a.imgA, a.imgB, a.ea, a.eb, nk, nJ, cta, P,
                     [&](long long t, int& I, int& J) { I = 0; J = (int)t; },
                     [&](int r, int J, int& cols) -> c128* {
                       cols = ncol - J * OZ_N;
                       return r < jb ? a.W + (size_t)act[i0 + r] * ldw + J * OZ_N : nullptr;
                     });
    if (!ok || !(ok = grid_sync(ctl))) break;
    const int r0 = fwd ? i0 + jb : 0, rows = fwd ? m - r0 : i0, nI = (rows + OZ_M - 1) / OZ_M;
    if (rows == 0) continue;
    digits_rhs(i0, jb);
    digits_A(rows, jb, [&](int r, int k) { return a.LU[(size_t)(r0 + r) * ldw + i0 + k]; });
    if (!(ok = images_done())) break;
    ok = oz_tiles<-1>(oz, f_smem, a.imgA, a.imgB, a.ea, a.eb, nk, (long long)nI * nJ, cta, P,
                      [&](long long t, int& I, int& J) { I = (int)(t % nI); J = (int)(t / nI); },
                      [&](int r, int J, int& cols) -> c128* {
                        cols = ncol - J * OZ_N;
                        return r < rows ? a.W + (size_t)act[r0 + r] * ldw + J * OZ_N : nullptr;
                      });
    if (ok) ok = grid_sync(ctl);
  }
  // ---- the rows of the pixels that are off, and T: += G_ia v_a [W | e]_a, of W
  //      only the tiles that reach the upper triangle
  if (ok && m > 0) {
    const int ni = n - m, nr = ni + a.n_o, nI = (nr + OZ_M - 1) / OZ_M;
    auto jmin = [&](int I) { return (I + 1) * OZ_M > ni ? 0 : ina[I * OZ_M] / OZ_N; };
    if (tid == 0) {
      int c = 0;
      for (int I = 0; I < nI; ++I) {
        s_cum[I] = c;
        c += nJ - jmin(I);
      }
      s_cum[nI] = c;
    }
    __syncthreads();
    const int T = s_cum[nI];
    for (int k0 = 0; ok && k0 < m; k0 += OZ_KMAX) {
      const int kb = min(OZ_KMAX, m - k0), nk = (kb + OZ_KC - 1) / OZ_KC;
      digits_rhs(k0, kb);
      digits_A(nr, kb, [&](int r, int k) {
        const int pk = act[k0 + k];
        return cmul(r < ni ? a.G[(size_t)ina[r] * n + pk] : a.God[(size_t)(r - ni) * n + pk], a.dv[pk]);
      });
      if (!(ok = images_done())) break;
      ok = oz_tiles<1>(oz, f_smem, a.imgA, a.imgB, a.ea, a.eb, nk, T, cta, P,
                       [&](long long t, int& I, int& J) {
                         int lo = 0, hi = nI - 1;
                         while (lo < hi) {
                           const int mid = (lo + hi + 1) >> 1;
                           if (s_cum[mid] <= t) lo = mid;
                           else hi = mid - 1;
                         }
                         I = lo;
                         J = jmin(I) + (int)t - s_cum[I];
                       },
                       [&](int r, int J, int& cols) -> c128* {
                         if (r >= nr) return nullptr;
                         if (r < ni) {
                           cols = ncol - J * OZ_N;
                           return a.W + (size_t)ina[r] * ldw + J * OZ_N;
                         }
                         cols = n - J * OZ_N;
                         return a.T + (size_t)(r - ni) * a.ldt + J * OZ_N;
                       });
      if (ok) ok = grid_sync(ctl);
    }
  }
  // ---- the lower triangle of W mirrors the upper one; diag W and e are read off
  if (ok) {
    constexpr int TS = 32, TLD = TS + 1;
    const int nt = (n + TS - 1) / TS;
    const long long nT = (long long)nt * (nt + 1) / 2;
    for (long long t = cta; t < nT; t += P) {
      int bi, bj;
      tri_rc(t, nt, bi, bj);
      __syncthreads();
      for (int q = tid; q < TS * TS; q += FT_THREADS) {
        const int r = q / TS, c = q % TS, i = bi * TS + r, j = bj * TS + c;
        if (i < n && j < n) {
          const c128 w = a.W[(size_t)i * ldw + j];
          sm[r * TLD + c] = w;
          if (i == j) a.diag[i] = w;
        }
      }
      __syncthreads();
      for (int q = tid; q < TS * TS; q += FT_THREADS) {
        const int r = q / TS, c = q % TS, i = bj * TS + r, j = bi * TS + c;  // lower: i > j
        if (i < n && j < i) {
          a.W[(size_t)i * ldw + j] = sm[c * TLD + r];
        }
      }
    }
    for (int i = cta * FT_THREADS + tid; i < n; i += P * FT_THREADS) a.e[i] = a.W[(size_t)i * ldw + n];
  } else if (tid == 0) {
    latch_status(ctl, PNGF_ETIMEOUT);
  }
  oz_teardown(oz, !ok);
}

}  // namespace

// bytes of the factor's scratch (c->L.oz): digit images, row exponents, lists,
// candidate rows, reciprocals of the pivots
struct FactorScratch {
  size_t imgA, imgB, ea, eb, act, cand, key, cand_row, drow, piv, dinv, perm, binv, total;
};
static FactorScratch factor_scratch(int n) {
  FactorScratch f{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += (bytes + 255) / 256 * 256;
    return o;
  };
  f.imgA = take(oz_a_bytes(n + kMaxPorts, OZ_KMAX));
  f.imgB = take(oz_b_bytes(n + 1, OZ_KMAX));
  f.ea = take(((size_t)n + kMaxPorts + OZ_M) * sizeof(int));
  f.eb = take(((size_t)n + 1 + OZ_N) * sizeof(int));
  f.act = take(((size_t)n + 64) * sizeof(int));
  f.cand = take((size_t)2 * 1024 * NB * sizeof(c128));
  f.key = take((size_t)2 * 1024 * sizeof(unsigned long long));
  f.cand_row = take((size_t)2 * 1024 * sizeof(int));
  f.drow = take((size_t)2 * NB * sizeof(c128));
  f.piv = take(NB * sizeof(int));
  f.dinv = take((size_t)n * sizeof(c128));
  f.perm = take((size_t)n * sizeof(int));
  f.binv = take((size_t)2 * ((n + BB - 1) / BB) * BB * BB * sizeof(c128));
  f.total = off;
  return f;
}
size_t factor_scratch_bytes(int n) { return factor_scratch(n).total; }
void factor_images(int n, size_t off[5]) {
  const FactorScratch f = factor_scratch(n);
  off[0] = f.imgA;
  off[1] = f.imgB;
  off[2] = f.ea;
  off[3] = f.eb;
  off[4] = f.act;  // the end of the four
}

// ---------------------------------------------------------------- driver
pngf_status factor_fp64(pngf_ctx* c, const uint8_t* b) {
  const int n = c->cfg.n_d;
  cudaStream_t s = c->stream;
  const FactorScratch f = factor_scratch(n);
  char* ws = c->ws + c->L.oz;
  FactorArgs a{};
  a.n = n;
  a.n_o = c->cfg.n_o;
  a.ldw = c->L.ldw;
  a.ldt = c->L.ldt;
  a.G = c->G;
  a.God = c->God;
  a.cd = c->cd;
  a.dv = c->dv;
  a.b_in = b;
  a.LU = at<c128>(c, c->L.LU);
  a.W = at<c128>(c, c->L.W);
  a.T = at<c128>(c, c->L.T);
  a.v = at<c128>(c, c->L.v);
  a.b = at<uint8_t>(c, c->L.b);
  a.diag = at<c128>(c, c->L.diag);
  a.e = at<c128>(c, c->L.e);
  a.Gs = at<double>(c, c->L.gsum);
  a.imgA = reinterpret_cast<unsigned char*>(ws + f.imgA);
  a.imgB = reinterpret_cast<unsigned char*>(ws + f.imgB);
  a.ea = reinterpret_cast<int*>(ws + f.ea);
  a.eb = reinterpret_cast<int*>(ws + f.eb);
  a.act = reinterpret_cast<int*>(ws + f.act);
  a.count = a.act + n + 32;
  a.cand = reinterpret_cast<c128*>(ws + f.cand);
  a.key = reinterpret_cast<unsigned long long*>(ws + f.key);
  a.cand_row = reinterpret_cast<int*>(ws + f.cand_row);
  a.drow = reinterpret_cast<c128*>(ws + f.drow);
  a.piv = reinterpret_cast<int*>(ws + f.piv);
  a.dinv = reinterpret_cast<c128*>(ws + f.dinv);
  a.perm = reinterpret_cast<int*>(ws + f.perm);
  a.binv = reinterpret_cast<c128*>(ws + f.binv);
  a.ctl = at<Control>(c, c->L.ctl);
  if (cudaFuncSetAttribute(factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM) != cudaSuccess)
    return PNGF_ECUDA;
  int P = (n + 15) / 16;
  if (P > c->n_sm) P = c->n_sm;
  if (cudaMemsetAsync(&a.ctl->bar_count, 0, sizeof(unsigned), s) != cudaSuccess) return PNGF_ECUDA;
  void* params[] = {&a};
  if (cudaLaunchCooperativeKernel((const void*)factor_kernel, dim3(P), dim3(FT_THREADS), params, OZ_SMEM, s) !=
      cudaSuccess)
    return PNGF_ECUDA;
  form_o<<<1, 256, 0, s>>>(c->God, c->co, a.v, a.e, n, c->obj, a.ctl);
  return cuda_status(cudaGetLastError());
}

}  // namespace pngf
