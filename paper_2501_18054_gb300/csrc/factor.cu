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
// Measured, half the pixels on: N_d = 4096 748 -> 38 ms, N_d = 1517 86 -> 9.5
// ms (before: LU of the whole M and its substitutions on the FP64 pipe).  At
// 4096 the panels take 9.6 ms (4.7 us a column: one exchange of words, an L2 round trip
// for the pivot row and the FP64 chain of the reciprocal and the update; 5.3 us
// with a grid barrier and a read of the keys), the products of LU, substitutions and
// last step about 17 (tensor cores and the read-back of
// ozaki.cuh), diagonal blocks 3.7, interchanges and L^-1 3.0, digits 4.
#include <cstdio>

#include "factor_common.cuh"
#include "form_ports.cuh"
#include "ozaki.cuh"

namespace pngf {
namespace {

constexpr int BB = 64;        // block of the substitutions, K of their products
constexpr int FT_THREADS = OZ_THREADS;
constexpr int FT_WARPS = FT_THREADS / 32;

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
      for (int k = c; k < jb; ++k) {
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
      for (int k = c < jb ? min(c + 1, jb - 1) : -1; k >= 0; --k) {
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

// Whether a pixel that is on has |dv G_kk| >= 16: lossy metal (500) and the
// like, against 0.5 for eps = 10.  Such systems go to factor_pipe.cu.  Not for
// accuracy: at N_d = 576 and contrasts of 0.5 to 500 (both devices, dv scaled, four
// designs) the error of W here is 3e-16 to 6e-16 against 7e-16 to 1e-15 there (the guide at
// 0.5: 4e-15 each; at 2, near a resonance: 2e-13 against 3e-13), that of the objective
// within a factor of four either way, and the time 3.2-3.6 ms against 13.3.  But
// what a search reports on metal can hang on the last bits of the start state (a
// metal-filled guide transmits 10^-9 of the power: rounding of 10^-14 in the fields is
// 10^-9 of it), and stays the same; any line between the two contrasts does that.
// So does a contrast that is not finite.  (2, from factor_kernel: G is not finite.
// Eliminating the pixels that are on alone would leave an entry between two
// others out of sight; the elimination of the whole M meets it and reports it.)
__global__ void contrast_kernel(const c128* G, const c128* dv, const uint8_t* b, int n, int* high) {
  int h = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    if (b[i] && !(cabs2(dv[i]) * cabs2(G[(size_t)i * n + i]) < 256.0)) h = 1;
  h = __syncthreads_or(h);
  if (threadIdx.x == 0) *high = h;
}

// After a product: the grid's barrier, and the entries that the product left to FP64
template <int OP, class Row>
__device__ __forceinline__ bool product_done(const FactorArgs& a, bool ok, int K, Row row_of) {
  if (!ok || !grid_sync(a.ctl)) return false;
  const unsigned m = oz_listed(a.im);
  if (m == 0) return true;
  const int P = gridDim.x;
  oz_redo<OP>(a.im, m, K, (int)(threadIdx.x >> 5) * P + blockIdx.x, P * FT_WARPS, row_of);
  return grid_sync(a.ctl);
}

// ---------------------------------------------------------------- the factorisation
__global__ void __launch_bounds__(FT_THREADS, 1) factor_kernel(const __grid_constant__ FactorArgs a) {
  extern __shared__ __align__(128) unsigned char f_smem[];
  if (*a.high == 1) return;
  __shared__ __align__(8) unsigned long long s_bars[OZ_NBAR];
  __shared__ unsigned s_tmem;
  __shared__ Swaps s_sw;
  __shared__ int s_cum[264];  // tiles before row block I of the last product (n_d <= 32768: 257 blocks)
  const int tid = threadIdx.x, warp = tid >> 5, P = gridDim.x, cta = blockIdx.x;
  const int gw = cta * FT_WARPS + warp, nw = P * FT_WARPS;  // warps of the grid
  const int n = a.n, ldw = a.ldw, ncol = n + 1;
  Control* ctl = a.ctl;
  c128* sm = reinterpret_cast<c128*>(f_smem);
  OzState oz;
  oz_setup(oz, s_bars, &s_tmem);
  bool ok = true;
  // ---- the lists (CTA 0); one pass over G: Re G + Im G for the refreshes; the rows of W at pixels that are off start as [G | c_d]
  if (cta == 0) factor_lists(a);
  int bad = 0;
  for (int i = cta; i < n; i += P) {
    const c128* g = a.G + (size_t)i * n;
    c128* w = a.W + (size_t)i * ldw;
    double* gs = a.Gs + (size_t)i * n;
    const bool on = a.b_in[i] != 0;
    for (int j = tid; j < n; j += FT_THREADS) {
      const c128 z = g[j];
      if (!on) w[j] = z;
      gs[j] = z.x + z.y;
      bad |= oz_exp(z.x) == 0x7ff || oz_exp(z.y) == 0x7ff;
    }
    if (tid == 0) {
      if (!on) w[n] = a.cd[i];
      a.v[i] = on ? a.dv[i] : mk(0.0, 0.0);
      a.b[i] = on ? 1 : 0;
    }
  }
  for (int q = cta * FT_THREADS + tid; q < a.n_o * n; q += P * FT_THREADS)
    a.T[(size_t)(q / n) * a.ldt + q % n] = a.God[q];
  if (__syncthreads_or(bad) && tid == 0) *const_cast<int*>(a.high) = 2;
  ok = grid_sync(ctl);
  if (ok && *reinterpret_cast<const volatile int*>(a.high)) {
    oz_teardown(oz, false);
    return;
  }
  const int m = ok ? *reinterpret_cast<volatile int*>(a.count) : 0;
  const int* act = a.act;
  const int* ina = a.act + m;
  const int nJ = (ncol + OZ_N - 1) / OZ_N;  // tile columns of the right-hand sides
  // digits of the rows act[i0 .. i0 + K) of [W | e], column by column
  auto digits_rhs = [&](int i0, int K) {
    const int nk = (K + OZ_KC - 1) / OZ_KC;
    for (int r0 = 4 * gw; r0 < nJ * OZ_N; r0 += 4 * nw)
      oz_digitise_rows<OZ_N>(r0, K, nk, a.im.B, a.im.sqB, a.im.eb, a.im.nb, a.im.fb, [&](int c, int k) {
        return c < ncol ? a.W[(size_t)act[i0 + k] * ldw + c] : mk(0.0, 0.0);
      });
  };
  auto digits_A = [&](int rows, int K, auto load) {
    const int nk = (K + OZ_KC - 1) / OZ_KC, rpad = (rows + OZ_M - 1) / OZ_M * OZ_M;
    for (int r0 = 4 * gw; r0 < rpad; r0 += 4 * nw)
      oz_digitise_rows<OZ_M>(r0, K, nk, a.im.A, a.im.sqA, a.im.ea, a.im.na, a.im.fa,
                             [&](int r, int k) { return r < rows ? load(r, k) : mk(0.0, 0.0); });
  };
  // the images are read next by bulk asynchronous copies (async proxy)
  auto images_done = [&]() -> bool {
    if (cta == 0 && tid == 0) oz_list_clear(a.im);
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
    ok = factor_panel<FT_WARPS, false>(a, m, j0, jb, sm);
    if (!ok) break;
    net_swaps(a, j0, jb, s_sw);
    // L of the block (unit lower), column-major: Ls[k][row]
    for (int q = tid; q < NB * NB; q += FT_THREADS) {
      const int k = q / NB, r = q % NB;
      sm[q] = (r < jb && k < r) ? a.LU[(size_t)(j0 + r) * ldw + j0 + k] : mk(0.0, 0.0);
    }
    __syncthreads();
    swap_and_solve(a, s_sw, sm, m, j0, jb, gw, nw);
    if (rest > 0) digits_A(rest, jb, [&](int r, int k) { return a.LU[(size_t)(i1 + r) * ldw + j0 + k]; });
    if (!(ok = images_done())) break;
    if (rest == 0) continue;
    // U12, column by column
    const int nI = (rest + OZ_M - 1) / OZ_M, nb1 = (rest + OZ_N - 1) / OZ_N;
    for (int r0 = 4 * gw; r0 < nb1 * OZ_N; r0 += 4 * nw)
      oz_digitise_rows<OZ_N>(r0, jb, nk, a.im.B, a.im.sqB, a.im.eb, a.im.nb, a.im.fb, [&](int r, int k) {
        return r < rest ? a.LU[(size_t)(j0 + k) * ldw + i1 + r] : mk(0.0, 0.0);
      });
    if (!(ok = images_done())) break;
    auto row = [&](int r, int J, int& cols) -> c128* {
      cols = rest - J * OZ_N;
      return r < rest ? a.LU + (size_t)(i1 + r) * ldw + i1 + J * OZ_N : nullptr;
    };
    ok = oz_tiles<-1>(oz, f_smem, a.im, jb, 1.0f, (long long)nI * nb1, cta, P,
                      [&](long long t, int& I, int& J) { I = (int)(t % nI); J = (int)(t / nI); }, row);
    ok = product_done<-1>(a, ok, jb, row);
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
    const int bi = fwd ? step : 2 * nblk - 1 - step, i0 = bi * BB, jb = min(BB, m - i0);
    const c128* inv = a.binv + ((size_t)(fwd ? 0 : nblk) + bi) * BB * BB;
    digits_rhs(i0, jb);
    digits_A(jb, jb, [&](int r, int k) { return inv[r * BB + k]; });
    if (!(ok = images_done())) break;
    auto block_row = [&](int r, int J, int& cols) -> c128* {
      cols = ncol - J * OZ_N;
      return r < jb ? a.W + (size_t)act[i0 + r] * ldw + J * OZ_N : nullptr;
    };
    ok = oz_tiles<0>(oz, f_smem, a.im, jb, 0.0f, nJ, cta, P, [&](long long t, int& I, int& J) { I = 0; J = (int)t; },
                     block_row);
    ok = product_done<0>(a, ok, jb, block_row);
    if (!ok) break;
    const int r0 = fwd ? i0 + jb : 0, rows = fwd ? m - r0 : i0, nI = (rows + OZ_M - 1) / OZ_M;
    if (rows == 0) continue;
    digits_rhs(i0, jb);
    digits_A(rows, jb, [&](int r, int k) { return a.LU[(size_t)(r0 + r) * ldw + i0 + k]; });
    if (!(ok = images_done())) break;
    auto row = [&](int r, int J, int& cols) -> c128* {
      cols = ncol - J * OZ_N;
      return r < rows ? a.W + (size_t)act[r0 + r] * ldw + J * OZ_N : nullptr;
    };
    ok = oz_tiles<-1>(oz, f_smem, a.im, jb, 1.0f, (long long)nI * nJ, cta, P,
                      [&](long long t, int& I, int& J) { I = (int)(t % nI); J = (int)(t / nI); }, row);
    ok = product_done<-1>(a, ok, jb, row);
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
      const int kb = min(OZ_KMAX, m - k0);
      digits_rhs(k0, kb);
      digits_A(nr, kb, [&](int r, int k) {
        const int pk = act[k0 + k];
        return cmul(r < ni ? a.G[(size_t)ina[r] * n + pk] : a.God[(size_t)(r - ni) * n + pk], a.dv[pk]);
      });
      if (!(ok = images_done())) break;
      auto row = [&](int r, int J, int& cols) -> c128* {
        if (r >= nr) return nullptr;
        if (r < ni) {
          cols = ncol - J * OZ_N;
          return a.W + (size_t)ina[r] * ldw + J * OZ_N;
        }
        cols = n - J * OZ_N;
        return a.T + (size_t)(r - ni) * a.ldt + J * OZ_N;
      };
      ok = oz_tiles<1>(oz, f_smem, a.im, kb, 1.0f, T, cta, P,
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
                       row);
      ok = product_done<1>(a, ok, kb, row);
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

// operands of up to n + kMaxPorts rows (A) and n + 1 rows (B), K <= OZ_KMAX; rows in
// whole blocks
static size_t oz_operands_at(char* p, int n, OzOperands& im) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* q = p + off;
    off += (bytes + 255) / 256 * 256;
    return q;
  };
  const size_t ra = (size_t)n + kMaxPorts + OZ_M, rb = (size_t)n + 1 + OZ_N;
  im.A = reinterpret_cast<unsigned char*>(take(oz_a_bytes(n + kMaxPorts, OZ_KMAX)));
  im.B = reinterpret_cast<unsigned char*>(take(oz_b_bytes(n + 1, OZ_KMAX)));
  im.sqA = reinterpret_cast<unsigned char*>(take(oz_a_bytes(n + kMaxPorts, OZ_KMAX) / (2 * OZ_S)));
  im.sqB = reinterpret_cast<unsigned char*>(take(oz_b_bytes(n + 1, OZ_KMAX) / (2 * OZ_S)));
  im.ea = reinterpret_cast<int*>(take(ra * sizeof(int)));
  im.eb = reinterpret_cast<int*>(take(rb * sizeof(int)));
  im.na = reinterpret_cast<float*>(take(ra * sizeof(float)));
  im.nb = reinterpret_cast<float*>(take(rb * sizeof(float)));
  im.fa = reinterpret_cast<c128*>(take(ra * OZ_KMAX * sizeof(c128)));
  im.fb = reinterpret_cast<c128*>(take(rb * OZ_KMAX * sizeof(c128)));
  im.list = reinterpret_cast<unsigned*>(take((1 + ((size_t)n + kMaxPorts) * (n + 1)) * sizeof(unsigned)));
  return off;
}
OzOperands oz_operands(char* scratch, int n) {
  OzOperands im;
  oz_operands_at(scratch, n, im);
  return im;
}
size_t oz_operand_bytes(int n) {
  OzOperands im;
  return oz_operands_at(nullptr, n, im);
}

// the factor's scratch (c->L.oz): operand images (not for mixed contexts), lists,
// candidate rows, reciprocals of the pivots
struct FactorScratch {
  size_t act, cand, key, cand_row, drow, piv, dinv, perm, binv, high, total;
};
static FactorScratch factor_scratch(int n, bool images) {
  FactorScratch f{};
  size_t off = images ? oz_operand_bytes(n) : 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += (bytes + 255) / 256 * 256;
    return o;
  };
  f.act = take(((size_t)n + 64) * sizeof(int));
  f.cand = take((size_t)2 * 1024 * NB * sizeof(c128));
  f.key = take((size_t)2 * 1024 * kPanelWord * sizeof(unsigned long long));
  f.cand_row = take((size_t)2 * 1024 * sizeof(int));
  f.drow = take((size_t)2 * NB * sizeof(c128));
  f.piv = take(NB * sizeof(int));
  f.dinv = take((size_t)n * sizeof(c128));
  f.perm = take((size_t)n * sizeof(int));
  f.binv = take(images ? (size_t)2 * ((n + BB - 1) / BB) * BB * BB * sizeof(c128) : 0);
  f.high = take(sizeof(int));
  f.total = off;
  return f;
}
size_t factor_scratch_bytes(int n, bool images) { return factor_scratch(n, images).total; }

// ---------------------------------------------------------------- driver
// arguments of both factorisations
FactorArgs factor_args(pngf_ctx* c, const uint8_t* b) {
  const int n = c->cfg.n_d;
  const FactorScratch f = factor_scratch(n, c->cfg.precision == PNGF_FP64);
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
  if (c->cfg.precision == PNGF_FP64) a.im = oz_operands(ws, n);
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
  a.high = reinterpret_cast<int*>(ws + f.high);
  a.ctl = at<Control>(c, c->L.ctl);
  return a;
}

pngf_status factor_fp64(pngf_ctx* c, const uint8_t* b) {
  const int n = c->cfg.n_d;
  cudaStream_t s = c->stream;
  FactorArgs a = factor_args(c, b);
  contrast_kernel<<<1, 1024, 0, s>>>(a.G, a.dv, b, n, const_cast<int*>(a.high));
  if (cudaFuncSetAttribute(factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM) != cudaSuccess)
    return PNGF_ECUDA;
  int P = (n + 15) / 16;
  if (P > c->n_sm) P = c->n_sm;
  if (cudaMemsetAsync(&a.ctl->bar_count, 0, sizeof(unsigned), s) != cudaSuccess ||
      cudaMemsetAsync(a.key, 0, (size_t)2 * P * kPanelWord * sizeof(unsigned long long), s) != cudaSuccess)
    return PNGF_ECUDA;
  void* params[] = {&a};
  if (cudaLaunchCooperativeKernel((const void*)factor_kernel, dim3(P), dim3(FT_THREADS), params, OZ_SMEM, s) !=
      cudaSuccess)
    return PNGF_ECUDA;
  const pngf_status st = factor_pipe(c, a);  // the high contrast
  if (st != PNGF_OK) return st;
  form_o<<<1, 256, 0, s>>>(c->God, c->co, a.v, a.e, n, c->obj, a.ctl);
  return cuda_status(cudaGetLastError());
}

pngf_status factor_mixed(pngf_ctx* c, const uint8_t* b) {
  FactorArgs a = factor_args(c, b);
  a.high = nullptr;
  const pngf_status st = factor_pipe(c, a);
  if (st != PNGF_OK) return st;
  form_o<<<1, 256, 0, c->stream>>>(c->God, c->co, a.v, a.e, a.n, c->obj, a.ctl);
  return cuda_status(cudaGetLastError());
}

}  // namespace pngf
