// Factorisation of the reduced system on the FP64 pipe, for mixed contexts and
// for high contrast:
//
//   M = I - G diag(v),  v = dv .* b
//   LU = P M            blocked right-looking LU with partial pivoting, FP64
//   [W | e] = M^-1 [G | c_d]   forward / backward substitution, blocked
//   T = G_od + (G_od diag(v)) W,  o = c_o + G_od (v .* e),  diag(W)
//
// The elimination of factor.cu is as accurate and twenty times as fast, but its
// W differs in the last bits.  The mixed search keeps the FP32 rounding of W: at
// N_d = 4096 a few of the 17 million entries then round the other way, and each
// moves what a search reports for its pixel by up to 2e-7.  High contrast:
// contrast_kernel in factor.cu.  Their results stay the same to the last bit
// this way.
//
// The trailing updates are complex GEMMs on the FP64 pipe (four DFMA per complex
// multiply-add, 1.25 TFLOP/s): N_d = 4096 697 ms, 1517 59, 1024 29, in
// one cooperative launch (747, 86 and 48 ms in a launch per step, with two grid
// barriers per panel column and a one-thread permutation).
#include <cstdio>

#include "factor_common.cuh"

namespace pngf {
namespace {

constexpr int FP_THREADS = 512, FP_WARPS = FP_THREADS / 32;
constexpr int GT = 64, GK = 16;  // product tile, K chunk
// rows of the panel (n_d <= 32768 on 152 SMs: 216 of 512 bytes), or the tile's operands
constexpr int FP_SMEM = 216 * NB * (int)sizeof(c128);
static_assert(FP_SMEM >= 2 * GK * GT * (int)sizeof(c128), "operands");

// C[M x N] -= A[M x K] B[K x N], K <= NB: 64 x 64 tiles over the grid, a thread
// owning rows ty + 16 r and columns tx, tx + 32
__device__ void pipe_gemm_sub(int M, int N, int K, const c128* A, const c128* B, c128* C, int ld, c128* sm) {
  c128(*As)[GT] = reinterpret_cast<c128(*)[GT]>(sm);
  c128(*Bs)[GT] = reinterpret_cast<c128(*)[GT]>(sm + GK * GT);
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, nM = (M + GT - 1) / GT, nN = (N + GT - 1) / GT;
  for (int t = blockIdx.x; t < nM * nN; t += gridDim.x) {
    const int m0 = t % nM * GT, n0 = t / nM * GT;
    c128 acc[4][2];
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r][0] = acc[r][1] = mk(0.0, 0.0);
    for (int k0 = 0; k0 < K; k0 += GK) {
      __syncthreads();
#pragma unroll
      for (int q = 0; q < GT * GK / FP_THREADS; ++q) {
        const int idx = threadIdx.x + q * FP_THREADS;
        int mm = idx >> 4, kk = idx & 15;
        As[kk][mm] = (m0 + mm < M && k0 + kk < K) ? A[(size_t)(m0 + mm) * ld + k0 + kk] : mk(0.0, 0.0);
        kk = idx >> 6;
        mm = idx & 63;
        Bs[kk][mm] = (k0 + kk < K && n0 + mm < N) ? B[(size_t)(k0 + kk) * ld + n0 + mm] : mk(0.0, 0.0);
      }
      __syncthreads();
#pragma unroll 4
      for (int kk = 0; kk < GK; ++kk) {
        const c128 b0 = Bs[kk][tx], b1 = Bs[kk][tx + 32];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const c128 x = As[kk][ty + 16 * r];
          acc[r][0] = cfma(x, b0, acc[r][0]);
          acc[r][1] = cfma(x, b1, acc[r][1]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int gm = m0 + ty + 16 * r, gn = n0 + tx + 32 * h;
        if (gm < M && gn < N) {
          c128* p = C + (size_t)gm * ld + gn;
          *p = csub(*p, acc[r][h]);
        }
      }
  }
}

__global__ void __launch_bounds__(FP_THREADS, 1) factor_pipe_kernel(const __grid_constant__ FactorArgs a) {
  extern __shared__ __align__(16) unsigned char p_smem[];
  if (a.high && !*a.high) return;
  __shared__ Swaps s_sw;
  c128* sm = reinterpret_cast<c128*>(p_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, P = gridDim.x, cta = blockIdx.x;
  const int gw = warp * P + cta, nw = P * FP_WARPS;  // neighbouring warps of the grid on different SMs
  const int n = a.n, ldw = a.ldw, ncol = n + 1;
  Control* ctl = a.ctl;
  bool ok = true;
  for (int i = cta; i < n; i += P) {
    const c128* g = a.G + (size_t)i * n;
    for (int j = tid; j < n; j += FP_THREADS) {
      const c128 vj = a.b_in[j] ? a.dv[j] : mk(0.0, 0.0), gij = g[j];
      c128 mij = mk(-(gij.x * vj.x - gij.y * vj.y), -(gij.x * vj.y + gij.y * vj.x));
      if (j == i) mij.x += 1.0;
      a.LU[(size_t)i * ldw + j] = mij;
    }
    if (tid == 0) {
      const bool on = a.b_in[i] != 0;
      a.v[i] = on ? a.dv[i] : mk(0.0, 0.0);
      a.b[i] = on ? 1 : 0;
      a.perm[i] = i;
    }
  }
  ok = grid_sync(ctl);
  auto load_L = [&](int j0, int jb) {  // the unit lower block, column-major
    __syncthreads();
    for (int q = tid; q < NB * NB; q += FP_THREADS) {
      const int k = q / NB, r = q % NB;
      sm[q] = (r < jb && k < r) ? a.LU[(size_t)(j0 + r) * ldw + j0 + k] : mk(0.0, 0.0);
    }
    __syncthreads();
  };
  for (int j0 = 0; ok && j0 < n; j0 += NB) {
    const int jb = min(NB, n - j0), i1 = j0 + jb;
    if (!(ok = factor_panel<FP_WARPS, true>(a, n, j0, jb, sm))) break;
    net_swaps(a, j0, jb, s_sw);
    load_L(j0, jb);
    swap_and_solve(a, s_sw, sm, n, j0, jb, gw, nw);
    if (!(ok = grid_sync(ctl))) break;
    if (i1 == n) continue;
    pipe_gemm_sub(n - i1, n - i1, jb, a.LU + (size_t)i1 * ldw + j0, a.LU + (size_t)j0 * ldw + i1,
                  a.LU + (size_t)i1 * ldw + i1, ldw, sm);
    ok = grid_sync(ctl);
  }
  // the pivoted right-hand sides
  if (ok) {
    for (int i = cta; i < n; i += P) {
      const int src = a.perm[i];
      for (int j = tid; j < n; j += FP_THREADS) a.W[(size_t)i * ldw + j] = a.G[(size_t)src * n + j];
      if (tid == 0) a.W[(size_t)i * ldw + n] = a.cd[src];
    }
    ok = grid_sync(ctl);
  }
  // forward substitution: two columns per warp, lane = row
  for (int i0 = 0; ok && i0 < n; i0 += NB) {
    const int jb = min(NB, n - i0), rest = n - i0 - jb;
    load_L(i0, jb);
    for (int u = gw; u < (ncol + 1) / 2; u += nw) {
      const bool two = 2 * u + 1 < ncol;
      c128* p = a.W + (size_t)(i0 + lane) * ldw + 2 * u;
      c128 x0 = lane < jb ? p[0] : mk(0.0, 0.0), x1 = lane < jb && two ? p[1] : mk(0.0, 0.0);
      for (int k = 0; k + 1 < jb; ++k) {
        const c128 l = sm[k * NB + lane];
        const c128 s0 = shfl_c(x0, k), s1 = shfl_c(x1, k);
        x0 = cfms(l, s0, x0);
        x1 = cfms(l, s1, x1);
      }
      if (lane < jb) {
        p[0] = x0;
        if (two) p[1] = x1;
      }
    }
    if (!(ok = grid_sync(ctl))) break;
    if (rest > 0) {
      pipe_gemm_sub(rest, ncol, jb, a.LU + (size_t)(i0 + jb) * ldw + i0, a.W + (size_t)i0 * ldw,
                    a.W + (size_t)(i0 + jb) * ldw, ldw, sm);
      ok = grid_sync(ctl);
    }
  }
  // backward substitution: one column per thread, each row summed from the diagonal outwards
  for (int i0 = (n - 1) / NB * NB; ok && i0 >= 0; i0 -= NB) {
    const int jb = min(NB, n - i0);
    __syncthreads();
    for (int q = tid; q < NB * NB; q += FP_THREADS) {
      const int r = q / NB, k = q % NB;
      sm[q] = (r < jb && k < jb) ? a.LU[(size_t)(i0 + r) * ldw + i0 + k] : mk(0.0, 0.0);
    }
    c128* di = sm + NB * NB;
    if (tid < NB) di[tid] = tid < jb ? a.dinv[i0 + tid] : mk(0.0, 0.0);
    __syncthreads();
    for (int u = gw; u < (ncol + 31) / 32; u += nw) {
      const int c = 32 * u + lane;
      if (c >= ncol) continue;
      c128 x[NB];
      for (int i = 0; i < jb; ++i) x[i] = a.W[(size_t)(i0 + i) * ldw + c];
      for (int i = jb - 1; i >= 0; --i) {
        c128 s = x[i];
        for (int l = i + 1; l < jb; ++l) s = cfms(sm[i * NB + l], x[l], s);
        x[i] = cmul(s, di[i]);
        a.W[(size_t)(i0 + i) * ldw + c] = x[i];
      }
    }
    if (!(ok = grid_sync(ctl))) break;
    if (i0 > 0) {
      pipe_gemm_sub(i0, ncol, jb, a.LU + i0, a.W + (size_t)i0 * ldw, a.W, ldw, sm);
      ok = grid_sync(ctl);
    }
  }
  if (!ok && tid == 0) latch_status(ctl, PNGF_ETIMEOUT);
}

// ---------------------------------------------------------------- state formation
// T[p][j] = G_od[p][j] + sum_i (G_od[p][i] v_i) W[i][j]; one thread per column j.
__global__ void __launch_bounds__(256) form_T(const c128* __restrict__ W, int n, int ldw,
                                              const c128* __restrict__ God, const c128* __restrict__ v,
                                              int n_o, c128* __restrict__ T, int ldt, const int* high) {
  if (high && !*high) return;
  __shared__ c128 gv[kMaxPorts][64];
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  c128 acc[kMaxPorts];
  for (int p = 0; p < kMaxPorts; ++p) acc[p] = mk(0.0, 0.0);
  for (int i0 = 0; i0 < n; i0 += 64) {
    __syncthreads();
    for (int idx = threadIdx.x; idx < n_o * 64; idx += blockDim.x) {
      int p = idx / 64, ii = idx % 64, i = i0 + ii;
      gv[p][ii] = (i < n) ? cmul(God[(size_t)p * n + i], v[i]) : mk(0.0, 0.0);
    }
    __syncthreads();
    if (j < n) {
      int iend = min(64, n - i0);
      for (int ii = 0; ii < iend; ++ii) {
        c128 w = W[(size_t)(i0 + ii) * ldw + j];
        FOR_PORTS(p, n_o) acc[p] = cfma(gv[p][ii], w, acc[p]);
      }
    }
  }
  if (j < n)
    FOR_PORTS(p, n_o) T[(size_t)p * ldt + j] = cadd(God[(size_t)p * n + j], acc[p]);
}

// diag(W), e = column n of the solved RHS
__global__ void extract_diag_e(const c128* __restrict__ W, int n, int ldw, c128* __restrict__ diag,
                               c128* __restrict__ e, const int* high) {
  if (high && !*high) return;
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) {
    diag[j] = W[(size_t)j * ldw + j];
    e[j] = W[(size_t)j * ldw + n];
  }
}

// S = Re G + Im G (n x n, row-major), the third real matrix of the refresh's
// three-multiplication complex products
__global__ void gsum_kernel(const c128* __restrict__ G, long long nn, double* __restrict__ S, const int* high) {
  if (high && !*high) return;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nn; i += (long long)gridDim.x * blockDim.x) {
    const c128 g = G[i];
    S[i] = g.x + g.y;
  }
}

// G as unevaluated sums of two FP32 values per real part, hi = fl32(g) and
// lo = fl32(g - hi) (48 significant bits), for the double-float refresh
// residual of the mixed search: (Re hi, Im hi, Re lo, Im lo), so that the
// (Re, Im) pairs of the hi and of the lo parts are 64-bit operands
__global__ void gsplit_kernel(const c128* __restrict__ G, long long nn, float4* __restrict__ G2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nn; i += (long long)gridDim.x * blockDim.x) {
    const c128 g = G[i];
    const float rh = (float)g.x, ih = (float)g.y;
    G2[i] = make_float4(rh, ih, (float)(g.x - (double)rh), (float)(g.y - (double)ih));
  }
}

__global__ void to_planar_fp32(const c128* __restrict__ W, int n, int ldw, float* __restrict__ Wr,
                               float* __restrict__ Wi, int ldl) {
  int i = blockIdx.y;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    c128 w = W[(size_t)i * ldw + j];
    Wr[(size_t)i * ldl + j] = (float)w.x;
    Wi[(size_t)i * ldl + j] = (float)w.y;
  }
}

}  // namespace

// everything but the ports (form_o); a.high: run only where the flag is set (nullptr: always)
pngf_status factor_pipe(pngf_ctx* c, const FactorArgs& args) {
  FactorArgs a = args;
  const int n = a.n;
  cudaStream_t s = c->stream;
  if (cudaFuncSetAttribute(factor_pipe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FP_SMEM) != cudaSuccess ||
      cudaMemsetAsync(&a.ctl->bar_count, 0, sizeof(unsigned), s) != cudaSuccess)
    return PNGF_ECUDA;
  int P = (n + 31) / 32;
  if (P > c->n_sm) P = c->n_sm;
  if (n > 512 && P < c->n_sm) P = c->n_sm;  // products of several tiles per SM
  void* params[] = {&a};
  if (cudaLaunchCooperativeKernel((const void*)factor_pipe_kernel, dim3(P), dim3(FP_THREADS), params, FP_SMEM, s) !=
      cudaSuccess)
    return PNGF_ECUDA;
  gsum_kernel<<<c->n_sm * 4, 256, 0, s>>>(a.G, (long long)n * n, a.Gs, a.high);
  extract_diag_e<<<(n + 255) / 256, 256, 0, s>>>(a.W, n, a.ldw, a.diag, a.e, a.high);
  form_T<<<(n + 255) / 256, 256, 0, s>>>(a.W, n, a.ldw, a.God, a.v, a.n_o, a.T, a.ldt, a.high);
  if (c->cfg.precision == PNGF_MIXED) {
    gsplit_kernel<<<c->n_sm * 4, 256, 0, s>>>(a.G, (long long)n * n, at<float4>(c, c->L.gsplit));
    dim3 grid((n + 255) / 256 > 8 ? 8 : (n + 255) / 256, n);
    to_planar_fp32<<<grid, 256, 0, s>>>(a.W, n, a.ldw, at<float>(c, c->L.Wlo_re), at<float>(c, c->L.Wlo_im), c->L.ldl);
  }
  return cuda_status(cudaGetLastError());
}

}  // namespace pngf
