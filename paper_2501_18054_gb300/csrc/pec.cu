// Direct binary search over perfect-conductor (PEC) pixels: the paper's own
// binary system, Eq. 2, [(I - P) + P G] j = P e_inc, in this code's sign of G
// (total field e = c_d + G j; on a metal pixel e = 0, on an empty one j = 0).
//
// For metal set M the solution is j_M = -(G_MM)^-1 c_M.  With
//   H = (G_MM)^-1 padded with zeros,  Q = G H,  W = G - G H G (zero on M),
//   R = G_od H,  T = G_od - G_od H G,  o = c_o + G_od j,
// adding pixel k is a rank-1 change with pivot W_kk and removing it one with
// pivot H_kk (Eqs. 9 and 14 for dP = +-e_k e_k^T).  W lives on the empty
// pixels, H on the metal ones and Q between them, so the three fit one complex
// symmetric matrix (the principal pivot transform of G on M),
//   S_jk = W_jk (both empty), H_jk (both metal), i Q_jk (j empty, k metal),
// and likewise one field u = e (empty), -i j (metal) and one set of port rows
// v = T (empty), i R (metal).  In these a flip of k in either direction is the
// same symmetric update as a flip of the field form,
//   alpha = -1 / S_kk,  c = S[:, k],
//   S += alpha c c^T,  u += alpha u_k c,  v += alpha v_k c^T,  o += alpha u_k v_k,
// and pixel k itself, now on the other side, restarts from
//   S_kj = +-i c_j / S_kk,  u_k, v_k times +-i / S_kk,  S_kk' = 1 / S_kk
// (+: metal put in).  So the delayed search kernel of the FP64 path runs it
// (delayed_search.cuh), one triangle instead of two and a full matrix.
//
// The initial state of a design is built from the empty design (S = G, u =
// c_d, v = G_od) by adding its metal pixels one by one (forced flips).
// N_d = 1024, start built and three sweeps: 54.1 ms with H, Q and W updated one
// flip at a time, 15.1 ms now (the chain of the search for each flip).
#include <cstdio>

#include "delayed_search.cuh"

namespace pngf {
namespace {

// the empty design's state: S = G (upper triangle), u = c_d, v = G_od, b = 0
__global__ void pec_empty_kernel(SweepArgs a) {
  const int n = a.n;
  for (int i = blockIdx.x; i < n; i += gridDim.x)
    for (int c = threadIdx.x; c < n; c += blockDim.x)
      a.W[(size_t)i * a.ldw + c] = c >= i ? a.G[(size_t)i * n + c] : mk(0.0, 0.0);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    a.diag[i] = a.G[(size_t)i * n + i];
    a.e[i] = a.cd[i];
    a.b[i] = 0;
    a.v[i] = mk(0.0, 0.0);
    for (int p = 0; p < a.n_o; ++p) a.T[(size_t)p * a.ldt + i] = a.God[(size_t)p * n + i];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    Control* ctl = a.ctl;
    FOR_PORTS(p, a.n_o) ctl->o[p] = a.co[p];
    ctl->f = objective_of(a.op, a.co);
    ctl->since_refresh = 0;
    ctl->n_acc_total = 0;
  }
}

// list of the metal pixels of design b (ascending), and its length
__global__ void pec_list_kernel(const uint8_t* __restrict__ b, int n, int* list, int* count) {
  __shared__ int s_base;
  if (threadIdx.x == 0) s_base = 0;
  __syncthreads();
  for (int i0 = 0; i0 < n; i0 += blockDim.x) {
    const int i = i0 + threadIdx.x;
    const int on = i < n && b[i] != 0;
    // block-wide exclusive scan of `on` in thread order (one block)
    __shared__ int s_cnt[1024];
    s_cnt[threadIdx.x] = on;
    __syncthreads();
    for (int off = 1; off < (int)blockDim.x; off <<= 1) {
      const int v = threadIdx.x >= (unsigned)off ? s_cnt[threadIdx.x - off] : 0;
      __syncthreads();
      s_cnt[threadIdx.x] += v;
      __syncthreads();
    }
    if (on) list[s_base + s_cnt[threadIdx.x] - 1] = i;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) s_base += s_cnt[threadIdx.x];
    __syncthreads();
  }
  if (threadIdx.x == 0) *count = s_base;
}

__global__ void pec_score_kernel(SweepArgs a, const int32_t* __restrict__ pixels, int m, double* __restrict__ f_new) {
  __shared__ ObjParams s_op;
  __shared__ c128 o[kMaxPorts];
  if (threadIdx.x == 0) {
    s_op = a.op;
    FOR_PORTS(p, a.n_o) o[p] = a.ctl->o[p];
  }
  __syncthreads();
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < m; q += gridDim.x * blockDim.x) {
    const int i = pixels[q];
    double fn = NAN;
    c128 al, co, idv;
    const bool ok = i >= 0 && i < a.n &&
                    score_pec(s_op, a.b[i] != 0, a.diag[i], a.e[i], [&](int p) { return a.T[(size_t)p * a.ldt + i]; }, o,
                              fn, al, co, idv);
    f_new[q] = ok ? fn : NAN;
  }
}

// what pngf_get_state gives: W, diag W, e and T, zero at metal pixels (any may be nullptr)
__global__ void pec_state_kernel(SweepArgs a, c128* W, c128* diag, c128* e, c128* T) {
  const int n = a.n;
  if (W)
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
      const bool mi = a.b[i] != 0;
      for (int c = threadIdx.x; c < n; c += blockDim.x)
        W[(size_t)i * n + c] = mi || a.b[c] ? mk(0.0, 0.0) : a.W[(size_t)i * a.ldw + c];
    }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const bool mi = a.b[i] != 0;
    if (diag) diag[i] = mi ? mk(0.0, 0.0) : a.diag[i];
    if (e) e[i] = mi ? mk(0.0, 0.0) : a.e[i];
    if (T)
      for (int p = 0; p < a.n_o; ++p) T[(size_t)p * n + i] = mi ? mk(0.0, 0.0) : a.T[(size_t)p * a.ldt + i];
  }
}

}  // namespace

pngf_status factor_pec(pngf_ctx* c, const uint8_t* b) {
  SweepArgs a = make_args(c);
  const int n = c->cfg.n_d;
  const int blocks = n < 4 * c->n_sm ? n : 4 * c->n_sm;
  pec_empty_kernel<<<blocks, 256, 0, c->stream>>>(a);
  int* list = at<int>(c, c->L.pos_of);  // scratch until the search sets it
  int* count = at<int>(c, c->L.actg);
  pec_list_kernel<<<1, 1024, 0, c->stream>>>(b, n, list, count);
  if (cudaGetLastError() != cudaSuccess) return PNGF_ECUDA;
  return launch_delayed<true>(c, DelayedArgs{a, list, count, -1}, delayed64_grid(c));
}

pngf_status run_sweep_pec(pngf_ctx* c, int n_sweeps, const int32_t* order, int32_t* trace, double* trace_f,
                          int32_t trace_cap, int64_t* counters) {
  SweepArgs a = make_args(c);
  a.n_sweeps = n_sweeps;
  a.order = order;
  a.trace = trace;
  a.trace_f = trace_f;
  a.trace_cap = trace_cap;
  a.counters = counters;
  return launch_delayed<true>(c, DelayedArgs{a, nullptr, nullptr, -1}, delayed64_grid(c));
}

pngf_status accept_flip_pec(pngf_ctx* c, int pixel) {
  return launch_delayed<true>(c, DelayedArgs{make_args(c), nullptr, nullptr, pixel}, delayed64_grid(c));
}

pngf_status score_flips_pec(pngf_ctx* c, const int32_t* pixels, int m, double* f_new) {
  if (m <= 0) return PNGF_OK;
  int blocks = (m + 255) / 256;
  if (blocks > 4 * c->n_sm) blocks = 4 * c->n_sm;
  pec_score_kernel<<<blocks, 256, 0, c->stream>>>(make_args(c), pixels, m, f_new);
  return cuda_status(cudaGetLastError());
}

pngf_status pec_state(pngf_ctx* c, double* W, double* diag, double* e, double* T) {
  const int n = c->cfg.n_d;
  pec_state_kernel<<<n < 4 * c->n_sm ? n : 4 * c->n_sm, 256, 0, c->stream>>>(
      make_args(c), reinterpret_cast<c128*>(W), reinterpret_cast<c128*>(diag), reinterpret_cast<c128*>(e),
      reinterpret_cast<c128*>(T));
  return cuda_status(cudaGetLastError());
}

}  // namespace pngf
