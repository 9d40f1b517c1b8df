// Last step of both factorisations: the ports and the objective of the design.
#pragma once

#include "sweep_common.cuh"

namespace pngf {
namespace {

// o = c_o + G_od (v .* e), objective, reset of the sweep counters.  One CTA.
__global__ void __launch_bounds__(256) form_o(const c128* __restrict__ God, const c128* __restrict__ co,
                                              const c128* __restrict__ v, const c128* __restrict__ e,
                                              int n, ObjParams op, Control* __restrict__ ctl) {
  __shared__ c128 red[kMaxPorts][256];
  c128 acc[kMaxPorts];
  for (int p = 0; p < kMaxPorts; ++p) acc[p] = mk(0.0, 0.0);
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    c128 ve = cmul(v[j], e[j]);
    FOR_PORTS(p, op.n_o) acc[p] = cfma(God[(size_t)p * n + j], ve, acc[p]);
  }
  FOR_PORTS(p, op.n_o) red[p][threadIdx.x] = acc[p];
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      FOR_PORTS(p, op.n_o) red[p][threadIdx.x] = cadd(red[p][threadIdx.x], red[p][threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    c128 o[kMaxPorts];
    FOR_PORTS(p, op.n_o) {
      o[p] = cadd(co[p], red[p][0]);
      ctl->o[p] = o[p];
    }
    ctl->f = objective_of(op, o);
    ctl->factored = 1;
    ctl->n_acc_total = 0;
    ctl->since_refresh = 0;
    ctl->r_delay = 0;
  }
}

}  // namespace
}  // namespace pngf
