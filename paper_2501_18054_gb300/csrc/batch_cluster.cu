// FP64 batch in sequential (FIRST) mode where the large runs are few: a cluster
// of kRunCtas CTAs advances one run at a time with the persistent search's own
// code (delayed_search.cuh; a run's result does not depend on how many CTAs
// share it).  One CTA per run (batch.cu) leaves SMs idle while the large runs
// last, each bound by the latency of its chain of flips: a 1024-pixel run
// takes 100 ms on one SM and 50 ms here (96 runs of 256, 576 and 1024 pixels:
// 109 -> 50 ms).
//
// In a file of its own: with this kernel and batch.cu's in one file the latter's
// folds lacked their product (nvcc 13.0.88; the cause is not known).  Each file has one kernel
// that calls the fold's out-of-line functions.
#include <cooperative_groups.h>
#include <algorithm>

#include "delayed_search.cuh"

namespace pngf {
namespace {

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

}  // namespace

// Clusters for a batch of n_runs, `large` of which have at least half the
// largest region's max_n pixels, or 0: one CTA per run.  Measured (ms, clusters
// against one CTA per run; n_d pixels, 4 / 38 / 76 equal runs of 10 sweeps, refresh
// every 64 kept flips):
//   1024: 60 / 109 / 170 against 172 / 198 / 209     100: 0.73 / 2.4 / 3.6 against 1.1 / 3.0 / 3.9
//    576: 16 / 31 / 49 against 41 / 51 / 52           64: 0.48 / 1.6 / 2.9 against 0.58 / 1.5 / 2.4
//    256: 2.4 / 6.2 / 10 against 4.6 / 9.3 / 10       16: 0.29 / 1.2 / 2.1 against 0.25 / 1.0 / 1.8
// so up to two rounds of clusters over the large runs, and from 96 pixels on.
// Every CTA holds a share of every run: at least one pixel, at most kOwn64.
int batch_clusters(int n_runs, int large, int min_n, int max_n, int n_sm) {
  if (large * kRunCtas > 2 * n_sm || max_n < 96 || max_n > kRunCtas * kOwn64 || min_n < kRunCtas) return 0;
  return std::min(n_runs, n_sm / kRunCtas);
}

pngf_status launch_batch_clusters(const void* runs, int n_runs, int* queue, int max_n, int max_o, int clusters,
                                  cudaStream_t stream) {
  if (cudaFuncSetAttribute(dbs_batch_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kDelayed64MaxSmem) != cudaSuccess)
    return PNGF_ECUDA;
  dbs_batch_cluster_kernel<<<clusters * kRunCtas, OZ_THREADS, delayed64_smem(max_o, own64_stride(max_n, kRunCtas)),
                             stream>>>(static_cast<const SweepArgs*>(runs), n_runs, queue);
  return cuda_status(cudaGetLastError());
}

}  // namespace pngf
