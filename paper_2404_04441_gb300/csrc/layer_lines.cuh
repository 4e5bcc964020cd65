// The unrolled line ends of the CPML layer (cpml.cuh) for one storage type:
// for one grid, and batched over the shot server's resident shots.
#pragma once

#include "cpml.cuh"

namespace gbw {

// The shot of a batched launch's block: the last whose first block is not
// past it.
__device__ __forceinline__ int cpml_batch_find(const CpmlBatchShot *shots, int nshots, int which,
                                               int blk) {
  int lo = 0, hi = nshots - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (shots[mid].blk_begin[which] <= blk) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// The pass of batch step k of a shot; false outside its steps.
__device__ __forceinline__ bool cpml_batch_pass(const CpmlBatchShot &sh, long long k,
                                                CpmlPass &a) {
  const long long n = k - sh.b0;
  if (n < 0 || n >= sh.nsteps) return false;
  const int cur = (int)(n & 1);
  a.u = sh.buf[cur];
  a.unext = sh.buf[cur ^ 1];
  a.c = sh.c;
  a.dout = nullptr;
  a.d = sh.desc;
  a.koff = (int)n;
  return true;
}

// Every axis's lines of the shots of a group (ax < 0), or one axis's. The
// shot's profile is staged in shared memory (read with immediate offsets where
// the single-grid kernel takes it from its parameters). A cluster's CTAs
// belong to one shot: its first block is a multiple of the cluster.
template <class OP>
__global__ void __launch_bounds__(kCpmlThreads, cpml_ctas(OP::NPML))
    cpml_lines_batched_kernel(const CpmlBatchShot *__restrict__ shots, int nshots, long long k,
                              int ax) {
  const int which = ax < 0 ? 0 : ax;
  const CpmlBatchShot &sh = shots[cpml_batch_find(shots, nshots, which, blockIdx.x)];
  CpmlPass a;
  if (!cpml_batch_pass(sh, k, a)) return;
  __shared__ CpmlProf<OP::NPML> pf;
  for (int i = threadIdx.x; i < 6 * OP::NPML; i += kCpmlThreads) {
    const int j = i % OP::NPML, f = i / OP::NPML;
    pf.b[f >> 1][f & 1][j] = sh.plan.prof.b[f >> 1][f & 1][j];
    pf.a[f >> 1][f & 1][j] = sh.plan.prof.a[f >> 1][f & 1][j];
  }
  __syncthreads();
  cpml_lines<OP>(sh.plan.g, ax < 0 ? sh.plan.all : sh.plan.one[ax], pf, a,
                 (int)(blockIdx.x - sh.blk_begin[which]) / kCpmlCluster);
}

// Launch of `blocks` CTAs, in clusters where several axes' lines meet (one
// axis's lines need no barrier).
template <class K, class... Args>
void cpml_launch_grid(K kernel, int blocks, bool clusters, cudaStream_t st, const Args &...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(kCpmlThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kCpmlCluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = clusters ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <class OP>
void cpml_launch(const CpmlPlan &p, const CpmlTiles &t, const CpmlPass &a, bool record,
                 cudaStream_t st) {
  CpmlProf<OP::NPML> pf;
  for (int f = 0; f < 6; ++f)
    for (int j = 0; j < OP::NPML; ++j) {
      pf.b[f >> 1][f & 1][j] = p.prof.b[f >> 1][f & 1][j];
      pf.a[f >> 1][f & 1][j] = p.prof.a[f >> 1][f & 1][j];
    }
  const int clusters = t.start[7] + (OP::kRecords && record ? kCpmlRecClusters : 0);
  cpml_launch_grid(cpml_lines_kernel<OP>, clusters * kCpmlCluster, t.all, st, p.g, t, pf, a);
}

template <class T, bool kStoreD>
void cpml_launch_lines(const CpmlPlan &p, const CpmlTiles &t, const CpmlPass &a, bool record,
                       cudaStream_t st) {
  switch (p.variant) {
    case 0: return cpml_launch<CpmlForward<8, T, kStoreD>>(p, t, a, record, st);
    case 1: return cpml_launch<CpmlForward<10, T, kStoreD>>(p, t, a, record, st);
    case 2: return cpml_launch<CpmlForward<16, T, kStoreD>>(p, t, a, record, st);
    default: return cpml_launch<CpmlForward<20, T, kStoreD>>(p, t, a, record, st);
  }
}

template <class T>
void cpml_launch_batched_lines(int variant, int ax, const CpmlBatchShot *shots, int n, int blocks,
                               long long k, cudaStream_t st) {
  switch (variant) {
    case 0:
      cpml_launch_grid(cpml_lines_batched_kernel<CpmlForward<8, T, false>>, blocks, ax < 0, st,
                       shots, n, k, ax);
      return;
    case 1:
      cpml_launch_grid(cpml_lines_batched_kernel<CpmlForward<10, T, false>>, blocks, ax < 0, st,
                       shots, n, k, ax);
      return;
    case 2:
      cpml_launch_grid(cpml_lines_batched_kernel<CpmlForward<16, T, false>>, blocks, ax < 0, st,
                       shots, n, k, ax);
      return;
    default:
      cpml_launch_grid(cpml_lines_batched_kernel<CpmlForward<20, T, false>>, blocks, ax < 0, st,
                       shots, n, k, ax);
  }
}

}  // namespace gbw
