// Launches of the CPML layer's passes (cpml.cuh): the unrolled line ends where
// they apply, the line walks on the other axes, and the shell receivers, for
// one grid and batched over the shot server's resident shots.
#include "layer_lines.cuh"

using namespace gbw;

namespace {

template <int AX, class T, bool kD>
void walk(const CpmlPlan &p, const CpmlPass &a, cudaStream_t st) {
  const int inner = AX == 0 ? p.g.ny : p.g.nx, outer = AX == 2 ? p.g.ny : p.g.nz;
  cpml_line_kernel<AX, T, kD><<<dim3((inner + 127) / 128, outer), 128, 0, st>>>(
      p.g, static_cast<const T *>(a.u), static_cast<T *>(a.unext), a.c, a.dout, a.d, a.koff);
}

template <int AX>
void walk_adjoint(const CpmlPlan &p, const CpmlPass &a, cudaStream_t st) {
  const int inner = AX == 0 ? p.g.ny : p.g.nx, outer = AX == 2 ? p.g.ny : p.g.nz;
  cpml_adjoint_line_kernel<AX><<<dim3((inner + 127) / 128, outer), 128, 0, st>>>(
      p.g, static_cast<const float *>(a.u), static_cast<float *>(a.unext), a.c, a.nus[AX],
      a.mus[AX]);
}

template <class T>
void record(const CpmlPlan &p, const CpmlPass &a, int sms, cudaStream_t st) {
  cpml_record_kernel<T><<<sms, 256, 0, st>>>(p.g, static_cast<const T *>(a.unext), a.d, a.srec,
                                             a.nsrec, a.koff);
}

template <class T, bool kD>
void forward(const CpmlPlan &p, const CpmlPass &a, int sms, cudaStream_t st) {
  const bool all = p.axes == 7 && !p.by_axis;
  if (all) cpml_launch_lines<T, kD>(p, p.all, a, true, st);
  for (int ax = 0; ax < 3 && !all; ++ax) {
    if ((p.axes >> ax) & 1)
      cpml_launch_lines<T, kD>(p, p.one[ax], a, p.axes == 7 && ax == 0, st);
    else if (ax == 0)
      walk<0, T, kD>(p, a, st);
    else if (ax == 1)
      walk<1, T, kD>(p, a, st);
    else
      walk<2, T, kD>(p, a, st);
  }
  if (!kD && p.axes != 7) record<T>(p, a, sms, st);
}

template <int AX, class T>
__global__ void __launch_bounds__(kCpmlThreads)
    walk_batched_kernel(const CpmlBatchShot *__restrict__ shots, int nshots, long long k) {
  const CpmlBatchShot &sh = shots[cpml_batch_find(shots, nshots, 3 + AX, blockIdx.x)];
  CpmlPass a;
  if (!cpml_batch_pass(sh, k, a)) return;
  const CpmlGeom &g = sh.plan.g;
  const int local = blockIdx.x - sh.blk_begin[3 + AX];
  const int across = AX == 0 ? g.ny : g.nx;
  const int bpr = (across + kCpmlThreads - 1) / kCpmlThreads;  // blocks per row of lines
  const int q = local / bpr;
  cpml_line_walk<AX, T, false>(g, (local - q * bpr) * kCpmlThreads + threadIdx.x, q,
                               static_cast<const T *>(a.u), static_cast<T *>(a.unext), a.c,
                               nullptr, a.d, a.koff);
}

// Shell receivers of batch step k: blocks_per_shot blocks per shot (a
// receiver plane inside the layer puts all of a shot's receivers here).
template <class T>
__global__ void record_batched_kernel(const CpmlBatchShot *__restrict__ shots, long long k,
                                      int blocks_per_shot) {
  const CpmlBatchShot &sh = shots[blockIdx.x / blocks_per_shot];
  CpmlPass a;
  if (sh.nsrec == 0 || !cpml_batch_pass(sh, k, a)) return;
  CpmlScale<T> sc;
  sc.init(a.d, a.koff);
  const T *un = static_cast<const T *>(a.unext);
  for (int r = blockIdx.x % blocks_per_shot * blockDim.x + threadIdx.x; r < sh.nsrec;
       r += blocks_per_shot * blockDim.x) {
    const int4 e = sh.srec[r];
    a.d->traces[(size_t)(a.d->n + a.koff) * a.d->nrec + e.w] =
        cpml_get(un + ((size_t)e.z * sh.plan.g.ny + e.y) * sh.plan.g.pxu + e.x, sc.so);
  }
}

template <class T>
void step(int group, const CpmlBatchShot *shots, int n, const int blocks[6], int rec_blocks,
          long long k, cudaStream_t st) {
  if (group < kCpmlVariants) {
    cpml_launch_batched_lines<T>(group, -1, shots, n, blocks[0], k, st);
  } else {
    for (int ax = 0; ax < 3; ++ax) {
      const int b = blocks[3 + ax];
      if (blocks[ax] > 0)
        cpml_launch_batched_lines<T>(group - kCpmlVariants, ax, shots, n, blocks[ax], k, st);
      if (b > 0 && ax == 0) walk_batched_kernel<0, T><<<b, kCpmlThreads, 0, st>>>(shots, n, k);
      if (b > 0 && ax == 1) walk_batched_kernel<1, T><<<b, kCpmlThreads, 0, st>>>(shots, n, k);
      if (b > 0 && ax == 2) walk_batched_kernel<2, T><<<b, kCpmlThreads, 0, st>>>(shots, n, k);
    }
  }
  record_batched_kernel<T><<<n * rec_blocks, 128, 0, st>>>(shots, k, rec_blocks);
}

}  // namespace

namespace gbw {

void cpml_forward(int storage, bool store_d, const CpmlPlan &p, const CpmlPass &a, int sms,
                  cudaStream_t st) {
  if (storage == WAVE_STORAGE_BF16)
    forward<__nv_bfloat16, false>(p, a, sms, st);
  else if (storage == WAVE_STORAGE_F16)
    forward<__half, false>(p, a, sms, st);
  else if (store_d)
    forward<float, true>(p, a, sms, st);
  else
    forward<float, false>(p, a, sms, st);
}

void cpml_record_last(int storage, const CpmlPlan &p, const CpmlPass &a, int sms,
                      cudaStream_t st) {
  if (p.axes != 7) return;
  if (storage == WAVE_STORAGE_BF16)
    record<__nv_bfloat16>(p, a, sms, st);
  else if (storage == WAVE_STORAGE_F16)
    record<__half>(p, a, sms, st);
  else
    record<float>(p, a, sms, st);
}

void cpml_adjoint(const CpmlPlan &p, const CpmlPass &a, cudaStream_t st) {
  const bool all = p.axes == 7 && !p.by_axis;
  if (all) cpml_launch_adjoint_lines(p, p.all, a, st);
  for (int ax = 0; ax < 3 && !all; ++ax) {
    if ((p.axes >> ax) & 1)
      cpml_launch_adjoint_lines(p, p.one[ax], a, st);
    else if (ax == 0)
      walk_adjoint<0>(p, a, st);
    else if (ax == 1)
      walk_adjoint<1>(p, a, st);
    else
      walk_adjoint<2>(p, a, st);
  }
}

int cpml_batch_blocks(const CpmlBatchShot &s, int which, bool by_axis) {
  const CpmlPlan &p = s.plan;
  const int ax = which % 3;
  if (p.axes == 7 && !by_axis) return which == 0 ? p.all.start[7] * kCpmlCluster : 0;
  if ((p.axes >> ax) & 1) return which < 3 ? p.one[ax].start[7] * kCpmlCluster : 0;
  if (which < 3) return 0;
  const int across = ax == 0 ? p.g.ny : p.g.nx, rows = ax == 2 ? p.g.ny : p.g.nz;
  return rows * ((across + kCpmlThreads - 1) / kCpmlThreads);
}

void cpml_batch_step(int storage, int group, const CpmlBatchShot *shots, int n,
                     const int blocks[6], int rec_blocks, long long k, cudaStream_t st) {
  if (storage == WAVE_STORAGE_BF16)
    step<__nv_bfloat16>(group, shots, n, blocks, rec_blocks, k, st);
  else if (storage == WAVE_STORAGE_F16)
    step<__half>(group, shots, n, blocks, rec_blocks, k, st);
  else
    step<float>(group, shots, n, blocks, rec_blocks, k, st);
}

}  // namespace gbw
