// stage.cu - the end of a residual or Runge-Kutta stage whose direction passes ran as one launch
// (each into its own accumulator): the sum of the directions' residuals, in the order of the passes, scaled into
// dQ/dt or applied as the stage update.  The same operations as the last pass's own epilogue.
#include <cuda_runtime.h>

#include "sweep.cuh"

namespace fpk {

namespace {

// Bound by memory latency at these sizes (a few hundred thousand points, all in L2): one point per
// thread, all its loads in flight at once.
template <typename T>
__global__ void __launch_bounds__(256) k_finish(const BlockDev *__restrict__ blk, unsigned ncells, int ni, int nj,
                                                int dims, int rk, int stage, const double *__restrict__ dtp) {
  const unsigned idx = blockIdx.x * 256u + threadIdx.x;
  const unsigned i = idx % ni, r = idx / ni, j = r % nj, k = r / nj, qc = blk->qc;
  const DirDev *D = &blk->dir[0];      // lines along i: its transverse strides are those of j and k
  const T *kj = static_cast<const T *>(D->kj);
  const unsigned mo = blk->moff + i + j * D->mT1 + k * D->mT2;
  const bool in = idx < ncells;
  const T Jc = in ? Num<T>::rcp(*FPK_IN(kj + (4ULL * mo + 3), kj, 4LL * blk->mc, blk->status)) : T(0);
  chain_wait();
  chain_next();
  if (!in) return;
  T acc[3][5], R[5], qk[5], qn[5];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (d >= dims) continue;
    const T *a = static_cast<const T *>(blk->dir[d].racc);
    load4(FPK_IN(a + 4ULL * idx, a, 4LL * qc - 3, blk->status), acc[d]);
    acc[d][4] = *FPK_IN(comp_at(a, idx, qc, 4), a, 5LL * qc, blk->status);
  }
  const T *const q0 = static_cast<const T *>(blk->q[0]), *const qi = static_cast<const T *>(blk->q[stage]);
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    R[v] = acc[0][v] + acc[1][v];
    if (dims == 3) R[v] += acc[2][v];
    if (rk) qk[v] = *FPK_IN(qi + state_at(stage, idx, qc, v), qi, 5LL * qc, blk->status);
    qn[v] = rk && stage ? *FPK_IN(comp_at(q0, idx, qc, v), q0, 5LL * qc, blk->status) : T(0);
  }
  if (!rk) {
    T *const out = static_cast<T *>(blk->dqdt);
#pragma unroll
    for (int v = 0; v < 5; ++v) *FPK_IN(comp_at(out, idx, qc, v), out, 5LL * qc, blk->status) = -Jc * R[v];
    return;
  }
  const RkStage<T> update(stage, T(*dtp));
  T *qs = static_cast<T *>(blk->q[(stage + 1) % 3]);
  bool bad = false;
  T nv[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    nv[v] = update(qk[v], qn + v, -Jc * R[v]);
    bad |= !isfinite(nv[v]);
  }
  if (stage < 2) {
    store4(FPK_IN(qs + 4ULL * idx, qs, 4LL * qc - 3, blk->status), nv);
  } else {
#pragma unroll
    for (int v = 0; v < 4; ++v) *FPK_IN(comp_at(qs, idx, qc, v), qs, 5LL * qc, blk->status) = nv[v];
  }
  *FPK_IN(comp_at(qs, idx, qc, 4), qs, 5LL * qc, blk->status) = nv[4];
  if (bad) atomicOr(blk->status, ST_NONFINITE);
}

}  // namespace

cudaError_t launch_finish(const BlockDev *blk, int is_f32, long long ncells, const int *n, int dims, int rk,
                          int stage, const double *dt, cudaStream_t s) {
  const int grid = (int)((ncells + 255) / 256);
  // FP64 not chained: its early CTAs disturb the even placement of the sweep's (a 128^2 linear-upwind
  // step 226 us chained, 205 us not)
  return is_f32 ? launch_kernel(k_finish<float>, grid, 256, 0, s, 1, blk, (unsigned)ncells, n[0], n[1], dims, rk, stage, dt)
                : launch_kernel(k_finish<double>, grid, 256, 0, s, 0, blk, (unsigned)ncells, n[0], n[1], dims, rk, stage, dt);
}

}  // namespace fpk
