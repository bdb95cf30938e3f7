// cfl.cu - time-step bound: max over points of sum_d (|u . grad d| + c |grad d|),
// grad d = J (d_x, d_y, d_z)/J, reduced to one value per launch; the global Lax-Friedrichs
// speeds; and the packing of the cells a neighbouring process needs as its halo.
#include <cuda_runtime.h>
#include <math.h>

#include "sweep.cuh"

namespace fpk {

namespace {

// sum_d (|u . grad d| + c |grad d|) of one point in FP64, as |J| (sum_d |u . k_d| + c sum_d |k_d|)
template <typename T>
__device__ double cfl_point(const BlockDev *blk, const T *q, long long idx, long long mo, int dims) {
  const long long qc = blk->qc;
  const double g = blk->gamma;
  auto val = [&](int c) { return (double)*FPK_IN(q + (c * qc + idx), q, 5 * qc, blk->status); };
  const double rho = val(0);
  const double u = val(1) / rho, v = val(2) / rho, w = val(3) / rho;
  const double p = (g - 1.0) * (val(4) - 0.5 * rho * (u * u + v * v + w * w));
  const double c = sqrt(g * p / rho);
  double Jc = 0.0, U = 0.0, K = 0.0;
  for (int d = 0; d < dims; ++d) {
    const T *kj = static_cast<const T *>(blk->dir[d].kj);
    T k[4];
    load4(FPK_IN(kj + 4 * mo, kj, 4LL * blk->mc - 3, blk->status), k);
    if (d == 0) Jc = 1.0 / (double)k[3];
    const double kx = (double)k[0], ky = (double)k[1], kz = (double)k[2];
    U += fabs(u * kx + v * ky + w * kz);
    K += sqrt(kx * kx + ky * ky + kz * kz);
  }
  return fabs(Jc) * (U + c * K);
}

// x rounded towards zero to FP32 (relative error below 2^-23; 0 below 2^-126, infinity from 2^128 on
// and for a NaN) by integer operations: a conversion takes the FP64 pipe as long as an addition, and
// a point's 17 took the FP64 screen 26 us on 1.05M points
__device__ __forceinline__ float screen_value(float x) { return x; }
__device__ __forceinline__ float screen_value(double x) {
  const unsigned hi = __double2hiint(x), m = hi & 0x7fffffffu;
  const unsigned bits = __funnelshift_l((unsigned)__double2loint(x), m, 3) - (896u << 23);
  const unsigned mag = m < (897u << 20) ? 0u : (m >= (1151u << 20) ? 0x7f800000u : bits);
  return __uint_as_float(mag | (hi & 0x80000000u));
}

constexpr int kCflThreads = 256, kCflPoints = 4;   // points per thread

// The maximum of cfl_point over a block.  The FP64 pipe does two operations per clock and SM, and
// a point's four quotients and four roots cost about 120 (1.05M points: 220 us, 20 times their
// memory time), so every point is first enclosed in FP32 bounds.  k_cfl_bound keeps the largest
// lower bound of the block and each CTA's largest and smallest upper bound; k_cfl_max evaluates in
// FP64 the points whose upper bound reaches the former, so the result is the FP64 maximum.  (One
// kernel whose CTAs knew only their own lower bound evaluated a point in every CTA: 39 us.)  The
// bounds' relative width 4e-6 is more than three times the error of the FP32 evaluation (inputs to
// 2^-23, the approximate reciprocal and root 2^-23 each, at most 12 operations deep: 1.2e-6);
// cancellation in the pressure and in u . grad d is covered by adding that width of the summed
// magnitudes.  Points with an input, a squared sound speed or a sum outside [1e-30, 1e30], where a
// product could leave the FP32 range (p/rho of a dense cold gas rounds to zero), and anything not
// finite have the upper bound +inf.
// Measured, a call on 128 x 128 x 64 points (one FP64 kernel over all points | the screen): a smooth
// flow 268 | 46 us in FP32, 242 | 65 us in FP64.  Where every point ties (a uniform stream on a
// uniform grid) the screen rejects nothing and its pass comes on top: 292 | 294 us in FP32, 267 |
// 281 us in FP64.  So a tie is kept cheap: CTAs all of whose points pass do not look at the bounds
// again (26 us), and each CTA does one atomic (one per thread: 25 to 70 us).
template <typename T> struct CflScreen {
  const BlockDev *blk;
  const T *q;
  long long qc;
  int ni, nj, dims;
  float g1, gam;
  __device__ CflScreen(const BlockDev *b, int ni_, int nj_, int dims_)
      : blk(b), q(static_cast<const T *>(b->q[0])), qc(b->qc), ni(ni_), nj(nj_), dims(dims_), g1((float)(b->gamma - 1.0)), gam((float)b->gamma) {}
  __device__ long long place(long long idx) const {
    // (a block has fewer than 2^31 points)
    const unsigned r = (unsigned)idx / (unsigned)ni, i = (unsigned)idx - r * ni;
    const unsigned k = r / (unsigned)nj, j = r - k * nj;
    // lines of the xi direction run along i; their transverse strides are those of j and k
    return blk->moff + i + (long long)j * blk->dir[0].mT1 + (dims == 3 ? (long long)k * blk->dir[0].mT2 : 0);
  }
  // upper bound of the point, and its lower bound (0 if it has none)
  __device__ float bound(long long idx, long long mo, float &lo) const {
    constexpr float kW = 4e-6f, kLow = 1e-30f, kHigh = 1e30f;
    float Q[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) Q[v] = screen_value(*FPK_IN(q + (v * qc + idx), q, 5 * qc, blk->status));
    // the point's metric vectors and 1/J, the values of one direction side by side
    auto metric = [&](int d, T k[4]) {
      const T *kj = static_cast<const T *>(blk->dir[d].kj);
      load4(FPK_IN(kj + 4 * mo, kj, 4LL * blk->mc - 3, blk->status), k);
    };
    T kj[4];
    metric(0, kj);
    const float ij = fabsf(screen_value(kj[3]));
    bool ok = Q[0] > kLow && Q[0] < kHigh && Q[4] > kLow && Q[4] < kHigh && ij > kLow && ij < kHigh;
    const float ri = Num<float>::rcp(Q[0]), Jc = Num<float>::rcp(ij);
    const float u = Q[1] * ri, v = Q[2] * ri, w = Q[3] * ri;
    const float ke = 0.5f * (Q[1] * u + Q[2] * v + Q[3] * w);
    const float e = Q[4] - ke, de = kW * (Q[4] + ke);
    const float c2 = gam * g1 * fmaxf(e + de, 0.f) * ri;
    ok = ok && c2 > kLow;
    const float chi = Num<float>::sqrt_(c2), clo = Num<float>::sqrt_(gam * g1 * fmaxf(e - de, 0.f) * ri);
    float sh = 0.f, sl = 0.f;
    for (int d = 0; d < dims; ++d) {
      if (d) metric(d, kj);
      const float kx = screen_value(kj[0]), ky = screen_value(kj[1]), kz = screen_value(kj[2]);
      const float k2 = kx * kx + ky * ky + kz * kz, kn = Num<float>::sqrt_(k2);
      ok = ok && k2 > kLow && k2 < kHigh;
      const float U = fabsf(u * kx + v * ky + w * kz);
      const float dU = kW * (fabsf(u * kx) + fabsf(v * ky) + fabsf(w * kz));
      sh += U + dU + chi * kn;
      sl += U - dU + clo * kn;
    }
    sh *= Jc * (1.f + kW);
    sl *= Jc * (1.f - kW);
    ok = ok && sh > kLow && sh < kHigh;             // false for NaN as well
    lo = ok && e > de ? sl : 0.f;                   // a negative pressure has no value (NaN, ignored)
    return ok ? sh : __int_as_float(0x7f800000);
  }
};

// Blocks of at most one such CTA per SM: every point in FP64 by k_cfl_max alone, one per thread.  A
// second kernel costs 2 to 5 us there, more than the screen saves (us a call, one kernel | two:
// 4,320 points 30.6 | 34.5, 32,768 30.6 | 34.7, 65,120 42.6 | 34.3).
constexpr long long kCflSmall = 152 * kCflThreads;

template <typename T>
__global__ void __launch_bounds__(kCflThreads) k_cfl_bound(const BlockDev *blk, long long ncells, int ni, int nj, int dims,
                                                           CflScratch *out, float2 *cta_hi) {
  __shared__ float red[3][kCflThreads / 32];
  const CflScreen<T> screen(blk, ni, nj, dims);
  const long long base = (long long)blockIdx.x * (kCflThreads * kCflPoints) + threadIdx.x;
  float hi = -1.f, lo = 0.f, least = __int_as_float(0x7f800000);
#pragma unroll
  for (int m = 0; m < kCflPoints; ++m) {
    const long long idx = base + m * kCflThreads;
    if (idx >= ncells) continue;
    float l;
    const float h = screen.bound(idx, screen.place(idx), l);
    hi = fmaxf(hi, h);
    least = fminf(least, h);
    lo = fmaxf(lo, l);
  }
  for (int h = 16; h; h >>= 1) {
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, h));
    lo = fmaxf(lo, __shfl_xor_sync(0xffffffffu, lo, h));
    least = fminf(least, __shfl_xor_sync(0xffffffffu, least, h));
  }
  if (threadIdx.x % 32 == 0) {
    red[0][threadIdx.x / 32] = hi;
    red[1][threadIdx.x / 32] = lo;
    red[2][threadIdx.x / 32] = least;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kCflThreads / 32; ++w) {
      hi = fmaxf(hi, red[0][w]);
      lo = fmaxf(lo, red[1][w]);
      least = fminf(least, red[2][w]);
    }
    cta_hi[blockIdx.x] = make_float2(hi, least);
    atomicMax(&out->lower_bits, __float_as_uint(lo));
  }
  chain_next();
}

template <typename T>
__global__ void __launch_bounds__(kCflThreads) k_cfl_max(const BlockDev *blk, long long ncells, int ni, int nj, int dims,
                                                         CflScratch *out, const float2 *cta_hi) {
  __shared__ long long red[kCflThreads / 32];
  chain_wait();
  float lo = 0.f;
  bool all = true;                                  // every point of the CTA, without another look
  if (cta_hi) {
    lo = __uint_as_float(*(volatile unsigned int *)&out->lower_bits);
    const float2 hi = cta_hi[blockIdx.x];
    if (hi.x < lo) return;
    all = hi.y >= lo;
  }
  const CflScreen<T> screen(blk, ni, nj, dims);
  const int points = cta_hi ? kCflPoints : 1;       // of a thread
  long long best = 0;                               // bits: non-negative doubles are ordered like them
  for (int m = 0; m < points; ++m) {
    const long long idx = (long long)blockIdx.x * (kCflThreads * points) + m * kCflThreads + threadIdx.x;
    if (idx >= ncells) break;
    const long long mo = screen.place(idx);
    float l;
    if (!all && screen.bound(idx, mo, l) < lo) continue;
    const long long s = __double_as_longlong(cfl_point(blk, screen.q, idx, mo, dims));
    if (s > best && s <= 0x7ff0000000000000LL) best = s;   // (a NaN is ignored)
  }
  for (int h = 16; h; h >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, h));
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kCflThreads / 32; ++w) best = max(best, red[w]);
    if (best > 0) atomicMax(&out->max_bits, (unsigned long long)best);
  }
}

template <typename T>
__global__ void k_lam_zero(const BlockDev *blocks, int nblocks) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < nblocks) {
    T *l = static_cast<T *>(blocks[b].lamg);
    for (int t = 0; t < 9; ++t) l[t] = T(0);
  }
}

__device__ __forceinline__ void atomic_max_nonneg(float *a, float v) {
  atomicMax(reinterpret_cast<unsigned int *>(a), __float_as_uint(v));
}
__device__ __forceinline__ void atomic_max_nonneg(double *a, double v) {
  atomicMax(reinterpret_cast<unsigned long long *>(a), (unsigned long long)__double_as_longlong(v));
}

// 1/x, in FP64 with a quarter of the operations of a quotient
__device__ __forceinline__ float reciprocal(float x) { return 1.0f / x; }
__device__ __forceinline__ double reciprocal(double x) { return Num<double>::rcp(x); }

// sqrt(a b) by correctly rounded roots, two in FP32 and one in FP64 (as Num::sqrt_product)
__device__ __forceinline__ float sqrt_product(float a, float b) { return sqrtf(a) * sqrtf(b); }
__device__ __forceinline__ double sqrt_product(double a, double b) { return sqrt(a * b); }

// Max over each block's points of |U - c|grad d||, |U|, |U + c|grad d|| for every direction.  A CTA
// takes a contiguous range of the items (kLamChunk points each), keeps its maxima in registers
// while the block stays the same, and then reduces them by warp and adds them to the block's.
// One point per thread and item, so that small blocks spread over the chip: 200^2 points in FP64
// (whose divisions and roots run on the two-lane FP64 pipe) took 230 us in five items of 8192
// (an RK3 step there 2008 -> 1168 us with one point per thread).
template <typename T>
__global__ void k_lam_max(const BlockDev *blocks, const int2 *items, int nitems, int charwise, int stage) {
  __shared__ T red[9][kLamChunk / 32];
  const int it0 = (int)((long long)nitems * blockIdx.x / gridDim.x);
  const int it1 = (int)((long long)nitems * (blockIdx.x + 1) / gridDim.x);
  T best[9];
  for (int t = 0; t < 9; ++t) best[t] = T(0);
  for (int it = it0; it < it1; ++it) {
    const int2 item = items[it];
    const BlockDev *B = blocks + item.x;
    const int dims = B->dims, ni = B->dir[0].nd, nj = B->dir[1].nd;
    const long long qc = B->qc;
    const T *q = static_cast<const T *>(B->q[stage]);
    const T g = T(B->gamma);
    const long long idx = (long long)item.y + threadIdx.x;
    if (idx < qc) {
      const int i = (int)(idx % ni);
      const long long r = idx / ni;
      const int j = (int)(r % nj);
      const int k = (int)(r / nj);
      const long long mo = B->moff + i + (long long)j * B->dir[0].mT1 + (dims == 3 ? (long long)k * B->dir[0].mT2 : 0);
      auto val = [&](int c) { return *FPK_IN(q + state_at(stage, idx, qc, c), q, 5 * qc, B->status); };
      const T rho = val(0), rinv = reciprocal(rho);
      const T u = val(1) * rinv, v = val(2) * rinv, w = val(3) * rinv;
      const T p = (g - T(1)) * (val(4) - T(0.5) * rho * (u * u + v * v + w * w));
      const T c2 = g * p * rinv;
      auto metric = [&](int d, T k[4]) {
        const T *kj = static_cast<const T *>(B->dir[d].kj);
        load4(FPK_IN(kj + 4 * mo, kj, 4LL * B->mc - 3, B->status), k);
      };
      T kj[4];
      metric(0, kj);
      const T Jc = reciprocal(kj[3]);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (d >= dims) continue;
        if (d) metric(d, kj);
        // grad d = J k: FP32 forms it first, whose square stays in range for any cell size; FP64
        // saves the operations
        const T j = sizeof(T) == 4 ? Jc : T(1), Jo = sizeof(T) == 4 ? T(1) : Jc;
        const T gx = j * kj[0], gy = j * kj[1], gz = j * kj[2];
        const T U = Jo * (u * gx + v * gy + w * gz), a = fabs(Jo) * sqrt_product(c2, gx * gx + gy * gy + gz * gz);
        T lm = fabs(U - a), l0 = fabs(U), lp = fabs(U + a);
        if (!charwise) { lm = fmax(lm, lp); l0 = lm; lp = lm; }
        best[3 * d] = fmax(best[3 * d], lm);
        best[3 * d + 1] = fmax(best[3 * d + 1], l0);
        best[3 * d + 2] = fmax(best[3 * d + 2], lp);
      }
    }
    if (it + 1 < it1 && items[it + 1].x == item.x) continue;
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      T b = best[t];
      for (int h = 16; h; h >>= 1) b = fmax(b, __shfl_xor_sync(0xffffffffu, b, h));
      if (threadIdx.x % 32 == 0) red[t][threadIdx.x / 32] = b;
      best[t] = T(0);
    }
    __syncthreads();
    if (threadIdx.x < 3 * dims) {
      T b = red[threadIdx.x][0];
      for (int w = 1; w < kLamChunk / 32; ++w) b = fmax(b, red[threadIdx.x][w]);
      atomic_max_nonneg(FPK_IN(static_cast<T *>(B->lamg) + threadIdx.x, static_cast<T *>(B->lamg), 9, B->status), b);
    }
    __syncthreads();
  }
}

// The G cells next to one side of a block, in the halo layout the receiving block reads:
// the state layout [5][nk][nj][ni] with the extent of direction `dir` replaced by G.  Low
// side: cells 0..G-1; high side: cells n-G..n-1 (index x - (n - G) in the buffer).
template <typename T>
__global__ void k_pack_halo(const T *__restrict__ q, int stage, T *__restrict__ out, int dir, int side, int G, int ni,
                            int nj, int nk, int *status) {
  int e[3] = {ni, nj, nk};
  const int nd = e[dir];
  e[dir] = G;
  const long long hc = (long long)e[0] * e[1] * e[2], qc = (long long)ni * nj * nk;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < 5 * hc;
       idx += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(idx / hc);
    long long r = idx - v * hc;
    int c[3];
    c[0] = (int)(r % e[0]);
    r /= e[0];
    c[1] = (int)(r % e[1]);
    c[2] = (int)(r / e[1]);
    c[dir] += side ? nd - G : 0;
    *FPK_IN(out + idx, out, 5 * hc, status) = *FPK_IN(q + state_at(stage, ((long long)c[2] * nj + c[1]) * ni + c[0], qc, v), q, 5 * qc, status);
  }
}

}  // namespace

cudaError_t launch_pack_halo(const void *q, int stage, int is_f32, int dir, int side, int G, const int *n, void *out,
                             int *status, cudaStream_t s) {
  int e[3] = {n[0], n[1], n[2]};
  e[dir] = G;
  const long long total = 5LL * e[0] * e[1] * e[2];
  const int threads = 256;
  const long long want = (total + threads - 1) / threads;
  const int grid = (int)(want < 4096 ? (want < 1 ? 1 : want) : 4096);
  if (is_f32)
    k_pack_halo<float><<<grid, threads, 0, s>>>(static_cast<const float *>(q), stage, static_cast<float *>(out), dir, side, G,
                                                n[0], n[1], n[2], status);
  else
    k_pack_halo<double><<<grid, threads, 0, s>>>(static_cast<const double *>(q), stage, static_cast<double *>(out), dir, side,
                                                 G, n[0], n[1], n[2], status);
  return cudaGetLastError();
}

cudaError_t launch_lambda(const BlockDev *blocks, int nblocks, const int2 *items, int nitems, int is_f32,
                          int charwise, int stage, cudaStream_t s) {
  const int zb = (nblocks + 127) / 128;
  int grid = nitems < 152 * 8 ? nitems : 152 * 8;
  if (grid < 1) grid = 1;
  if (is_f32) {
    k_lam_zero<float><<<zb, 128, 0, s>>>(blocks, nblocks);
    k_lam_max<float><<<grid, kLamChunk, 0, s>>>(blocks, items, nitems, charwise, stage);
  } else {
    k_lam_zero<double><<<zb, 128, 0, s>>>(blocks, nblocks);
    k_lam_max<double><<<grid, kLamChunk, 0, s>>>(blocks, items, nitems, charwise, stage);
  }
  return cudaGetLastError();
}

int cfl_ctas(long long ncells) { return (int)((ncells + kCflThreads * kCflPoints - 1) / (kCflThreads * kCflPoints)); }

cudaError_t launch_cfl(const BlockDev *blk, int is_f32, long long ncells, const int *n, int dims,
                       CflScratch *scratch, cudaStream_t s) {
  // small blocks: one kernel over all points
  const bool small = ncells <= kCflSmall;
  const int g = small ? (int)((ncells + kCflThreads - 1) / kCflThreads) : cfl_ctas(ncells);
  float2 *hi = reinterpret_cast<float2 *>(scratch + 1);
  if (!small) {
    cudaError_t e = launch_kernel(is_f32 ? k_cfl_bound<float> : k_cfl_bound<double>, g, kCflThreads, 0, s, 0, blk, ncells,
                                  n[0], n[1], dims, scratch, hi);
    if (e != cudaSuccess) return e;
  }
  return launch_kernel(is_f32 ? k_cfl_max<float> : k_cfl_max<double>, g, kCflThreads, 0, s, small ? 0 : 1, blk, ncells, n[0],
                       n[1], dims, scratch, small ? (const float2 *)nullptr : (const float2 *)hi);
}

}  // namespace fpk
