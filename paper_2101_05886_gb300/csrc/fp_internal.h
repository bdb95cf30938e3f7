// fp_internal.h - device-side descriptors shared by the kernels and the C ABI of
// libfpgb300.so.  Not part of the public interface (include/fp.h is).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fpk {

constexpr int kCellFields = 14;      // per-cell values staged in shared memory
constexpr int kFaceFields = 16;      // per-face values staged in shared memory, at most (sweep_face_fields)
constexpr int kNextFields = 21;      // staged per thread: next chunk's cell (Q, k, 1/J), face metrics and their change x2
constexpr int kEpiFields = 10;       // epilogue operands staged per thread (accumulator, Q^n)

// CTA shape of a sweep variant (precision, scheme, fix: 0 switches read at run time, 1 folded,
// 2 folded with the alternative shape, 3 component-wise, 4 states far from unit scale): its threads, which equal faces per chunk x
// lines per tile, whether the rings of the xi pass are padded (none is: turning the slots of
// every other group of lines keeps all tile shapes free of bank conflicts), and the CTAs one SM
// holds.
// The warps of a CTA meet at two or three barriers per chunk, so with fewer warps per CTA the phases
// of the chunk (staging, FMA-heavy faces, epilogue) of different CTAs overlap instead of running
// in step; large CTAs read wider rows in the eta and zeta passes (TT = 16 lines instead of 8).  The
// folded FP32 sweeps have both, and a batch runs the one sweep_batch_shape names:
//   WENO5-JS:       64 threads, 8 CTAs per SM             |  alternative 128, 4
//   linear upwind: 128 threads, 4                         |  alternative  64, 8
//   WENO7-JS:      128 threads, 2 (255 registers)         |  alternative  64, 4
// Every other sweep: 128 threads, 4 CTAs (FP32) or 2 (FP64, and WENO7).
// Measured, 64 | 128 threads, default tiles: WENO5 256^3 7.81 | 7.86 ms, 64-block batch 16.28 | 16.35;
// linear upwind 256^3 5.45 | 5.46, 20-block batch 2.29 | 2.32; WENO7 256^3 11.44 | 11.54, batch 4.86 |
// 4.85.  A batch runs one shape throughout (kernels of two shapes in its graph would not share SMs).
__host__ __device__ constexpr bool sweep_has_alt(bool f32, int scheme, int fix) {
  return f32 && (fix == 1 || fix == 2) && scheme >= 0 && scheme <= 2;
}
__host__ __device__ constexpr int sweep_batch_shape(bool f32, int scheme, int fix) {
  return sweep_has_alt(f32, scheme, fix) && scheme == 1 ? 1 : 0;
}
__host__ __device__ constexpr int sweep_threads(bool f32, int scheme, int fix) {
  return !sweep_has_alt(f32, scheme, fix) ? 128
         : ((scheme == 0) != (fix == 2) ? 64 : 128);   // WENO5 primary 64, the others' alternative 64
}
__host__ __device__ constexpr bool sweep_padded(bool, int, int) { return false; }
__host__ __device__ constexpr int sweep_ring(bool f32, int scheme, int fix) {
  return 2 * sweep_threads(f32, scheme, fix);
}
__host__ __device__ constexpr int sweep_min_ctas(bool f32, int scheme, int fix) {
  return (!f32 || scheme == 2 ? 256 : 512) / sweep_threads(f32, scheme, fix);
}

// Fields of the face ring: flux and reference-state increment, and for FP32 WENO7 (see the sweep) the
// lower cell's state and 1/J.
__host__ __device__ constexpr bool sweep_early(bool f32, int scheme) { return f32 && scheme == 2; }
__host__ __device__ constexpr int sweep_face_fields(bool f32, int scheme) {
  return sweep_early(f32, scheme) ? kFaceFields : 10;
}

// Shared-memory field indices of a staged cell.
enum : int {
  CF_Q = 0,      // 0..4 conserved variables
  CF_K = 5,      // 5..7 metric vector of the swept direction (d_x, d_y, d_z)/J
  CF_INVJ = 8,   // 1/J
  CF_RINV = 9,   // 1/rho
  CF_H = 10,     // total enthalpy
  CF_SQR = 11,   // sqrt(rho)
  CF_UC = 12,    // contravariant velocity u . grad(d), grad(d) = J k
  CF_AC = 13     // c |grad(d)|
};

// What a pass does with its part of the residual: write or add it to the accumulator, or finish
// dQ/dt or the RK stage with it.  Where all directions run in one launch, each writes an
// accumulator of its own and launch_finish sums them.
enum : int { MODE_WRITE = 0, MODE_ADD = 1, MODE_RHS = 2, MODE_RK = 3 };

// Status word bits set by the kernels.
enum : int { ST_NONFINITE = 1, ST_BOUNDS = 2 };

// Bounds-checking builds (compiled with -DFPK_BOUNDS_CHECK, libfpgb300_check.so): before every
// access of the sweep, the sum that ends a stage, the halo packing and the speed and time-step
// reductions to a block's arrays (states, halos, metrics, face metrics, accumulators, dQ/dt, speeds)
// the element is checked against the array, and every shared-ring offset against the ring.  (The
// lists that a launch is made of, descriptors and work items, are read by CTA number and link and
// not checked.)  An element outside records ST_BOUNDS in the status word and the access goes to
// the array's first element instead, so a wrong index shows as FP_ERR_BOUNDS, not as a fault.  In
// the normal build FPK_CHK_ONLY(...) expands to nothing and FPK_IN(p, ...) to p.
#ifdef FPK_BOUNDS_CHECK
#define FPK_CHK_ONLY(...) __VA_ARGS__
template <typename P>
__device__ __forceinline__ P fpk_in(P p, P base, long long n, int *status) {
  if (p >= base && p < base + n) return p;
  atomicOr(status, ST_BOUNDS);
  return base;
}
#define FPK_IN(p, base, n, status) ::fpk::fpk_in((p), (base), (long long)(n), (status))
#else
#define FPK_CHK_ONLY(...)
#define FPK_IN(p, base, n, status) (p)
#endif

// One swept direction of one block.  A "line" runs along the swept direction.  Strides of one
// grid index and component, and element offsets within a component, are 32-bit: a block holds
// fewer than 2^31 points (and fewer than 2^32 with its ghosts, or its metrics fit no device).
struct DirDev {
  int nd;              // points along the line
  int nt1;             // extent of the first transverse coordinate (lines are numbered t1 + nt1 t2)
  int nt2;             // extent of the second one (0 for a direction the block does not sweep)
  int qT1, qT2, qsd;   // state offsets: t1, t2 and along-line strides
  int mT1, mT2, msd;   // metric offsets (ghosted arrays)
  int fT1, fT2, fsd;   // face-metric offsets, face f+1/2 at (f+1)*fsd
  unsigned fc;         // faces of this direction
  int bclo, bchi;      // boundary codes at the two line ends
  int S, TT;           // faces per chunk, lines per tile (S * TT == the variant's sweep_threads)
  // Metrics of this direction, the values of a point side by side, so that the eta and zeta passes,
  // whose tiles are TT points wide, read rows of 16 TT and 24 TT bytes instead of 4 TT (FP32; with
  // the accumulator alike: 256^3 WENO5 step 8.52 -> 7.85 ms, 64-block batch 16.81 -> 16.33 ms,
  // linear batch 2.48 -> 2.33 ms).
  const void *kj;      // T [ghosted cells][4]: metric vector (d_x, d_y, d_z)/J and 1/J
  const void *fk;      // T [faces][6]: metric k of face x + 1/2; k_{x+1/2} - k_{x-1/2} of cell x (FP64-formed)
  void *racc;          // residual accumulator, T [cells][4] then T [cells] (the directions' own or the same one)
  // FP_BC_HALO sides: the caller's buffers of the G cells beyond each side, laid out like the
  // state with this direction's extent replaced by G (strides: t1, t2, along the line, component)
  const void *halo[2];
  int hT1, hT2, hsd;
  int nbr[2];          // FP_BC_BLOCK sides: index of the linked block in the launch's block table
  unsigned hc;
};

// 16-byte aligned and padded so that the sweep can copy a descriptor into shared memory in
// 16-byte cp.async pieces
struct alignas(16) BlockDev {
  DirDev dir[3];
  int dims;
  int G;               // metric ghost width
  unsigned qc;         // state component stride (ni*nj*nk)
  unsigned mc;         // ghosted cells
  unsigned moff;       // offset of point (0,0,0) in the metric arrays
  // stage states: 0 = Q^n (the caller's, T [5][cells]), 1 = Q^(1), 2 = Q^(2) (T [cells][4] then T [cells])
  void *q[3];
  void *dqdt;          // output of the rhs mode
  double gamma;
  // the sweep's constants in its arithmetic type (12 float or double values): reference (far-field)
  // state, its velocity and pressure, gamma - 1, gamma, 1/(gamma - 1)
  alignas(16) double cst[12];
  int *status;         // device status word: ST_NONFINITE, ST_BOUNDS
  int global_lf;       // 1: Lax-Friedrichs speeds from lamg instead of the stencil
  void *lamg;          // T [3 directions][3]: max |U - c|grad||, |U|, |U + c|grad|| over the block
  int cut;             // FP_BC_CUT sides: lines t1 < cut or t1 >= nt1 - cut meet across the cut
};

// A work item of the sweep: `len` consecutive positions (cells and the ghost positions between two
// lines) of one block's stream, the first one position u0 (0 .. nd + 2 G - 1) of tile `tile`;
// after the end of a tile's line the stream goes on with the tile `stride` further.  `dir` is the
// swept direction.  Item c is
// the first of CTA c, `next` the index of the CTA's next item (-1: none).  16-byte aligned:
// copied into shared memory in 16-byte pieces.
struct alignas(16) SweepItem {
  int block, tile, stride, u0;
  int len, next, dir, pad;
};

struct SweepLaunch {
  const BlockDev *blocks;
  const SweepItem *items;
  int mode;
  int stage;           // RK stage 0,1,2 (input q[stage], output q[(stage+1)%3])
  const double *dt;    // device scalar
  int grid;            // CTAs of the launch
  int bnd = 0;         // some block of the launch has a slip-wall or cut side in a swept direction
  int glf = 0;         // the blocks of the launch use global Lax-Friedrichs speeds
  int alt = 0;         // the blocks' tiles are of the alternative CTA shape
  int wide = 0;        // some block's state is far from unit scale (FP32: the sweep that squares no momenta)
  int chained = 0;     // the kernel before it in the stream may still run (launch_kernel)
};

// Launchers of the sweep, one per translation unit (sweep_<NAME>.cu): precision f32 / f64,
// `_bnd` with the slip-wall, cut, link and halo rules compiled in, `_fix` with the
// characteristic decomposition and the FP form fixed on, `_fix2` the same in the alternative
// CTA shape (FP32 only), `_comp` component-wise, `_wide` for states far from unit scale (FP32 only; `fp`
// there is 2 bits: the FP form, component-wise).  Each returns the cudaError_t of the
// launch; prepare_sweep_<NAME> opts in to the dynamic shared memory of its 16 (M, scheme)
// variants and returns the resident CTAs per SM of the given one.
cudaError_t launch_sweep_f32(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f32_fix(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f32_fix2(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f32_comp(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f32_wide(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f32_bnd(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f32_bnd_fix(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f32_bnd_fix2(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f32_bnd_comp(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f32_bnd_wide(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f64(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f64_fix(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f64_comp(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f64_bnd(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f64_bnd_fix(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
cudaError_t launch_sweep_f64_bnd_comp(const SweepLaunch &L, int M, int scheme, int fp, cudaStream_t s);
int prepare_sweep_f32(int M, int scheme);
int prepare_sweep_f32_fix(int M, int scheme);
int prepare_sweep_f32_fix2(int M, int scheme);
int prepare_sweep_f32_comp(int M, int scheme);
int prepare_sweep_f32_wide(int M, int scheme);
int prepare_sweep_f32_bnd(int M, int scheme);
int prepare_sweep_f32_bnd_fix(int M, int scheme);
int prepare_sweep_f32_bnd_fix2(int M, int scheme);
int prepare_sweep_f32_bnd_comp(int M, int scheme);
int prepare_sweep_f32_bnd_wide(int M, int scheme);
int prepare_sweep_f64(int M, int scheme);
int prepare_sweep_f64_fix(int M, int scheme);
int prepare_sweep_f64_comp(int M, int scheme);
int prepare_sweep_f64_bnd(int M, int scheme);
int prepare_sweep_f64_bnd_fix(int M, int scheme);
int prepare_sweep_f64_bnd_comp(int M, int scheme);

// Programmatic dependent launch: with `chained`, the kernel may be scheduled while the one before
// it in the stream is still running and has to execute chain_wait() before it touches anything
// that one reads or writes; chain_next() lets the kernel after it do the same.  Without, the
// launch waits as usual and both are no-ops.
template <typename... P, typename... A>
inline cudaError_t launch_kernel(void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t s, int chained,
                                 A... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#ifdef __CUDACC__
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

// Every device and page-locked allocation of the library goes through these two, so the
// host-side hook fp_debug_fail_allocation can make a chosen one fail as if the device (or
// the pinned host pool) were out of memory.  Defined in api.cu.
cudaError_t dev_malloc(void **p, size_t bytes);
cudaError_t host_malloc(void **p, size_t bytes);
template <typename P> inline cudaError_t dev_alloc(P **p, size_t bytes) {
  return dev_malloc(reinterpret_cast<void **>(p), bytes);
}

// Metric construction (metrics.cu), FP64.
struct MetricJob {
  int dims, M, G, Gn;
  int n[3];
  const double *nodes;     // device, [dims][..] with Gn ghosts
  double *met;             // device, [10][B3]
  double *fmet[3];         // device, face metrics per direction [3][faces]
  double *scratch;         // device, 9 * |B2| doubles
};
cudaError_t build_metrics(const MetricJob &J, cudaStream_t s);
// The sweep's arrays (DirDev kj and fk) of direction d from the FP64 ones, in its type.
cudaError_t pack_metrics(const MetricJob &J, int d, int is_f32, void *kj, cudaStream_t s);
cudaError_t pack_faces(const MetricJob &J, int d, int is_f32, void *fk, cudaStream_t s);
// The way back: values first .. first + n - 1 of the FP64 [components][points] array that packed arrays
// hold, `per` components in each of `arrays` of them and the first one's next value behind these
// (metrics: kj of three directions, per = 3, and 1/J; face metrics: one fk, per = 3).
cudaError_t unpack(const void *const a[3], int is_f32, int stride, int per, int arrays, long long points,
                   long long first, long long n, double *out, cudaStream_t s);

// Global Lax-Friedrichs speeds (cfl.cu): zero, then max over (block, first point) items of
// kLamChunk points each (the kernel's threads).
constexpr int kLamChunk = 256;
cudaError_t launch_lambda(const BlockDev *blocks, int nblocks, const int2 *items, int nitems,
                          int is_f32, int charwise, int stage, cudaStream_t s);

// Sum of the directions' accumulators of one block and the end of the pass (stage.cu): dQ/dt (rk = 0)
// or the RK stage (rk = 1).
cudaError_t launch_finish(const BlockDev *blk, int is_f32, long long ncells, const int *n, int dims, int rk,
                          int stage, const double *dt, cudaStream_t s);

// CFL reduction (cfl.cu): `scratch` holds CflScratch and a float2 per CTA (cfl_ctas of them).
struct CflScratch {
  unsigned long long max_bits;   // the result: bits of the FP64 maximum
  unsigned int lower_bits;       // bits of the largest FP32 lower bound
  unsigned int pad;
};
int cfl_ctas(long long ncells);
cudaError_t launch_cfl(const BlockDev *blk, int is_f32, long long ncells, const int *n, int dims,
                       CflScratch *scratch, cudaStream_t s);

// Halo packing (cfl.cu): the G cells of stage state `stage` next to side `side` of direction
// `dir` into `out`, in the halo layout of DirDev (the receiving block's view of them); `status`
// is the context's status word (bounds-checking builds record there).
cudaError_t launch_pack_halo(const void *q, int stage, int is_f32, int dir, int side, int G, const int *n, void *out,
                             int *status, cudaStream_t s);

}  // namespace fpk
