// sgp_launch.cuh -- host-side launchers for the pass kernels, dispatched on
// the line length N (a compile-time parameter of every kernel) and on the
// kernel variant V chosen by the autotuner.
#pragma once
#include <cuda_runtime.h>

#include <atomic>

#include "sgp_kernels.cuh"

namespace sgp {

// Elements per thread: 8 (FP32) / 4 (FP64) for powers of two, 6 for 3*2^k.
template <typename R, int N>
constexpr int elems_per_thread() {
  return (N % 3 == 0) ? 6 : (sizeof(R) == 4 ? 8 : 4);
}

// Line lengths with compiled kernels.
#define SGP_FOR_EACH_N(X) \
  X(16) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512) X(768) X(1024)
#define SGP_FOR_EACH_N_POW2(X) X(16) X(32) X(64) X(128) X(256) X(512) X(1024)

inline bool supported_n(int n) {
  switch (n) {
#define SGP_CASE(N) case N:
    SGP_FOR_EACH_N(SGP_CASE)
#undef SGP_CASE
    return true;
    default:
      return false;
  }
}

// Kernel variants of a pass (the tile and radix schedules the autotuner
// chooses from):
//   0  default geometry (x-pass: about 256 threads per CTA; line pass: up
//      to 512 threads, TILE >= 4 FP32 / 2 FP64 columns) and radix plan
//      (a context takes for it what suits its size: default_kernel below,
//      with the component-parallel passes of sgp_split.cuh)
//   1  CTAs of about half the threads (line pass: TILE down to 1)
//   2  CTAs of about a quarter of the threads
//   3  FP32 only.  N a power of two: radix-4 plan (4 elements per thread
//      instead of 8: more stages, half the registers per line element).
//      N = 3*2^k: 12 elements per thread, radix 6 then 4s (96 = 6*4*4 in
//      three stages instead of 6*2*2*2*2 in five), in CTAs of 128 threads
//      (x-pass geometry 1, line-pass geometry 2: a thread holds 120
//      registers of field data)
//   4  FP32 only.  Line pass: geometry 1 with the tile loaded by tensor
//      copies (TMA) into shared memory; x-pass: the same as variant 1
//   5  FP32, x-pass of 3D grids with NX = NY = 64 or 128 only: the steps'
//      x-passes become xy-plane passes (k_xyplane: one thread-block cluster
//      per z plane, the y transforms done there), so a step drops its
//      y-line passes; x-passes outside the steps are those of variant 1
//   6  x-pass: the rows of geometry 2 with the nonlinear flow shared by the
//      256 threads of the CTA (k_xpass_wide; for small grids, whose CTAs
//      are few); line pass: the same as variant 2
//   7  the default geometry itself, whatever the size (variant 0 of the groups
//      of an ensemble): a member's result does not depend on the batch
constexpr int kVariants = 8;

template <typename R, int N, int V>
constexpr int variant_elems() {
  return V == 3 ? (N % 3 == 0 ? 12 : 4) : elems_per_thread<R, N>();
}
// geometry of variant V for the x-pass (PART 0) and the line pass (PART 1)
template <int N, int V, int PART>
constexpr int variant_geom() {
  return V == 3 ? (N % 3 == 0 ? 1 + PART : 0) : (V == 4 || V == 5) ? 1 : V == 6 ? 2 : V == 7 ? 0 : V;
}

// Does variant V exist for line length N (prec_bytes 4 or 8)?
inline bool variant_exists(int prec_bytes, int N, int V) {
  if (!supported_n(N) || V < 0 || V >= kVariants) return false;
  if (V == 3 || V == 4) return prec_bytes == 4;
  return V != 5;       // variant 5 depends on the whole grid (plane_ok in the host runtime)
}
// Elements per thread of variant V (the twiddle table layout depends on it).
inline int variant_elems_rt(int prec_bytes, int N, int V) {
  if (V == 3) return N % 3 == 0 ? 12 : 4;
  return (N % 3 == 0) ? 6 : (prec_bytes == 4 ? 8 : 4);
}

// Launch geometry of one pass (for accounting and the observables scratch).
struct PassGeom {
  int threads;
  int rows_or_tile;   // rows per CTA (x-pass) or columns per CTA (line pass)
  size_t smem;
};

// Lets a kernel have more than 48 KB of dynamic shared memory on the current
// device; done: the device it was last done on (any number of host threads).
template <typename K>
inline cudaError_t opt_in(K kern, size_t smem, std::atomic<int>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || done.load(std::memory_order_acquire) == dev) return e;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) done.store(dev, std::memory_order_release);
  return e;
}

// Launch of a pass kernel; dependent: it may begin while the pass before it on
// the stream is at work (the kernel waits in pdl_wait before it touches the
// field).
template <typename K, typename... A>
inline cudaError_t launch_pass(K kern, dim3 grid, int threads, size_t smem, bool dependent, cudaStream_t s,
                               const A&... a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, a...);
}

// Per-variant entry points (explicitly instantiated in sgp_inst.cu).
template <typename R, int V> PassGeom xpass_geom_v(int N);
template <typename R, int V> PassGeom linepass_geom_v(int N);
template <typename R, int V> cudaError_t prepare_xpass_v(int N);
template <typename R, int V> cudaError_t prepare_linepass_v(int N);
template <typename R, int V>
cudaError_t launch_xpass_v(int N, const XPassArgs<R>& a, int members, bool dependent, cudaStream_t s);
template <typename R, int V>
cudaError_t launch_linepass_v(int N, const LPassArgs<R>& a, int planes, int members,
                              bool dependent, cudaStream_t s);
// Variant 4 of the line pass (tile loads by tensor copies over `map`).
cudaError_t launch_linepass_tma(int N, const LPassArgs<float>& a, const CUtensorMap& map, int planes,
                                int members, bool dependent, cudaStream_t s);
cudaError_t prepare_linepass_tma(int N);
PassGeom linepass_geom_tma(int N);
// Variant 5 of the x-pass: the xy-plane pass over `planes` z planes of
// `members` members (N = NX = NY; twy: the y twiddles; err: the word a
// bounded wait for a hand-over sets when it gives up).
cudaError_t launch_xyplane(int N, const XPassArgs<float>& a, const TwE<float>* twy, int* err, int planes,
                           int members, cudaStream_t s);
cudaError_t prepare_xyplane(int N);
// Variant 6 of the x-pass (k_xpass_wide).
template <typename R>
cudaError_t launch_xpass_wide(int N, const XPassArgs<R>& a, int members, bool dependent, cudaStream_t s);
template <typename R>
cudaError_t prepare_xpass_wide(int N);

// x-pass variants 4 and 5 are variant 1 (variant 5's plane pass has its own
// entry point) and variant 6 has the geometry of variant 2 (its own kernel,
// dispatched first), variant 7 is variant 0; the line pass has its own variant
// 4 and takes variant 2 for 6
#define SGP_VARIANT_SWITCH_X(V, CALL, FAIL)                  \
  switch (V) {                                               \
    case 0: return CALL(0);                                  \
    case 1: return CALL(1);                                  \
    case 2: return CALL(2);                                  \
    case 3:                                                  \
      if constexpr (sizeof(R) == 4) return CALL(3);          \
      return FAIL;                                           \
    case 4:                                                  \
    case 5:                                                  \
      if constexpr (sizeof(R) == 4) return CALL(1);          \
      return FAIL;                                           \
    case 6: return CALL(2);                                  \
    case 7: return CALL(0);                                  \
    default: return FAIL;                                    \
  }
#define SGP_VARIANT_SWITCH(V, CALL, FAIL)                    \
  switch (V) {                                               \
    case 0: return CALL(0);                                  \
    case 1: return CALL(1);                                  \
    case 2: return CALL(2);                                  \
    case 3:                                                  \
      if constexpr (sizeof(R) == 4) return CALL(3);          \
      return FAIL;                                           \
    case 6: return CALL(2);                                  \
    case 7: return CALL(0);                                  \
    default: return FAIL;                                    \
  }

template <typename R>
inline PassGeom xpass_geom(int N, int V = 0) {
#define SGP_C(v) xpass_geom_v<R, v>(N)
  SGP_VARIANT_SWITCH_X(V, SGP_C, (PassGeom{0, 0, 0}))
#undef SGP_C
}
template <typename R>
inline PassGeom linepass_geom(int N, int V = 0) {
  if constexpr (sizeof(R) == 4)
    if (V == 4) return linepass_geom_tma(N);
#define SGP_C(v) linepass_geom_v<R, v>(N)
  SGP_VARIANT_SWITCH(V, SGP_C, (PassGeom{0, 0, 0}))
#undef SGP_C
}
// Set the kernels' shared-memory attributes for line length N on the
// current device (done before any stream capture).
template <typename R>
inline cudaError_t prepare_xpass(int N, int V = 0) {
  if (V == 6) {
    const cudaError_t e = prepare_xpass_wide<R>(N);
    if (e != cudaSuccess) return e;
  }
#define SGP_C(v) prepare_xpass_v<R, v>(N)
  SGP_VARIANT_SWITCH_X(V, SGP_C, cudaErrorInvalidValue)
#undef SGP_C
}
template <typename R>
inline cudaError_t prepare_linepass(int N, int V = 0) {
  if constexpr (sizeof(R) == 4)
    if (V == 4) return prepare_linepass_tma(N);
#define SGP_C(v) prepare_linepass_v<R, v>(N)
  SGP_VARIANT_SWITCH(V, SGP_C, cudaErrorInvalidValue)
#undef SGP_C
}
template <typename R>
inline cudaError_t launch_xpass(int N, int V, const XPassArgs<R>& a, int members, bool dependent, cudaStream_t s) {
  if (V == 6) return launch_xpass_wide<R>(N, a, members, dependent, s);
#define SGP_C(v) launch_xpass_v<R, v>(N, a, members, dependent, s)
  SGP_VARIANT_SWITCH_X(V, SGP_C, cudaErrorInvalidValue)
#undef SGP_C
}
// Variants 0-3 of the line pass (variant 4 goes through launch_linepass_tma).
template <typename R>
inline cudaError_t launch_linepass(int N, int V, const LPassArgs<R>& a, int planes, int members,
                                   bool dependent, cudaStream_t s) {
#define SGP_C(v) launch_linepass_v<R, v>(N, a, planes, members, dependent, s)
  SGP_VARIANT_SWITCH(V, SGP_C, cudaErrorInvalidValue)
#undef SGP_C
}
#undef SGP_VARIANT_SWITCH
#undef SGP_VARIANT_SWITCH_X

// What variant 0 of an axis stands for, by the size of the whole batch (pts
// grid points), the precision and the line length; measured per TS2 step on
// the GB300 (plain variant 0 -> the choice, us):
//   component-parallel passes for grids of few lines (split_range): FP32 2D up
//     to 192 Ki points (64^2 22 -> 5, 256^2 32 -> 10, 384^2 44 -> 27; from 256
//     Ki points the others are ahead: 4 x 256^2 27 against 33), 3D below 128 Ki
//     (48^3 35 -> 28; 64 x 64 x 32 28 against 30).  Past 128 Ki points y-lines
//     shorter than 64, whose CTAs of two columns are one to three warps, take
//     geometry 2 unless the rows are the shortest (with component-parallel
//     rows, split -> geometry 2: 32 x 48 times 128 30.7 -> 25.5, times 96 24.1 ->
//     21.8, 64 x 32 times 72 19.0 -> 18.2, 96 x 16 times 128 27.0 -> 23.8, 1024 x
//     32 times 5 27.1 -> 26.1, times 4 16.8 -> 17.6; but 16 x 16 times 768 26.9 ->
//     37.5, and 64 x 64 times 40 20.0 -> 19.9);
//   FP64 everywhere (fixed-point transforms, sgp_fix.cuh: 64^2 229 -> 50, 8 x
//     512^2 5300 -> 2500, 128^3 5510 -> 2610), with one line per CTA while that
//     gives no more than four CTAs an SM;
//   FP32 2D otherwise: TMA tiles for the y-lines (768^2 104 -> 90 with x-pass
//     geometry 1), for the x-pass geometry 1 or that of long_row_geometry;
//   FP32 3D otherwise: geometry 1 on every axis (128^3 230 -> 190).
constexpr int kSplitPass = 100, kSplitMany = 101;

// x-pass geometry of FP32 rows of 512 or 1024 points, by the last wave: CTAs of
// 256 threads (geometry 0) cost less than twice as many of 128 (geometry 1)
// where they do not end later, that is where halving them saves no part of a
// wave of one CTA an SM; 1024 points past two CTAs an SM take geometry 1.  us per
// TS2 step with geometry 0 and 1, rows of 512: 512 rows 26.1 and 27.0, 640 38.5
// and 35.5, 1024 39.7 and 41.5, 1408 59.2 and 56.8, 2048 75.4 and 73.9, 4096
// 135.9 and 138.0; of 1024: 384 45.0 and 39.7, 512 45.6 and 47.0, 2048 156 and
// 150.  Shorter rows are within 1% at 256 and ahead with geometry 1 below (64:
// 23.8 and 22.9), those of 3*2^k ahead with it or level.
inline int long_row_geometry(int nx, long long rows, int sms) {
  const long long c0 = (rows + xpass_geom<float>(nx, 0).rows_or_tile - 1) / xpass_geom<float>(nx, 0).rows_or_tile;
  const long long c1 = (rows + xpass_geom<float>(nx, 1).rows_or_tile - 1) / xpass_geom<float>(nx, 1).rows_or_tile;
  const bool level = 2 * ((c0 + sms - 1) / sms) <= (c1 + sms - 1) / sms;
  return level && (nx <= 512 || c0 <= 2LL * sms) ? 0 : 1;
}

// FP32 grids (whole batches) of few lines
inline bool split_range(int dim, long long pts) { return pts <= (dim == 2 ? 3LL << 16 : (1LL << 17) - 1); }

inline int default_kernel(int prec_bytes, int dim, const int* n, int batch, int a, bool tensor_maps, int sms) {
  const long long pts = (long long)n[0] * n[1] * (dim == 3 ? n[2] : 1) * batch;
  if (prec_bytes == 8) return pts / n[a] > 4LL * sms ? kSplitMany : kSplitPass;
  if (split_range(dim, pts)) {
    const bool short_columns = dim == 2 && a == 1 && n[1] < 64 && n[0] >= 32;
    return short_columns && pts > 8LL << 14 ? 2 : kSplitPass;
  }
  if (dim == 3) return 1;
  if (a == 0) return n[0] >= 512 && n[0] % 3 != 0 ? long_row_geometry(n[0], pts / n[0], sms) : 1;
  return tensor_maps ? 4 : 1;
}

// Do a gradient's passes run component-parallel too?  In the range of split_range
// (24 TS2 steps with the sweep, us, plain -> split: 64^2 1820 -> 550, 2 x 256^2
// 2360 -> 1870, 48^3 3060 -> 2550) but for
//   rows of 1024 points, whose adjoint CTAs (640 threads of 128 registers) are one
//     to an SM: past one wave of rows (3 x 1024 x 48 2340 -> 2100, 4 x 1024 x 48
//     2660 -> 3030);
//   rows of 32 points, a CTA of one warp each: past 128 Ki points in 2D (32 x 64
//     times 64 2000 -> 1940, times 96 2440 -> 2730), past 112 Ki in 3D (32 x 16 x
//     16 times 15 2470 -> 2640).
inline bool gradient_split_pays(int dim, const int* n, int batch, int sms) {
  const long long pts = (long long)n[0] * n[1] * (dim == 3 ? n[2] : 1) * batch;
  if (n[0] == 1024 && pts / n[0] > sms) return false;
  return n[0] != 32 || pts <= (dim == 2 ? 8LL << 14 : 7LL << 14);
}

// Observables kernels (default geometry only).
template <typename R>
cudaError_t launch_obs_x(int N, const ObsXArgs<R>& a, int members, cudaStream_t s);
template <typename R>
cudaError_t launch_obs_line(int N, const ObsLArgs<R>& a, int planes, int members,
                            cudaStream_t s);

}  // namespace sgp
