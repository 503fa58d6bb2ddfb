// sgp_split.cu -- instantiation and launchers of the FP32 component-parallel
// passes; see sgp_split.cuh.
#include "sgp_split.cuh"

#include "sgp_launch.cuh"

namespace sgp {
namespace {

template <typename K>
cudaError_t opt_in(K kern, size_t smem, int* done_dev) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (*done_dev == dev) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) *done_dev = dev;
  return e;
}

template <int N>
cudaError_t xsplit_prepare_n() {
  constexpr int E = split_elems<float, N>(), G = split_rows<float, N>();
  static int done = -1;
  return opt_in(k_xsplit<float, N, E, G, false>, SplitCfg<float, N, E, G>::SMEM, &done);
}

template <int N>
cudaError_t xsplit_n(const XPassArgs<float>& a, int members, bool dependent, cudaStream_t s) {
  constexpr int E = split_elems<float, N>(), G = split_rows<float, N>();
  typedef SplitCfg<float, N, E, G> Cfg;
  const cudaError_t e = xsplit_prepare_n<N>();
  if (e != cudaSuccess) return e;
  return launch_pass(k_xsplit<float, N, E, G, false>, dim3((a.rows + G - 1) / G, members), Cfg::THREADS, Cfg::SMEM,
                     dependent, s, a);
}

template <int N>
cudaError_t lsplit_prepare_n() {
  constexpr int E = split_elems<float, N>(), G = split_cols<float, N>();
  static int done = -1;
  return opt_in(k_lsplit<float, N, E, G>, SplitCfg<float, N, E, G>::SMEM, &done);
}

template <int N>
cudaError_t lsplit_n(const LPassArgs<float>& a, int planes, int members, bool dependent, cudaStream_t s) {
  constexpr int E = split_elems<float, N>(), G = split_cols<float, N>();
  typedef SplitCfg<float, N, E, G> Cfg;
  const cudaError_t e = lsplit_prepare_n<N>();
  if (e != cudaSuccess) return e;
  return launch_pass(k_lsplit<float, N, E, G>, dim3((a.nx + G - 1) / G, planes, members), Cfg::THREADS, Cfg::SMEM,
                     dependent, s, a);
}

}  // namespace

#define SGP_SWITCH(CALL, FAIL) \
  switch (N) {                 \
    SGP_FOR_EACH_N(CALL)       \
    default:                   \
      return FAIL;             \
  }

template <>
bool split_exists<float>(int N) {
  return supported_n(N);
}

template <>
int split_elems_rt<float>(int N) {
#define SGP_CASE(NN) case NN: return split_elems<float, NN>();
  SGP_SWITCH(SGP_CASE, 0)
#undef SGP_CASE
}

template <>
cudaError_t prepare_xsplit<float>(int N, bool) {
#define SGP_CASE(NN) case NN: return xsplit_prepare_n<NN>();
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

template <>
cudaError_t prepare_lsplit<float>(int N, bool) {
#define SGP_CASE(NN) case NN: return lsplit_prepare_n<NN>();
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

template <>
cudaError_t launch_xsplit<float>(int N, bool, const XPassArgs<float>& a, int members, bool dependent,
                                 cudaStream_t s) {
#define SGP_CASE(NN) case NN: return xsplit_n<NN>(a, members, dependent, s);
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

template <>
cudaError_t launch_lsplit<float>(int N, bool, const LPassArgs<float>& a, int planes, int members, bool dependent,
                                 cudaStream_t s) {
#define SGP_CASE(NN) case NN: return lsplit_n<NN>(a, planes, members, dependent, s);
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

}  // namespace sgp
