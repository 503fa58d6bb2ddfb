// sgp_split.cu -- instantiation and launchers of the component-parallel passes
// for one precision (SGP_REAL); see sgp_split.cuh.
#include "sgp_split.cuh"

#include "sgp_launch.cuh"

#ifndef SGP_REAL
#error "define SGP_REAL (float or double)"
#endif

namespace sgp {
namespace {

typedef SGP_REAL Real;

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
  if constexpr (split_has<Real, N>()) {
    constexpr int E = split_elems<Real, N>(), G = split_rows<Real, N>();
    static int done = -1;
    return opt_in(k_xsplit<Real, N, E, G, false>, SplitCfg<Real, N, E, G>::SMEM, &done);
  } else {
    return cudaErrorInvalidValue;
  }
}

template <int N>
cudaError_t xsplit_n(const XPassArgs<Real>& a, int members, bool dependent, cudaStream_t s) {
  if constexpr (split_has<Real, N>()) {
    constexpr int E = split_elems<Real, N>(), G = split_rows<Real, N>();
    typedef SplitCfg<Real, N, E, G> Cfg;
    const cudaError_t e = xsplit_prepare_n<N>();
    if (e != cudaSuccess) return e;
    return launch_pass(k_xsplit<Real, N, E, G, false>, dim3((a.rows + G - 1) / G, members), Cfg::THREADS, Cfg::SMEM,
                  dependent, s, a);
  } else {
    return cudaErrorInvalidValue;
  }
}

template <int N>
cudaError_t lsplit_prepare_n() {
  if constexpr (split_has<Real, N>()) {
    constexpr int E = split_elems<Real, N>(), G = split_cols<Real, N>();
    static int done = -1;
    return opt_in(k_lsplit<Real, N, E, G>, SplitCfg<Real, N, E, G>::SMEM, &done);
  } else {
    return cudaErrorInvalidValue;
  }
}

template <int N>
cudaError_t lsplit_n(const LPassArgs<Real>& a, int planes, int members, bool dependent, cudaStream_t s) {
  if constexpr (split_has<Real, N>()) {
    constexpr int E = split_elems<Real, N>(), G = split_cols<Real, N>();
    typedef SplitCfg<Real, N, E, G> Cfg;
    const cudaError_t e = lsplit_prepare_n<N>();
    if (e != cudaSuccess) return e;
    return launch_pass(k_lsplit<Real, N, E, G>, dim3((a.nx + G - 1) / G, planes, members), Cfg::THREADS, Cfg::SMEM,
                  dependent, s, a);
  } else {
    return cudaErrorInvalidValue;
  }
}

}  // namespace

#define SGP_SWITCH(CALL, FAIL) \
  switch (N) {                 \
    SGP_FOR_EACH_N(CALL)       \
    default:                   \
      return FAIL;             \
  }

template <>
bool split_exists<Real>(int N) {
#define SGP_CASE(NN) case NN: return split_has<Real, NN>();
  SGP_SWITCH(SGP_CASE, false)
#undef SGP_CASE
}

template <>
int split_elems_rt<Real>(int N) {
#define SGP_CASE(NN) case NN: return split_elems<Real, NN>();
  SGP_SWITCH(SGP_CASE, 0)
#undef SGP_CASE
}

template <>
cudaError_t prepare_xsplit<Real>(int N) {
#define SGP_CASE(NN) case NN: return xsplit_prepare_n<NN>();
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

template <>
cudaError_t prepare_lsplit<Real>(int N) {
#define SGP_CASE(NN) case NN: return lsplit_prepare_n<NN>();
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

template <>
cudaError_t launch_xsplit<Real>(int N, const XPassArgs<Real>& a, int members, bool dependent, cudaStream_t s) {
#define SGP_CASE(NN) case NN: return xsplit_n<NN>(a, members, dependent, s);
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

template <>
cudaError_t launch_lsplit<Real>(int N, const LPassArgs<Real>& a, int planes, int members, bool dependent,
                                cudaStream_t s) {
#define SGP_CASE(NN) case NN: return lsplit_n<NN>(a, planes, members, dependent, s);
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

}  // namespace sgp
