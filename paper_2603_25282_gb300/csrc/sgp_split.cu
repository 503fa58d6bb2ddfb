// sgp_split.cu -- instantiation and launchers of the FP32 component-parallel
// passes; see sgp_split.cuh.
#include "sgp_split.cuh"

#include "sgp_launch.cuh"

namespace sgp {
namespace {

template <int N>
cudaError_t xsplit_prepare_n() {
  constexpr int E = split_elems<float, N>(), G = split_rows<float, N>();
  static std::atomic<int> done{-1};
  return opt_in(k_xsplit<float, N, E, G, false>, SplitCfg<float, N, E, G>::SMEM, done);
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
  static std::atomic<int> done{-1};
  return opt_in(k_lsplit<float, N, E, G, false, NoAdj>, SplitCfg<float, N, E, G>::SMEM, done);
}

template <int N>
cudaError_t lsplit_n(const LPassArgs<float>& a, int planes, int members, bool dependent, cudaStream_t s) {
  constexpr int E = split_elems<float, N>(), G = split_cols<float, N>();
  typedef SplitCfg<float, N, E, G> Cfg;
  const cudaError_t e = lsplit_prepare_n<N>();
  if (e != cudaSuccess) return e;
  return launch_pass(k_lsplit<float, N, E, G, false, NoAdj>, dim3((a.nx + G - 1) / G, planes, members), Cfg::THREADS, Cfg::SMEM,
                     dependent, s, a, NoAdj{});
}

// ---- the passes of a gradient ----
template <int N>
cudaError_t xadj_prepare_n() {
  constexpr int E = split_elems<float, N>(), G = split_rows<float, N>();
  static std::atomic<int> done{-1}, done_t{-1};
  const cudaError_t e = opt_in(k_xadj_split<float, N, E, G>, SplitCfg<float, N, E, G>::SMEM, done);
  if (e != cudaSuccess) return e;
  return opt_in(k_xsplit<float, N, E, G, true>, SplitCfg<float, N, E, G>::SMEM, done_t);
}
template <int N>
cudaError_t ladj_prepare_n() {
  constexpr int E = split_elems<float, N>(), G = split_cols<float, N>();
  static std::atomic<int> done{-1};
  return opt_in(k_lsplit<float, N, E, G, true, AdjHook<float>>, SplitCfg<float, N, E, G>::SMEM, done);
}
template <int N>
cudaError_t xtap_n(const XPassArgs<float>& a, int members, bool dependent, cudaStream_t s) {
  constexpr int E = split_elems<float, N>(), G = split_rows<float, N>();
  typedef SplitCfg<float, N, E, G> Cfg;
  const cudaError_t e = xadj_prepare_n<N>();
  if (e != cudaSuccess) return e;
  return launch_pass(k_xsplit<float, N, E, G, true>, dim3((a.rows + G - 1) / G, members), Cfg::THREADS, Cfg::SMEM,
                     dependent, s, a);
}
template <int N>
cudaError_t xadj_n(const XAdjArgs<float>& a, int members, bool dependent, cudaStream_t s) {
  constexpr int E = split_elems<float, N>(), G = split_rows<float, N>();
  typedef SplitCfg<float, N, E, G> Cfg;
  const cudaError_t e = xadj_prepare_n<N>();
  if (e != cudaSuccess) return e;
  return launch_pass(k_xadj_split<float, N, E, G>, dim3((a.rows + G - 1) / G, members), Cfg::THREADS, Cfg::SMEM,
                     dependent, s, a);
}
template <int N>
cudaError_t ladj_n(const LPassArgs<float>& a, const AdjHook<float>& h, int planes, int members, bool dependent,
                   cudaStream_t s) {
  constexpr int E = split_elems<float, N>(), G = split_cols<float, N>();
  typedef SplitCfg<float, N, E, G> Cfg;
  const cudaError_t e = ladj_prepare_n<N>();
  if (e != cudaSuccess) return e;
  return launch_pass(k_lsplit<float, N, E, G, true, AdjHook<float>>, dim3((a.nx + G - 1) / G, planes, members),
                     Cfg::THREADS, Cfg::SMEM, dependent, s, a, h);
}

}  // namespace

#define SGP_SWITCH(CALL, FAIL) \
  switch (N) {                 \
    SGP_FOR_EACH_N(CALL)       \
    default:                   \
      return FAIL;             \
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

cudaError_t prepare_adj_split(int NX, int NL) {
  auto x = [](int N) -> cudaError_t {
#define SGP_CASE(NN) case NN: return xadj_prepare_n<NN>();
    SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
  };
  auto l = [](int N) -> cudaError_t {
#define SGP_CASE(NN) case NN: return ladj_prepare_n<NN>();
    SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
  };
  const cudaError_t e = x(NX);
  return e != cudaSuccess ? e : l(NL);
}

cudaError_t launch_xsplit_tap(int N, const XPassArgs<float>& a, int members, bool dependent, cudaStream_t s) {
#define SGP_CASE(NN) case NN: return xtap_n<NN>(a, members, dependent, s);
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

cudaError_t launch_xadj_split(int N, const XAdjArgs<float>& a, int members, bool dependent, cudaStream_t s) {
#define SGP_CASE(NN) case NN: return xadj_n<NN>(a, members, dependent, s);
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

cudaError_t launch_lsplit_adj(int N, const LPassArgs<float>& a, const AdjHook<float>& h, int planes, int members,
                              bool dependent, cudaStream_t s) {
#define SGP_CASE(NN) case NN: return ladj_n<NN>(a, h, planes, members, dependent, s);
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

int xsplit_ctas(int N, int rows) {
#define SGP_CASE(NN) case NN: return (rows + split_rows<float, NN>() - 1) / split_rows<float, NN>();
  SGP_SWITCH(SGP_CASE, 0)
#undef SGP_CASE
}

int lsplit_tiles(int N, int nx) {
#define SGP_CASE(NN) case NN: return (nx + split_cols<float, NN>() - 1) / split_cols<float, NN>();
  SGP_SWITCH(SGP_CASE, 0)
#undef SGP_CASE
}

}  // namespace sgp
