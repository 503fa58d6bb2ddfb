// sgp_fix.cu -- instantiation, twiddles and launchers of the FP64 passes with
// fixed-point transforms; see sgp_fix.cuh.
#include "sgp_fix.cuh"

#include "sgp_launch.cuh"

namespace sgp {
namespace {

// ----------------------------------------------------------------------------
// twiddles to 2^-62: double-double arithmetic (a value is the unevaluated sum
// h + l), Taylor series on [0, pi/4] and the octant symmetries
// ----------------------------------------------------------------------------
struct DD { double h, l; };
__device__ __forceinline__ DD dd_norm(double a, double b) {
  const double s = a + b;
  return DD{s, b - (s - a)};
}
__device__ __forceinline__ DD dd_add(DD a, DD b) {
  const double s = a.h + b.h, t = s - a.h;
  const double e = (a.h - (s - t)) + (b.h - t);
  return dd_norm(s, e + a.l + b.l);
}
__device__ __forceinline__ DD dd_mul(DD a, DD b) {
  const double p = a.h * b.h;
  return dd_norm(p, fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
__device__ __forceinline__ DD dd_div(DD a, double d) {
  const double q = a.h / d;
  return dd_norm(q, (fma(-q, d, a.h) + a.l) / d);
}
// sin and cos of 2 pi k / n, 0 <= k <= n / 8
__device__ void dd_sincos(int k, int n, DD* s, DD* c) {
  const DD two_pi = {6.283185307179586, 2.4492935982947064e-16};
  const DD x = dd_mul(two_pi, dd_div(DD{(double)k, 0.0}, (double)n));
  const DD x2 = dd_mul(x, x);
  DD ts = x, tc = {1.0, 0.0};
  *s = x;
  *c = tc;
  for (int m = 1; m <= 14; ++m) {
    tc = dd_div(dd_mul(tc, x2), -(2.0 * m - 1.0) * (2.0 * m));
    ts = dd_div(dd_mul(ts, x2), -(2.0 * m) * (2.0 * m + 1.0));
    *c = dd_add(*c, tc);
    *s = dd_add(*s, ts);
  }
}
// h + l in units of 2^-62 as hi 2^32 + lo, lo signed and its negative
// representable
__device__ __forceinline__ void fix_store(DD v, int* hi, int* lo) {
  const double a = v.h * 0x1p62, r = rint(a);
  long long q = (long long)r + (long long)rint((a - r) + v.l * 0x1p62);
  if ((int)(unsigned)(unsigned long long)q == INT_MIN) ++q;
  *hi = fix_hi(q);
  *lo = fix_lo(q);
}

__global__ void k_fix_twiddles(int N, int E, FixTw* out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= N) return;
  int num = 0, den = 1, off = 0, ns = radix_at(N, E, 0), st = 1;
  while (true) {
    const int rd = radix_at(N, E, st);
    if (rd <= 0) break;                // past the table's last entry: 1
    const int cnt = (rd - 1) * ns;
    if (k < off + cnt) {
      const int r = (k - off) / ns + 1, j = (k - off) % ns;
      num = j * r;
      den = ns * rd;
      break;
    }
    off += cnt;
    ns *= rd;
    ++st;
  }
  // the angle 2 pi num / den in eighths of a turn: den is a multiple of 8 or
  // den / 8 need not be whole, so the octant is taken of 8 num
  num %= den;
  const int oct = 8 * num / den;                       // 0..7
  // reduced numerator over 8 den: the angle to the nearest quarter turn
  const int quarter = (oct + 1) / 2;                   // nearest multiple of a quarter turn
  int red = 4 * num - quarter * den;                   // over 4 den, |red| <= den / 2
  const bool neg = red < 0;
  if (neg) red = -red;
  DD s, c;
  dd_sincos(red, 4 * den, &s, &c);
  if (neg) s = DD{-s.h, -s.l};
  // rotate by the quarter turns
  DD cs = c, sn = s;
  const int q4 = quarter & 3;
  if (q4 == 1) {
    cs = DD{-s.h, -s.l};
    sn = c;
  } else if (q4 == 2) {
    cs = DD{-c.h, -c.l};
    sn = DD{-s.h, -s.l};
  } else if (q4 == 3) {
    cs = s;
    sn = DD{-c.h, -c.l};
  }
  FixTw w;
  fix_store(cs, &w.ch, &w.cl);
  fix_store(DD{-sn.h, -sn.l}, &w.sh, &w.sl);
  out[k] = w;
}

template <int N, int G>
cudaError_t xfix_prepare() {
  static std::atomic<int> done{-1};
  return opt_in(k_xfix<N, G>, FixCfg<N, G>::SMEM, done);
}
template <int N, int G>
cudaError_t lfix_prepare() {
  static std::atomic<int> done{-1};
  return opt_in(k_lfix<N, G>, FixCfg<N, G>::SMEM, done);
}

template <int N, int G>
cudaError_t xfix(const XPassArgs<double>& a, int members, bool dependent, cudaStream_t s) {
  const cudaError_t e = xfix_prepare<N, G>();
  if (e != cudaSuccess) return e;
  return launch_pass(k_xfix<N, G>, dim3((a.rows + G - 1) / G, members), FixCfg<N, G>::THREADS, FixCfg<N, G>::SMEM,
                     dependent, s, a);
}
template <int N, int G>
cudaError_t lfix(const LPassArgs<double>& a, int planes, int members, bool dependent, cudaStream_t s) {
  const cudaError_t e = lfix_prepare<N, G>();
  if (e != cudaSuccess) return e;
  return launch_pass(k_lfix<N, G>, dim3((a.nx + G - 1) / G, planes, members), FixCfg<N, G>::THREADS,
                     FixCfg<N, G>::SMEM, dependent, s, a);
}

}  // namespace

#define SGP_SWITCH(CALL, FAIL) \
  switch (N) {                 \
    SGP_FOR_EACH_N(CALL)            \
    default:                   \
      return FAIL;             \
  }

cudaError_t launch_fix_twiddles(int N, FixTw* out, cudaStream_t s) {
  int E = 0;
  switch (N) {
#define SGP_CASE(NN) case NN: E = fix_elems<NN>(); break;
    SGP_FOR_EACH_N(SGP_CASE)
#undef SGP_CASE
    default: return cudaErrorInvalidValue;
  }
  k_fix_twiddles<<<(N + 63) / 64, 64, 0, s>>>(N, E, out);
  return cudaGetLastError();
}

template <>
cudaError_t prepare_xsplit<double>(int N, bool many) {
#define SGP_CASE(NN) case NN: return many ? xfix_prepare<NN, fix_lines<NN>(true)>() : xfix_prepare<NN, 1>();
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

template <>
cudaError_t prepare_lsplit<double>(int N, bool many) {
#define SGP_CASE(NN) case NN: return many ? lfix_prepare<NN, fix_lines<NN>(true)>() : lfix_prepare<NN, 1>();
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

template <>
cudaError_t launch_xsplit<double>(int N, bool many, const XPassArgs<double>& a, int members, bool dependent,
                                  cudaStream_t s) {
#define SGP_CASE(NN)                                                                          \
  case NN:                                                                                    \
    return many ? xfix<NN, fix_lines<NN>(true)>(a, members, dependent, s)                     \
                : xfix<NN, 1>(a, members, dependent, s);
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

template <>
cudaError_t launch_lsplit<double>(int N, bool many, const LPassArgs<double>& a, int planes, int members,
                                  bool dependent, cudaStream_t s) {
#define SGP_CASE(NN)                                                                          \
  case NN:                                                                                    \
    return many ? lfix<NN, fix_lines<NN>(true)>(a, planes, members, dependent, s)             \
                : lfix<NN, 1>(a, planes, members, dependent, s);
  SGP_SWITCH(SGP_CASE, cudaErrorInvalidValue)
#undef SGP_CASE
}

}  // namespace sgp
