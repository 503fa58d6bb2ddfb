// sgp_fix.cuh -- FP64 passes with their transforms in 64-bit fixed point.
//
// The FP64 pipe of this GPU runs at 1/64 of the FP32 and integer rates (two
// results per clock and SM), and the transforms of a pass are more than half
// of its FP64 operations.  They are linear and keep the norm of a line, so
// they need no exponent per value: here a line is brought to integers with
// one common exponent, transformed in 64-bit integer arithmetic (an addition
// is two instructions, a complex twiddle product twelve 32 x 32 -> 64 bit
// multiply-adds), and brought back to doubles.  The common exponent follows
// the line from stage to stage, so that its largest value has a modulus of 2^56
// or more before every butterfly.  A line enters with 58 bits for its largest
// component and 58 - k for one 2^-k of it, truncated; a twiddle product errs by
// up to 1.5 units, one by sqrt(1/2) or sqrt(3)/2 by up to 2.5, and the floors add
// up: an element of a random line of 768 comes out off by up to 2^-52.4 of the
// line's largest value.  In relative L2 a transform is closer to the exact one
// than in FP64 (an emulation of the integers: 2e-17 to 6e-17 for random lines, up
// to 1.3e-16 for smooth ones of 768 and 1024; FP64 1.4e-16 to 2.4e-16).  The
// pointwise flow and the mode mix stay in FP64, with fewer operations than the
// forms that FP32 shares (flow_point, mix_mode).
//
// Measured (GB300; relative L2 of a forward and inverse 2D transform, and us
// per launch): 256^2 3.3e-16 in FP64, 1.0e-16 here; 192 x 128 4.0e-16, 1.4e-16.
// 512^2, one member: x-pass 467 -> 281 (the FP64 pipe 71% busy, 380 of its
// operations a point instead of 783), line pass 302 -> 188 (55%; 191 of 510; the
// rest is integer issue between the pipe's phases); 96 x 64 x 48: x-pass 645 ->
// 272, y-lines, without a mix, 61 -> 21, z-lines 248 -> 155.
//
// Work split as in sgp_split.cuh: a line of one component to T threads (of one
// warp up to T = 32), the points (modes) shared out over all threads.  A line whose
// input is not finite comes out as NaN.
#pragma once
#include "sgp_split.cuh"

namespace sgp {

// ----------------------------------------------------------------------------
// radix 3 and 6 butterflies in integers (2, 4 and 8 are those of sgp_fft.cuh)
// ----------------------------------------------------------------------------
template <int DIR> struct Dft<3, DIR, longlong2> {
  __device__ __forceinline__ static void run(longlong2 (&x)[3]) {
    const longlong2 t = cadd(x[1], x[2]), u = csub(x[1], x[2]);
    const longlong2 m = mkc(x[0].x - (t.x >> 1), x[0].y - (t.y >> 1));
    const long long sx = mul_rt3_half(u.x), sy = mul_rt3_half(u.y);
    const longlong2 iu = DIR < 0 ? mkc(sy, -sx) : mkc(-sy, sx);
    x[0] = cadd(x[0], t);
    x[1] = cadd(m, iu);
    x[2] = csub(m, iu);
  }
};
template <int DIR> struct Dft<6, DIR, longlong2> {
  __device__ __forceinline__ static void run(longlong2 (&x)[6]) {
    longlong2 e[3] = {x[0], x[2], x[4]};
    longlong2 o[3] = {x[1], x[3], x[5]};
    Dft<3, DIR, longlong2>::run(e);
    Dft<3, DIR, longlong2>::run(o);
    // W6^1 = 1/2 -+ i s3, W6^2 = -1/2 -+ i s3
    constexpr int sg = DIR < 0 ? -1 : 1;
    const longlong2 o1 = mkc((o[1].x >> 1) - sg * mul_rt3_half(o[1].y), (o[1].y >> 1) + sg * mul_rt3_half(o[1].x));
    const longlong2 o2 = mkc(-(o[2].x >> 1) - sg * mul_rt3_half(o[2].y), -(o[2].y >> 1) + sg * mul_rt3_half(o[2].x));
    x[0] = cadd(e[0], o[0]);
    x[3] = csub(e[0], o[0]);
    x[1] = cadd(e[1], o1);
    x[4] = csub(e[1], o1);
    x[2] = cadd(e[2], o2);
    x[5] = csub(e[2], o2);
  }
};

// Twiddle exp(-2 pi i j r / (NS RD)) in units of 2^-62: (cos, -sin), each
// as hi 2^32 + lo with lo signed.  Table order as in sgp_fft.cuh.
struct FixTw { int ch, cl, sh, sl; };
static_assert(sizeof(FixTw) == sizeof(TwE<double>), "one table entry size");

// x W / 4 (W conjugated for DIR > 0).  The low halves' products are left out
// (below one unit); |x| < 2^62 componentwise keeps every sum in 64 bits.
template <int DIR>
__device__ __forceinline__ longlong2 fix_twiddle(longlong2 x, FixTw w) {
  const int rh = fix_hi(x.x), rl = fix_lo(x.x), ih = fix_hi(x.y), il = fix_lo(x.y);
  const int sh = DIR < 0 ? w.sh : -w.sh, sl = DIR < 0 ? w.sl : -w.sl;
  const int nh = -sh, nl = -sl;
  long long tr = (long long)rl * w.ch, ti = (long long)rl * sh;
  tr = mad_wide(rh, w.cl, tr);
  ti = mad_wide(rh, sl, ti);
  tr = mad_wide(il, nh, tr);
  ti = mad_wide(il, w.ch, ti);
  tr = mad_wide(ih, nl, tr);
  ti = mad_wide(ih, w.cl, ti);
  long long r = mad_wide(rh, w.ch, tr >> 32);
  long long i = mad_wide(rh, sh, ti >> 32);
  r = mad_wide(ih, nh, r);
  i = mad_wide(ih, w.ch, i);
  return mkc(r, i);
}

// ----------------------------------------------------------------------------
// doubles to integers of a common exponent and back
// ----------------------------------------------------------------------------
// A line's components start below 2^kFixStart and are brought below 2^kFixTw
// (the largest to half of that or more) before each twiddle stage, so below
// 2^57.5 before its butterflies: radix 8 stays below 8 sqrt2 2^58 < 2^62, which
// the twiddle product of the next stage accepts.
constexpr int kFixStart = 58, kFixTw = 59;
constexpr int kFixBad = 1 << 20;        // exponent of a line that is not finite

__device__ __forceinline__ int fix_exp(double d) { return (__double2hiint(d) >> 20) & 0x7ff; }

// d / 2^(emax - 1022 - kFixStart) for |d| < 2^(emax - 1022): below 2^kFixStart
__device__ __forceinline__ long long fix_from(double d, int emax) {
  const int hi = __double2hiint(d);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned mh = (unsigned)(hi & 0xfffff) | (e ? 0x100000u : 0u);
  const unsigned long long m = ((unsigned long long)mh << 32 | (unsigned)__double2loint(d)) << (kFixStart - 53);
  int sh = emax - (e ? e : 1);
  sh = sh > 63 ? 63 : sh;
  const long long q = (long long)(m >> sh);
  const long long s = (long long)hi >> 63;
  return (q ^ s) - s;
}

// q 2^ex, rounded to nearest (ties away).  Exponents near the ends of the
// range, and a line that is not finite, take the second branch.
__device__ __forceinline__ double fix_to(long long q, int ex) {
  if (ex >= -1022 && ex <= 959) {
    const long long s = q >> 63;
    unsigned long long m = (unsigned long long)((q ^ s) - s);
    const int lz = __clzll((long long)m);
    const unsigned long long n = m << (lz & 63);
    const unsigned long long b = ((unsigned long long)(unsigned)(ex + 63 - lz + 1022) << 52) + (n >> 11) + ((n >> 10) & 1);
    return __longlong_as_double((long long)((m ? b : 0) | ((unsigned long long)s & 0x8000000000000000ull)));
  }
  if (ex >= kFixBad) return __longlong_as_double(0x7ff8000000000000LL);
  const int a = ex / 2, c = ex - a;
  return (double)q * __longlong_as_double((long long)(a + 1023) << 52) * __longlong_as_double((long long)(c + 1023) << 52);
}

// ----------------------------------------------------------------------------
// the transform
// ----------------------------------------------------------------------------
// Lines of up to 32 threads lie in one warp (threads side by side for G = 1,
// every G-th of G T when G lines are interleaved); longer ones are two warps
// (G = 1), which meet at named barrier `bid` and through two words `red`.
struct FixLine {
  int bid;
  unsigned* red;
};
template <int T>
__device__ __forceinline__ void fix_sync(const FixLine& l) {
  if constexpr (T <= 32) __syncwarp();
  else group_sync<T>(l.bid);
}
// bitwise or, and maximum, over the line of the calling thread; the words are
// free again after the line's next barrier
template <int T, int G>
__device__ __forceinline__ unsigned fix_line_or(unsigned v, const FixLine& l) {
#pragma unroll
  for (int o = G; o < (G * T < 32 ? G * T : 32); o *= 2) v |= __shfl_xor_sync(0xffffffffu, v, o);
  if constexpr (T > 32) {
    if ((threadIdx.x & 31) == 0) l.red[(threadIdx.x >> 5) & 1] = v;
    fix_sync<T>(l);
    v = l.red[0] | l.red[1];
  }
  return v;
}
template <int T, int G>
__device__ __forceinline__ int fix_line_max(int v, const FixLine& l) {
#pragma unroll
  for (int o = G; o < (G * T < 32 ? G * T : 32); o *= 2) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if constexpr (T > 32) {
    if ((threadIdx.x & 31) == 0) l.red[(threadIdx.x >> 5) & 1] = (unsigned)v;
    fix_sync<T>(l);
    v = max((int)l.red[0], (int)l.red[1]);
  }
  return v;
}

// Stages S.. of the transform of a line whose thread i holds elements i + T e
// in v; top: the or of the components' magnitudes' high words after the last
// stage, ex: the line's exponent.  b: the line's exchange buffer.
template <int N, int E, int DIR, int G, int S, int NS>
struct FixStages {
  __device__ __forceinline__ static void run(longlong2 (&v)[E], int i, const FixTw* tw, longlong2* b,
                                             const FixLine& l, int& ex) {
    constexpr int RD = radix_at(N, E, S);
    if constexpr (RD > 0) {
      constexpr int T = N / E;
      constexpr int B = E / RD;
      constexpr bool LAST = (NS * RD == N);
      constexpr int TOFF = tw_offset(N, E, S);
      if constexpr (S > 0) {
        // the line to kFixTw bits for its largest component (a shift up is
        // exact; where no line of the warp needs one it is skipped): the
        // twiddle product of a value below 2^kFixTw is below 2^(kFixTw - 1.5)
        unsigned m = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int hx = (int)(v[e].x >> 32), hy = (int)(v[e].y >> 32);
          m |= (unsigned)(hx ^ (hx >> 31)) | (unsigned)(hy ^ (hy >> 31));
        }
        m = fix_line_or<T, G>(m, l);
        const int L = 64 - __clz((int)m);
        const int up = L < kFixTw ? kFixTw - L : 0, down = L > kFixTw ? L - kFixTw : 0;
        ex += 2 + down - up;
        if (__any_sync(0xffffffffu, up != 0)) {
#pragma unroll
          for (int e = 0; e < E; ++e) v[e] = mkc(v[e].x << up, v[e].y << up);
        }
        if (__any_sync(0xffffffffu, down != 0)) {
          const long long half = (1LL << down) >> 1;
#pragma unroll
          for (int e = 0; e < E; ++e) v[e] = mkc((v[e].x + half) >> down, (v[e].y + half) >> down);
        }
#pragma unroll
        for (int k = 0; k < B; ++k) {
          const int j = (i + T * k) % NS;
          v[k] = mkc((v[k].x + 2) >> 2, (v[k].y + 2) >> 2);
#pragma unroll
          for (int r = 1; r < RD; ++r) v[k + r * B] = fix_twiddle<DIR>(v[k + r * B], tw[TOFF + (r - 1) * NS + j]);
        }
      }
#pragma unroll
      for (int k = 0; k < B; ++k) {
        longlong2 x[RD];
#pragma unroll
        for (int r = 0; r < RD; ++r) x[r] = v[k + r * B];
        Dft<RD, DIR, longlong2>::run(x);
#pragma unroll
        for (int r = 0; r < RD; ++r) v[k + r * B] = x[r];
      }
      if constexpr (!LAST) {
        fix_sync<T>(l);                 // earlier reads of the buffer are done
#pragma unroll
        for (int k = 0; k < B; ++k) {
          const int q = i + T * k;
          const int d = (q / NS) * NS * RD + (q % NS);
          // one slot in nine is padding: the offsets are constants where NS is a
          // multiple of 8, or d is and r stays below 8
          constexpr bool LIN = NS % 8 == 0 || (NS == 1 && RD == 8);
#pragma unroll
          for (int r = 0; r < RD; ++r)
            b[LIN ? padx<double>(d) + r * NS + (NS % 8 == 0 ? r * (NS / 8) : 0) : padx<double>(d + r * NS)] = v[k + r * B];
        }
        fix_sync<T>(l);
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = b[T % 8 == 0 ? padx<double>(i) + e * (T + T / 8) : padx<double>(i + T * e)];
        FixStages<N, E, DIR, G, S + 1, NS * RD>::run(v, i, tw, b, l, ex);
      }
    }
  }
};

// The transform of the calling thread's line, doubles in and out (layout as
// in sgp_fft.cuh, no normalisation).  Whole warps call it.
template <int N, int E, int DIR, int G>
__device__ __forceinline__ void fix_fft(double2 (&v)[E], int i, const FixTw* tw, double2* buf, const FixLine& l) {
  constexpr int T = N / E;
  static_assert(plan_ok(N, E) && ((T * G <= 32 && 32 % (T * G) == 0) || (T == 64 && G == 1)),
                "fixed-point transform: lines within a warp, or of two");
  if constexpr (T > 32) fix_sync<T>(l);   // the words of an earlier transform have been read
  int emax = 1;
#pragma unroll
  for (int e = 0; e < E; ++e) emax = max(emax, max(fix_exp(v[e].x), fix_exp(v[e].y)));
  emax = fix_line_max<T, G>(emax, l);
  longlong2 q[E];
#pragma unroll
  for (int e = 0; e < E; ++e) q[e] = mkc(fix_from(v[e].x, emax), fix_from(v[e].y, emax));
  int ex = emax == 0x7ff ? kFixBad : emax - 1022 - kFixStart;
  FixStages<N, E, DIR, G, 0, 1>::run(q, i, tw, reinterpret_cast<longlong2*>(buf), l, ex);
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = make_double2(fix_to(q[e].x, ex), fix_to(q[e].y, ex));
}

// ----------------------------------------------------------------------------
// the nonlinear flow at one point and the linear flow of one mode, FP64
// ----------------------------------------------------------------------------
// (K t) for K = k.f with the real kz and complex kp = kx + i ky, sk = sqrt6/2 kp
// (spin-2 matrices of Sec. 1): tridiagonal, see spin_dot.
__device__ __forceinline__ void fix_spin_dot(double kz, double2 kp, double2 sk, const double2 (&t)[5],
                                             double2 (&o)[5]) {
  const double k2 = 2.0 * kz;
  o[0] = mkc(fma(kp.y, t[1].y, fma(kp.x, t[1].x, k2 * t[0].x)), fma(-kp.y, t[1].x, fma(kp.x, t[1].y, k2 * t[0].y)));
  o[1] = mkc(fma(sk.y, t[2].y, fma(sk.x, t[2].x, fma(-kp.y, t[0].y, fma(kp.x, t[0].x, kz * t[1].x)))),
             fma(-sk.y, t[2].x, fma(sk.x, t[2].y, fma(kp.y, t[0].x, fma(kp.x, t[0].y, kz * t[1].y)))));
  o[2] = mkc(fma(sk.y, t[3].y, fma(sk.x, t[3].x, fma(-sk.y, t[1].y, sk.x * t[1].x))),
             fma(-sk.y, t[3].x, fma(sk.x, t[3].y, fma(sk.y, t[1].x, sk.x * t[1].y))));
  o[3] = mkc(fma(kp.y, t[4].y, fma(kp.x, t[4].x, fma(-sk.y, t[2].y, fma(sk.x, t[2].x, -kz * t[3].x)))),
             fma(-kp.y, t[4].x, fma(kp.x, t[4].y, fma(sk.y, t[2].x, fma(sk.x, t[2].y, -kz * t[3].y)))));
  o[4] = mkc(fma(-kp.y, t[3].y, fma(kp.x, t[3].x, -k2 * t[4].x)), fma(kp.y, t[3].x, fma(kp.x, t[3].y, -k2 * t[4].y)));
}

// Constants of the flow over delta for one member.
struct FlowPrm {
  double ph, k1, k2;        // delta (c0 + c2/5), delta c1, delta c2/5
};

// Exact nonlinear flow over delta at one point (Sec. 3.2, Eq. (solution2)): the
// singlet rotation, exp(-i c1 delta F.f), the scalar phase, applied as
// v + increment as in nonlinear_point; dV = delta V.  About 360 FP64
// operations instead of 520: angles that are small take their Taylor series,
// each to a remainder below 1e-17 (no square root, no SU(2) factors), others
// the library's sine and cosine and the SU(2) image (spin_rotation); products
// share their terms.
__device__ __forceinline__ void flow_point(double2 (&v)[5], double dV, const FlowPrm& P) {
  const double r6h = 1.22474487139158904910;
  const double a0 = cabs2(v[0]), a1 = cabs2(v[1]), a3 = cabs2(v[3]), a4 = cabs2(v[4]);
  const double rho = ((a0 + a4) + (a1 + a3)) + cabs2(v[2]);
  const double Fz = fma(2.0, a0 - a4, a1 - a3);
  // F+ / 2 = conj(v0) v1 + conj(v3) v4 + sqrt6/2 (conj(v1) v2 + conj(v2) v3)
  double hx = v[1].x * v[2].x, hy = v[1].x * v[2].y;
  hx = fma(v[1].y, v[2].y, hx);
  hy = fma(-v[1].y, v[2].x, hy);
  hx = fma(v[2].x, v[3].x, hx);
  hy = fma(v[2].x, v[3].y, hy);
  hx = fma(v[2].y, v[3].y, hx);
  hy = fma(-v[2].y, v[3].x, hy);
  double gx = v[0].x * v[1].x, gy = v[0].x * v[1].y;
  gx = fma(v[0].y, v[1].y, gx);
  gy = fma(-v[0].y, v[1].x, gy);
  gx = fma(v[3].x, v[4].x, gx);
  gy = fma(v[3].x, v[4].y, gy);
  gx = fma(v[3].y, v[4].y, gx);
  gy = fma(-v[3].y, v[4].x, gy);
  gx = fma(r6h, hx, gx);
  gy = fma(r6h, hy, gy);
  // A = sqrt5 A00 = 2 (v0 v4 - v1 v3) + v2^2
  double ax = v[0].x * v[4].x, ay = v[0].x * v[4].y;
  ax = fma(-v[0].y, v[4].y, ax);
  ay = fma(v[0].y, v[4].x, ay);
  ax = fma(-v[1].x, v[3].x, ax);
  ay = fma(-v[1].x, v[3].y, ay);
  ax = fma(v[1].y, v[3].y, ax);
  ay = fma(-v[1].y, v[3].x, ay);
  ay = 2.0 * fma(v[2].x, v[2].y, ay);
  ax = fma(2.0, ax, fma(-v[2].y, v[2].y, v[2].x * v[2].x));
  // (1) b = cos th v + i (sin th / th) k2 (rho v - A A' conj v), th = k2 D,
  //     D^2 = rho^2 - |A|^2, with A' conj v = (conj v4, -conj v3, conj v2, -conj v1, conj v0)
  double D2 = fma(-ay, ay, fma(-ax, ax, rho * rho));
  D2 = D2 > 0.0 ? D2 : 0.0;
  const double x1 = P.k2 * P.k2 * D2;
  double cm, sn;             // cos th - 1, sin th / th
  if (x1 < 0x1p-10) {
    cm = x1 * fma(x1, fma(x1, fma(x1, 1.0 / 40320.0, -1.0 / 720.0), 1.0 / 24.0), -0.5);
    sn = fma(x1, fma(x1, fma(x1, fma(x1, 1.0 / 362880.0, -1.0 / 5040.0), 1.0 / 120.0), -1.0 / 6.0), 1.0);
  } else {
    const double th = sqrt(x1);
    double sh, ch;
    sincos(0.5 * th, &sh, &ch);
    cm = -2.0 * sh * sh;
    sn = 2.0 * sh * ch / th;
  }
  sn *= P.k2;
  const double al = sn * rho, bx = -sn * ay, by = sn * ax;       // be = i sn A
  double2 inc[5], b[5];
  {
    const double2 ac[5] = {cconj(v[4]), cneg(cconj(v[3])), cconj(v[2]), cneg(cconj(v[1])), cconj(v[0])};
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      inc[k] = mkc(fma(-bx, ac[k].x, fma(by, ac[k].y, fma(-al, v[k].y, cm * v[k].x))),
                   fma(-bx, ac[k].y, fma(-by, ac[k].x, fma(al, v[k].x, cm * v[k].y))));
      b[k] = cadd(v[k], inc[k]);
    }
  }
  // (2) e = (exp(-iK) - 1) b, K = k1 F.f, |K| = 2 k1 |F|: the Taylor polynomial
  //     whose remainder |K|^(n+1)/(n+1)! is below 1e-17, in Horner's form
  const double kz = P.k1 * Fz;
  const double2 kp = mkc(2.0 * P.k1 * gx, 2.0 * P.k1 * gy);
  const double K2 = 4.0 * fma(kz, kz, fma(kp.x, kp.x, kp.y * kp.y));
  const int n = K2 <= 1.21e-8 ? 3 : K2 <= 1.0e-6 ? 4 : K2 <= 1.76e-5 ? 5 : K2 <= 1.21e-4 ? 6 : 0;
  double2 t[5];
  if (n > 0) {
    const double2 sk = mkc(r6h * kp.x, r6h * kp.y);
    double2 o[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) t[k] = b[k];
#pragma unroll 1
    for (int j = n; j > 1; --j) {
      const double f = j == 2 ? 0.5 : j == 3 ? 1.0 / 3.0 : j == 4 ? 0.25 : j == 5 ? 0.2 : 1.0 / 6.0;
      fix_spin_dot(f * kz, mkc(f * kp.x, f * kp.y), mkc(f * sk.x, f * sk.y), t, o);
#pragma unroll
      for (int k = 0; k < 5; ++k) t[k] = mkc(b[k].x + o[k].y, b[k].y - o[k].x);
    }
    fix_spin_dot(kz, kp, sk, t, o);
#pragma unroll
    for (int k = 0; k < 5; ++k) t[k] = mkc(o[k].y, -o[k].x);
  } else {
    SpinRot<double> sr;
#pragma unroll
    for (int k = 0; k < 5; ++k) t[k] = mkc(0.0, 0.0);
    if (spin_rotation<double>(Fz, mkc(2.0 * gx, 2.0 * gy), P.k1, 1.0, sr))
      spin2_increment<double>(b, sr.am1, sr.bhat, sr.cpm1, sr.sp, t);
  }
  // (3) exp(-i ph) - 1, ph = delta V + delta (c0 + c2/5) rho
  const double ph = fma(P.ph, rho, dV);
  double c, s;               // cos ph - 1, sin ph
  if (fabs(ph) < 0.25) {
    const double x = ph * ph;
    c = x * fma(x, fma(x, fma(x, fma(x, fma(x, 1.0 / 479001600.0, -1.0 / 3628800.0), 1.0 / 40320.0), -1.0 / 720.0),
                       1.0 / 24.0), -0.5);
    s = ph * fma(x, fma(x, fma(x, fma(x, fma(x, fma(x, 1.0 / 6227020800.0, -1.0 / 39916800.0), 1.0 / 362880.0),
                                      -1.0 / 5040.0), 1.0 / 120.0), -1.0 / 6.0), 1.0);
  } else {
    double sh, ch;
    sincos(0.5 * ph, &sh, &ch);
    c = -2.0 * sh * sh;
    s = 2.0 * sh * ch;
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const double2 be = cadd(b[k], t[k]), q = cadd(inc[k], t[k]);
    v[k] = mkc(v[k].x + fma(s, be.y, fma(c, be.x, q.x)), v[k].y + fma(-s, be.x, fma(c, be.y, q.y)));
  }
}

// Linear flow of one mode with its table entry, kinetic factor 1 + kh and the
// 1/(NX NY [NZ]) of the forward transforms (inv): v <- (v + e + kh (v + e)) inv,
// e = (D - I) v, D - I = diag(w^m) (d - I) diag(z^m) + diag(ahat^(2m) - 1) as in
// spin2_increment.  d is the rotation by beta (cos beta = c^2 - s^2) of spin 2: on
// u0 + u4, u1 - u3, u2 and on u0 - u4, u1 + u3 it is a 3 x 3 and a 2 x 2 block.
// About 180 FP64 operations against 230 in mix_entry.
__device__ __forceinline__ void mix_mode(double2 (&v)[5], const ModeEntry<double>& m, int ps, int qs, double2 kh,
                                         double inv) {
  const double r6 = 2.44948974278317809820;
  const double ar = 1.0 + m.am1r, ai = m.am1i;
  const double bx = ps < 0 ? -m.bx : m.bx, by = qs < 0 ? m.by : -m.by;
  const double p1 = ar * bx, p3 = ar * by;
  const double2 w = mkc(fma(-ai, by, p1), fma(ai, bx, p3));      // ahat bhat
  const double2 z = mkc(fma(ai, by, p1), fma(ai, bx, -p3));      // ahat conj(bhat)
  const double2 z2 = mkc(fma(-z.y, z.y, z.x * z.x), 2.0 * z.x * z.y);
  const double2 wh = mkc(0.5 * w.x, 0.5 * w.y);                  // w / 2, w^2 / 2
  const double2 w2h = mkc(fma(-wh.y, w.y, wh.x * w.x), 2.0 * wh.x * w.y);
  const double2 am1 = mkc(m.am1r, m.am1i);
  const double2 g2 = cmul(am1, mkc(2.0 + am1.x, am1.y));         // ahat^2 - 1
  const double2 g4 = cmul(g2, mkc(2.0 + g2.x, g2.y));            // ahat^4 - 1
  const double2 u0 = cmul(z2, v[0]), u1 = cmul(z, v[1]), u2 = v[2];
  const double2 u3 = cmulc(v[3], z), u4 = cmulc(v[4], z2);
  const double2 sp = cadd(u0, u4), sm = csub(u0, u4), tp = cadd(u1, u3), tm = csub(u1, u3);
  const double cbm = -2.0 * m.sp * m.sp;                         // cos beta - 1
  const double sb = 2.0 * m.sp * (1.0 + m.cm1);                  // sin beta
  const double q = sb * sb, sc = fma(sb, cbm, sb);
  const double R = 0.25 * r6 * q, S = 0.5 * r6 * sc;
  // twice the rows 0 +- 4 and 1 -+ 3 of (d - I) u; row 2
  const double2 e0 = caxpy(caxpy(cscale(sp, -0.5 * q), tm, sc), u2, 2.0 * R);
  const double2 e1 = caxpy(caxpy(cscale(tm, -2.0 * q), sp, -sc), u2, 2.0 * S);
  const double2 o2 = caxpy(caxpy(cscale(u2, -1.5 * q), sp, R), tm, -S);
  const double2 f0 = caxpy(cscale(sm, cbm), tp, sb);
  const double2 f1 = caxpy(cscale(tp, cbm), sm, -sb);
  double2 e[5];
  {
    const double2 y0 = cadd(e0, f0), y1 = cadd(f1, e1), y3 = csub(f1, e1), y4 = csub(e0, f0);
    e[0] = mkc(fma(-w2h.y, y0.y, fma(w2h.x, y0.x, fma(-g4.y, v[0].y, g4.x * v[0].x))),
               fma(w2h.y, y0.x, fma(w2h.x, y0.y, fma(g4.y, v[0].x, g4.x * v[0].y))));
    e[1] = mkc(fma(-wh.y, y1.y, fma(wh.x, y1.x, fma(-g2.y, v[1].y, g2.x * v[1].x))),
               fma(wh.y, y1.x, fma(wh.x, y1.y, fma(g2.y, v[1].x, g2.x * v[1].y))));
    e[2] = o2;
    e[3] = mkc(fma(wh.y, y3.y, fma(wh.x, y3.x, fma(g2.y, v[3].y, g2.x * v[3].x))),
               fma(-wh.y, y3.x, fma(wh.x, y3.y, fma(-g2.y, v[3].x, g2.x * v[3].y))));
    e[4] = mkc(fma(w2h.y, y4.y, fma(w2h.x, y4.x, fma(g4.y, v[4].y, g4.x * v[4].x))),
               fma(-w2h.y, y4.x, fma(w2h.x, y4.y, fma(-g4.y, v[4].x, g4.x * v[4].y))));
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const double2 x = cadd(v[k], e[k]);
    v[k] = mkc(inv * (v[k].x + fma(-kh.y, x.y, fma(kh.x, x.x, e[k].x))),
               inv * (v[k].y + fma(kh.y, x.x, fma(kh.x, x.y, e[k].y))));
  }
}

// ----------------------------------------------------------------------------
// geometry
// ----------------------------------------------------------------------------
// Elements per thread: radix 8 stages (16 elements from 512 on, so that a line
// of 512 stays within a warp), radix 6 then 4s for N = 3*2^k.
template <int N>
constexpr int fix_elems() { return N % 3 == 0 ? 12 : N >= 512 ? 16 : 8; }

// G lines of each component per CTA: one for grids of few lines; as many as make
// a warp per component otherwise (a CTA of fewer threads spends more of its time
// on its constants and barriers).
template <int N>
constexpr int fix_lines(bool many) { return many && N / fix_elems<N>() < 32 ? 32 / (N / fix_elems<N>()) : 1; }

template <int N, int G>
struct FixCfg {
  static constexpr int E = fix_elems<N>();
  static constexpr int T = N / E;
  static constexpr int GC = G * T;
  static constexpr int FTP = (5 * GC + 31) / 32 * 32;
  static constexpr int LINES = FTP / T;
  static constexpr int PTS = G * N;
  // small CTAs: 256 threads or one per point; else just the lines' threads, so
  // that three CTAs share an SM and one's transforms overlap another's flow
  static constexpr int PW = GC >= 32 ? 160 : PTS < 256 ? (PTS + 31) / 32 * 32 : 256;
  static constexpr int THREADS = FTP > PW ? FTP : PW;
  static constexpr int LP = line_pad_tile<double>(N, G);
  static constexpr size_t SMEM = sizeof(FixTw) * (size_t)N + sizeof(double2) * (size_t)(LINES * LP);
  static constexpr int MINB0 = 65536 / (THREADS * 128);
  static constexpr int MINB1 = (int)(220 * 1024 / SMEM);
  static constexpr int MINB = MINB0 < 1 ? 1 : MINB0 < MINB1 ? MINB0 : MINB1 < 1 ? 1 : MINB1;
};

// ----------------------------------------------------------------------------
// x-pass
// ----------------------------------------------------------------------------
template <int N, int G>
__global__ void __launch_bounds__(FixCfg<N, G>::THREADS, FixCfg<N, G>::MINB) k_xfix(XPassArgs<double> a) {
  typedef double2 C;
  typedef FixCfg<N, G> Cfg;
  constexpr int T = Cfg::T, E = Cfg::E;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FixTw* tw = reinterpret_cast<FixTw*>(smem_raw);
  C* xb = reinterpret_cast<C*>(tw + N);
  __shared__ double s_prm[8];
  __shared__ unsigned s_red[10];
  const bool early = gridDim.x * gridDim.y <= kSplitEarly;
  if (early) pdl_trigger();
  const int tid = threadIdx.x;
  const int member = blockIdx.y;
  for (int k = tid; k < N; k += Cfg::THREADS) tw[k] = reinterpret_cast<const FixTw*>(a.tw)[k];
  if ((a.mode & XP_NL) && tid == 0) {
    const MemberPrm& P = a.mp[member];
    const double t = a.t_base ? *a.t_base + a.t_off : a.t_off;
    sincos(P.omega * t, &s_prm[1], &s_prm[0]);
    s_prm[2] = a.delta * (P.c0 + P.c2 / 5.0);
    s_prm[3] = a.delta * P.c1;
    s_prm[4] = a.delta * (P.c2 / 5.0);
    s_prm[5] = a.delta * P.gx2h;
    s_prm[6] = a.delta * P.gy2h;
    s_prm[7] = a.delta * P.gz2h;
  }
  const int line = tid / T;             // component * G + row of the CTA
  const int i = tid - line * T;
  const int comp = line / G, g = line - comp * G;
  const int row = blockIdx.x * G + g;
  const bool lane = tid < Cfg::FTP;     // whole warps
  const bool valid = line < 5 * G && row < a.rows;
  C* base = a.field + ((size_t)member * 5 + (valid ? comp : 0)) * a.ntot + (size_t)(valid ? row : 0) * N + i;
  C* b = xb + line * Cfg::LP;
  const FixLine fl = {1 + line, s_red + 2 * (T > 32 ? line : 0)};
  C v[E];
  pdl_wait();
  if (lane) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = valid ? base[T * e] : make_double2(0.0, 0.0);
  }
  __syncthreads();                      // twiddles, s_prm
  if (lane && (a.mode & XP_INV)) fix_fft<N, E, +1, 1>(v, i, tw, b, fl);
  if (a.mode & XP_NL) {
    if (lane) {
      fix_sync<T>(fl);                  // the exchanges' reads are done
#pragma unroll
      for (int e = 0; e < E; ++e) b[padx<double>(i + T * e)] = v[e];
    }
    __syncthreads();                    // the rows are staged
    const double co = s_prm[0], si = s_prm[1];
    const FlowPrm P = {s_prm[2], s_prm[3], s_prm[4]};
    const double gx2h = s_prm[5], gy2h = s_prm[6], gz2h = s_prm[7];
#pragma unroll 1
    for (int p = tid; p < Cfg::PTS; p += Cfg::THREADS) {
      const int r = p / N, j = p - r * N;
      const int rr = blockIdx.x * G + r;
      if (rr >= a.rows) break;          // p only grows
      const double y = a.y0 + (double)(rr % a.ny) * a.hy;
      const double z = a.z0 + (double)(rr / a.ny) * a.hz;
      const double x = a.x0 + (double)j * a.hx;
      const double xr = co * x + si * y;
      const double yr = co * y - si * x;
      const double dV = gx2h * xr * xr + gy2h * yr * yr + gz2h * z * z;
      constexpr int CS = G * Cfg::LP;
      C* pp = xb + r * Cfg::LP + padx<double>(j);
      C q[5] = {pp[0], pp[CS], pp[2 * CS], pp[3 * CS], pp[4 * CS]};
      flow_point(q, dV, P);
#pragma unroll
      for (int c = 0; c < 5; ++c) pp[c * CS] = q[c];
    }
    __syncthreads();                    // every point is done
    if (lane) {
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = b[padx<double>(i + T * e)];
    }
  }
  if (lane) {
    if (!early) pdl_trigger();
    if (a.mode & XP_FWD) fix_fft<N, E, -1, 1>(v, i, tw, b, fl);
    if (valid) {
#pragma unroll
      for (int e = 0; e < E; ++e) base[T * e] = v[e];
    }
  }
}

// ----------------------------------------------------------------------------
// line pass
// ----------------------------------------------------------------------------
// G columns side by side: thread i * G + column of its component's G T
template <int N, int G>
__global__ void __launch_bounds__(FixCfg<N, G>::THREADS, FixCfg<N, G>::MINB) k_lfix(LPassArgs<double> a) {
  typedef double2 C;
  typedef FixCfg<N, G> Cfg;
  constexpr int T = Cfg::T, E = Cfg::E;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FixTw* tw = reinterpret_cast<FixTw*>(smem_raw);
  C* xb = reinterpret_cast<C*>(tw + N);
  __shared__ unsigned s_red[10];
  const bool early = gridDim.x * gridDim.y * gridDim.z <= kSplitEarly;
  if (early) pdl_trigger();
  const int tid = threadIdx.x;
  const int plane = blockIdx.y, member = blockIdx.z;
  for (int k = tid; k < N; k += Cfg::THREADS) tw[k] = reinterpret_cast<const FixTw*>(a.tw)[k];
  const int comp = tid / Cfg::GC;
  const int rem = tid - comp * Cfg::GC;
  const int i = rem / G, col = rem - i * G;
  const int xcol = blockIdx.x * G + col;
  const bool lane = tid < Cfg::FTP;
  const bool valid = comp < 5 && xcol < a.nx;
  C* base = a.field + ((size_t)member * 5 + (valid ? comp : 0)) * a.ntot + (size_t)plane * a.plane_stride +
            (valid ? xcol : 0) + (size_t)i * a.line_stride;
  const size_t step = (size_t)T * a.line_stride;
  C* b = xb + (comp * G + col) * Cfg::LP;
  const FixLine fl = {1 + comp, s_red + 2 * (T > 32 ? comp : 0)};
  C v[E];
  pdl_wait();
  if (lane) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = valid ? base[e * step] : make_double2(0.0, 0.0);
  }
  __syncthreads();                      // twiddles
  if (lane && (a.mode & LP_FWD)) fix_fft<N, E, -1, G>(v, i, tw, b, fl);
  if (a.mode & LP_MIX) {
    if (lane) {
      fix_sync<T>(fl);                  // the exchanges' reads are done
#pragma unroll
      for (int e = 0; e < E; ++e) b[padx<double>(i + T * e)] = v[e];
    }
    __syncthreads();                    // the columns are staged
#pragma unroll 1
    for (int p = tid; p < Cfg::PTS; p += Cfg::THREADS) {
      const int pos = p / G, cl = p - pos * G;
      const int px = blockIdx.x * G + cl;
      if (px >= a.nx) continue;         // idle columns of a ragged tile
      const int ps = px < a.NX / 2 ? px : px - a.NX;
      const int q = a.axis == 1 ? pos : plane;
      const int qs = q < a.NY / 2 ? q : q - a.NY;
      const int ap = ps < 0 ? -ps : ps, aq = qs < 0 ? -qs : qs;
      const ModeEntry<double> m =
          load_mode_shared(a.mt + (size_t)member * a.mt_member, ap * (a.NY / 2 + 1) + aq);
      constexpr int CS = G * Cfg::LP;
      C* pp = xb + cl * Cfg::LP + padx<double>(pos);
      C u[5] = {pp[0], pp[CS], pp[2 * CS], pp[3 * CS], pp[4 * CS]};
      const C kh = make_double2(m.khr, m.khi);
      mix_mode(u, m, ps, qs, a.axis == 2 ? kinetic_z(kh, a.kz[pos]) : kh, a.inv_hi);
#pragma unroll
      for (int c = 0; c < 5; ++c) pp[c * CS] = u[c];
    }
    __syncthreads();                    // every mode is done
    if (lane) {
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = b[padx<double>(i + T * e)];
    }
  }
  if (lane) {
    if (!early) pdl_trigger();
    if (a.mode & LP_INV) fix_fft<N, E, +1, G>(v, i, tw, b, fl);
    if (valid) {
#pragma unroll
      for (int e = 0; e < E; ++e) base[e * step] = v[e];
    }
  }
}

// Fixed-point twiddles of a length-N line (fix_elems<N>() elements per thread).
cudaError_t launch_fix_twiddles(int N, FixTw* out, cudaStream_t s);

}  // namespace sgp
