// sgp_split.cuh -- component-parallel passes for grids of few lines.
//
// The passes of sgp_kernels.cuh hold all five components of a line in the
// same threads.  A grid of few lines then leaves the GPU nearly empty, and a
// pass lasts as long as one thread's chain: five transforms of E elements and
// the flow (or the mix) at E points, one after the other.  Here the five
// components of a line go to five groups of threads, each transforming one
// component, and the points (modes) of the CTA's lines are shared out again
// over all threads for the nonlinear flow (the mix), staged in the exchange
// buffers in between.  A CTA holds as few lines as fill its warps.  Per line
// and per point the arithmetic is that of the other passes with the same
// radix plan.
//
// Every constant a pass needs (twiddles, the rotation at its time, its mode
// entries) is fetched before griddepcontrol.wait, while the previous pass of
// the same run is still at work (programmatic dependent launch); the field is
// read and written only after it.
#pragma once
#include "sgp_adjoint.cuh"
#include "sgp_kernels.cuh"

namespace sgp {

// Launches of at most this many CTAs let the next pass onto the SMs at once:
// both then have SMs of their own (half the 152 of a GB300; a hint, on a device
// with other numbers only the overlap differs).  Larger ones wait until their
// points or modes are done, or the next pass crowds onto a few SMs (TS2 step,
// one FP32 member: at 64^2 4.3 us early, 5.4 us late; at 256^2 12.0 and 10.4).
constexpr unsigned kSplitEarly = 76;

// Geometry.  G lines of each component per CTA: the rows of an x-pass, the
// columns of a line pass.
template <typename R, int N, int E, int G>
struct SplitCfg {
  static constexpr int T = N / E;                       // threads per line
  static constexpr int GC = G * T;                      // threads per component
  static constexpr int FT = 5 * GC;                     // threads with a line
  // whole warps take part in the transforms: the lines past 5 G in the last
  // warp are zeros and go nowhere
  static constexpr int FTP = (FT + 31) / 32 * 32;
  static constexpr int LINES = FTP / T;
  static constexpr int PTS = G * N;                     // points (modes) of the CTA
  static constexpr int PW = PTS < 256 ? (PTS + 31) / 32 * 32 : 256;
  static constexpr int THREADS = FTP > PW ? FTP : PW;
  // consecutive lines start in different banks
  static constexpr int LP = line_pad_tile<R>(N, G);
  static constexpr int XCH = (LINES > 5 * G ? LINES : 5 * G) * LP;
  static constexpr size_t SMEM = sizeof(TwE<R>) * (size_t)N + sizeof(cplx<R>) * (size_t)XCH;
  // registers: about 96 a thread
  static constexpr int MINB0 = 65536 / (THREADS * 96);
  static constexpr int MINB1 = (int)(220 * 1024 / SMEM);
  static constexpr int MINB = MINB0 < 1 ? 1 : (MINB0 < MINB1 ? MINB0 : (MINB1 < 1 ? 1 : MINB1));
};

// one shared-memory slot per (line, position), padded as the exchanges are
template <typename R, typename Cfg>
__device__ __forceinline__ int split_slot(int line, int pos) {
  return line * Cfg::LP + padx<R>(pos);
}

// transform of the calling thread's line (buffer b, thread i of the line)
template <typename R, int N, int E, int DIR, int GT>
__device__ __forceinline__ void split_fft(cplx<R> (&v)[1][E], int i, const TwE<R>* tw, cplx<R>* b, int bid) {
  fft_lines<R, N, E, DIR, 1, 1, GT>(v, i, tw, b, 0, bid);
}

// ----------------------------------------------------------------------------
// x-pass
// ----------------------------------------------------------------------------
template <typename R, int N, int E, int G, bool TAP>
__global__ void __launch_bounds__(SplitCfg<R, N, E, G>::THREADS, SplitCfg<R, N, E, G>::MINB)
k_xsplit(XPassArgs<R> a) {
  typedef cplx<R> C;
  typedef SplitCfg<R, N, E, G> Cfg;
  constexpr int T = Cfg::T;
  // lines of up to a warp exchange within the warp, wider ones through a
  // named barrier of the line's threads
  constexpr int GT = T <= 32 ? 32 : T;
  static_assert(T <= 32 || 5 * G <= 15, "named barriers");
  static_assert(Cfg::PTS % 32 == 0, "whole warps in the flow");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TwE<R>* tw = reinterpret_cast<TwE<R>*>(smem_raw);
  C* xb = reinterpret_cast<C*>(tw + N);
  __shared__ R s_prm[8];
  const bool early = gridDim.x * gridDim.y * gridDim.z <= kSplitEarly;
  if (early) pdl_trigger();
  const int tid = threadIdx.x;
  const int member = blockIdx.y;
  for (int k = tid; k < N; k += Cfg::THREADS) tw[k] = a.tw[k];
  if ((a.mode & XP_NL) && tid == 0) {
    const MemberPrm& P = a.mp[member];
    const double t = a.t_base ? *a.t_base + a.t_off : a.t_off;
    double sn, cs;
    sincos(P.omega * t, &sn, &cs);
    s_prm[0] = (R)cs;
    s_prm[1] = (R)sn;
    s_prm[2] = coupling<R>(P);
    s_prm[3] = (R)P.c1;
    s_prm[4] = (R)P.c2;
    s_prm[5] = (R)P.gx2h;
    s_prm[6] = (R)P.gy2h;
    s_prm[7] = (R)P.gz2h;
  }
  const int line = tid / T;             // component * G + row of the CTA
  const int i = tid - line * T;
  const int comp = line / G, g = line - comp * G;
  const int row = blockIdx.x * G + g;
  const bool lane = tid < Cfg::FTP;     // whole warps
  const bool valid = line < 5 * G && row < a.rows;
  C* base = a.field + ((size_t)member * 5 + (valid ? comp : 0)) * a.ntot + (size_t)(valid ? row : 0) * N + i;
  C* b = xb + line * Cfg::LP;
  const int bid = 1 + line;
  C v[1][E];
  pdl_wait();
  if (lane) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[0][e] = valid ? base[T * e] : mkc((R)0, (R)0);
  }
  __syncthreads();                      // twiddles, s_prm
  if (lane && (a.mode & XP_INV)) split_fft<R, N, E, +1, GT>(v, i, tw, b, bid);
  if (a.mode & XP_NL) {
    if (lane) {
      group_sync<GT>(bid);              // the exchanges' reads are done
#pragma unroll
      for (int e = 0; e < E; ++e) b[padx<R>(i + T * e)] = v[0][e];
    }
    __syncthreads();                    // the rows are staged
    const R co = s_prm[0], si = s_prm[1];
    const R c0p = s_prm[2], c1 = s_prm[3], c2 = s_prm[4];
    const R gx2h = s_prm[5], gy2h = s_prm[6], gz2h = s_prm[7];
    // PTS is a multiple of 32: every warp is whole here
#pragma unroll 1
    for (int p = tid; p < Cfg::PTS; p += Cfg::THREADS) {
      const int r = p / N, j = p - r * N;
      const int rr = blockIdx.x * G + r;
      const R y = a.y0 + (R)(rr % a.ny) * a.hy;
      const R z = a.z0 + (R)(rr / a.ny) * a.hz;
      const R x = a.x0 + (R)j * a.hx;
      const R xr = co * x + si * y;
      const R yr = co * y - si * x;
      const R V = gx2h * xr * xr + gy2h * yr * yr + gz2h * z * z;
      C* pp = xb + split_slot<R, Cfg>(r, j);
      constexpr int CS = G * Cfg::LP;
      C q[5] = {pp[0], pp[CS], pp[2 * CS], pp[3 * CS], pp[4 * CS]};
      nonlinear_point<R>(q, V, a.delta, c0p, c1, c2);
#pragma unroll
      for (int c = 0; c < 5; ++c) pp[c * CS] = q[c];
    }
    __syncthreads();                    // every point is done
    if (lane) {
#pragma unroll
      for (int e = 0; e < E; ++e) v[0][e] = b[padx<R>(i + T * e)];
      if constexpr (TAP) {
        if (valid) {
          C* tp = a.tap + (base - a.field);
#pragma unroll
          for (int e = 0; e < E; ++e) tp[T * e] = v[0][e];
        }
      }
    }
  }
  if (lane) {
    if (!early) pdl_trigger();
    if (a.mode & XP_FWD) split_fft<R, N, E, -1, GT>(v, i, tw, b, bid);
    if (valid) {
#pragma unroll
      for (int e = 0; e < E; ++e) base[T * e] = v[0][e];
    }
  }
}

// ----------------------------------------------------------------------------
// line pass
// ----------------------------------------------------------------------------
// ADJ: the line pass of a gradient, with the work of AdjHook at every mode: the
// sweep adds the Omega and gamma terms before the mix (h.spec, fetched with the
// table entry), the recomputation keeps a copy after it (h.tap).
struct NoAdj {};
template <typename R, int N, int E, int G, bool ADJ, class H>
__global__ void __launch_bounds__(SplitCfg<R, N, E, G>::THREADS, SplitCfg<R, N, E, G>::MINB)
k_lsplit(LPassArgs<R> a, H h) {
  typedef cplx<R> C;
  typedef SplitCfg<R, N, E, G> Cfg;
  constexpr int T = Cfg::T;
  // a component's G columns side by side: thread i * G + column of its group
  constexpr int GT = Cfg::GC <= 32 ? 32 : Cfg::GC;
  static_assert(Cfg::GC % 32 == 0 || 32 % Cfg::GC == 0, "line groups in whole warps");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TwE<R>* tw = reinterpret_cast<TwE<R>*>(smem_raw);
  C* xb = reinterpret_cast<C*>(tw + N);
  const bool early = gridDim.x * gridDim.y * gridDim.z <= kSplitEarly;
  if (early) pdl_trigger();
  const int tid = threadIdx.x;
  const int plane = blockIdx.y, member = blockIdx.z;
  for (int k = tid; k < N; k += Cfg::THREADS) tw[k] = a.tw[k];
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
  const int bid = 1 + comp;
  // the thread's first mode: its table entry is on the way during the
  // transform
  const bool mix = a.mode & LP_MIX;
  auto entry = [&](int p, int& ps, int& qs, C& kz) -> ModeEntry<R> {
    const int pos = p / G;
    int px = blockIdx.x * G + (p - pos * G);
    px = px < a.nx ? px : 0;            // idle columns of a ragged tile
    ps = px < a.NX / 2 ? px : px - a.NX;
    const int q = a.axis == 1 ? pos : plane;
    qs = q < a.NY / 2 ? q : q - a.NY;
    const int ap = ps < 0 ? -ps : ps, aq = qs < 0 ? -qs : qs;
    kz = a.axis == 2 ? a.kz[pos] : mkc((R)0, (R)0);
    return load_mode_shared(a.mt + (size_t)member * a.mt_member, ap * (a.NY / 2 + 1) + aq);
  };
  // element offset of mode p of component 0
  auto element = [&](int p) -> size_t {
    const int pos = p / G;
    return (size_t)member * 5 * a.ntot + (size_t)plane * a.plane_stride + (size_t)pos * a.line_stride +
           blockIdx.x * G + (p - pos * G);
  };
  ModeEntry<R> m0{};
  int ps0 = 0, qs0 = 0;
  C kz0 = mkc((R)0, (R)0);
  if (mix && tid < Cfg::PTS) m0 = entry(tid, ps0, qs0, kz0);
  // the transform of Phi_out at the mode: not written by the pass before
  C sv[5];
  if constexpr (ADJ) {
    if (h.spec && tid < Cfg::PTS && blockIdx.x * G + tid % G < a.nx) {
#pragma unroll
      for (int c = 0; c < 5; ++c) sv[c] = h.spec[element(tid) + (size_t)c * a.ntot];
    }
  }
  double acc[LPA_NT] = {0.0, 0.0};
  C v[1][E];
  pdl_wait();
  if (lane) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[0][e] = valid ? base[e * step] : mkc((R)0, (R)0);
  }
  __syncthreads();                      // twiddles
  if (lane && (a.mode & LP_FWD)) split_fft<R, N, E, -1, GT>(v, i, tw, b, bid);
  if (mix) {
    if (lane) {
      group_sync<GT>(bid);              // the exchanges' reads are done
#pragma unroll
      for (int e = 0; e < E; ++e) b[padx<R>(i + T * e)] = v[0][e];
    }
    __syncthreads();                    // the columns are staged
#pragma unroll 1
    for (int p = tid; p < Cfg::PTS; p += Cfg::THREADS) {
      const int pos = p / G, cl = p - pos * G;
      if (p != tid) m0 = entry(p, ps0, qs0, kz0);
      C* pp = xb + split_slot<R, Cfg>(cl, pos);
      constexpr int CS = G * Cfg::LP;
      C q[5] = {pp[0], pp[CS], pp[2 * CS], pp[3 * CS], pp[4 * CS]};
      const C kh = mkc(m0.khr, m0.khi);
      if constexpr (ADJ) {
        if (h.spec && blockIdx.x * G + cl < a.nx) {
          if (p != tid) {
#pragma unroll
            for (int c = 0; c < 5; ++c) sv[c] = h.spec[element(p) + (size_t)c * a.ntot];
          }
          const MemberPrm& P = h.mp[member];
          constexpr double kPi = 3.14159265358979323846;
          lin_param_mode<R>(q, sv, ps0, qs0, (R)P.gamma, (R)P.omega, (R)h.delta, (R)(kPi / h.Lx), (R)(kPi / h.Ly),
                            acc);
        }
      }
      mix_entry<R>(q, a, m0, ps0, qs0, a.axis == 2 ? kinetic_z(kh, kz0) : kh);
#pragma unroll
      for (int c = 0; c < 5; ++c) pp[c * CS] = q[c];
      if constexpr (ADJ) {
        if (h.tap && blockIdx.x * G + cl < a.nx) {
#pragma unroll
          for (int c = 0; c < 5; ++c) h.tap[element(p) + (size_t)c * a.ntot] = q[c];
        }
      }
    }
    __syncthreads();                    // every mode is done
    if (lane) {
#pragma unroll
      for (int e = 0; e < E; ++e) v[0][e] = b[padx<R>(i + T * e)];
    }
  }
  if (lane) {
    if (!early) pdl_trigger();
    if (a.mode & LP_INV) split_fft<R, N, E, +1, GT>(v, i, tw, b, bid);
    if (valid) {
#pragma unroll
      for (int e = 0; e < E; ++e) base[e * step] = v[0][e];
    }
  }
  if constexpr (ADJ) {
    if (h.spec) {                       // the same for every thread of the launch
      __shared__ double red[(Cfg::THREADS / 32) * LPA_NT];
      __shared__ double out[LPA_NT];
      block_sums<LPA_NT>(acc, out, red);
      if (tid < LPA_NT) {
        double* row = h.partials + ((size_t)member * h.prows + h.prow0 + (size_t)plane * h.tiles + blockIdx.x) * GP_N;
        row[tid == 0 ? GP_OMEGA : GP_GAMMA] += out[tid] * h.scale;
      }
    }
  }
}

// ----------------------------------------------------------------------------
// x-pass of the adjoint sweep (k_xadj with the components split)
// ----------------------------------------------------------------------------
template <typename R, int N, int E, int G>
__global__ void __launch_bounds__(SplitCfg<R, N, E, G>::THREADS, 65536 / (SplitCfg<R, N, E, G>::THREADS * 128))
k_xadj_split(XAdjArgs<R> a) {
  typedef cplx<R> C;
  typedef SplitCfg<R, N, E, G> Cfg;
  constexpr int T = Cfg::T;
  constexpr int GT = T <= 32 ? 32 : T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TwE<R>* tw = reinterpret_cast<TwE<R>*>(smem_raw);
  C* xb = reinterpret_cast<C*>(tw + N);
  __shared__ double s_rot[3];
  __shared__ double red[(Cfg::THREADS / 32) * NLA_NT];
  __shared__ double out[NLA_NT];
  const bool early = gridDim.x * gridDim.y <= kSplitEarly;
  if (early) pdl_trigger();
  const int tid = threadIdx.x;
  const int member = blockIdx.y;
  for (int k = tid; k < N; k += Cfg::THREADS) tw[k] = a.tw[k];
  if (tid == 0) {
    const double t = *a.t_base + a.t_off;
    sincos(a.mp[member].omega * t, &s_rot[1], &s_rot[0]);
    s_rot[2] = t;
  }
  const size_t mo = (size_t)member * 5 * a.ntot;
  const int line = tid / T;
  const int i = tid - line * T;
  const int comp = line / G, g = line - comp * G;
  const int row = blockIdx.x * G + g;
  const bool lane = tid < Cfg::FTP;
  const bool valid = line < 5 * G && row < a.rows;
  C* base = a.g + mo + (size_t)(valid ? comp : 0) * a.ntot + (size_t)(valid ? row : 0) * N + i;
  C* b = xb + line * Cfg::LP;
  const int bid = 1 + line;
  C v[1][E];
  // Phi_out at the thread's first point: not written by the pass before
  C psi[5];
  if (tid < Cfg::PTS && blockIdx.x * G + tid / N < a.rows) {
    const C* pr = a.phi + mo + (size_t)(blockIdx.x * G) * N + tid;
#pragma unroll
    for (int c = 0; c < 5; ++c) psi[c] = pr[(size_t)c * a.ntot];
  }
  pdl_wait();
  if (lane) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[0][e] = valid ? base[T * e] : mkc((R)0, (R)0);
  }
  __syncthreads();                      // twiddles, s_rot
  if (lane) {
    if (a.mode & XP_INV) split_fft<R, N, E, +1, GT>(v, i, tw, b, bid);
    group_sync<GT>(bid);                // the exchanges' reads are done
#pragma unroll
    for (int e = 0; e < E; ++e) b[padx<R>(i + T * e)] = v[0][e];
  }
  __syncthreads();                      // the rows are staged
  double acc[NLA_NT] = {0.0, 0.0, 0.0, 0.0};
  {
    const MemberPrm& P = a.mp[member];
    NLAdjPrm<R> q;
    q.d = (R)a.delta;
    q.c0p = coupling<R>(P);
    q.c1 = (R)P.c1;
    q.c2 = (R)P.c2;
    q.tdgg = (R)(s_rot[2] * 2.0 * (P.gx2h - P.gy2h));
    const R co = (R)s_rot[0], si = (R)s_rot[1];
    const R gx2h = (R)P.gx2h, gy2h = (R)P.gy2h, gz2h = (R)P.gz2h;
#pragma unroll 1
    for (int p = tid; p < Cfg::PTS; p += Cfg::THREADS) {
      const int r = p / N, j = p - r * N;
      const int rw = blockIdx.x * G + r;
      if (rw >= a.rows) break;          // p only grows
      const int iy = rw % a.ny, iz = rw / a.ny;
      const R x = a.x0 + (R)j * a.hx, y = a.y0 + (R)iy * a.hy, z = a.z0 + (R)iz * a.hz;
      const R xr = co * x + si * y, yr = co * y - si * x;
      const R V = gx2h * xr * xr + gy2h * yr * yr + gz2h * z * z;
      if (p != tid) {
        const C* pr = a.phi + mo + (size_t)rw * N + j;
#pragma unroll
        for (int c = 0; c < 5; ++c) psi[c] = pr[(size_t)c * a.ntot];
      }
      constexpr int CS = G * Cfg::LP;
      C* sp = xb + split_slot<R, Cfg>(r, j);
      C gp[5] = {sp[0], sp[CS], sp[2 * CS], sp[3 * CS], sp[4 * CS]};
      nl_adjoint_point<R>(psi, gp, V, xr * yr, q, acc);
#pragma unroll
      for (int c = 0; c < 5; ++c) sp[c * CS] = gp[c];
    }
  }
  __syncthreads();                      // every point is done
  if (lane) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[0][e] = b[padx<R>(i + T * e)];
    if (!early) pdl_trigger();
    if (a.mode & XP_FWD) split_fft<R, N, E, -1, GT>(v, i, tw, b, bid);
    if (valid) {
#pragma unroll
      for (int e = 0; e < E; ++e) base[T * e] = v[0][e];
    }
  }
  block_sums<NLA_NT>(acc, out, red);
  if (tid < NLA_NT) {
    const int slot[NLA_NT] = {GP_OMEGA, GP_C0, GP_C1, GP_C2};
    a.partials[((size_t)member * a.prows + blockIdx.x) * GP_N + slot[tid]] += out[tid];
  }
}

// Lines per CTA: one row; two where one is not whole warps of points.  Two
// columns (a line element's 16 bytes together); one where the threads of two
// are too many.
template <typename R, int N>
constexpr int split_rows() { return N % 32 == 0 ? 1 : 2; }
template <typename R, int N>
constexpr int split_cols() { return N <= 512 ? 2 : 1; }
// Elements per thread: those of the other passes, except 12 for N = 3*2^k:
// radix 6 then 4s (192 = 6*4*4*2) instead of 6 then 2s (192 = 6*2*2*2*2*2), one
// stage fewer for every factor 4; one component's 12 elements are few registers.
template <typename R, int N>
constexpr int split_elems() { return N % 3 == 0 ? 12 : 8; }
// Launchers: FP32 here (sgp_split.cu); in FP64 the component-parallel passes
// are those of sgp_fix.cuh (sgp_fix.cu).  dependent: the launch may begin
// while the pass before it on the stream is at work.  many (FP64): enough
// lines for CTAs of several.
template <typename R> int split_elems_rt(int N);
template <typename R> cudaError_t prepare_xsplit(int N, bool many);
template <typename R> cudaError_t prepare_lsplit(int N, bool many);
template <typename R>
cudaError_t launch_xsplit(int N, bool many, const XPassArgs<R>& a, int members, bool dependent, cudaStream_t s);
template <typename R>
cudaError_t launch_lsplit(int N, bool many, const LPassArgs<R>& a, int planes, int members, bool dependent,
                          cudaStream_t s);
// The passes of a gradient (FP32): the x-pass that copies its rows after the
// flow to a.tap, the adjoint x-pass, the line pass with its hooks; CTAs per
// member of the x-passes and columns' tiles per plane (rows of the partials).
cudaError_t prepare_adj_split(int NX, int NL);
cudaError_t launch_xsplit_tap(int N, const XPassArgs<float>& a, int members, bool dependent, cudaStream_t s);
cudaError_t launch_xadj_split(int N, const XAdjArgs<float>& a, int members, bool dependent, cudaStream_t s);
cudaError_t launch_lsplit_adj(int N, const LPassArgs<float>& a, const AdjHook<float>& h, int planes, int members,
                              bool dependent, cudaStream_t s);
int xsplit_ctas(int N, int rows);
int lsplit_tiles(int N, int nx);

}  // namespace sgp
