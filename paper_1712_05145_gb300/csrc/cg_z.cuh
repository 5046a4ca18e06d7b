// z passes of the FP32 CG and BiCGSTAB iterations in Fourier space (see spectral_cg.h).
//
// A CTA owns TC consecutive spectrum columns (flat index of the x-y half-spectrum plane) over all N3
// planes and walks through the six Kelvin components.  A thread keeps E values of one column in
// registers through the whole z FFT: the stages exchange through shared memory, the first stage's
// inputs come straight from global memory and the last stage's outputs go straight back (TC
// consecutive values per plane, 64 to 512 bytes).  The component loop accumulates w = tau_hat q in
// registers, so no component has to wait for the others in shared memory and no cluster is needed.
//
// Bound by latency: a column's values, the next component and w take 128 registers a thread, 16 warps an
// SM (80 and 96 registers spill; 16 values a thread, one exchange fewer, spill or take 168).  Inverse and forward pass,
// ms per launch: 128^3, six loads, 0.241 and 0.203 (4.4 and 3.0 TB/s of their own traffic); 256^3, two loads,
// 0.640 and 0.571; 512x256x512, one load, 1.29 and 1.39.  With the passes between them an iteration of 128^3
// takes 0.75 ms; with the vectors as real fields its three passes took 1.00 ms.
#pragma once
#include "ls_common.cuh"
#include "spectral.cuh"
#include "spectral_cg.h"

namespace hom {

namespace {

template <int... Rs> struct Radices {};
// values per thread, radices (each divides E) of the z lengths
template <int N> struct ZPlan;
#define HOM_ZPLAN(N_, E_, ...) \
  template <> struct ZPlan<N_> { static constexpr int E = E_; using Seq = Radices<__VA_ARGS__>; };
HOM_ZPLAN(1, 1, 1)
HOM_ZPLAN(2, 2, 2)
HOM_ZPLAN(3, 3, 3)
HOM_ZPLAN(4, 4, 4)
HOM_ZPLAN(6, 6, 6)
HOM_ZPLAN(8, 8, 8)
HOM_ZPLAN(12, 12, 12)
HOM_ZPLAN(16, 8, 4, 4)
HOM_ZPLAN(24, 12, 6, 4)
HOM_ZPLAN(32, 8, 8, 4)
HOM_ZPLAN(48, 12, 12, 4)
HOM_ZPLAN(64, 8, 8, 8)
HOM_ZPLAN(96, 12, 6, 4, 4)
HOM_ZPLAN(128, 8, 8, 4, 4)
HOM_ZPLAN(192, 12, 12, 4, 4)
HOM_ZPLAN(256, 8, 8, 8, 4)
HOM_ZPLAN(384, 12, 6, 4, 4, 4)
HOM_ZPLAN(512, 8, 8, 8, 8)
#undef HOM_ZPLAN

template <typename Seq> struct FirstLast;
template <int R> struct FirstLast<Radices<R>> { static constexpr int first = R, last = R, count = 1; };
template <int R, int... Rs> struct FirstLast<Radices<R, Rs...>> {
  static constexpr int first = R, last = FirstLast<Radices<Rs...>>::last, count = 1 + FirstLast<Radices<Rs...>>::count;
};

// element n of an exchange buffer: rows of TC values, padded so that the first stage's strided rows of a
// warp (8 values apart) fall in different banks
template <int TC>
__device__ __forceinline__ int zpos(int n, int tc) {
  if constexpr (TC >= 16) return n * TC + tc;
  else return (n + (n >> 3)) * TC + tc;
}
constexpr int zbuf_elems(int n, int tc) { return tc >= 16 ? n * tc : (n + (n >> 3) + 1) * tc; }

// Stockham FFT of one column spread over N / E threads (thread u), in registers.  On entry
// v[b * R + r] is element u + b N/E + r N/R for the first radix R; on return the same for the last one.
// Exchanges alternate between two buffers, so one barrier each suffices: a buffer is written again
// only after the barrier of the exchange through the other one, when all its reads are done.  A stage's
// twiddles are fetched before the barrier in front of it, while the registers of v are free.
template <int N, int E, int TC, int DIR, int NS, typename Seq> struct RegFFT;
template <int N, int E, int TC, int DIR, int NS, int R, int... Rest>
struct RegFFT<N, E, TC, DIR, NS, Radices<R, Rest...>> {
  static constexpr int U = N / E, B = E / R;
  // W_(NS R)^(k r) of this stage's butterflies; where U is a multiple of NS they are the same for all b
  static constexpr bool kSameTw = U % NS == 0;
  static constexpr int kTw = kSameTw ? 1 : B;
  __device__ __forceinline__ static void run(cx<float> (&v)[E], int u, int tc, cx<float>*& b0, cx<float>*& b1,
                                             const cx<float>* tw) {
    cx<float> w[kTw][R];
    run_tw(v, u, tc, b0, b1, tw, w);
  }
  __device__ __forceinline__ static void load_tw(int u, const cx<float>* tw, cx<float> (&w)[kTw][R]) {
    constexpr int tstep = N / (NS * R);
#pragma unroll
    for (int b = 0; b < kTw; ++b) {
      const int st = ((u + b * U) % NS) * tstep;
#pragma unroll
      for (int r = 1; r < R; ++r) {
        w[b][r] = tw[st * r];
        if (DIR > 0) w[b][r].im = -w[b][r].im;
      }
    }
  }
  __device__ __forceinline__ static void run_tw(cx<float> (&v)[E], int u, int tc, cx<float>*& b0, cx<float>*& b1,
                                                const cx<float>* tw, const cx<float> (&w)[kTw][R]) {
#pragma unroll
    for (int b = 0; b < B; ++b) {
      if constexpr (NS > 1) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[b * R + r] = cmul(v[b * R + r], w[kSameTw ? 0 : b][r]);
      }
      SmallDFT<float, R, DIR>::run(v + b * R);
    }
    if constexpr (sizeof...(Rest) > 0) {
      using Next = RegFFT<N, E, TC, DIR, NS * R, Radices<Rest...>>;
      constexpr int R2 = FirstLast<Radices<Rest...>>::first, B2 = E / R2;
#pragma unroll
      for (int b = 0; b < B; ++b) {
        const int j = u + b * U, k = j % NS, base = (j - k) * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) b0[zpos<TC>(base + r * NS, tc)] = v[b * R + r];
      }
      cx<float> wn[Next::kTw][R2];
      Next::load_tw(u, tw, wn);
      __syncthreads();
#pragma unroll
      for (int b = 0; b < B2; ++b)
#pragma unroll
        for (int r = 0; r < R2; ++r) v[b * R2 + r] = b0[zpos<TC>(u + b * U + r * (N / R2), tc)];
      cx<float>* t = b0;
      b0 = b1;
      b1 = t;
      Next::run_tw(v, u, tc, b0, b1, tw, wn);
    }
  }
};

// shared memory of a z CTA: two exchange buffers (none for single-stage lengths; the reduction's
// per-thread sums at the end), twiddles, (cz, sz)
template <int N, int TC> struct ZSmem {
  static constexpr int kBuf = FirstLast<typename ZPlan<N>::Seq>::count > 1 ? zbuf_elems(N, TC) : 0;
  static constexpr int kRed = 2 * (N / ZPlan<N>::E * TC);   // doubles, the size of one complex value
  static constexpr int kArea = 2 * kBuf > kRed ? 2 * kBuf : kRed;
  static constexpr size_t bytes = (size_t)(kArea + 2 * N) * sizeof(cx<float>);
};
// Resident threads per SM: 512 at 8 values per thread (128 registers), 384 at 12 (168 registers; with
// 128 they spill up to 500 bytes).
template <int N, int TC> struct ZLaunch {
  static constexpr int threads = N / ZPlan<N>::E * TC;
  static constexpr int resident = ZPlan<N>::E > 8 ? 384 : 512;
  static constexpr int min_blocks = threads >= resident ? 1 : resident / threads;
};

// wave vector q = (a1 cz(n), a2 cz(n), a3 sz(n)), see cg_column_factors: the column factors, and the table over n
struct ColumnQ {
  float a1, a2, a3;
};
// (In FP32 throughout: a warp instruction takes 16 cycles of the SM's FP64 pipe, and these run in every thread.)
__device__ __forceinline__ ColumnQ column_q(const CgZArgs& a, int kx, int ky) {
  ColumnQ q;
  cg_column_factors<float>(a.g, a.green, a.gtab, kx, ky, q.a1, q.a2, q.a3);
  return q;
}
__device__ __forceinline__ cx<float> z_factors(const CgZArgs& a, int n) {   // (cz, sz)
  cx<float> z;
  cg_z_factors<float>(a.g, a.green, a.gtab, n, z.re, z.im);
  return z;
}

__device__ __forceinline__ cx<float> fma_cx(cx<float> a, float s, cx<float> c) {
  return mk<float>(fmaf(a.re, s, c.re), fmaf(a.im, s, c.im));
}

constexpr float kR3f = 0.57735026918962576451f, kR2f = 0.70710678118654752440f, kR6f = 0.40824829046386301637f;

// w += k_c (M_c q) for the Kelvin basis tensors M_c
__device__ __forceinline__ void add_w(int c, cx<float> k, float q1, float q2, float q3, cx<float>& w1, cx<float>& w2,
                                      cx<float>& w3) {
  switch (c) {
    case 0: k = k * kR3f; w1 = fma_cx(k, q1, w1); w2 = fma_cx(k, q2, w2); w3 = fma_cx(k, q3, w3); break;
    case 1: k = k * kR2f; w1 = fma_cx(k, q1, w1); w2 = fma_cx(k, -q2, w2); break;
    case 2: k = k * kR6f; w1 = fma_cx(k, q1, w1); w2 = fma_cx(k, q2, w2); w3 = fma_cx(k, -2.0f * q3, w3); break;
    case 3: k = k * kR2f; w2 = fma_cx(k, q3, w2); w3 = fma_cx(k, q2, w3); break;
    case 4: k = k * kR2f; w1 = fma_cx(k, q3, w1); w3 = fma_cx(k, q1, w3); break;
    default: k = k * kR2f; w1 = fma_cx(k, q2, w1); w2 = fma_cx(k, q1, w2); break;
  }
}
// Kelvin component c of e = v (x) q + q (x) v, k_c = 2 v . (M_c q)
__device__ __forceinline__ cx<float> strain_k(int c, float q1, float q2, float q3, cx<float> v1, cx<float> v2,
                                              cx<float> v3) {
  switch (c) {
    case 0: return fma_cx(v3, q3, fma_cx(v2, q2, v1 * q1)) * (2.0f * kR3f);
    case 1: return fma_cx(v2, -q2, v1 * q1) * (2.0f * kR2f);
    case 2: return fma_cx(v3, -2.0f * q3, fma_cx(v2, q2, v1 * q1)) * (2.0f * kR6f);
    case 3: return fma_cx(v3, q2, v2 * q3) * (2.0f * kR2f);
    case 4: return fma_cx(v3, q1, v1 * q3) * (2.0f * kR2f);
    default: return fma_cx(v2, q1, v1 * q2) * (2.0f * kR2f);
  }
}

// kx, ky of the flat spectrum index f (0, 0 past the plane)
__device__ __forceinline__ void column_of(const Geo& g, unsigned f, bool valid, int& kx, int& ky) {
  const unsigned nmain = (unsigned)g.n2 * (unsigned)g.h;
  kx = ky = 0;
  if (f < nmain) { ky = (int)g.fd_h.div(f); kx = (int)f - ky * g.h; }
  else if (valid) { ky = (int)(f - nmain); kx = g.h; }
}

// Parseval weight of a half-spectrum column: columns 0 < kx < n1/2 stand for their conjugates too
__device__ __forceinline__ float parseval_weight(const Geo& g, int kx, bool valid) {
  return !valid ? 0.0f : (kx == 0 || kx == g.h) ? 1.0f : 2.0f;
}
// nn += |q|^2 Re(a . conj b), nd += Re((q . a) conj(q . b)): <e_a, e_b> = 2 nn + 2 nd
__device__ __forceinline__ void add_product(float q1, float q2, float q3, cx<float> a1, cx<float> a2, cx<float> a3,
                                            cx<float> b1, cx<float> b2, cx<float> b3, float& nn, float& nd) {
  const float q = fmaf(q1, q1, fmaf(q2, q2, q3 * q3));
  const cx<float> da = fma_cx(a3, q3, fma_cx(a2, q2, a1 * q1)), db = fma_cx(b3, q3, fma_cx(b2, q2, b1 * q1));
  const float m = a1.re * b1.re + a1.im * b1.im + a2.re * b2.re + a2.im * b2.im + a3.re * b3.re + a3.im * b3.im;
  nn = fmaf(q, m, nn);
  nd = fmaf(da.re, db.re, fmaf(da.im, db.im, nd));
}

// columns (within the plane) of this CTA's tiles
template <int TC>
__device__ __forceinline__ long long columns_of_cta(unsigned pc, int ntiles) {
  long long cols = 0;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const long long left = (long long)pc - (long long)t * TC;
    cols += left < TC ? left : TC;
  }
  return cols;
}

// The vectors lie tile by tile, [rhs][tile][3][N3][TC]: a CTA reads and writes them as one contiguous
// block (in the spectrum's layout, TC values of every plane, they moved at half the rate).
//
// A CTA takes tiles blockIdx.x, + gridDim.x, ...: neighbouring tiles run at the same time, so the parts
// of a cache line are written together.  Of the next one it prefetches the vectors into L2 while it
// transforms the current one: otherwise a tile's vector reads (2.5 of the pass's 3.5 sweeps) would wait
// for DRAM with nothing else to do in the CTA.
template <int N, int TC, int MODE>
__global__ void __launch_bounds__(ZLaunch<N, TC>::threads, ZLaunch<N, TC>::min_blocks)
    cg_z_inv_kernel(const CgZArgs a, int ntiles) {
  constexpr int E = ZPlan<N>::E, U = N / E, THREADS = ZLaunch<N, TC>::threads;
  using Seq = typename ZPlan<N>::Seq;
  constexpr int RF = FirstLast<Seq>::first, RL = FirstLast<Seq>::last;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Geo& g = a.g;
  const int lrhs = blockIdx.y, rhs = a.rhs0 + lrhs;
  grid_dep_launch();
  cx<float>* b0 = reinterpret_cast<cx<float>*>(smem_raw);
  cx<float>* b1 = b0 + ZSmem<N, TC>::kBuf;
  cx<float>* tw = b0 + ZSmem<N, TC>::kArea;
  cx<float>* zt = tw + N;
  const int tid = threadIdx.x, tc = tid % TC, u = tid / TC;
  for (int i = tid; i < N; i += THREADS) {
    tw[i] = ldg_cx(a.tw_n3 + i);
    zt[i] = z_factors(a, i);
  }
  grid_dep_wait();
  const RhsState& s = a.st[rhs];
  if (s.active == 0) return;
  const unsigned pc = (unsigned)g.plane_c;
  const size_t comp = (size_t)N * pc;
  const bool restart = s.restart != 0;
  const bool addx = MODE == CGI_STEP ? !restart : MODE == CGI_OUT && s.xpend != 0;
  const float beta = restart ? 0.0f : (float)s.beta;
  const float alpha = addx || MODE == CGI_BI_S ? (float)s.alpha : 0.0f;
  const float omega = MODE == CGI_BI_P ? (float)s.omega : 0.0f;
  double sum_n = 0.0, sum_d = 0.0;   // CGI_BI_S: weighted sums of |q|^2 |s|^2 and |q . s|^2
  __syncthreads();   // tables
  const int step = gridDim.x;
#pragma unroll 1
  for (int tile = blockIdx.x; tile < ntiles; tile += step) {
    const unsigned f = (unsigned)tile * TC + tc;
    const bool valid = f < pc;
    int kx, ky;
    column_of(g, f, valid, kx, ky);
    const ColumnQ cq = column_q(a, kx, ky);
    // element e = b * RF + r of this thread is plane u + b U + r N / RF
    cx<float> v[3][E];
    const size_t block = ((size_t)rhs * ntiles + tile) * (3 * N * TC);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const size_t off = block + i * N * TC + u * TC + tc;
      cx<float>* pp = a.p + off;
      cx<float>* xp = a.x + off;
      const cx<float>* rp = a.r + off;
      cx<float> pv[E], xv[E];   // BiCGSTAB: xv holds v
      const cx<float>* vp = a.v + off;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int o = ((e / RF) * U + (e % RF) * (N / RF)) * TC;
        v[i][e] = pv[e] = xv[e] = mk<float>(0.0f, 0.0f);
        if (MODE != CGI_OUT) v[i][e] = rp[o];
        if (addx || (MODE == CGI_BI_P && !restart)) pv[e] = pp[o];
        if (addx || MODE == CGI_OUT) xv[e] = xp[o];
        if (MODE == CGI_BI_S || (MODE == CGI_BI_P && !restart)) xv[e] = vp[o];
      }
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int o = ((e / RF) * U + (e % RF) * (N / RF)) * TC;
        if (MODE == CGI_BI_P) {   // p = r + beta (p - omega v); a restart also sets r_hat
          v[i][e] = fma_cx(fma_cx(xv[e], -omega, pv[e]), beta, v[i][e]);
          pp[o] = v[i][e];
          if (restart) a.rh[off + o] = v[i][e];
          continue;
        }
        if (MODE == CGI_BI_S) {   // s = r - alpha v
          v[i][e] = fma_cx(xv[e], -alpha, v[i][e]);
          a.s[off + o] = v[i][e];
          continue;
        }
        const cx<float> xn = fma_cx(pv[e], alpha, xv[e]);
        if (MODE == CGI_STEP) {
          v[i][e] = fma_cx(pv[e], beta, v[i][e]);
          if (addx) xp[o] = xn;
          pp[o] = v[i][e];
        } else {
          v[i][e] = xn;
        }
      }
    }
    if (tid == 0 && tile + step < ntiles) {
      const size_t next = block + (size_t)step * (3 * N * TC);
      constexpr unsigned bytes = 3 * N * TC * sizeof(cx<float>);
      if (MODE != CGI_OUT) prefetch_l2(a.r + next, bytes);
      if (addx || (MODE == CGI_BI_P && !restart)) prefetch_l2(a.p + next, bytes);
      if (addx || MODE == CGI_OUT) prefetch_l2(a.x + next, bytes);
      if (MODE == CGI_BI_S || (MODE == CGI_BI_P && !restart)) prefetch_l2(a.v + next, bytes);
    }
    if (MODE == CGI_BI_S) {
      float nn = 0.0f, nd = 0.0f;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const cx<float> z = zt[u + (e / RF) * U + (e % RF) * (N / RF)];
        add_product(cq.a1 * z.re, cq.a2 * z.re, cq.a3 * z.im, v[0][e], v[1][e], v[2][e], v[0][e], v[1][e], v[2][e], nn, nd);
      }
      const float wt = parseval_weight(g, kx, valid);
      sum_n += (double)(wt * nn);
      sum_d += (double)(wt * nd);
    }
#pragma unroll 1
    for (int c = 0; c < 6; ++c) {
      cx<float> k[E];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const cx<float> z = zt[u + (e / RF) * U + (e % RF) * (N / RF)];
        k[e] = strain_k(c, cq.a1 * z.re, cq.a2 * z.re, cq.a3 * z.im, v[0][e], v[1][e], v[2][e]);
      }
      RegFFT<N, E, TC, +1, 1, Seq>::run(k, u, tc, b0, b1, tw);
      if (valid) {
        cx<float>* Sc = a.S + (size_t)(lrhs * 6 + c) * comp + f;
#pragma unroll
        for (int e = 0; e < E; ++e) Sc[(unsigned)(u + (e / RL) * U + (e % RL) * (N / RL)) * pc] = k[e];
      }
    }
  }
  if (a.prof != nullptr && tid == 0) {
    const long long cols = columns_of_cta<TC>(pc, ntiles);
    // 3-component sweeps of the vectors
    const int sweeps = MODE == CGI_STEP   ? (restart ? 2 : 5)
                       : MODE == CGI_BI_P ? (restart ? 3 : 4)
                       : MODE == CGI_BI_S ? 3
                                          : (addx ? 2 : 1);
    atomicAdd(a.prof, (unsigned long long)((3 * sweeps + 6) * N * cols * (long long)sizeof(cx<float>)));
  }
  if (MODE == CGI_BI_S) {
    double* red = reinterpret_cast<double*>(smem_raw);
    __syncthreads();   // the exchange buffers are free
    red[tid] = sum_n;
    red[THREADS + tid] = sum_d;
    __syncthreads();
    if (tid < 32) {
      const double sn = warp_sum_f64(red, THREADS), sd = warp_sum_f64(red + THREADS, THREADS);
      double vv[2] = {2.0 * (sn + sd), 0.0};
      const int ncta = gridDim.x;
      if (warp_publish_and_collect<2>(vv, a.part + (long long)rhs * 2 * ncta, a.cnt + rhs, ncta, blockIdx.x) && tid == 0)
        bicg_finalize(BI_S, a.st[rhs], vv, 1.0);
    }
  }
}

template <int N, int TC, int MODE>
__global__ void __launch_bounds__(ZLaunch<N, TC>::threads, ZLaunch<N, TC>::min_blocks)
    cg_z_fwd_kernel(const CgZArgs a, int ntiles) {
  constexpr int E = ZPlan<N>::E, U = N / E, THREADS = ZLaunch<N, TC>::threads;
  using Seq = typename ZPlan<N>::Seq;
  constexpr int RF = FirstLast<Seq>::first, RL = FirstLast<Seq>::last;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Geo& g = a.g;
  const int lrhs = blockIdx.y, rhs = a.rhs0 + lrhs;
  grid_dep_launch();
  cx<float>* b0 = reinterpret_cast<cx<float>*>(smem_raw);
  cx<float>* b1 = b0 + ZSmem<N, TC>::kBuf;
  cx<float>* tw = b0 + ZSmem<N, TC>::kArea;
  cx<float>* zt = tw + N;
  const int tid = threadIdx.x, tc = tid % TC, u = tid / TC;
  const unsigned pc = (unsigned)g.plane_c;
  const size_t comp = (size_t)N * pc;
  const cx<float>* Sl = a.S + (size_t)(lrhs * 6) * comp;
  const int step = gridDim.x;
  cx<float> nx[E];   // the next component, loaded while the current one is transformed
  auto fetch = [&](int tile, int c) {
    const unsigned f = (unsigned)tile * TC + tc;
    if (f < pc) {
      const cx<float>* Sc = Sl + c * comp + f;
#pragma unroll
      for (int e = 0; e < E; ++e) nx[e] = Sc[(unsigned)(u + (e / RF) * U + (e % RF) * (N / RF)) * pc];
    } else {
#pragma unroll
      for (int e = 0; e < E; ++e) nx[e] = mk<float>(0.0f, 0.0f);
    }
  };
  for (int i = tid; i < N; i += THREADS) {
    tw[i] = ldg_cx(a.tw_n3 + i);
    zt[i] = z_factors(a, i);
  }
  // v = Gamma0_hat(q) : tau_hat from w = tau_hat q (STEP, RHS), or the components of a compatible strain (INIT)
  __shared__ float gc[2];
  const int rve = rve_of(rhs, a.rve_loads);
  if (MODE != CGF_INIT) green_consts_shared<float>(gc, a.c0, rve, a.lam0, a.mu0);
  else if (tid == 0) gc[0] = 1.0f, gc[1] = 0.5f;
  grid_dep_wait();
  const int active = a.st[rhs].active;
  fetch(blockIdx.x, 0);   // with the state on its way: a launch rarely holds loads that have ended
  if (active == 0) return;
  const float alpha = MODE == CGF_STEP ? (float)a.st[rhs].alpha : 0.0f;
  // weighted sums of |q|^2 |v|^2 and |q . v|^2 over the new r (BiCGSTAB: of the products above)
  double sum_n = 0.0, sum_d = 0.0, sum_t = 0.0;
  __syncthreads();   // tables
  const float c1 = gc[0] * a.scale, c2h = gc[1] * a.scale;
#pragma unroll 1
  for (int tile = blockIdx.x; tile < ntiles; tile += step) {
    const unsigned f = (unsigned)tile * TC + tc;
    const bool valid = f < pc;
    int kx, ky;
    column_of(g, f, valid, kx, ky);
    const ColumnQ cq = column_q(a, kx, ky);
    const size_t block = ((size_t)rhs * ntiles + tile) * (3 * N * TC);
    // this tile's r (BiCGSTAB: r_hat or s), needed after the transforms
    constexpr bool kBi = MODE == CGF_BI_V || MODE == CGF_BI_T;
    const cx<float>* ol = (MODE == CGF_BI_V ? a.rh : MODE == CGF_BI_T ? a.s : a.r) + block;
    if ((MODE == CGF_STEP || kBi) && tid == 0) prefetch_l2(ol, 3 * N * TC * sizeof(cx<float>));
    ol += u * TC + tc;
    cx<float>* rl = (MODE == CGF_BI_V ? a.v : MODE == CGF_BI_T ? a.t : a.r) + block + u * TC + tc;
    cx<float> w[3][E];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int e = 0; e < E; ++e) w[i][e] = mk<float>(0.0f, 0.0f);
#pragma unroll 1
    for (int c = 0; c < 6; ++c) {
      cx<float> k[E];
#pragma unroll
      for (int e = 0; e < E; ++e) k[e] = nx[e];
      if (c < 5) fetch(tile, c + 1);
      else if (tile + step < ntiles) fetch(tile + step, 0);
      RegFFT<N, E, TC, -1, 1, Seq>::run(k, u, tc, b0, b1, tw);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const cx<float> z = zt[u + (e / RL) * U + (e % RL) * (N / RL)];
        add_w(c, k[e], cq.a1 * z.re, cq.a2 * z.re, cq.a3 * z.im, w[0][e], w[1][e], w[2][e]);
      }
    }
    float nn = 0.0f, nd = 0.0f, tn = 0.0f, td = 0.0f;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int n = u + (e / RL) * U + (e % RL) * (N / RL);
      const int o = (n - u) * TC;
      constexpr int comp_v = N * TC;
      const cx<float> z = zt[n];
      const float q1 = cq.a1 * z.re, q2 = cq.a2 * z.re, q3 = cq.a3 * z.im;
      const float q = fmaf(q1, q1, fmaf(q2, q2, q3 * q3));
      const float iq = q > 0.0f ? 1.0f / q : 0.0f;
      const float f1 = c1 * iq, f2 = c2h * iq * iq;
      const cx<float> sq = fma_cx(w[2][e], q3, fma_cx(w[1][e], q2, w[0][e] * q1)) * f2;
      cx<float> v1 = fma_cx(sq, -q1, w[0][e] * f1), v2 = fma_cx(sq, -q2, w[1][e] * f1), v3 = fma_cx(sq, -q3, w[2][e] * f1);
      if (MODE == CGF_STEP) {
        v1 = fma_cx(v1, -alpha, rl[o]);
        v2 = fma_cx(v2, -alpha, rl[o + comp_v]);
        v3 = fma_cx(v3, -alpha, rl[o + 2 * comp_v]);
      } else if (MODE == CGF_RHS) {
        v1 = v1 * -1.0f;
        v2 = v2 * -1.0f;
        v3 = v3 * -1.0f;
      }
      rl[o] = v1;
      rl[o + comp_v] = v2;
      rl[o + 2 * comp_v] = v3;
      if (kBi) {   // the sums of <r_hat, v>, or of <t, s> and <t, t>
        const cx<float> o1 = ol[o], o2 = ol[o + comp_v], o3 = ol[o + 2 * comp_v];
        add_product(q1, q2, q3, v1, v2, v3, o1, o2, o3, nn, nd);
        if (MODE == CGF_BI_T) add_product(q1, q2, q3, v1, v2, v3, v1, v2, v3, tn, td);
      } else if (MODE != CGF_INIT) {
        add_product(q1, q2, q3, v1, v2, v3, v1, v2, v3, nn, nd);
      }
    }
    if (MODE != CGF_INIT) {
      const float wt = parseval_weight(g, kx, valid);
      sum_n += (double)(wt * nn);
      sum_d += (double)(wt * nd);
      if (MODE == CGF_BI_T) {
        sum_t += (double)(wt * tn);
        sum_t += (double)(wt * td);
      }
    }
  }
  if (a.prof != nullptr && tid == 0) {
    const long long cols = columns_of_cta<TC>(pc, ntiles);
    atomicAdd(a.prof, (unsigned long long)((6 + (MODE == CGF_STEP ? 6 : 3)) * N * cols * (long long)sizeof(cx<float>)));
    atomicAdd(a.prof + 1, (unsigned long long)(N * cols));
  }
  if (MODE != CGF_INIT) {
    // |e|^2 = 2 |q|^2 |v|^2 + 2 |q . v|^2 and tr e = 2 q . v give ||e||^2 and <e, e>_C0
    double* red = reinterpret_cast<double*>(smem_raw);
    __syncthreads();   // the exchange buffers are free
    constexpr bool kBi = MODE == CGF_BI_V || MODE == CGF_BI_T;
    red[tid] = kBi ? sum_n + sum_d : sum_n;
    red[THREADS + tid] = kBi ? sum_t : sum_d;
    __syncthreads();
    if (tid < 32) {
      const double sn = warp_sum_f64(red, THREADS), sd = warp_sum_f64(red + THREADS, THREADS);
      const double lam0 = a.c0 ? a.c0[4 * rve] : a.lam0, mu0 = a.c0 ? a.c0[4 * rve + 1] : a.mu0;
      const double e2 = 2.0 * (sn + sd);
      double vv[2] = {kBi ? 2.0 * sn : 2.0 * mu0 * e2 + 4.0 * lam0 * sd, kBi ? 2.0 * sd : e2};
      const int ncta = gridDim.x;
      if (warp_publish_and_collect<2>(vv, a.part + (long long)rhs * 2 * ncta, a.cnt + rhs, ncta, blockIdx.x) && tid == 0) {
        if (kBi) bicg_finalize(MODE == CGF_BI_V ? BI_ALPHA : BI_OMEGA, a.st[rhs], vv, 1.0);
        else finalize_state(MODE == CGF_RHS ? FIN_RHS : FIN_CG, a.st[rhs], vv, 1.0);
      }
    }
  }
}

// Tile width per depth: 128 to 256 threads per CTA (512 at N3 = 256 and 512, for runs of at least 64 bytes:
// at 512, 8 columns 1.29 and 1.39 ms against 1.36 and 1.53 with 4; at 256, 16 columns 0.640 and 0.571 against 0.640
// and 0.618 with 8; at 128, 16 columns 0.241 and 0.203 against 0.252 and 0.226 with 8).
// Spectra of less than two wide tiles per SM take the narrow form.  Width and grouping depend on the
// grid alone: a load's sums are grouped the same way in launches of any number of loads.
constexpr int wide_tc(int n) {
  return n == 256 ? 16 : n >= 192 ? 8 : n >= 96 ? 16 : n == 64 ? 32 : n == 48 ? 32 : n >= 16 ? 64 : 128;
}
constexpr int narrow_tc(int n) { return n >= 64 ? 8 : n >= 16 ? 16 : 32; }
int tile_width(const Geo& g) {
  const int w = wide_tc(g.n3);
  return g.plane_c >= 2 * 152 * w ? w : narrow_tc(g.n3);
}
// tiles per CTA: up to 4, of launches of one load that still fill the SMs
int tile_group(const Geo& g, int tc) {
  const long long tiles = (g.plane_c + tc - 1) / tc;
  long long k = tiles / 200;
  return (int)(k < 1 ? 1 : k > 4 ? 4 : k);
}

template <int N, int TC, int MODE>
cudaError_t run_inv_mode(const CgZArgs& a, int nrhs, cudaStream_t s) {
  const int tiles = (int)((a.g.plane_c + TC - 1) / TC), group = tile_group(a.g, TC);
  cudaError_t e = set_smem(cg_z_inv_kernel<N, TC, MODE>, ZSmem<N, TC>::bytes);
  if (e != cudaSuccess) return e;
  return launch_dependent(cg_z_inv_kernel<N, TC, MODE>, dim3((unsigned)((tiles + group - 1) / group), (unsigned)nrhs),
                          ZLaunch<N, TC>::threads, ZSmem<N, TC>::bytes, s, a, tiles);
}
template <int N, int TC, int MODE>
cudaError_t run_fwd_mode(const CgZArgs& a, int nrhs, cudaStream_t s) {
  const int tiles = (int)((a.g.plane_c + TC - 1) / TC), group = tile_group(a.g, TC);
  cudaError_t e = set_smem(cg_z_fwd_kernel<N, TC, MODE>, ZSmem<N, TC>::bytes);
  if (e != cudaSuccess) return e;
  return launch_dependent(cg_z_fwd_kernel<N, TC, MODE>, dim3((unsigned)((tiles + group - 1) / group), (unsigned)nrhs),
                          ZLaunch<N, TC>::threads, ZSmem<N, TC>::bytes, s, a, tiles);
}

// every z length
#define HOM_Z_LENGTHS(X) \
  X(1) X(2) X(3) X(4) X(6) X(8) X(12) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512)

}  // namespace

}  // namespace hom
