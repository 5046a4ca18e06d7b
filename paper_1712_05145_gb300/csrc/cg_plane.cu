// Middle pass of the FP32 CG iteration in Fourier space (see spectral_cg.h): one CTA takes one
// (z-plane, component, load) of the chunk spectrum through the inverse y and x transforms, the
// material law tau = C : p with the energy <p, C p>, and the forward x and y transforms.
//
// The direction p exists only here: the plane is read and written once.  The y stages next to global
// memory load and store it directly, the row transforms merge, multiply and split in registers
// (cg_xy.cuh), and every stage works in place, so the plane crosses shared memory six times and the
// CTA meets at seven barriers; separate forward and inverse plane kernels took it through twelve
// times (the vectors and their update traffic besides).
#include "cg_xy.cuh"
#include "spectral_cg.h"

namespace hom {

namespace {

// y length n2 = RA RB: the radix-RA stage touches global memory, the radix-RB stage runs on blocks of RB
// consecutive rows.  Between them position P holds index P / RB + RA (P % RB).
template <int N> struct ColPlan;
#define HOM_COLPLAN(N_, A_, B_) \
  template <> struct ColPlan<N_> { static constexpr int RA = A_, RB = B_; };
HOM_COLPLAN(2, 2, 1)
HOM_COLPLAN(3, 3, 1)
HOM_COLPLAN(4, 4, 1)
HOM_COLPLAN(6, 6, 1)
HOM_COLPLAN(8, 8, 1)
HOM_COLPLAN(12, 12, 1)
HOM_COLPLAN(16, 4, 4)
HOM_COLPLAN(24, 6, 4)
HOM_COLPLAN(32, 8, 4)
HOM_COLPLAN(48, 8, 6)
HOM_COLPLAN(64, 8, 8)
HOM_COLPLAN(96, 12, 8)
HOM_COLPLAN(128, 16, 8)
HOM_COLPLAN(192, 16, 12)
HOM_COLPLAN(256, 16, 16)
#undef HOM_COLPLAN

constexpr int kMaxPlane = 8192;   // values of a plane one CTA holds

struct PlaneSmem {
  cx<float>* pl;       // [n2][P]
  cx<float>* col;      // [n2] column 0 of the forward transform, before its separation
  cx<float>*twh, *twy, *tw1;
  float* tab;          // [n_phase] half the component's modulus
  uint8_t* ph;         // [n2][php] phase rows by position
  float* red;          // [threads] energy
  int php;
};
// row pitch of the plane in shared memory: odd, so that consecutive rows fall in distinct banks
template <int H> constexpr int kPitch = (H & 1) ? H : H + 1;

template <int N2, int H>
__device__ __forceinline__ void y_inverse(const PlaneSmem& m, const cx<float>* Sp) {
  constexpr int RA = ColPlan<N2>::RA, RB = ColPlan<N2>::RB, h = H, P = kPitch<H>;
  const cx<float>* nyq = Sp + (unsigned)(N2 * h);
  for (int t = threadIdx.x; t < RB * h; t += blockDim.x) {
    const int j = t / h, col = t % h;
    cx<float> v[RA];
#pragma unroll
    for (int r = 0; r < RA; ++r) v[r] = Sp[(unsigned)((j + r * RB) * h + col)];
    if (col == 0) {   // columns 0 and n1/2 travel together as A + i B
#pragma unroll
      for (int r = 0; r < RA; ++r) {
        const cx<float> b = nyq[j + r * RB];
        v[r] = mk<float>(v[r].re - b.im, v[r].im + b.re);
      }
    }
    SmallDFT<float, RA, +1>::run(v);
#pragma unroll
    for (int r = 0; r < RA; ++r) {
      if (RB > 1 && r > 0) v[r] = cmul(v[r], conj(m.twy[j * r]));
      m.pl[(j + r * RB) * P + col] = v[r];
    }
  }
  __syncthreads();
  if constexpr (RB > 1) {
    for (int t = threadIdx.x; t < RA * h; t += blockDim.x) {
      const int b = t / h, col = t % h;
      cx<float>* q = m.pl + (b * RB) * P + col;
      cx<float> v[RB];
#pragma unroll
      for (int s = 0; s < RB; ++s) v[s] = q[s * P];
      SmallDFT<float, RB, +1>::run(v);
#pragma unroll
      for (int s = 0; s < RB; ++s) q[s * P] = v[s];
    }
    __syncthreads();
  }
}

template <int N2, int H>
__device__ __forceinline__ void y_forward(const PlaneSmem& m, cx<float>* Sp) {
  constexpr int RA = ColPlan<N2>::RA, RB = ColPlan<N2>::RB, h = H, P = kPitch<H>;
  if constexpr (RB > 1) {
    for (int t = threadIdx.x; t < RA * h; t += blockDim.x) {
      const int b = t / h, col = t % h;
      cx<float>* q = m.pl + (b * RB) * P + col;
      cx<float> v[RB];
#pragma unroll
      for (int s = 0; s < RB; ++s) v[s] = q[s * P];
      SmallDFT<float, RB, -1>::run(v);
#pragma unroll
      for (int s = 0; s < RB; ++s) {
        if (s > 0) v[s] = cmul(v[s], m.twy[b * s]);
        q[s * P] = v[s];
      }
    }
    __syncthreads();
  }
  for (int t = threadIdx.x; t < RB * h; t += blockDim.x) {
    const int j = t / h, col = t % h;
    cx<float> v[RA];
#pragma unroll
    for (int r = 0; r < RA; ++r) v[r] = m.pl[(j + r * RB) * P + col];
    SmallDFT<float, RA, -1>::run(v);
    if (col == 0) {
#pragma unroll
      for (int r = 0; r < RA; ++r) m.col[j + r * RB] = v[r];
    } else {
#pragma unroll
      for (int r = 0; r < RA; ++r) Sp[(unsigned)((j + r * RB) * h + col)] = v[r];
    }
  }
  __syncthreads();
  // column 0 holds the transforms of two real columns: A = (P + conj P(-k)) / 2, B = (P - conj P(-k)) / 2i
  cx<float>* nyq = Sp + (unsigned)(N2 * h);
  for (int ky = threadIdx.x; ky < N2; ky += blockDim.x) {
    const cx<float> p = m.col[ky], q = conj(m.col[ky == 0 ? 0 : N2 - ky]);
    Sp[(unsigned)(ky * h)] = (p + q) * 0.5f;
    nyq[ky] = mul_i<float, -1>(p - q) * 0.5f;
  }
}

// the rows of the plane: inverse, material law, forward (times 1/2 times 2, see cg_xy.cuh); returns the sum of
// c p^2 / 2, at most 32 terms in a row in FP32 before a butterfly's sum joins the thread's others.  Consecutive
// threads take consecutive rows: the odd row pitch keeps them in distinct banks.
template <int H>
__device__ __forceinline__ float rows(const PlaneSmem& m, const Geo& g) {
  constexpr int R1 = RowPlan<H>::R1, R2 = RowPlan<H>::R2, NP = row_pair_tasks<H>(), P = kPitch<H>;
  const int n2 = g.n2;
  float sum = 0.0f;
  for (int t = threadIdx.x; t < NP * n2; t += blockDim.x) {
    const int jp = (int)g.fd_n2.div((unsigned)t), row = t - jp * n2;
    cx<float>* q = m.pl + row * P;
    const int jb = jp == 0 ? R2 / 2 : R2 - jp;
    cx<float> A[R1], B[R1];
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      A[r] = q[jp + r * R2];
      if (R2 > 1) B[r] = q[jb + r * R2];
    }
    merge_and_stage<H>(A, B, jp, m.tw1);
    row_twiddle<R1, R2, +1>(A, jp, m.twh);
    if (R2 > 1) row_twiddle<R1, R2, +1>(B, jb, m.twh);
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      q[jp + r * R2] = A[r];
      if (R2 > 1) q[jb + r * R2] = B[r];
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < R1 * n2; t += blockDim.x) {
    const int b = (int)g.fd_n2.div((unsigned)t), row = t - b * n2;
    cx<float>* q = m.pl + row * P + b * R2;
    const uint8_t* ph = m.ph + row * m.php + 2 * b;
    cx<float> v[R2];
#pragma unroll
    for (int s = 0; s < R2; ++s) v[s] = q[s];
    SmallDFT<float, R2, +1>::run(v);
    float acc = 0.0f;
#pragma unroll
    for (int s = 0; s < R2; ++s) {
      const uchar2 f = *reinterpret_cast<const uchar2*>(ph + 2 * R1 * s);
      const cx<float> tau = mk<float>(m.tab[f.x] * v[s].re, m.tab[f.y] * v[s].im);
      acc = fmaf(tau.re, v[s].re, fmaf(tau.im, v[s].im, acc));
      v[s] = tau;
    }
    sum += acc;
    SmallDFT<float, R2, -1>::run(v);
#pragma unroll
    for (int s = 0; s < R2; ++s) {
      if (s > 0) v[s] = cmul(v[s], m.twh[b * s]);
      q[s] = v[s];
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < NP * n2; t += blockDim.x) {
    const int jp = (int)g.fd_n2.div((unsigned)t), row = t - jp * n2;
    cx<float>* q = m.pl + row * P;
    const int jb = jp == 0 ? R2 / 2 : R2 - jp;
    cx<float> A[R1], B[R1];
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      A[r] = q[jp + r * R2];
      if (R2 > 1) B[r] = q[jb + r * R2];
    }
    stage_and_split<H>(A, B, jp, m.tw1);
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      q[jp + r * R2] = A[r];
      if (R2 > 1) q[jb + r * R2] = B[r];
    }
  }
  __syncthreads();
  return sum;
}

#define HOM_PLANE_N2(X) X(2) X(3) X(4) X(6) X(8) X(12) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256)
#define HOM_PLANE_H(X) X(2) X(3) X(4) X(6) X(8) X(12) X(16) X(24) X(32) X(48) X(64) X(96) X(128)

// position -> y index between the y stages, and back
__device__ __forceinline__ int col_rb(int n2) {
  switch (n2) {
#define HOM_CASE(N) case N: return ColPlan<N>::RB;
    HOM_PLANE_N2(HOM_CASE)
#undef HOM_CASE
    default: return 1;
  }
}

// Shared memory holds two planes of 8192 values per SM (with their phases), three of 6144, four of 4608.
// The kernel waits at barriers and for shared memory, so CTAs that run independently of each other are worth more
// than threads of one.  Measured with six loads, ms per launch:
//   2304 to 4608 values: 256 threads of 64 registers, four CTAs: 96^3 0.132 (two of 512 threads: 0.182; three
//     of 80 registers: 0.148), 128x64x64 0.071 (0.096), 96x48x96 0.078 (0.091)
//   6144: 256 threads of 80 registers, three CTAs: 128x96x96 0.153 (two of 512: 0.203), 192x64x64 0.125 (0.147)
//   8192: two CTAs.  Three shapes have that size, and the launch shape is a choice per shape, measured at one depth
//     and six loads each, not a rule: 128x128 takes 80 registers and 256 threads (128^3 0.309, 512 threads of 64: 0.335),
//     256x64 and 64x256 keep 512 of 64 (256x64x64 0.181 with 256 of 80, 0.170; 64x256x64 0.215, 0.210)
// Below 2304 values 8 values per thread are best (32x64x128 0.055, with 256 threads 0.076).
template <int N2, int H>
constexpr bool kWidePlane = N2 * H >= 6144 && (N2 * H < kMaxPlane || N2 == 2 * H);   // 80 registers
bool wide_plane(const Geo& g) {
  const long long e = (long long)g.n2 * g.h;
  return e >= 6144 && (e < kMaxPlane || g.n2 == 2 * g.h);
}
template <int N2, int H, bool Wide>
constexpr bool is_plane = N2 * H <= kMaxPlane && kWidePlane<N2, H> == Wide;
template <int H, bool Wide>
__global__ void __launch_bounds__(Wide ? 256 : 512, Wide ? 3 : 2) cg_plane_kernel(const CgPlaneArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Geo& g = a.g;
  const int z = blockIdx.x, c = blockIdx.y, lrhs = blockIdx.z, rhs = a.rhs0 + lrhs;
  grid_dep_launch();
  constexpr int h = H, n1 = 2 * H, P = kPitch<H>;
  const int n2 = g.n2;
  PlaneSmem m;
  m.php = n1 + 4;   // 2 bytes per value and a word of padding: rows start in distinct banks
  m.pl = reinterpret_cast<cx<float>*>(smem_raw);
  m.col = m.pl + n2 * P;
  m.twh = m.col + n2;
  m.twy = m.twh + h;
  m.tw1 = m.twy + n2;
  const int tid = threadIdx.x, nthr = blockDim.x;
  m.tab = reinterpret_cast<float*>(m.tw1 + h + 1);
  m.red = m.tab + 256;
  m.ph = reinterpret_cast<uint8_t*>(m.red + nthr);
  for (int i = tid; i < h; i += nthr) m.twh[i] = ldg_cx(a.tw_h + i);
  for (int i = tid; i < n2; i += nthr) m.twy[i] = ldg_cx(a.tw_n2 + i);
  for (int i = tid; i <= h; i += nthr) m.tw1[i] = ldg_cx(a.tw_n1 + i);
  const int rve = rve_of(rhs, a.rve_loads);
  const float* mat = a.mat + (long long)rve * kRveTable;
  for (int i = tid; i < a.n_phase; i += nthr) m.tab[i] = 0.5f * mat[i * 4 + (c == 0 ? 2 : 3)];
  // phase rows in the order of the row positions: index y = b + RA s lies at position b RB + s
  const uint8_t* php = a.phase + (long long)rve * g.M + (long long)z * n2 * n1;
  const int rb = col_rb(n2), ra = n2 / rb;
  if ((n1 & 3) == 0) {
    const int words = n1 >> 2;
    for (int y = tid / 32; y < n2; y += nthr / 32) {
      const unsigned* src = reinterpret_cast<const unsigned*>(php + (long long)y * n1);
      unsigned* dst = reinterpret_cast<unsigned*>(m.ph + ((y % ra) * rb + y / ra) * m.php);
      for (int i = tid & 31; i < words; i += 32) dst[i] = src[i];
    }
  } else {
    for (int y = tid / 32; y < n2; y += nthr / 32) {
      const uint8_t* src = php + (long long)y * n1;
      uint8_t* dst = m.ph + ((y % ra) * rb + y / ra) * m.php;
      for (int i = tid & 31; i < n1; i += 32) dst[i] = src[i];
    }
  }
  __syncthreads();
  grid_dep_wait();
  if (a.st[rhs].active == 0) return;
  cx<float>* Sp = a.S + ((long long)(lrhs * 6 + c) * g.n3 + z) * g.plane_c;
  // pairs of lengths of the other kind are not instantiated
  switch (n2) {
#define HOM_CASE(N)                                                    \
  case N:                                                              \
    if constexpr (is_plane<N, H, Wide>) y_inverse<N, H>(m, Sp);       \
    break;
    HOM_PLANE_N2(HOM_CASE)
#undef HOM_CASE
  }
  m.red[tid] = rows<H>(m, g);
  switch (n2) {
#define HOM_CASE(N)                                                    \
  case N:                                                              \
    if constexpr (is_plane<N, H, Wide>) y_forward<N, H>(m, Sp);       \
    break;
    HOM_PLANE_N2(HOM_CASE)
#undef HOM_CASE
  }
  if (a.prof != nullptr && tid == 0) {
    atomicAdd(a.prof, (unsigned long long)(2 * g.plane_c * (long long)sizeof(cx<float>) + (long long)n2 * n1));
    atomicAdd(a.prof + 1, (unsigned long long)((long long)n2 * n1));
  }
  if (tid < 32 && a.fin == FIN_ENERGY) {   // y_forward's barriers have made red complete
    double v[1] = {2.0 * warp_sum_f64(m.red, nthr)};
    const int ncta = 6 * g.n3;
    if (warp_publish_and_collect<1>(v, a.part + (long long)rhs * 2 * ncta, a.cnt + rhs, ncta, c * g.n3 + z) && tid == 0)
      finalize_state(FIN_ENERGY, a.st[rhs], v, 1.0 / (double)g.M);
  }
}

int plane_threads_cg(const Geo& g) {
  const long long e = (long long)g.n2 * g.h;
  if (e >= 2304) return e < kMaxPlane || wide_plane(g) ? 256 : 512;
  int thr = (int)((e + 7) / 8);
  thr = ((thr + 31) / 32) * 32;
  return thr < 64 ? 64 : thr;
}

template <int H, bool Wide>
cudaError_t run_plane(const CgPlaneArgs& a, int nrhs, cudaStream_t s) {
  const Geo& g = a.g;
  const int thr = plane_threads_cg(g);
  const size_t smem = (size_t)(g.n2 * kPitch<H> + 2 * g.n2 + 2 * H + 1) * sizeof(cx<float>) +
                      (256 + thr) * sizeof(float) + (size_t)g.n2 * (g.n1 + 4);
  cudaError_t err = set_smem(cg_plane_kernel<H, Wide>, smem);
  if (err != cudaSuccess) return err;
  return launch_dependent(cg_plane_kernel<H, Wide>, dim3(g.n3, 6, nrhs), thr, smem, s, a);
}

}  // namespace

bool cg_plane_fits(const Geo& g) {
  bool y = false, x = false;
#define HOM_CASE(N) y = y || g.n2 == N;
  HOM_PLANE_N2(HOM_CASE)
#undef HOM_CASE
#define HOM_CASE(N) x = x || g.h == N;
  HOM_PLANE_H(HOM_CASE)
#undef HOM_CASE
  return x && y && (long long)g.n2 * g.h <= kMaxPlane;
}

cudaError_t launch_cg_plane(const CgPlaneArgs& a, int nrhs, cudaStream_t s) {
  if (!cg_plane_fits(a.g) || nrhs < 1 || a.n_phase > 256) return cudaErrorInvalidValue;
  count_launch();
  switch (a.g.h) {
#define HOM_CASE(N)                                                                          \
  case N:                                                                                    \
    if constexpr (256 * N >= 6144)                                                           \
      if (wide_plane(a.g)) return run_plane<N, true>(a, nrhs, s);                            \
    return run_plane<N, false>(a, nrhs, s);
    HOM_PLANE_H(HOM_CASE)
#undef HOM_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace hom
