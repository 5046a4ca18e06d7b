// Row pass of the FP32 CG iteration in Fourier space (see spectral_cg.h) for planes larger than one
// CTA: a block of rows of the chunk spectrum, between the inverse and the forward y passes (ypass.cu),
// goes through the inverse row transform, the material law with the energy <p, C p>, and the forward
// row transform, in place (cg_xy.cuh).  Rows move straight between global memory and registers:
// consecutive threads take consecutive butterflies of a row, and the task pairs (j, R2 - j) cover whole
// 32-byte sectors.  One radix-R2 block is padded by one value, so that a warp's blocks fall in
// different banks.  Column 0 holds X[0] + i X[n1/2] here, as the y passes leave it.
#include "cg_xy.cuh"
#include "spectral_cg.h"

namespace hom {

namespace {

constexpr int kRowThreads = 128;
// rows of a CTA: the radix-R2 stage (R1 tasks per row) has a task per thread
template <int H> struct RowBlock {
  static constexpr int R1 = RowPlan<H>::R1, R2 = RowPlan<H>::R2;
  static constexpr int rows = kRowThreads / R1;
  static constexpr int pitch = R1 * (R2 + 1);
  static constexpr size_t tables = (size_t)(2 * H + 1) * sizeof(cx<float>);
  static constexpr size_t smem = (size_t)rows * pitch * sizeof(cx<float>) + tables + (256 + kRowThreads) * sizeof(float);
};

// Resident CTAs: latency-bound, so as many as fit with next to no spills, five (96 registers), six up to
// 256-point rows.  512x256x512, one load: 1.054 ms with four, 1.000 with five (1.16 with two of 256 threads, 1.19
// with eight of 64); 384x192x64, two loads: 0.185 -> 0.172; 256^3, two loads: 0.610, 0.550 with five, 0.518 with six.
template <int H> constexpr int row_blocks() { return H > 128 ? 5 : 6; }
template <int H>
__global__ void __launch_bounds__(kRowThreads, row_blocks<H>()) cg_rows_kernel(const CgPlaneArgs a) {
  using RB = RowBlock<H>;
  constexpr int R1 = RB::R1, R2 = RB::R2, NP = row_pair_tasks<H>(), ROWS = RB::rows;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Geo& g = a.g;
  const int c = blockIdx.y, lrhs = blockIdx.z, rhs = a.rhs0 + lrhs;
  grid_dep_launch();
  cx<float>* pl = reinterpret_cast<cx<float>*>(smem_raw);
  cx<float>* twh = pl + ROWS * RB::pitch;
  cx<float>* tw1 = twh + H;
  float* tab = reinterpret_cast<float*>(tw1 + H + 1);   // [256] half the component's modulus
  float* red = tab + 256;                               // [kRowThreads] energy
  const int tid = threadIdx.x;
  const unsigned nrows = (unsigned)g.n2 * (unsigned)g.n3, row0 = blockIdx.x * ROWS;
  const int nr = (int)(nrows - row0 < (unsigned)ROWS ? nrows - row0 : ROWS);
  cx<float>* Sc = a.S + (long long)(lrhs * 6 + c) * g.n3 * g.plane_c;
  const int rve = rve_of(rhs, a.rve_loads);
  const uint8_t* phase = a.phase + (long long)rve * g.M + (long long)row0 * g.n1;
  if (tid == 0) prefetch_l2_if_aligned(phase, (unsigned)(nr * g.n1));
  for (int i = tid; i < H; i += kRowThreads) twh[i] = ldg_cx(a.tw_h + i);
  for (int i = tid; i <= H; i += kRowThreads) tw1[i] = ldg_cx(a.tw_n1 + i);
  const float* mat = a.mat + (long long)rve * kRveTable;
  for (int i = tid; i < a.n_phase; i += kRowThreads) tab[i] = 0.5f * mat[i * 4 + (c == 0 ? 2 : 3)];
  __syncthreads();
  grid_dep_wait();
  if (a.st[rhs].active == 0) return;
  // row r of the block: start of its half spectrum in S
  auto row_ptr = [&](int r) {
    const unsigned gr = row0 + (unsigned)r, z = g.fd_n2.div(gr), y = gr - z * (unsigned)g.n2;
    return Sc + (long long)z * g.plane_c + (long long)y * H;
  };
  for (int t = tid; t < NP * nr; t += kRowThreads) {
    const int row = t / NP, jp = t % NP, jb = jp == 0 ? R2 / 2 : R2 - jp;
    const cx<float>* src = row_ptr(row);
    cx<float> A[R1], B[R1];
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      A[r] = src[jp + r * R2];
      if (R2 > 1) B[r] = src[jb + r * R2];
    }
    merge_and_stage<H>(A, B, jp, tw1);
    row_twiddle<R1, R2, +1>(A, jp, twh);
    if (R2 > 1) row_twiddle<R1, R2, +1>(B, jb, twh);
    cx<float>* q = pl + row * RB::pitch;
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      q[jp + r * (R2 + 1)] = A[r];
      if (R2 > 1) q[jb + r * (R2 + 1)] = B[r];
    }
  }
  __syncthreads();
  cx<float> acc = mk<float>(0.0f, 0.0f);   // of even and odd voxels, at most 32 terms in a row each
  for (int t = tid; t < R1 * nr; t += kRowThreads) {
    const int row = t / R1, b = t % R1;
    cx<float>* q = pl + row * RB::pitch + b * (R2 + 1);
    const uint8_t* ph = phase + (long long)row * g.n1 + 2 * b;
    cx<float> v[R2];
#pragma unroll
    for (int s = 0; s < R2; ++s) v[s] = q[s];
    SmallDFT<float, R2, +1>::run(v);
#pragma unroll
    for (int s = 0; s < R2; ++s) {
      const uchar2 f = *reinterpret_cast<const uchar2*>(ph + 2 * R1 * s);
      const cx<float> tau = mk<float>(tab[f.x] * v[s].re, tab[f.y] * v[s].im);
      acc.re = fmaf(tau.re, v[s].re, acc.re);
      acc.im = fmaf(tau.im, v[s].im, acc.im);
      v[s] = tau;
    }
    SmallDFT<float, R2, -1>::run(v);
#pragma unroll
    for (int s = 0; s < R2; ++s) {
      if (s > 0) v[s] = cmul(v[s], twh[b * s]);
      q[s] = v[s];
    }
  }
  red[tid] = acc.re + acc.im;
  __syncthreads();
  for (int t = tid; t < NP * nr; t += kRowThreads) {
    const int row = t / NP, jp = t % NP, jb = jp == 0 ? R2 / 2 : R2 - jp;
    cx<float>* dst = row_ptr(row);
    const cx<float>* q = pl + row * RB::pitch;
    cx<float> A[R1], B[R1];
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      A[r] = q[jp + r * (R2 + 1)];
      if (R2 > 1) B[r] = q[jb + r * (R2 + 1)];
    }
    stage_and_split<H>(A, B, jp, tw1);
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      dst[jp + r * R2] = A[r];
      if (R2 > 1) dst[jb + r * R2] = B[r];
    }
  }
  if (a.prof != nullptr && tid == 0) {
    const long long vox = (long long)nr * g.n1;
    atomicAdd(a.prof, (unsigned long long)(2LL * nr * H * (long long)sizeof(cx<float>) + vox));
    atomicAdd(a.prof + 1, (unsigned long long)vox);
  }
  if (tid < 32 && a.fin == FIN_ENERGY) {
    double v[1] = {2.0 * warp_sum_f64(red, kRowThreads)};
    const int ncta = 6 * gridDim.x;
    if (warp_publish_and_collect<1>(v, a.part + (long long)rhs * 2 * ncta, a.cnt + rhs, ncta,
                                    c * gridDim.x + blockIdx.x) && tid == 0)
      finalize_state(FIN_ENERGY, a.st[rhs], v, 1.0 / (double)g.M);
  }
}

template <int H>
cudaError_t run_rows(const CgPlaneArgs& a, int nrhs, cudaStream_t s) {
  cudaError_t e = set_smem(cg_rows_kernel<H>, RowBlock<H>::smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(cg_rows_kernel<H>, dim3(cg_row_blocks(a.g), 6, nrhs), kRowThreads, RowBlock<H>::smem, s, a);
}

#define HOM_ROW_LENGTHS(X) \
  X(2) X(3) X(4) X(6) X(8) X(12) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512)

}  // namespace

int cg_row_blocks(const Geo& g) {
  int rows = 1;
  switch (g.h) {
#define HOM_CASE(N) case N: rows = RowBlock<N>::rows; break;
    HOM_ROW_LENGTHS(HOM_CASE)
#undef HOM_CASE
  }
  return (int)(((long long)g.n2 * g.n3 + rows - 1) / rows);
}

cudaError_t launch_cg_rows(const CgPlaneArgs& a, int nrhs, cudaStream_t s) {
  if (nrhs < 1 || a.n_phase > 256) return cudaErrorInvalidValue;
  count_launch();
  switch (a.g.h) {
#define HOM_CASE(N) case N: return run_rows<N>(a, nrhs, s);
    HOM_ROW_LENGTHS(HOM_CASE)
#undef HOM_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace hom
