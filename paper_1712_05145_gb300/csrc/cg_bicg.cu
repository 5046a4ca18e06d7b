// FP32 BiCGSTAB (see bicgstab.cu) with its vectors in Fourier space (spectral_cg.h): the z passes of the CG
// iteration in four more modes carry the vector updates and sums that surround the two operator
// applications,
//   CGI_BI_P  p = r + beta (p - omega v) (a restart: r_hat = r, p = r), strain of p -> S
//   CGF_BI_V  v = A p, alpha = rho / <r_hat, v>
//   CGI_BI_S  s = r - alpha v, ||s||^2, strain of s -> S
//   CGF_BI_T  t = A s, omega = <t, s> / <t, t>
// and cg_bicg_x, pointwise, ends the iteration: x += alpha p + omega s, r = s - omega t, <r_hat, r> and
// <r, r> by Parseval.  17 spectrum sweeps of 24 B per voxel, load and iteration, where real fields moved 30
// (two LS passes of 6, five vector kernels of 18 together): 32x64x128, six loads, 10.1 -> 6.1 ms per solve.
// The kernel here is a plain stream of 7 vector sweeps, bound by memory.
#include "cg_z.cuh"

namespace hom {

namespace {

template <int N, int TC>
__global__ void __launch_bounds__(ZLaunch<N, TC>::threads) cg_bicg_x_kernel(const CgZArgs a, int ntiles) {
  constexpr int E = ZPlan<N>::E, U = N / E, THREADS = ZLaunch<N, TC>::threads;
  __shared__ double red[2 * THREADS];
  const Geo& g = a.g;
  const int rhs = a.rhs0 + blockIdx.y;
  const int tid = threadIdx.x, tc = tid % TC, u = tid / TC;
  grid_dep_launch();
  grid_dep_wait();
  const RhsState& s = a.st[rhs];
  if (s.active == 0) return;
  const float alpha = (float)s.alpha, omega = (float)s.omega;
  const unsigned pc = (unsigned)g.plane_c;
  double sum_h = 0.0, sum_r = 0.0;   // weighted sums of <r_hat, r> and <r, r>
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const unsigned f = (unsigned)tile * TC + tc;
    const bool valid = f < pc;
    int kx, ky;
    column_of(g, f, valid, kx, ky);
    const ColumnQ cq = column_q(a, kx, ky);
    float hn = 0.0f, hd = 0.0f, rn = 0.0f, rd = 0.0f;
    const size_t block = ((size_t)rhs * ntiles + tile) * (3 * N * TC) + u * TC + tc;
#pragma unroll 4
    for (int e = 0; e < E; ++e) {
      const int n = u + e * U;
      cx<float> r[3], h[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const size_t o = block + i * N * TC + e * U * TC;
        const cx<float> sv = a.s[o];
        a.x[o] = fma_cx(a.p[o], alpha, fma_cx(sv, omega, a.x[o]));
        r[i] = fma_cx(a.t[o], -omega, sv);
        h[i] = a.rh[o];
        a.r[o] = r[i];
      }
      const cx<float> z = z_factors(a, n);
      const float q1 = cq.a1 * z.re, q2 = cq.a2 * z.re, q3 = cq.a3 * z.im;
      add_product(q1, q2, q3, h[0], h[1], h[2], r[0], r[1], r[2], hn, hd);
      add_product(q1, q2, q3, r[0], r[1], r[2], r[0], r[1], r[2], rn, rd);
    }
    const float wt = parseval_weight(g, kx, valid);
    sum_h += (double)(wt * hn) + (double)(wt * hd);
    sum_r += (double)(wt * rn) + (double)(wt * rd);
  }
  red[tid] = sum_h;
  red[THREADS + tid] = sum_r;
  __syncthreads();
  if (tid < 32) {
    double vv[2] = {2.0 * warp_sum_f64(red, THREADS), 2.0 * warp_sum_f64(red + THREADS, THREADS)};
    const int ncta = gridDim.x;
    if (warp_publish_and_collect<2>(vv, a.part + (long long)rhs * 2 * ncta, a.cnt + rhs, ncta, blockIdx.x) && tid == 0)
      bicg_finalize(BI_X, a.st[rhs], vv, 1.0);
  }
}

template <int N, int TC>
cudaError_t run_bicg(const CgZArgs& a, int step, int nrhs, cudaStream_t s) {
  switch (step) {
    case BI_P: return run_inv_mode<N, TC, CGI_BI_P>(a, nrhs, s);
    case BI_ALPHA: return run_fwd_mode<N, TC, CGF_BI_V>(a, nrhs, s);
    case BI_S: return run_inv_mode<N, TC, CGI_BI_S>(a, nrhs, s);
    case BI_OMEGA: return run_fwd_mode<N, TC, CGF_BI_T>(a, nrhs, s);
    case BI_X: {
      const int tiles = (int)((a.g.plane_c + TC - 1) / TC), group = tile_group(a.g, TC);
      return launch_dependent(cg_bicg_x_kernel<N, TC>, dim3((unsigned)((tiles + group - 1) / group), (unsigned)nrhs),
                              ZLaunch<N, TC>::threads, 0, s, a, tiles);
    }
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_cg_bicg(const CgZArgs& a, int step, int nrhs, cudaStream_t s) {
  if (nrhs < 1) return cudaErrorInvalidValue;
  const int tc = tile_width(a.g);
  count_launch();
  switch (a.g.n3) {
#define HOM_CASE(N)                                                               \
  case N:                                                                         \
    if (tc == wide_tc(N)) return run_bicg<N, wide_tc(N)>(a, step, nrhs, s);       \
    return run_bicg<N, narrow_tc(N)>(a, step, nrhs, s);
    HOM_Z_LENGTHS(HOM_CASE)
#undef HOM_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace hom
