// z passes at FP64 accuracy (double-float) around the FP32 CG sweeps in Fourier space (spectral_cg.h).
//
// cg_df_residual: the residual r = b - Gamma0 * (C : (x + E)) only has to reach CG's vectors, so the
// forward x-y transforms of the stress end here: z FFT, contraction to the components v of
// Gamma0 * sigma, r = -v in FP32 and its norms by Parseval.  The inverse z FFT, the inverse x-y pass and
// an FP32 transform of r back to Fourier space are not run.
// cg_df_out: the correction of a sweep, strain of x in double-float and inverse z FFT.  Its x-y
// transforms add it to the FP64 solution free of the FP32 transform's incompatible rounding.
//
// Bound by the double-float chains (a product is two dependent operations, a sum six).  Ending the residual
// here took 16.5 ms per solve of 96^3 spheres, six loads, to 15.1; the FP64 solution from double-float transforms saves
// tight solves a projection and a second residual (256^3, 2e-7: 613 -> 538 ms).
//
// Tiles are those of the cluster z pass (zcluster.cu): 2^lg columns over all planes, one CTA per Kelvin
// component; the residual's contraction reads the six components through distributed shared memory.
#include <cooperative_groups.h>

#include "ls_common.cuh"
#include "spectral.cuh"
#include "spectral_cg.h"

namespace cg = cooperative_groups;

namespace hom {

namespace {

constexpr int kDfEPT = kEptOf<df64>;
constexpr int kDfThreads = 512 * (kEPT / kDfEPT);

// kx, ky of the flat spectrum index f
__device__ __forceinline__ void freq_of(const Geo& g, long long f, int& kx, int& ky) {
  const long long nmain = (long long)g.n2 * g.h;
  if (f < nmain) { ky = (int)g.fd_h.div((unsigned)f); kx = (int)f - ky * g.h; }
  else { ky = (int)(f - nmain); kx = g.h; }
}
// offset of component 0 of frequency (f, n) in a CG vector (see cg_z.cu), components cs apart
__device__ __forceinline__ size_t vec_index(const CgDfArgs& a, int rhs, long long f, int n, int& cs) {
  const int lg = a.vec_lg, N = a.g.n3;
  cs = N << lg;
  return ((size_t)rhs * a.vec_tiles + (size_t)(f >> lg)) * 3 * cs + ((size_t)n << lg) + (size_t)(f & ((1 << lg) - 1));
}

__global__ void __cluster_dims__(6, 1, 1) __launch_bounds__(kDfThreads, 1) cg_df_residual_kernel(const CgDfArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cg::cluster_group cl = cg::this_cluster();
  const Geo& g = a.g;
  const int comp = (int)cl.block_rank();
  const int tile = blockIdx.x / 6, lrhs = blockIdx.y, rhs = a.rhs0 + lrhs;
  if (a.st[rhs].active == 0) return;   // the whole cluster leaves together
  const int lg = a.tc_log2, TC = 1 << lg, n3 = g.n3, per = n3 * TC;
  const long long f0 = (long long)tile * TC;
  cx<df64>* buf = reinterpret_cast<cx<df64>*>(smem_raw);   // [n3][TC]
  cx<df64>* twz = buf + per;
  double* red = reinterpret_cast<double*>(twz + n3);       // [2][threads]
  const int tid = threadIdx.x, nthr = blockDim.x;
  const cx<df64>* Sc = a.S + (long long)(lrhs * 6 + comp) * n3 * g.plane_c;
  for (int e = tid; e < per; e += nthr) {
    const long long f = f0 + (e & (TC - 1));
    if (f < g.plane_c) cp_async_elem<sizeof(cx<df64>)>(buf + e, Sc + (long long)(e >> lg) * g.plane_c + f);
    else buf[e] = mk<df64>(0, 0);
  }
  for (int i = tid; i < n3; i += nthr) twz[i] = ldg_cx(a.tw_n3 + i);
  if (a.prof != nullptr && tid == 0) {
    const long long cols = (g.plane_c - f0 < TC) ? g.plane_c - f0 : TC;
    atomicAdd(a.prof, (unsigned long long)(n3 * cols * (long long)(sizeof(cx<df64>) + sizeof(cx<float>) / 2)));
    if (comp == 0) atomicAdd(a.prof + 1, (unsigned long long)(n3 * cols));
  }
  __shared__ df64 gc[2];
  green_consts_shared<df64>(gc, a.c0, rve_of(rhs, a.rve_loads), a.lam0, a.mu0);
  cp_async_wait_all();
  __syncthreads();
  fft_pencils<df64, -1, kDfEPT>(buf, ColAddr{TC}, n3, TC, a.fd_in, twz);
  cl.sync();   // every component of the tile is transformed along z
  df64 nn = 0, nd = 0;   // weighted sums of |q|^2 |v|^2 and |q . v|^2
  {
    const cx<df64>* part[6];
#pragma unroll
    for (int r = 0; r < 6; ++r) part[r] = cl.map_shared_rank(buf, r);
    const df64 c1 = gc[0], c2h = gc[1];
    const df64 scale = (df64)a.scale;
    const int share = (per + 5) / 6;
    const int q0 = comp * share, q1 = (q0 + share < per) ? q0 + share : per;
    for (int e = q0 + tid; e < q1; e += nthr) {
      const int n = e >> lg;
      const long long f = f0 + (e & (TC - 1));
      if (f >= g.plane_c) continue;
      cx<df64> k[6], tt[6], w1, w2, w3;
#pragma unroll
      for (int i = 0; i < 6; ++i) k[i] = part[i][e];
      int kx, ky;
      freq_of(g, f, kx, ky);
      df64 x1, x2, x3;
      cg_wave_vector<df64>(g, a.green, a.gtab, kx, ky, n, x1, x2, x3);
      kelvin_to_tensor<df64>(k, tt);
      tensor_dot_xi<df64>(tt, x1, x2, x3, w1, w2, w3);
      const df64 q = x1 * x1 + x2 * x2 + x3 * x3;
      cx<df64> v1 = mk<df64>(0, 0), v2 = v1, v3 = v1;
      if (q != (df64)0) {
        const df64 iq = (df64)1 / q, iqs = iq * scale, a1 = c1 * iqs;
        const cx<df64> s = w1 * x1 + w2 * x2 + w3 * x3, sa = s * (c2h * iq * iqs);
        v1 = sa * x1 - w1 * a1;   // r = -v
        v2 = sa * x2 - w2 * a1;
        v3 = sa * x3 - w3 * a1;
        const cx<df64> d = s * ((c2h - c1) * iqs);
        const df64 wt = (kx == 0 || kx == g.h) ? (df64)1 : (df64)2;
        nn += wt * q * (v1.re * v1.re + v1.im * v1.im + v2.re * v2.re + v2.im * v2.im + v3.re * v3.re + v3.im * v3.im);
        nd += wt * (d.re * d.re + d.im * d.im);
      }
      int cs;
      const size_t o = vec_index(a, rhs, f, n, cs);
      a.r[o] = mk<float>((float)v1.re, (float)v1.im);
      a.r[o + cs] = mk<float>((float)v2.re, (float)v2.im);
      a.r[o + 2 * cs] = mk<float>((float)v3.re, (float)v3.im);
    }
  }
  if (tile == a.ntiles - 1) {
    // The vector's last tile may hold columns past the plane.  The FP32 passes carry them along (with weight 0 in
    // the sums, which a NaN would survive): zeros, whatever the buffer held before.
    const int cols = (int)(((long long)a.vec_tiles << a.vec_lg) - g.plane_c);
    for (int e = comp * nthr + tid; e < 3 * n3 * cols; e += 6 * nthr) {
      const int rest = e / cols, i = rest / n3, n = rest - i * n3;
      int cs;
      const size_t o = vec_index(a, rhs, g.plane_c + (e - rest * cols), n, cs);
      a.r[o + (size_t)i * cs] = mk<float>(0.0f, 0.0f);
    }
  }
  // |e|^2 = 2 |q|^2 |v|^2 + 2 |q . v|^2 and tr e = 2 q . v, as in cg_z_fwd
  red[tid] = (double)nn;
  red[nthr + tid] = (double)nd;
  __syncthreads();
  if (tid < 32) {
    const double sn = warp_sum_f64(red, nthr), sd = warp_sum_f64(red + nthr, nthr);
    const int rve = rve_of(rhs, a.rve_loads), ncta = gridDim.x;
    const double lam0 = a.c0 ? a.c0[4 * rve] : a.lam0, mu0 = a.c0 ? a.c0[4 * rve + 1] : a.mu0;
    const double e2 = 2.0 * (sn + sd);
    double v[2] = {2.0 * mu0 * e2 + 4.0 * lam0 * sd, e2};
    if (warp_publish_and_collect<2>(v, a.part + (long long)rhs * 2 * ncta, a.cnt + rhs, ncta, blockIdx.x) && tid == 0)
      finalize_state(a.fin, a.st[rhs], v, 1.0);
  }
  cl.sync();   // the others have read this CTA's buffer
}

__global__ void __launch_bounds__(kDfThreads, 1) cg_df_out_kernel(const CgDfArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Geo& g = a.g;
  const int comp = blockIdx.x % 6, tile = blockIdx.x / 6, lrhs = blockIdx.y, rhs = a.rhs0 + lrhs;
  if (a.st[rhs].active == 0) return;
  const int lg = a.tc_log2, TC = 1 << lg, n3 = g.n3, per = n3 * TC;
  const long long f0 = (long long)tile * TC;
  cx<df64>* buf = reinterpret_cast<cx<df64>*>(smem_raw);
  cx<df64>* twz = buf + per;
  const int tid = threadIdx.x, nthr = blockDim.x;
  const float alpha = a.st[rhs].xpend ? (float)a.st[rhs].alpha : 0.0f;
  const df64 r3 = (df64)(2.0 * 0.57735026918962576451), r2 = (df64)1.41421356237309504880,
             r6 = (df64)(2.0 * 0.40824829046386301637);
  for (int e = tid; e < per; e += nthr) {
    const int n = e >> lg;
    const long long f = f0 + (e & (TC - 1));
    cx<df64> k = mk<df64>(0, 0);
    if (f < g.plane_c) {
      int kx, ky, cs;
      freq_of(g, f, kx, ky);
      df64 q1, q2, q3;
      cg_wave_vector<df64>(g, a.green, a.gtab, kx, ky, n, q1, q2, q3);
      const size_t o = vec_index(a, rhs, f, n, cs);
      cx<df64> v[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {   // x += alpha p where the last update is pending, in FP32 as the iterations
        const cx<float> x = a.x[o + i * cs], p = alpha != 0.0f ? a.p[o + i * cs] : mk<float>(0.0f, 0.0f);
        v[i] = mk<df64>(df64(fmaf(p.re, alpha, x.re)), df64(fmaf(p.im, alpha, x.im)));
      }
      // Kelvin component of v (x) q + q (x) v
      switch (comp) {
        case 0: k = (v[0] * q1 + v[1] * q2 + v[2] * q3) * r3; break;
        case 1: k = (v[0] * q1 - v[1] * q2) * r2; break;
        case 2: k = (v[0] * q1 + v[1] * q2 - v[2] * ((df64)2 * q3)) * r6; break;
        case 3: k = (v[1] * q3 + v[2] * q2) * r2; break;
        case 4: k = (v[0] * q3 + v[2] * q1) * r2; break;
        default: k = (v[0] * q2 + v[1] * q1) * r2; break;
      }
    }
    buf[e] = k;
  }
  for (int i = tid; i < n3; i += nthr) twz[i] = ldg_cx(a.tw_n3 + i);
  __syncthreads();
  fft_pencils<df64, +1, kDfEPT>(buf, ColAddr{TC}, n3, TC, a.fd_in, twz);
  cx<df64>* Sc = a.S + (long long)(lrhs * 6 + comp) * n3 * g.plane_c;
  for (int e = tid; e < per; e += nthr) {
    const long long f = f0 + (e & (TC - 1));
    if (f < g.plane_c) Sc[(long long)(e >> lg) * g.plane_c + f] = buf[e];
  }
  if (a.prof != nullptr && tid == 0) {
    const long long cols = (g.plane_c - f0 < TC) ? g.plane_c - f0 : TC;
    atomicAdd(a.prof, (unsigned long long)(n3 * cols * (long long)(sizeof(cx<df64>) + sizeof(cx<float>) / 2)));
    if (comp == 0) atomicAdd(a.prof + 1, (unsigned long long)(n3 * cols));
  }
}

size_t df_smem(const CgDfArgs& a) {
  return (((size_t)a.g.n3 << a.tc_log2) + a.g.n3) * sizeof(cx<df64>) + 2 * (size_t)a.nthr * sizeof(double);
}
bool df_args_ok(const CgDfArgs& a, int nrhs) {
  return nrhs >= 1 && a.nthr >= 32 && a.nthr <= kDfThreads && ((long long)a.g.n3 << a.tc_log2) <= (long long)kDfEPT * a.nthr &&
         (long long)a.ntiles * 6 <= 0x7fffffffLL;
}

}  // namespace

cudaError_t launch_cg_df_residual(const CgDfArgs& a, int nrhs, cudaStream_t s) {
  if (!df_args_ok(a, nrhs)) return cudaErrorInvalidValue;
  const size_t smem = df_smem(a);
  cudaError_t e = set_smem(cg_df_residual_kernel, smem);
  if (e != cudaSuccess) return e;
  count_launch();
  cg_df_residual_kernel<<<dim3((unsigned)(a.ntiles * 6), (unsigned)nrhs), a.nthr, smem, s>>>(a);
  return cudaGetLastError();
}
cudaError_t launch_cg_df_out(const CgDfArgs& a, int nrhs, cudaStream_t s) {
  if (!df_args_ok(a, nrhs)) return cudaErrorInvalidValue;
  const size_t smem = df_smem(a);
  cudaError_t e = set_smem(cg_df_out_kernel, smem);
  if (e != cudaSuccess) return e;
  count_launch();
  cg_df_out_kernel<<<dim3((unsigned)(a.ntiles * 6), (unsigned)nrhs), a.nthr, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace hom
