// Pointwise spectral helpers shared by the z pass (Green contraction) and the equilibrium
// check: the Kelvin basis of symmetric tensors, the product with a wave vector, and the
// discrete wave numbers of the half spectrum.
#pragma once
#include "internal.h"

namespace hom {

// Kelvin components -> symmetric tensor (t11, t22, t33, t23, t13, t12)
template <typename T>
__device__ __forceinline__ void kelvin_to_tensor(const cx<T>* k, cx<T>* t) {
  const T r3 = (T)0.57735026918962576451, r2 = (T)0.70710678118654752440, r6 = (T)0.40824829046386301637;
  t[0] = k[0] * r3 + k[1] * r2 + k[2] * r6;
  t[1] = k[0] * r3 - k[1] * r2 + k[2] * r6;
  t[2] = k[0] * r3 - k[2] * ((T)2 * r6);
  t[3] = k[3] * r2;
  t[4] = k[4] * r2;
  t[5] = k[5] * r2;
}

// w = t xi for a symmetric tensor t
template <typename T>
__device__ __forceinline__ void tensor_dot_xi(const cx<T>* t, T x1, T x2, T x3, cx<T>& w1, cx<T>& w2, cx<T>& w3) {
  w1 = t[0] * x1 + t[5] * x2 + t[4] * x3;
  w2 = t[5] * x1 + t[1] * x2 + t[3] * x3;
  w3 = t[4] * x1 + t[3] * x2 + t[2] * x3;
}

// integer wave number of DFT index j on an axis of length n, Nyquist -> 0 (discrete derivative)
__device__ __forceinline__ int wave(int j, int n) {
  int k = (j >= (n + 1) / 2) ? j - n : j;
  if ((n & 1) == 0 && 2 * j == n) k = 0;
  return k;
}

// Constants of green_from_w for the reference medium (lam0, mu0), or for c0[rve] when c0 is given:
// c1 = 1 / (2 mu0), c2h = (lam0 + mu0) / (2 mu0 (lam0 + 2 mu0))
template <typename T>
__device__ __forceinline__ void green_consts(const double* c0, int rve, double lam0, double mu0, T& c1, T& c2h) {
  if (c0 != nullptr) {
    lam0 = c0[4 * rve];
    mu0 = c0[4 * rve + 1];
  }
  c1 = (T)(1.0 / (2.0 * mu0));
  c2h = (T)((lam0 + mu0) / (2.0 * mu0 * (lam0 + 2.0 * mu0)));
}

// The same by the CTA's thread 0 into shared memory (dst[2]); a barrier follows in the caller.  (In every
// thread, the two FP64 divisions kept the FP32 z passes waiting for the FP64 pipe.)
template <typename T>
__device__ __forceinline__ void green_consts_shared(T* dst, const double* c0, int rve, double lam0, double mu0) {
  if (threadIdx.x == 0) {
    T c1, c2h;
    green_consts<T>(c0, rve, lam0, mu0, c1, c2h);
    dst[0] = c1;
    dst[1] = c2h;
  }
}

// physical frequency of the integer wave number k on axis i: k xs, rounded to T as an FP64 product would be,
// without the FP64 pipe in FP32 and double-float (|k| <= 256 has 9 bits: k times 15 bits is exact)
template <typename T> __device__ __forceinline__ T wave_scaled(const Geo& g, int i, int k) {
  return (T)(k * (i == 0 ? g.xs1 : i == 1 ? g.xs2 : g.xs3));
}
template <> __device__ __forceinline__ float wave_scaled<float>(const Geo& g, int i, int k) {
  const float f = (float)k;
  return fmaf(f, g.xsw[i][0], fmaf(f, g.xsw[i][1], f * g.xsw[i][2]));
}
template <> __device__ __forceinline__ df64 wave_scaled<df64>(const Geo& g, int i, int k) {
  const float f = (float)k;
  const df64 s = df_fast_two_sum(__fmul_rn(f, g.xsw[i][0]), __fmul_rn(f, g.xsw[i][1]));
  return df_fast_two_sum(s.hi, fmaf(f, g.xsw[i][2], s.lo));
}

// The vector at which Gamma0_hat is evaluated for the half-spectrum frequency (kx, ky, n):
//  green == 0: the discrete wave vector xi (Nyquist components 0);
//  green == 1: the rotated finite-difference symbol q_j = sin(xi_j h/2) prod_{l != j} cos(xi_l h/2)
//  from gtab = [sin | cos](pi j / N1), j <= N1/2, then [sin | cos](pi j / N2), [sin | cos](pi j / N3),
//  j < N, by DFT index (cos exactly 0 at N/2).  Indices past N/2 flip sin and cos of an axis
//  together, which flips q as a whole; Gamma0_hat is even, so the operator is unchanged.
template <typename T>
__device__ __forceinline__ void wave_vector(const Geo& g, int green, const double* gtab, int kx, int ky, int n,
                                            T& x1, T& x2, T& x3) {
  if (green == 0) {
    x1 = wave_scaled<T>(g, 0, kx == g.h ? 0 : kx);
    x2 = wave_scaled<T>(g, 1, wave(ky, g.n2));
    x3 = wave_scaled<T>(g, 2, wave(n, g.n3));
  } else {
    const double* t2 = gtab + 2 * (g.h + 1);
    const double* t3 = t2 + 2 * g.n2;
    const double s1 = __ldg(gtab + kx), c1 = __ldg(gtab + g.h + 1 + kx);
    const double s2 = __ldg(t2 + ky), c2 = __ldg(t2 + g.n2 + ky);
    const double s3 = __ldg(t3 + n), c3 = __ldg(t3 + g.n3 + n);
    x1 = (T)(s1 * c2 * c3);
    x2 = (T)(c1 * s2 * c3);
    x3 = (T)(c1 * c2 * s3);
  }
}

// The vector q of CG's vectors in Fourier space (strain v (x) q + q (x) v), q = (a1 cz, a2 cz, a3 sz) with the factors
// of a spectrum column and of a z index.  Gamma0_hat depends on the direction of q alone, so any multiple will
// do, as long as every pass takes the same:
//  green == 0: xi, (a1, a2, a3) = (xi1, xi2, 1), (cz, sz) = (1, xi3);
//  green == 1: the rotated symbol over cos cos cos, the tangents tan(pi j / N), which follow sin and cos in gtab:
//  (t1, t2, 1) and (1, t3).  At a Nyquist index, where the tangent is infinite, the symbol's limit: the axis itself
//  if it is the only one there, else 0.
// So every component is one number rounded once to T, with either operator (as products of three rounded sines and
// cosines those of the rotated one were off by up to 2.5 ulp in FP32).
template <typename T> __device__ __forceinline__ T cg_tangent(const double* t) { return to_compute<T>(__ldg(t)); }
template <typename T>
__device__ __forceinline__ void cg_column_factors(const Geo& g, int green, const double* gtab, int kx, int ky, T& a1, T& a2,
                                                  T& a3) {
  if (green == 0) {
    a1 = wave_scaled<T>(g, 0, kx == g.h ? 0 : kx);
    a2 = wave_scaled<T>(g, 1, wave(ky, g.n2));
    a3 = (T)1;
  } else {
    const double* t = gtab + 2 * (g.h + 1 + g.n2 + g.n3);
    const bool nx = kx == g.h, ny = 2 * ky == g.n2;
    a1 = ny ? (T)0 : nx ? (T)1 : cg_tangent<T>(t + kx);
    a2 = nx ? (T)0 : ny ? (T)1 : cg_tangent<T>(t + g.h + 1 + ky);
    a3 = nx || ny ? (T)0 : (T)1;
  }
}
template <typename T>
__device__ __forceinline__ void cg_z_factors(const Geo& g, int green, const double* gtab, int n, T& cz, T& sz) {
  if (green == 0) {
    cz = (T)1;
    sz = wave_scaled<T>(g, 2, wave(n, g.n3));
  } else {
    const bool nz = 2 * n == g.n3;
    cz = nz ? (T)0 : (T)1;
    sz = nz ? (T)1 : cg_tangent<T>(gtab + 2 * (g.h + 1 + g.n2 + g.n3) + g.h + 1 + g.n2 + n);
  }
}
template <typename T>
__device__ __forceinline__ void cg_wave_vector(const Geo& g, int green, const double* gtab, int kx, int ky, int n, T& q1,
                                               T& q2, T& q3) {
  T cz, sz;
  cg_column_factors<T>(g, green, gtab, kx, ky, q1, q2, q3);
  cg_z_factors<T>(g, green, gtab, n, cz, sz);
  if (green != 0) {   // cz and q3 are 0 or 1
    q1 = cz == (T)0 ? (T)0 : q1;
    q2 = cz == (T)0 ? (T)0 : q2;
  }
  q3 = q3 == (T)0 ? (T)0 : sz;
}

// eta_hat = -Gamma0_hat(xi) : tau_hat in Kelvin components, given w = tau_hat xi.
// Gamma0_hat : tau_hat = v (x) xi + xi (x) v with
// v = w / (2 mu0 |xi|^2) - (lam0 + mu0) / (2 mu0 (lam0 + 2 mu0)) (xi . w) xi / |xi|^4,
// the four-index formula of Sec. 2 contracted with a symmetric tau_hat.
template <typename T>
__device__ __forceinline__ void green_from_w(cx<T>* k, cx<T> w1, cx<T> w2, cx<T> w3, T x1, T x2, T x3, T c1,
                                             T c2h, T scale) {
  const T r3 = (T)0.57735026918962576451, r2 = (T)0.70710678118654752440,
          r6 = (T)0.40824829046386301637, s2 = (T)1.41421356237309504880;
  const T q = x1 * x1 + x2 * x2 + x3 * x3;
  if (q == (T)0) {
#pragma unroll
    for (int i = 0; i < 6; ++i) k[i] = mk<T>(0, 0);
    return;
  }
  const cx<T> s = w1 * x1 + w2 * x2 + w3 * x3;
  const T iq = (T)1 / q;
  const T a1 = c1 * iq * scale;
  const T a2 = c2h * iq * iq * scale;
  const cx<T> v1 = w1 * a1 - s * (a2 * x1);
  const cx<T> v2 = w2 * a1 - s * (a2 * x2);
  const cx<T> v3 = w3 * a1 - s * (a2 * x3);
  const cx<T> e11 = v1 * ((T)-2 * x1), e22 = v2 * ((T)-2 * x2), e33 = v3 * ((T)-2 * x3);
  k[0] = (e11 + e22 + e33) * r3;
  k[1] = (e11 - e22) * r2;
  k[2] = (e11 + e22 - e33 * (T)2) * r6;
  k[3] = (v2 * x3 + v3 * x2) * (-s2);
  k[4] = (v1 * x3 + v3 * x1) * (-s2);
  k[5] = (v1 * x2 + v2 * x1) * (-s2);
}

}  // namespace hom
