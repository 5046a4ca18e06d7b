// FP32 CG iteration with its vectors in Fourier space (host interface; kernels in cg_z.cu,
// cg_plane.cu and cg_rows.cu).
//
// Every vector of the CG form (Eq. cg_form) is a compatible strain, e_hat(xi) = v (x) q + q (x) v with
// the wave vector q of the Green operator, so r, p and x are kept as the three complex components v
// per frequency.  One iteration of a chunk of loads is three passes over its spectrum scratch S:
//   cg_z_inv : x += alpha p, p = r + beta p (per frequency), strain of p, inverse z FFT      -> S
//   cg_plane : inverse y and x transforms, tau = C : p with <p, C p>, forward transforms     S -> S
//              (planes above one CTA: the y pass, cg_rows on blocks of rows, the y pass)
//   cg_z_fwd : forward z FFT, v = Gamma0_hat(q) : tau_hat, r -= alpha v, the norms of r      <- S
// A spectrum sweep is 24 B per voxel and load.  The passes move 3.5 + 2 + 2 of them where vectors held
// as six real components moved 6 + 2 + 3, and CG's vectors stay compatible exactly.
#pragma once
#include "internal.h"

namespace hom {

struct CgZArgs {
  Geo g;
  cx<float>* S;            // chunk spectrum [load][6][n3][plane_c]
  cx<float>* r;            // [rhs][tile of columns][3][n3][columns] each (cg_vector_elems per rhs)
  cx<float>* p;
  cx<float>* x;
  cx<float>*rh, *v, *s, *t;  // BiCGSTAB: r_hat, v = A p, s, t = A s
  int rhs0;
  RhsState* st;
  double lam0, mu0;
  int rve_loads;
  const double* c0;        // several RVE slots: [rve][4], see ZArgs
  float scale;             // 1 / M, the factor of the forward transform
  int green;
  const double* gtab;
  const cx<float>* tw_n3;
  double* part;            // cg_z_fwd: [rhs][2][CTAs]
  unsigned* cnt;
  unsigned long long* prof;
};
// cg_z_inv: CGI_STEP the iteration's first pass; CGI_OUT x += alpha p where pending, strain of x -> S
// cg_z_fwd: CGF_STEP the iteration's last pass; CGF_INIT r = the components v of a compatible strain;
//           CGF_RHS r = -Gamma0_hat : tau_hat with its norms (the right-hand side, from tau = (C - C0) : E)
// The BI modes are BiCGSTAB's (cg_bicg.cu).
enum CgInvMode { CGI_STEP = 0, CGI_OUT = 1, CGI_BI_P = 2, CGI_BI_S = 3 };
enum CgFwdMode { CGF_STEP = 0, CGF_INIT = 1, CGF_RHS = 2, CGF_BI_V = 3, CGF_BI_T = 4 };

// z passes in double-float around a sweep (cg_df.cu), with the tiles of the cluster z pass
struct CgDfArgs {
  Geo g;
  cx<df64>* S;             // chunk spectrum [load][6][n3][plane_c]
  cx<float>* r;            // cg_df_residual writes r
  const cx<float>* p;      // cg_df_out reads x and p
  const cx<float>* x;
  int vec_lg;              // log2 of the vectors' tile width, and tiles per load (cg_vector_tile)
  int vec_tiles;
  int rhs0;
  RhsState* st;
  int fin;                 // cg_df_residual: FIN_RHS or FIN_RESID
  double lam0, mu0;
  int rve_loads;
  const double* c0;
  double scale;            // 1 / M
  int green;
  const double* gtab;
  const cx<df64>* tw_n3;
  int tc_log2, ntiles, nthr;   // tiling of zcluster_tiling<df64>
  FastDiv fd_in;
  double* part;            // cg_df_residual: [rhs][2][6 ntiles]
  unsigned* cnt;
  unsigned long long* prof;
};
// r = -v(tau_hat) and its norms, from the x-y transforms of tau = C : (x + E) - C0 : b: r = b - Gamma0 * (C : (x + E))
cudaError_t launch_cg_df_residual(const CgDfArgs& a, int nrhs, cudaStream_t s);
// strain of x (with its pending update), inverse z FFT -> S
cudaError_t launch_cg_df_out(const CgDfArgs& a, int nrhs, cudaStream_t s);

struct CgPlaneArgs {
  Geo g;
  cx<float>* S;
  int fin;                 // FIN_ENERGY: reduce <p, C p>; FIN_NONE (BiCGSTAB)
  int rhs0;
  RhsState* st;
  const uint8_t* phase;    // [rve][n3][n2][n1]
  const float* mat;        // [rve][256][4]
  int n_phase;
  int rve_loads;
  const cx<float>* tw_h;
  const cx<float>* tw_n1;
  const cx<float>* tw_n2;
  double* part;
  unsigned* cnt;
  unsigned long long* prof;
};

long long cg_vector_elems(const Geo& g);  // complex values of one load's vector
int cg_vector_tile(const Geo& g);         // columns of one of its tiles (a power of two)
int cg_z_blocks(const Geo& g);            // CTAs of one load in the z passes
cudaError_t launch_cg_z_inv(const CgZArgs& a, int mode, int nrhs, cudaStream_t s);
cudaError_t launch_cg_z_fwd(const CgZArgs& a, int mode, int nrhs, cudaStream_t s);
// one of BiCGSTAB's passes (BI_P, BI_ALPHA, BI_S, BI_OMEGA, BI_X; cg_bicg.cu)
cudaError_t launch_cg_bicg(const CgZArgs& a, int step, int nrhs, cudaStream_t s);
// whether one CTA holds a plane of the grid in cg_plane (else the y pass and cg_rows run)
bool cg_plane_fits(const Geo& g);
cudaError_t launch_cg_plane(const CgPlaneArgs& a, int nrhs, cudaStream_t s);
int cg_row_blocks(const Geo& g);          // CTAs of one (load, component) in cg_rows
cudaError_t launch_cg_rows(const CgPlaneArgs& a, int nrhs, cudaStream_t s);

}  // namespace hom
