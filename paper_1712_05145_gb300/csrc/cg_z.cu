// z passes of the FP32 CG iteration in Fourier space: instantiation and dispatch over the z length
// (kernels in cg_z.cuh).
#include "cg_z.cuh"

namespace hom {

namespace {

template <int N, int TC>
cudaError_t run_inv(const CgZArgs& a, int mode, int nrhs, cudaStream_t s) {
  return mode == CGI_STEP ? run_inv_mode<N, TC, CGI_STEP>(a, nrhs, s) : run_inv_mode<N, TC, CGI_OUT>(a, nrhs, s);
}
template <int N, int TC>
cudaError_t run_fwd(const CgZArgs& a, int mode, int nrhs, cudaStream_t s) {
  return mode == CGF_STEP   ? run_fwd_mode<N, TC, CGF_STEP>(a, nrhs, s)
         : mode == CGF_INIT ? run_fwd_mode<N, TC, CGF_INIT>(a, nrhs, s)
                            : run_fwd_mode<N, TC, CGF_RHS>(a, nrhs, s);
}

}  // namespace

long long cg_vector_elems(const Geo& g) {
  const int tc = tile_width(g);
  return (g.plane_c + tc - 1) / tc * tc * 3 * g.n3;
}
int cg_vector_tile(const Geo& g) { return tile_width(g); }
int cg_z_blocks(const Geo& g) {
  const int tc = tile_width(g);
  const long long tiles = (g.plane_c + tc - 1) / tc, group = tile_group(g, tc);
  return (int)((tiles + group - 1) / group);
}

cudaError_t launch_cg_z_inv(const CgZArgs& a, int mode, int nrhs, cudaStream_t s) {
  if (nrhs < 1) return cudaErrorInvalidValue;
  const int tc = tile_width(a.g);
  count_launch();
  switch (a.g.n3) {
#define HOM_CASE(N)                                                               \
  case N:                                                                         \
    if (tc == wide_tc(N)) return run_inv<N, wide_tc(N)>(a, mode, nrhs, s);        \
    return run_inv<N, narrow_tc(N)>(a, mode, nrhs, s);
    HOM_Z_LENGTHS(HOM_CASE)
#undef HOM_CASE
    default: return cudaErrorInvalidValue;
  }
}
cudaError_t launch_cg_z_fwd(const CgZArgs& a, int mode, int nrhs, cudaStream_t s) {
  if (nrhs < 1) return cudaErrorInvalidValue;
  const int tc = tile_width(a.g);
  count_launch();
  switch (a.g.n3) {
#define HOM_CASE(N)                                                               \
  case N:                                                                         \
    if (tc == wide_tc(N)) return run_fwd<N, wide_tc(N)>(a, mode, nrhs, s);        \
    return run_fwd<N, narrow_tc(N)>(a, mode, nrhs, s);
    HOM_Z_LENGTHS(HOM_CASE)
#undef HOM_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace hom
