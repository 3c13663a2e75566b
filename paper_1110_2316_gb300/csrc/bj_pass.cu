// bj_pass.cu -- one unit of the one-pass element-block products per precision
// (a generated translation unit defines BJP_F64 for FP64, then includes this).
#if defined(BJP_F64)
#include "bj_pass.cuh"

cudaError_t bj_pass_f64(const BjArgs &a, const double *X, const double *r, double *z, int32_t *err, cudaStream_t s) {
  if (a.n_group <= 0 || a.n_rhs <= 0) return cudaSuccess;
  if (a.n_rhs == 1) return bjp_by_size<double, 1>(a, X, r, z, err, s);
  // eight right-hand sides per pass where they fit beside one stage of X
  if (a.n_rhs <= 4 || BjpLayout<double, 8>::bytes(a.n, 1) > 225 * 1024) return bjp_by_size<double, 4>(a, X, r, z, err, s);
  return bjp_by_size<double, 8>(a, X, r, z, err, s);
}
#else
#include "bj_mma.cuh"

cudaError_t bj_pass_f32(const BjArgs &a, const float *X, const float *r, float *z, int32_t *err, cudaStream_t s) {
  if (a.n_group <= 0 || a.n_rhs <= 0) return cudaSuccess;
  if (a.n_rhs == 1) return bjp_by_size<float, 1>(a, X, r, z, err, s);
  if (a.n_rhs <= 4) return bjp_by_size<float, 4>(a, X, r, z, err, s);
  if (a.n_rhs <= 8) return bjm_by_size<1>(a, X, r, z, err, s);
  return bjm_by_size<2>(a, X, r, z, err, s);
}
#endif
