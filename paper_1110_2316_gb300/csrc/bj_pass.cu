// bj_pass.cu -- one unit of the one-pass element-block products per precision
// (a generated translation unit defines BJP_F64 for FP64, then includes this).
#if defined(BJP_F64)
#include "bj_pass.cuh"

// eight right-hand sides per pass where they fit beside one stage of X
int bj_pass_rhs_f64(int n, int n_rhs) {
  return n_rhs == 1 ? 1 : (n_rhs <= 4 || BjpLayout<double, 8>::bytes(n, 1) > 225 * 1024 ? 4 : 8);
}
cudaError_t bj_pass_f64(const BjArgs &a, const double *X, const double *r, double *z, cudaStream_t s) {
  if (a.n_group <= 0 || a.n_rhs <= 0) return cudaSuccess;
  const int rt = bj_pass_rhs_f64(a.n, a.n_rhs);
  if (rt == 1) return bjp_by_size<double, 1>(a, X, r, z, s);
  return rt == 4 ? bjp_by_size<double, 4>(a, X, r, z, s) : bjp_by_size<double, 8>(a, X, r, z, s);
}
#else
#include "bj_mma.cuh"

// blocks up to W = 5 keep FP32 FMAs for any count: their sums are short, and the split of
// the matrix instructions would be the larger error (against the FP64 factor, 1 to 512
// elements, mma / chain of FMAs of the tiles: n = 8, 27, 64 1.2e-7, 1.3e-7, 1.46e-7 / 0.6e-7,
// 0.97e-7, 1.38e-7, n = 125 1.27..1.61e-7 / 1.06..1.88e-7, up to 1.33 times, n = 216 up to
// 1.08 times; n = 343 and more 0.4 to 0.88 times), although they would be faster on many
// elements (8,192 of 64, 16 rhs: 90 us, 243 here; 512 of 125 and of 216: 19 and 60 us, 40 and
// 99 here, the tiles 52 and 130)
int bj_pass_rhs_f32(int n, int n_rhs) {
  if (n_rhs == 1) return 1;
  return n_rhs <= 4 || n <= 256 ? 4 : (n_rhs <= 8 ? 8 : 16);
}
cudaError_t bj_pass_f32(const BjArgs &a, const float *X, const float *r, float *z, cudaStream_t s) {
  if (a.n_group <= 0 || a.n_rhs <= 0) return cudaSuccess;
  switch (bj_pass_rhs_f32(a.n, a.n_rhs)) {
    case 1: return bjp_by_size<float, 1>(a, X, r, z, s);
    case 4: return bjp_by_size<float, 4>(a, X, r, z, s);
    case 8: return bjm_by_size<1>(a, X, r, z, s);
    default: return bjm_by_size<2>(a, X, r, z, s);
  }
}
#endif
