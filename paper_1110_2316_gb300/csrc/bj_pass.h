// bj_pass.h -- arguments of the element-block preconditioner's kernels and the
// entry points of its one-pass product (bj_pass.cu, one unit per precision).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

struct BjArgs {
  const int32_t *elems;    // element ids of one degree group
  int32_t n_group;         // elements in the group
  int32_t n;               // block size (W+1)^3
  int32_t n_rhs;
  int64_t ndof;            // stride between right-hand sides of a vector
  const int64_t *dof_off;  // per element
  const int64_t *blk_off;  // per element: offset of its packed block
  int32_t *err;            // host-mapped, set when a bounded wait expired
  int32_t polls;           // polls after which a wait gives up
};

// Waits of the block products are bounded: BJ_POLLS polls (about a second; tests
// lower the limit of the first wait, never that of the one before the CTA ends).
// An expired wait sets *err, lets what the CTA still has in flight land (bounded
// too) and leaves NaN in the CTA's part of z.
constexpr int BJ_POLLS = 1 << 22;
#if defined(__CUDACC__)
__device__ __forceinline__ void bj_flag(int32_t *err) {
  *(volatile int32_t *)err = 1;
  __threadfence_system();
}
#endif

// z = X^T (X r) for the group's elements and all right-hand sides (bj_pass.cuh).
// X is read in whole 16-byte words: its allocation extends to the next one.
cudaError_t bj_pass_f32(const BjArgs &a, const float *X, const float *r, float *z, cudaStream_t s);
cudaError_t bj_pass_f64(const BjArgs &a, const double *X, const double *r, double *z, cudaStream_t s);
// right-hand sides that one CTA of the above takes, for blocks of size n
int bj_pass_rhs_f32(int n, int n_rhs);
int bj_pass_rhs_f64(int n, int n_rhs);
