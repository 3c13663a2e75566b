// registry.h -- interface between the host library and the per-(precision,
// degree) kernel translation units.  Each unit compiles kernels.cuh for one
// (REAL, WDEG) pair and fills a KernelSet with launchers.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace hpse {

// FP32 -> FP64, exact, by moving the bits: the conversion instruction runs on the
// FP64 pipe (two lanes per clock and SM) and would bound the FP64 sums of FP32
// vectors.  Subnormals go through an exact FP32 scaling by 2^24.
__device__ __forceinline__ double widen(float v) {
  const uint32_t b = __float_as_uint(v), s = b & 0x80000000u, a = b & 0x7fffffffu;
  uint32_t hi = (a >> 3) + 0x38000000u, lo = b << 29;  // exponent bias 127 -> 1023
  if (a - 0x00800000u >= 0x7f000000u) {                // zero, subnormal, infinity, NaN
    if (a >= 0x7f800000u) {
      hi = (a >> 3) + 0x70000000u;
    } else if (a == 0) {
      hi = lo = 0;
    } else {
      const uint32_t u = __float_as_uint(__uint_as_float(a) * 16777216.f);
      hi = (u >> 3) + 0x38000000u - (24u << 20);
      lo = u << 29;
    }
  }
  return __hiloint2double((int)(s | hi), (int)lo);
}
__device__ __forceinline__ double widen(double v) { return v; }

// COEF_EDGE: -(u_11 + u_22 + kappa(x_1) u_33) in the edge neighbourhood's
// modified coordinates, kappa = e^{2 tau} per x-point of the element
// COEF_VERTEX: the variable-coefficient form with per-point weights and
// first-order terms, u_22 scaled by 1/sin^2(x_1) per x-point (vertex
// neighbourhood, modified coordinates (phi, theta, ln rho))
// COEF_VERTEX_EDGE: the variable-coefficient form with the mixed term u_13 in
// place of u_2 (vertex-edge neighbourhood, (ln tan phi, theta, ln x3)):
// per-point m and coefficients of (u_1, u_13, u_3), u_11 scaled by 1 + kappa
// and u_33 by kappa per x-point, kappa = e^{2 psi}
// COEF_GENERAL: the ten-term operator of eq. (5.45) with per-point
// coefficients (weight and C's, GEN_NC = 12 per point; general.cuh)
enum { COEF_LAPLACE = 0, COEF_SCALAR = 1, COEF_EDGE = 2, COEF_VERTEX = 3, COEF_VERTEX_EDGE = 4, COEF_GENERAL = 5 };
// KAPPA_STRIDE = 2 * HPSE_MAX_W + 1, CSCR_STRIDE = HPSE_MAX_W + 1 (checked in the host library)
enum { KAPPA_STRIDE = 21, CSCR_STRIDE = 11, FACE_W = 10, ZEIG_STRIDE = 132 };
// MODE_RESIDUAL: z = sqrt(w J) (L u - f) at the volume points, no transpose (COEF_LAPLACE, COEF_SCALAR)
// MODE_PROBE: column probe0 + (the item's right-hand side) of the element's diagonal block
// A_ee (FP64, COEF_LAPLACE, COEF_SCALAR; with self_only), rows at and below the diagonal
enum { MODE_PLAIN = 0, MODE_PCG = 1, MODE_TRANSPOSE = 2, MODE_RESIDUAL = 3, MODE_PROBE = 4 };

template <typename T>
struct ApplyArgsT {
  const T *u;
  T *y;
  const int32_t *elems;
  int32_t n_group;
  int32_t n_rhs;
  int64_t ndof;
  const int64_t *dof_off;
  const int32_t *nbr;
  const T *geo;
  const int32_t *prob;
  const T *coef;            // [nquad][4]: m, d_x, d_y (COEF_VERTEX_EDGE: d_xz), d_z per volume point;
                            // COEF_GENERAL: [nquad][12] (w |J|, C_11 .. C_0, 0)
  const int64_t *coef_off;
  int64_t nquad;
  const T *z;
  const double *beta;
  T *pnew;
  double *partial;
  const double *rho;        // MODE_TRANSPOSE: the weighted point values, or null with zin
  // residual map: w J, a at the points ([2][nquad] of the mesh's FP64 data), the
  // source f, the point values written (MODE_RESIDUAL) or transposed (MODE_TRANSPOSE)
  const double *aux;
  const double *f;
  const double *sqw64;      // [nquad] square root of w J
  const T *sqw;
  T *zout;
  const T *zin;
  int32_t skip_faces;
  int32_t self_only;        // 1: neighbour traces taken as zero (diagonal blocks of A)
  int32_t probe0;           // MODE_PROBE: the first column of the launch
  // edge neighbourhood (COEF_EDGE); null / 0 for box meshes
  int32_t n_elem;           // corner set c's values start at dof_off[n_elem + c]
  const T *kappa;           // [E][KAPPA_STRIDE]: per x-point factor (e^{2 tau}, 1/sin^2 phi, e^{2 psi})
  const T *fw;              // [E][6][10] face-norm weights (null: all 1)
  const int32_t *cslot;     // [E][2] slot of the element's corner face 0 / face 4, or -1
  T *cscr;                  // [slots][n_rhs][CSCR_STRIDE] corner-side face contributions
  // outer-face conditions of box meshes of the Laplacian; null: every outer face Dirichlet
  const int32_t *fbc;       // [E][6]: 0 Dirichlet, 1 Neumann, 2 Robin
  const T *fgam;            // [E][6]: the Robin gamma (0 elsewhere)
};

template <typename T>
struct PrecArgsT {
  const int32_t *elems;
  int32_t n_group;
  int32_t n_rhs;
  int64_t ndof;
  const int64_t *dof_off;
  const int32_t *prob;
  const T *rin;
  T *zout;
  T *x;
  T *r;
  const T *p;
  const T *q;
  const double *alpha;
  double *part_rr;
  double *part_rz;
  // edge neighbourhood, C* form (eq. 5.30): per element the x3 eigenbasis
  // S_z (P x P, node-major) then its eigenvalues nu (P), ZEIG_STRIDE apart;
  // null for box meshes (the master C-form in every direction)
  const T *zeig;
};

// Packed FP64 tables for one degree, in the order of the device struct:
// B0, B1, B2 (Q*P each), D (P*P), S (P*P), MP (P*P), KP (P*P), WQ (Q), MU (P),
// then DQ (Q*Q, the differentiation matrix of the Q-point grid).
inline int packed_table_size(int W) {
  const int P = W + 1, Q = 2 * W + 1;
  return 3 * Q * P + 4 * P * P + Q + P + Q * Q;
}

// Second FP64 launch shape of the apply kernels (units f64b, HPSE_APPLY_ONLY):
// the threads per CTA that suit the other end of the item counts than the
// first one.  W = 2..5: more threads (128, 128, 192, 256 for 64, 64, 96, 128),
// for launches of at most one item per SM, where an item's latency counts and
// the extra warps shorten the line stages and the face phase (Laplacian / variable
// coefficient, one item per SM: W = 3 22.7 -> 18.7 / 31.0 -> 26.8 us, W = 4 31.5 ->
// 24.8 / 45.4 -> 37.1); with two and more items per SM they cost up to 20 %.
// W = 6, 7: fewer (128 for 192, 256), for launches of more items than SMs, where
// the registers then allow two CTAs per SM and one's barriers hide behind the
// other (1,024 items: W = 6 387 -> 346 / 605 -> 564 us, W = 7 537 -> 503 / 887 ->
// 843); a lone item is slower (57.6 -> 65.7 us).
constexpr int ALT_W0 = 2, ALT_W1 = 7;
constexpr int ALT_THREADS[ALT_W1 - ALT_W0 + 1] = {128, 128, 192, 256, 128, 128};
inline bool alt_shape(int W, long long items, long long all_items, int sms) {
  if (W < ALT_W0 || W > ALT_W1) return false;
  return W <= 5 ? all_items <= sms : items > sms;  // all_items: over every degree of the launch
}

struct KernelSet {
  int W;
  int is_double;
  cudaError_t (*upload)(const double *packed);
  // coef: COEF_*, mode: MODE_*; args points to ApplyArgsT<T>
  cudaError_t (*apply)(int coef, int mode, const void *args, int n_items, int threads, cudaStream_t s);
  size_t (*apply_smem)(int coef);
  int (*apply_max_threads)(int coef);
  // mode: MODE_PLAIN or MODE_PCG; args points to PrecArgsT<T>; sms: SMs of the device
  cudaError_t (*precond)(int mode, const void *args, int n_items, int sms, cudaStream_t s);
  // volume transpose in integration-by-parts form (COEF_LAPLACE, COEF_SCALAR;
  // args as for MODE_TRANSPOSE); ibp_smem: its shared memory, 0 where the
  // instance is not built
  cudaError_t (*transpose_ibp)(int coef, const void *args, int n_items, cudaStream_t s);
  size_t (*ibp_smem)(int coef);
};

}  // namespace hpse
