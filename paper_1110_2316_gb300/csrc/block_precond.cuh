// Element-block preconditioner: z_e = A_ee^{-1} r_e with A_ee the diagonal
// block of the normal operator A = S^T M S of eq. (4.2) for element e (its
// volume term and its own side of every face term).  Not the thesis's
// preconditioner (Section 5.2, eq. 5.19-5.20, which is kept as the default);
// a block-Jacobi alternative on the same element blocks.
//
// Set-up (FP64): A_ee is formed column by column with the operator kernel in
// self-only mode (neighbour traces taken as zero; MODE_PROBE, or MODE_PLAIN on
// unit vectors for the general, curved and neighbourhood operators), gathered into packed
// lower-triangular storage (row i holds columns 0..i at offset i(i+1)/2),
// factored A_ee = L L^T and X = L^{-1} is formed, both in 64 x 64 tiles.  The preconditioner is z = X^T (X r): two
// triangular products, kept in FP64 and rounded to FP32.  Storing the factor
// rather than A_ee^{-1} keeps the FP32 operator X~^T X~ symmetric positive
// definite whatever the rounding of X (A_ee^{-1} itself rounded to FP32 loses
// definiteness once eps32 * kappa(A_ee) approaches 1).
#pragma once

#include "bj_pass.h"

// offset of (i, j), j <= i, inside one packed block (n <= 1331: fits 32 bits)
__device__ __forceinline__ int pk(int i, int j) { return i * (i + 1) / 2 + j; }

// u[c][off_e + i] = (i == j0 + c) for the group's elements, c < nc
__global__ void k_bj_probe(BjArgs A, int j0, int nc, double *u) {
  const int item = blockIdx.x;
  const int ge = item / nc, c = item - ge * nc;
  const int e = A.elems[ge];
  const int64_t base = (int64_t)c * A.ndof + A.dof_off[e];
  for (int i = threadIdx.x; i < A.n; i += blockDim.x) u[base + i] = (i == j0 + c) ? 1.0 : 0.0;
}

// column j = j0 + c of every block: rows i >= j into packed storage
__global__ void k_bj_gather(BjArgs A, int j0, int nc, const double *y, double *blk) {
  const int item = blockIdx.x;
  const int ge = item / nc, c = item - ge * nc;
  const int e = A.elems[ge], j = j0 + c;
  const int64_t base = (int64_t)c * A.ndof + A.dof_off[e];
  double *B = blk + A.blk_off[e];
  for (int i = j + threadIdx.x; i < A.n; i += blockDim.x) B[pk(i, j)] = y[base + i];
}

// ---------------------------------------------------------------------------
// Factorisation A_ee = L L^T and X = L^{-1} in 64 x 64 tiles of the packed
// blocks, every step one launch over all elements of the group:
//   for block column p: k_bj_diag   L_pp by columns, X_pp = L_pp^{-1}
//                       k_bj_panel  L_ip = A_ip X_pp^T,            i > p
//                       k_bj_syrk   A_ij -= L_ip L_jp^T,       i >= j > p
//   for block row i:    k_bj_xrow   X_ij = -X_ii sum_{j <= m < i} L_im X_mj
// Bound by the FP64 pipe (2 x n^3 / 6 multiply-adds per block).  One CTA per
// block, column by column through global memory, took 119 + 41 ms for 64
// blocks of 729: the tiles spread a block over the SMs and read each operand
// once per 64 multiply-adds (20 ms, of which 13 are the pipe's).
// fail[0] is set (block index + 1) on a non-positive or non-finite pivot; the
// factorisation then goes on with pivot 1 and its result is not used.
// ---------------------------------------------------------------------------
constexpr int BJB = 64;                      // tile edge
constexpr int BJB_LD = BJB + 1;              // leading dimension of a whole tile in shared memory
constexpr int BJB_KC = 32;                   // K chunk of the tile products
constexpr size_t BJB_SMEM2 = 2 * (size_t)BJB * BJB_LD * sizeof(double);
constexpr size_t BJB_SMEM_X = ((size_t)BJB * BJB_LD + 2 * (size_t)BJB * (BJB_KC + 1)) * sizeof(double);

__global__ void __launch_bounds__(256) k_bj_diag(BjArgs A, int p, double *blk, double *xout, int32_t *fail) {
  extern __shared__ double bjb_sm[];
  double *L = bjb_sm, *V = bjb_sm + BJB * BJB_LD;
  __shared__ double s_inv[BJB];
  __shared__ int s_bad;
  const int e = A.elems[blockIdx.x], n = A.n, i0 = BJB * p, m = min(BJB, n - i0);
  double *B = blk + A.blk_off[e], *X = xout + A.blk_off[e];
  const int tid = threadIdx.x;
  for (int t = tid; t < BJB * BJB; t += 256) {
    const int i = t / BJB, j = t - i * BJB;
    L[i * BJB_LD + j] = (i < m && j <= i) ? B[pk(i0 + i, i0 + j)] : 0.0;
    V[i * BJB_LD + j] = i == j ? 1.0 : 0.0;
  }
  if (tid == 0) s_bad = 0;
  __syncthreads();
  const int ri = tid >> 2, rc = tid & 3;
  for (int k = 0; k < m; ++k) {
    if (tid == 0) {
      double d = L[k * BJB_LD + k];
      if (!(d > 0.0) || !isfinite(d)) {
        s_bad = 1;
        d = 1.0;
      }
      d = sqrt(d);
      L[k * BJB_LD + k] = d;
      s_inv[k] = 1.0 / d;
    }
    __syncthreads();
    if (tid > k && tid < m) L[tid * BJB_LD + k] *= s_inv[k];
    __syncthreads();
    if (ri > k && ri < m) {
      const double li = L[ri * BJB_LD + k];
      for (int j = k + 1 + rc; j <= ri; j += 4) L[ri * BJB_LD + j] -= li * L[j * BJB_LD + k];
    }
    __syncthreads();
  }
  // X_pp by forward substitution on the identity, row by row
  for (int k = 0; k < m; ++k) {
    if (tid <= k) V[k * BJB_LD + tid] *= s_inv[k];
    __syncthreads();
    if (ri > k && ri < m) {
      const double li = L[ri * BJB_LD + k];
      for (int j = rc; j <= k; j += 4) V[ri * BJB_LD + j] -= li * V[k * BJB_LD + j];
    }
    __syncthreads();
  }
  for (int t = tid; t < BJB * BJB; t += 256) {
    const int i = t / BJB, j = t - i * BJB;
    if (i < m && j <= i) {
      B[pk(i0 + i, i0 + j)] = L[i * BJB_LD + j];
      X[pk(i0 + i, i0 + j)] = V[i * BJB_LD + j];
    }
  }
  if (tid == 0 && s_bad) atomicCAS(fail, 0, blockIdx.x + 1);
}

// rows r0.. (BJB of them), columns c0 .. c0 + BJB_KC of a packed lower triangle
// into S[row][BJB_KC + 1]; zero above the diagonal and beyond n
__device__ __forceinline__ void bjb_load(const double *B, int n, int r0, int c0, double *S) {
  for (int t = threadIdx.x; t < BJB * BJB_KC; t += 256) {
    const int i = t / BJB_KC, j = t - i * BJB_KC;
    const int r = r0 + i, c = c0 + j;
    S[i * (BJB_KC + 1) + j] = (r < n && c <= r) ? B[pk(r, c)] : 0.0;
  }
}
// the same transposed: rows c0 .. c0 + BJB_KC, columns r0.. into S[column][row]
__device__ __forceinline__ void bjb_load_t(const double *B, int n, int r0, int c0, double *S) {
  for (int t = threadIdx.x; t < BJB * BJB_KC; t += 256) {
    const int j = t / BJB, i = t - j * BJB;
    const int r = c0 + j, c = r0 + i;
    S[i * (BJB_KC + 1) + j] = (r < n && c <= r) ? B[pk(r, c)] : 0.0;
  }
}
// acc[a][b] += sum_k P[ty + 16 a][k] Q[tx + 16 b][k] over one chunk
__device__ __forceinline__ void bjb_mac(const double *P, int ldp, const double *Q, double (&acc)[4][4]) {
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll 4
  for (int k = 0; k < BJB_KC; ++k) {
    double p[4], q[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      p[a] = P[(ty + 16 * a) * ldp + k];
      q[a] = Q[(tx + 16 * a) * (BJB_KC + 1) + k];
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] += p[a] * q[b];
  }
}

// L_ip = A_ip X_pp^T.  grid: n_group * (blocks below p)
__global__ void __launch_bounds__(256) k_bj_panel(BjArgs A, int p, double *blk, const double *xin) {
  __shared__ double P[BJB * (BJB_KC + 1)], Q[BJB * (BJB_KC + 1)];
  const int n = A.n, nt = (n + BJB - 1) / BJB - 1 - p;
  const int ge = blockIdx.x / nt, i = p + 1 + blockIdx.x - ge * nt;
  const int e = A.elems[ge];
  double *B = blk + A.blk_off[e];
  const double *X = xin + A.blk_off[e];
  double acc[4][4] = {};
  for (int c = 0; c < BJB; c += BJB_KC) {
    bjb_load(B, n, BJB * i, BJB * p + c, P);
    bjb_load(X, n, BJB * p, BJB * p + c, Q);
    __syncthreads();
    bjb_mac(P, BJB_KC + 1, Q, acc);
    __syncthreads();
  }
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int r = BJB * i + ty + 16 * a;
      if (r < n) B[pk(r, BJB * p + tx + 16 * b)] = acc[a][b];
    }
}

// A_ij -= L_ip L_jp^T on the trailing tiles.  grid: n_group * T (T + 1) / 2, T = blocks below p
__global__ void __launch_bounds__(256) k_bj_syrk(BjArgs A, int p, double *blk) {
  __shared__ double P[BJB * (BJB_KC + 1)], Q[BJB * (BJB_KC + 1)];
  const int n = A.n, nt = (n + BJB - 1) / BJB - 1 - p, tiles = nt * (nt + 1) / 2;
  const int ge = blockIdx.x / tiles, t = blockIdx.x - ge * tiles;
  int ti = 0;
  while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
  const int i = p + 1 + ti, j = p + 1 + t - ti * (ti + 1) / 2;
  double *B = blk + A.blk_off[A.elems[ge]];
  double acc[4][4] = {};
  for (int c = 0; c < BJB; c += BJB_KC) {
    bjb_load(B, n, BJB * i, BJB * p + c, P);
    bjb_load(B, n, BJB * j, BJB * p + c, Q);
    __syncthreads();
    bjb_mac(P, BJB_KC + 1, Q, acc);
    __syncthreads();
  }
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int r = BJB * i + ty + 16 * a, c = BJB * j + tx + 16 * b;
      if (r < n && c <= r) B[pk(r, c)] -= acc[a][b];
    }
}

// X_ij = -X_ii sum_{j <= m < i} L_im X_mj.  grid: n_group * i (j = 0, the longest sum, first)
__global__ void __launch_bounds__(256) k_bj_xrow(BjArgs A, int i, const double *blk, double *xout) {
  extern __shared__ double bjb_sm[];
  double *S = bjb_sm, *P = bjb_sm + BJB * BJB_LD, *Q = P + BJB * (BJB_KC + 1);
  const int n = A.n;
  const int j = blockIdx.x / A.n_group, ge = blockIdx.x - j * A.n_group;
  const int e = A.elems[ge];
  const double *B = blk + A.blk_off[e];
  double *X = xout + A.blk_off[e];
  double acc[4][4] = {};
  for (int k = BJB * j; k < BJB * i; k += BJB_KC) {
    bjb_load(B, n, BJB * i, k, P);
    bjb_load_t(X, n, BJB * j, k, Q);
    __syncthreads();
    bjb_mac(P, BJB_KC + 1, Q, acc);
    __syncthreads();
  }
  // the sum transposed (S[column][row]) as the right factor of X_ii S
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) S[(tx + 16 * b) * BJB_LD + ty + 16 * a] = acc[a][b];
  double out[4][4] = {};
  for (int c = 0; c < BJB; c += BJB_KC) {
    __syncthreads();
    bjb_load(X, n, BJB * i, BJB * i + c, P);
    __syncthreads();
    // P: X_ii rows; S read as rows tx + 16 b at columns c + k
#pragma unroll 4
    for (int k = 0; k < BJB_KC; ++k) {
      double p[4], q[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        p[a] = P[(ty + 16 * a) * (BJB_KC + 1) + k];
        q[a] = S[(tx + 16 * a) * BJB_LD + c + k];
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) out[a][b] += p[a] * q[b];
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int r = BJB * i + ty + 16 * a;
      if (r < n) X[pk(r, BJB * j + tx + 16 * b)] = -out[a][b];
    }
}

template <typename T>
__global__ void k_bj_convert(const double *in, T *out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (T)in[i];
}

// out_e = X_e in_e (TRANS = false, lower) or X_e^T in_e (TRANS = true) for
// every element of the group and every right-hand side.  CTA tile: TM rows
// of one element x RT right-hand sides, k in chunks of 32; thread tile MR x MC
// with rows tr + TR m and right-hand sides tc + TC c (tr = tid % TR fastest, so
// the shared reads are conflict-free and the stores coalesced; FP32 4 x 4
// tiles instead take 4 consecutive rows / right-hand sides per thread and read
// them with one 16-byte shared load each).  The next
// chunk is fetched into registers while the current one is used.
// grid: n_group * ceil(n / TM) row tiles (row tile fastest, so the tiles of an
// element run together and share its vector segment in L2), ceil(n_rhs / RT).
template <typename T, bool TRANS, int TM, int RT, int TR, int TC>
__global__ void __launch_bounds__(TR *TC) k_bj_tri(BjArgs A, const T *X, const T *in, T *out) {
  constexpr int KC = 32, MR = TM / TR, MC = RT / TC, NT = TR * TC;
  constexpr int NA = (TM * KC + NT - 1) / NT, NB = (KC * RT + NT - 1) / NT;
  // FP32 4 x 4 thread tiles read their operands as float4: rows 4 tr + m and
  // right-hand sides 4 tc + c, rows of the tiles padded to 16 bytes
  constexpr bool VEC = sizeof(T) == 4 && MR == 4 && MC == 4;
  constexpr int PADA = VEC ? 4 : 1, PADB = VEC ? 4 : 1;
  __shared__ __align__(16) T As[KC][TM + PADA];
  __shared__ __align__(16) T Bs[KC][RT + PADB];
  const int n = A.n, nrt = (n + TM - 1) / TM;
  const int ge = blockIdx.x / nrt, rt = blockIdx.x - ge * nrt;
  const int e = A.elems[ge];
  const int i0 = rt * TM, r0 = blockIdx.y * RT;
  const T *Xe = X + A.blk_off[e];
  const int64_t vb = A.dof_off[e];
  const int tid = threadIdx.x, tr = tid % TR, tc = tid / TR;
  T acc[MR][MC];
#pragma unroll
  for (int a = 0; a < MR; ++a)
#pragma unroll
    for (int b = 0; b < MC; ++b) acc[a][b] = (T)0;
  const int kbeg = TRANS ? (i0 / KC) * KC : 0;
  const int kend = TRANS ? n : min(n, i0 + TM);
  T ra[NA], rb[NB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int idx = tid + q * NT;
      int row, kk;
      if (!TRANS) {
        row = idx / KC;
        kk = idx - row * KC;
      } else {
        kk = idx / TM;
        row = idx - kk * TM;
      }
      const int i = i0 + row, k = k0 + kk;
      T v = (T)0;
      if (idx < TM * KC && i < n && k < n) {
        if (!TRANS) {
          if (k <= i) v = Xe[pk(i, k)];
        } else {
          if (i <= k) v = Xe[pk(k, i)];
        }
      }
      ra[q] = v;
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int idx = tid + q * NT;
      const int rr = idx / KC, kk = idx - rr * KC;
      const int k = k0 + kk, rhs = r0 + rr;
      rb[q] = (idx < KC * RT && k < n && rhs < A.n_rhs) ? in[(int64_t)rhs * A.ndof + vb + k] : (T)0;
    }
  };
  if (kbeg < kend) fetch(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += KC) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int idx = tid + q * NT;
      if (idx < TM * KC) {
        if (!TRANS) As[idx % KC][idx / KC] = ra[q];
        else As[idx / TM][idx % TM] = ra[q];
      }
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int idx = tid + q * NT;
      if (idx < KC * RT) Bs[idx % KC][idx / KC] = rb[q];
    }
    __syncthreads();
    if (k0 + KC < kend) fetch(k0 + KC);
#pragma unroll 8
    for (int kk = 0; kk < KC; ++kk) {
      T a[MR], b[MC];
      if constexpr (VEC) {
        const float4 av = *reinterpret_cast<const float4 *>(&As[kk][4 * tr]);
        const float4 bv = *reinterpret_cast<const float4 *>(&Bs[kk][4 * tc]);
        a[0] = av.x; a[1] = av.y; a[2] = av.z; a[3] = av.w;
        b[0] = bv.x; b[1] = bv.y; b[2] = bv.z; b[3] = bv.w;
      } else {
#pragma unroll
        for (int m = 0; m < MR; ++m) a[m] = As[kk][tr + TR * m];
#pragma unroll
        for (int c = 0; c < MC; ++c) b[c] = Bs[kk][tc + TC * c];
      }
#pragma unroll
      for (int m = 0; m < MR; ++m)
#pragma unroll
        for (int c = 0; c < MC; ++c) acc[m][c] += a[m] * b[c];
    }
    __syncthreads();
  }
#pragma unroll
  for (int m = 0; m < MR; ++m) {
    const int i = i0 + (VEC ? 4 * tr + m : tr + TR * m);
    if (i >= n) continue;
#pragma unroll
    for (int c = 0; c < MC; ++c) {
      const int rhs = r0 + (VEC ? 4 * tc + c : tc + TC * c);
      if (rhs < A.n_rhs) out[(int64_t)rhs * A.ndof + vb + i] = acc[m][c];
    }
  }
}

// Vector kernels of the PCG step, one warp per (element, rhs) item, eight items
// per CTA: the FP64 sums are bound by the FP64 pipe, and a warp that keeps its
// item's whole sum adds five values in the end, where a CTA per item added five
// per warp (512 blocks of 729, 16 rhs: 46 + 48 us for the pair, HBM 21 + 7).
constexpr int BJ_VEC_ITEMS = 8;
inline unsigned bj_vec_grid(int items) { return (unsigned)((items + BJ_VEC_ITEMS - 1) / BJ_VEC_ITEMS); }

// PCG update x += alpha p, r -= alpha q on the group's blocks, partial r.r per
// (element, rhs).  grid: bj_vec_grid(n_group * n_rhs), 32 * BJ_VEC_ITEMS threads.
template <typename T>
__global__ void __launch_bounds__(32 * BJ_VEC_ITEMS)
    k_bj_update(BjArgs A, const int32_t *prob, const double *alpha, T *x, T *r, const T *p, const T *q, double *part_rr) {
  const int item = blockIdx.x * BJ_VEC_ITEMS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (item >= A.n_group * A.n_rhs) return;
  const int ge = item / A.n_rhs, rr = item - ge * A.n_rhs;
  const int e = A.elems[ge];
  const int64_t base = (int64_t)rr * A.ndof + A.dof_off[e];
  const T al = (T)alpha[prob[e] * A.n_rhs + rr];
  double s = 0.0;
#pragma unroll 4
  for (int t = lane; t < A.n; t += 32) {
    if (x) x[base + t] += al * p[base + t];
    const T v = r[base + t] - al * q[base + t];
    r[base + t] = v;
    const double w = hpse::widen(v);
    s += w * w;
  }
  s = warp_sum(s);
  if (lane == 0) part_rr[(int64_t)e * A.n_rhs + rr] = s;
}

// partial z.r per (element, rhs) on the group's blocks.  grid and threads as k_bj_update.
template <typename T>
__global__ void __launch_bounds__(32 * BJ_VEC_ITEMS) k_bj_dot(BjArgs A, const T *z, const T *r, double *part) {
  const int item = blockIdx.x * BJ_VEC_ITEMS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (item >= A.n_group * A.n_rhs) return;
  const int ge = item / A.n_rhs, rr = item - ge * A.n_rhs;
  const int e = A.elems[ge];
  const int64_t base = (int64_t)rr * A.ndof + A.dof_off[e];
  double s = 0.0;
#pragma unroll 4
  for (int t = lane; t < A.n; t += 32) s += hpse::widen(z[base + t]) * hpse::widen(r[base + t]);
  s = warp_sum(s);
  if (lane == 0) part[(int64_t)e * A.n_rhs + rr] = s;
}

// Shapes of the two triangular products, picked per degree group and precision
// by timing the candidates of the right-hand-side count on the actual factors
// (bj_candidates).  bj_is_pass: both products in one pass over the factor
// (bj_pass.cuh, bj_mma.cuh); the other variants below 8 are tiles of k_bj_tri
// (rows x right-hand sides per CTA), variant 8 is the tensor-core form
// (bj_tc.cuh: 128 rows x 64 right-hand sides, 3xTF32), offered from 32
// right-hand sides on.  Variants 2 and 8 exist in FP32 only.
// 512 factors of n = 729, one application, tiles -> pass:
// FP32 270 -> 145 us (1 rhs), 468 -> 215 (4), 470 -> 242 (8), 871 -> 359 (16);
// FP64 4820 -> 2417 us (4), 4810 -> 4600 (8), and for 8 blocks 400 -> 98 us
// (4).  In FP64 many large blocks can be faster as tiles (128 blocks of n = 1000:
// 12 rhs 4506, 4805 us in one pass; one rhs 390 and 411), whose FP64 work is the
// same: there the 128 x 8 tile is timed beside the pass, from n = 729 and half the
// SMs on (32 blocks: 1786, 1198 in one pass), and two tiles at one right-hand side.
constexpr int BJ_NVAR = 9;
constexpr int BJ_TC = 8;
// (an entry of a one-pass variant serves the other precision's tile)
constexpr int BJ_TILE[BJ_NVAR][2] = {{64, 64}, {128, 32}, {0, 0},  {128, 8}, {128, 8},
                                     {128, 1}, {128, 1},  {64, 1}, {128, 64}};
inline bool bj_is_pass(int v, bool fp32) { return fp32 ? (v == 2 || v == 4 || v == 6) : (v == 3 || v == 5); }
inline bool bj_variant_ok(int v, bool fp32) { return v >= 0 && v < BJ_NVAR && (fp32 || (v != 2 && v != BJ_TC)); }
// candidates for n_group blocks of size n
inline int bj_candidates(int n, int n_group, int n_rhs, int sms, bool fp32, int *v) {
  int c = 0;
  const int all[3][4] = {{0, 1, 2, BJ_TC}, {3, 4, -1, -1}, {5, 6, 7, -1}};
  const int *a = all[n_rhs >= 32 ? 0 : (n_rhs >= 2 ? 1 : 2)];
  const bool tile = fp32 || (n_rhs >= 9 && n >= 729 && 2 * n_group >= sms);
  for (int i = 0; i < 4; ++i)
    if (a[i] >= 0 && bj_variant_ok(a[i], fp32) && (a[i] != 4 || tile)) v[c++] = a[i];
  return c;
}

template <typename T, int TM, int RT, int TR, int TC>
static void bj_pair(const BjArgs &a, const T *X, const T *r, T *t, T *z, cudaStream_t s) {
  dim3 g(a.n_group * ((a.n + TM - 1) / TM), (a.n_rhs + RT - 1) / RT);
  k_bj_tri<T, false, TM, RT, TR, TC><<<g, TR * TC, 0, s>>>(a, X, r, t);
  k_bj_tri<T, true, TM, RT, TR, TC><<<g, TR * TC, 0, s>>>(a, X, t, z);
}

// z = X^T (X r) for the group with a tile of k_bj_tri; t: scratch vector of the same layout.
template <typename T>
static cudaError_t bj_apply_group(const BjArgs &a, const T *X, const T *r, T *t, T *z, cudaStream_t s, int v) {
  if (a.n_group == 0) return cudaSuccess;
  if (v == 0) bj_pair<T, 64, 64, 16, 16>(a, X, r, t, z, s);
  else if (v == 1) bj_pair<T, 128, 32, 32, 8>(a, X, r, t, z, s);
  else if (v == 7) bj_pair<T, 64, 1, 64, 1>(a, X, r, t, z, s);
  else if (v == (sizeof(T) == 4 ? 3 : 4)) bj_pair<T, 128, 8, 64, 4>(a, X, r, t, z, s);
  else if (v == (sizeof(T) == 4 ? 5 : 6)) bj_pair<T, 128, 1, 128, 1>(a, X, r, t, z, s);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}
