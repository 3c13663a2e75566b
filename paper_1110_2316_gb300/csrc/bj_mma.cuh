// bj_mma.cuh -- the one-pass product z = X^T (X r) (bj_pass.cuh) for 5 to 31
// FP32 right-hand sides (variant 2: any count from 32 on) of blocks above n = 256:
// the same walk over blocks of 16 rows of X, with the products on mma.sync
// m16n8k8 (TF32).  At 8 and 16 right-hand sides the packed FMAs and their shared
// loads bound the pass (271 and 480 us for 512 blocks of 729); the matrix
// instructions cut the issued instructions, so that what is left is the latency
// of a block: split, MMA and addition chains, two barriers, 16 warps per SM, no
// pipe above 27 % (242 and 359 us; the two-product tiles took 470 and 871 us).  mma.sync and not
// tcgen05: the operand is a triangular, unaligned packed row block that is read
// once, at N = 8 or 16.
//
// FP32 accuracy: every operand is split, v = hi + lo (TF32 each), and a product
// takes lo hi + hi lo + hi hi.  The tensor core truncates its accumulator, so
// sums run over 16 terms only and are added up in FP32 registers: the error
// against 64 bits is 1.6e-7 at n = 729 (a chain of FP32 FMAs: 4.5e-7), where one
// long accumulation on the tensor core would lose a digit.
//
// Layout: the columns of a lane are chosen so that the packed rows need no
// padding: consecutive triangular numbers are distinct modulo 2^k, so lanes on
// 8 rows x columns 8 apart (t), or 4 rows x columns 4 apart (z), touch 32
// different banks.  r is kept as ready B fragments (hi, hi, lo, lo of the two
// k's of a lane), or as FP32 values split at each use where those do not fit; t
// of the block likewise; z stays in the accumulator layout.
// Block b + 1's t is formed in the same barrier interval as block b's z.
//
// Range: lo is 2^-11 of its value and keeps 11 bits, so a right-hand side whose entries are
// all below 2^-110 loses them to the subnormals (n = 729: error 1.3e-7 down to 2^-110,
// 3.5e-7 at 2^-115, 9e-6 at 2^-120; FP32 FMAs 2e-7), and hi is infinite from
// 2^128 (1 - 2^-12) on.  Scaling such right-hand sides by a power of two cost every product
// 3 to 6 %.
#pragma once
#include "bj_pass.cuh"

// shared memory: X stages | r fragments | partial t | t fragments
template <int NT8, int NW, bool PRE>
struct BjmLayout {
  static constexpr int RT = 8 * NT8;
  __host__ __device__ static int chunks(int n) { return (n + 31) / 32; }
  // floats of one X stage: 16 rows of up to n16 entries and the 16-byte slack at both ends
  __host__ __device__ static int stage(int n) { return BJP_BR * (((n + BJP_BR - 1) / BJP_BR) * BJP_BR) + 8; }
  __host__ __device__ static size_t bytes(int n, int stages) {
    return sizeof(float) * ((size_t)stages * stage(n) + (size_t)chunks(n) * 4 * NT8 * (PRE ? 128 : 64) + (size_t)NW * BJP_BR * RT +
                            2 * NT8 * 128);
  }
};

// v = hi + lo: hi = v rounded to TF32 (nearest, ties away), lo the exact rest
// (the tensor core reads its upper 11 significant bits)
__device__ __forceinline__ void bjm_split(float v, uint32_t &hi, uint32_t &lo) {
  hi = (__float_as_uint(v) + 0x1000u) & 0xffffe000u;
  lo = __float_as_uint(v - __uint_as_float(hi));
}
// d += a b, m16n8k8, TF32 operands
__device__ __forceinline__ void bjm_mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, "
      "%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float bjm_lds(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}
// B fragment i of r (hi, hi, lo, lo of the two k's of a lane): kept split (PRE), or as
// the FP32 values and split here
template <bool PRE>
__device__ __forceinline__ float4 bjm_frag(uint32_t rf, int i, int lane) {
  float4 v;
  if constexpr (PRE) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(rf + 16 * (32 * i + lane))
                 : "memory");
  } else {
    float x, y;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(x), "=f"(y) : "r"(rf + 8 * (32 * i + lane)) : "memory");
    uint32_t h0, l0, h1, l1;
    bjm_split(x, h0, l0);
    bjm_split(y, h1, l1);
    v = make_float4(__uint_as_float(h0), __uint_as_float(h1), __uint_as_float(l0), __uint_as_float(l1));
  }
  return v;
}
// the six products of two k-steps of one n8 tile (A hi/lo, B = (hi, hi, lo, lo) of the step), small terms apart
__device__ __forceinline__ void bjm_prod(const uint32_t (&ah)[2][4], const uint32_t (&al)[2][4], const float4 &b0,
                                         const float4 &b1, float (&acc)[4]) {
  float d[4] = {0.f, 0.f, 0.f, 0.f}, f[4] = {0.f, 0.f, 0.f, 0.f};
  bjm_mma(d, ah[0], __float_as_uint(b0.x), __float_as_uint(b0.y));
  bjm_mma(f, al[0], __float_as_uint(b0.x), __float_as_uint(b0.y));
  bjm_mma(d, ah[1], __float_as_uint(b1.x), __float_as_uint(b1.y));
  bjm_mma(f, al[1], __float_as_uint(b1.x), __float_as_uint(b1.y));
  bjm_mma(f, ah[0], __float_as_uint(b0.z), __float_as_uint(b0.w));
  bjm_mma(f, ah[1], __float_as_uint(b1.z), __float_as_uint(b1.w));
#pragma unroll
  for (int i = 0; i < 4; i += 2) {
    const float2 v = __fadd2_rn(__fadd2_rn(make_float2(acc[i], acc[i + 1]), make_float2(f[i], f[i + 1])),
                                make_float2(d[i], d[i + 1]));
    acc[i] = v.x;
    acc[i + 1] = v.y;
  }
}

// t = X r on one unit u of 16 columns of the block's 16 rows, added to acc.
// x0, x1: shared addresses of (row g or g + 8, column 8 t); lane column 32 (u / 2) + 4 (u % 2) + 8 t + 2 s2 + h
template <int NT8, bool PRE, bool GUARD>
__device__ __forceinline__ void bjm_fwd(uint32_t x0, uint32_t x1, uint32_t rf, int i0, int dn, int u, int lane,
                                        float (&acc)[NT8][4]) {
  const int k0 = 32 * (u >> 1) + 4 * (u & 1);
  uint32_t ah[2][4], al[2][4];
#pragma unroll
  for (int s2 = 0; s2 < 2; ++s2)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int o = 2 * s2 + (i >> 1);
      float x = 0.f;
      if (!GUARD) {
        x = bjm_lds(((i & 1) ? x1 : x0) + 4 * (k0 + o));
      } else {
        const int d = (lane >> 2) + 8 * (i & 1);
        if (d < dn && k0 + o + 8 * (lane & 3) <= i0 + d) x = bjm_lds(((i & 1) ? x1 : x0) + 4 * (k0 + o));
      }
      bjm_split(x, ah[s2][i], al[s2][i]);
    }
#pragma unroll
  for (int q = 0; q < NT8; ++q)
    bjm_prod(ah, al, bjm_frag<PRE>(rf, 2 * u * NT8 + q, lane), bjm_frag<PRE>(rf, (2 * u + 1) * NT8 + q, lane), acc[q]);
}

// z += X^T t on one group of 32 columns; ro: shared addresses of (row 8 s2 + 4 h + t, column 4 g)
template <int NT8, bool GUARD>
__device__ __forceinline__ void bjm_back(const uint32_t (&ro)[2][2], const float4 (&tf)[2][NT8], int i0, int dn, int gi,
                                         int lane, float (&z)[2][NT8][4]) {
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    uint32_t ah[2][4], al[2][4];
#pragma unroll
    for (int s2 = 0; s2 < 2; ++s2)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int o = 32 * gi + 2 * j + (i & 1);
        float x = 0.f;
        if (!GUARD) {
          x = bjm_lds(ro[s2][i >> 1] + 4 * o);
        } else {
          const int d = 8 * s2 + 4 * (i >> 1) + (lane & 3);
          if (d < dn && o + 4 * (lane >> 2) <= i0 + d) x = bjm_lds(ro[s2][i >> 1] + 4 * o);
        }
        bjm_split(x, ah[s2][i], al[s2][i]);
      }
#pragma unroll
    for (int q = 0; q < NT8; ++q) bjm_prod(ah, al, tf[0][q], tf[1][q], z[j][q]);
  }
}

template <int NT8, int NW, int CG, bool PRE>
__global__ void __launch_bounds__(32 * NW, NW >= 16 ? 1 : 16 / NW)
    k_bj_mma(BjArgs A, const float *X, const float *in, float *out, int stages, int cs) {
  typedef BjmLayout<NT8, NW, PRE> L;
  constexpr int RT = L::RT, NTH = 32 * NW;
  extern __shared__ __align__(16) unsigned char bjm_raw[];
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ int s_bad;
  const int n = A.n, nch = L::chunks(n), stage = L::stage(n);
  float *Xs = reinterpret_cast<float *>(bjm_raw);
  float *rf = Xs + (size_t)stages * stage;                // [chunk][k-step][n8][lane] of 4 (PRE) or 2 floats
  float *ps = rf + (size_t)nch * NT8 * (PRE ? 512 : 256);  // [warp][16][RT]
  float4 *ts = reinterpret_cast<float4 *>(ps + NW * BJP_BR * RT);          // [k-step][n8][lane]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = blockIdx.x % cs, ge = blockIdx.x / cs;
  const int e = A.elems[ge], r0 = blockIdx.y * RT;
  const int64_t vb = A.dof_off[e], xb = A.blk_off[e];
  const int nblk = (n + BJP_BR - 1) / BJP_BR;

  if (tid == 0) {
    s_bad = 0;
    for (int i = 0; i < 2; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bjp_saddr(&bar[i])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  // rows [16 b, 16 b + 16) of X are contiguous; the copy starts on the 16-byte boundary below
  auto issue = [&](int b, int st) {
    const int64_t s0 = xb + bjp_tri(b * BJP_BR), s1 = xb + bjp_tri(min(n, (b + 1) * BJP_BR));
    const int64_t a0 = s0 & ~(int64_t)3, a1 = (s1 + 3) & ~(int64_t)3;
    const uint32_t bytes = (uint32_t)((a1 - a0) * sizeof(float));
    const uint32_t mb = bjp_saddr(&bar[st]);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     bjp_saddr(Xs + (size_t)st * stage)),
                 "l"(X + a0), "r"(bytes), "r"(mb)
                 : "memory");
  };
  const int mine = rank < nblk ? (nblk - rank + cs - 1) / cs : 0;
  if (tid == 0)
    for (int s = 0; s < stages && s < mine; ++s) issue(rank + s * cs, s);
  // r as B fragments (hi, hi, lo, lo of the two k's of a lane), zero beyond n and n_rhs
  for (int w = warp; w < nch * (RT / 2); w += NW) {
    const int c = w / (RT / 2), qp = w - c * (RT / 2);
    const int t = lane & 3, q = 2 * qp + ((lane >> 2) & 1), s = lane >> 3;
    const int k = 32 * c + 8 * t + 2 * s;
    const float *src = in + (int64_t)(r0 + q) * A.ndof + vb;
    const bool ok = r0 + q < A.n_rhs;
    const float v0 = ok && k < n ? src[k] : 0.f, v1 = ok && k + 1 < n ? src[k + 1] : 0.f;
    const size_t at = ((size_t)(4 * c + s) * NT8 + (q >> 3)) * 32 + (q & 7) * 4 + t;
    if constexpr (PRE) {
      uint32_t h0, l0, h1, l1;
      bjm_split(v0, h0, l0);
      bjm_split(v1, h1, l1);
      reinterpret_cast<float4 *>(rf)[at] =
          make_float4(__uint_as_float(h0), __uint_as_float(h1), __uint_as_float(l0), __uint_as_float(l1));
    } else {
      reinterpret_cast<float2 *>(rf)[at] = make_float2(v0, v1);
    }
  }
  __syncthreads();

  const uint32_t rfa = bjp_saddr(rf);
  float z[CG][2][NT8][4];
#pragma unroll
  for (int c = 0; c < CG; ++c)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int q = 0; q < NT8; ++q)
#pragma unroll
        for (int i = 0; i < 4; ++i) z[c][j][q][i] = 0.f;

  auto block = [&](int it, int &i0, int &dn, int &st) -> uint32_t {
    i0 = (rank + it * cs) * BJP_BR;
    dn = min(BJP_BR, n - i0);
    st = stages == 2 ? (it & 1) : 0;
    const int64_t s0 = xb + bjp_tri(i0);
    return bjp_saddr(Xs) + 4 * (uint32_t)(st * stage + (int)(s0 & 3));  // entry (i0, 0)
  };
  for (int it = -1; it < mine; ++it) {
    if (it >= 0) {
      // z += X^T t on the columns of the warp's groups of 32
      int i0, dn, st;
      const uint32_t Xb = block(it, i0, dn, st);
      if (32 * warp < i0 + dn) {
        const int t = lane & 3, g = lane >> 2;
        float4 tf[2][NT8];
        uint32_t ro[2][2];
#pragma unroll
        for (int s2 = 0; s2 < 2; ++s2) {
#pragma unroll
          for (int q = 0; q < NT8; ++q) tf[s2][q] = ts[(s2 * NT8 + q) * 32 + lane];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int d = 8 * s2 + 4 * h + t;
            ro[s2][h] = Xb + 4 * (d * i0 + bjp_tri(d) + 4 * g);
          }
        }
        if (dn == BJP_BR && 32 * (warp + NW * (CG - 1)) + 31 <= i0) {
          // every group of the warp left of the diagonal: one straight run
#pragma unroll
          for (int c = 0; c < CG; ++c) bjm_back<NT8, false>(ro, tf, i0, dn, warp + NW * c, lane, z[c]);
        } else {
#pragma unroll
          for (int c = 0; c < CG; ++c) {
            const int gi = warp + NW * c;
            if (32 * gi < i0 + dn) {
              if (dn == BJP_BR && 32 * gi + 31 <= i0) bjm_back<NT8, false>(ro, tf, i0, dn, gi, lane, z[c]);
              else bjm_back<NT8, true>(ro, tf, i0, dn, gi, lane, z[c]);
            }
          }
        }
      }
      if (stages == 1 && it + 1 < mine) {
        __syncthreads();
        if (tid == 0) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          issue(rank + (it + 1) * cs, 0);
        }
      }
    }
    if (it + 1 >= mine) break;
    // t = X r of the next block: units of 16 columns dealt to the warps
    int i0, dn, st;
    const uint32_t Xb = block(it + 1, i0, dn, st);
    const int rg = lane >> 2, rt = lane & 3;
    const uint32_t x0 = Xb + 4 * (rg * i0 + bjp_tri(rg) + 8 * rt), x1 = Xb + 4 * ((rg + 8) * i0 + bjp_tri(rg + 8) + 8 * rt);
    if (!bjp_wait(bjp_saddr(&bar[st]), (stages == 2 ? (it + 1) >> 1 : it + 1) & 1, A.polls)) s_bad = 1;  // gives up after the barrier
    float acc[NT8][4];
#pragma unroll
    for (int q = 0; q < NT8; ++q)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[q][i] = 0.f;
    const int nu = 2 * ((i0 + dn + 31) / 32);
    const int nfull = dn == BJP_BR ? 2 * ((i0 + 1) / 32) : 0;  // units wholly left of the diagonal
    // in reverse warp order at 16 right-hand sides: the first warps have the most columns
    // of the other product (365 -> 359 us, 512 blocks of 729; at 8 no gain)
    int u = NT8 == 2 ? NW - 1 - warp : warp;
#pragma unroll 2
    for (; u < nfull; u += NW) bjm_fwd<NT8, PRE, false>(x0, x1, rfa, i0, dn, u, lane, acc);
    for (; u < nu; u += NW) bjm_fwd<NT8, PRE, true>(x0, x1, rfa, i0, dn, u, lane, acc);
    {
      const int g = lane >> 2, t = lane & 3;
#pragma unroll
      for (int q = 0; q < NT8; ++q) {
        float *p = ps + ((size_t)warp * BJP_BR + g) * RT + 8 * q + 2 * t;
        *reinterpret_cast<float2 *>(p) = make_float2(acc[q][0], acc[q][1]);
        *reinterpret_cast<float2 *>(p + 8 * RT) = make_float2(acc[q][2], acc[q][3]);
      }
    }
    __syncthreads();
    if (s_bad) {
      // the copies in flight land (bounded) before their memory is used again or the CTA
      // ends: this block's and, before the first block, the second stage's
      bjp_wait(bjp_saddr(&bar[st]), (stages == 2 ? (it + 1) >> 1 : it + 1) & 1, BJ_POLLS);
      if (stages == 2 && it < 0 && mine > 1) bjp_wait(bjp_saddr(&bar[1]), 0, BJ_POLLS);
#pragma unroll
      for (int c = 0; c < CG; ++c)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int q = 0; q < NT8; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) z[c][j][q][i] = __int_as_float(0x7fffffff);
      break;
    }
    if (stages == 2 && it >= 0 && it + 2 < mine && tid == 0) {
      // the generic reads of block it precede the copy that overwrites its stage
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(rank + (it + 2) * cs, st ^ 1);
    }
    for (int idx = tid; idx < BJP_BR * RT; idx += NTH) {
      float s = ps[idx];
#pragma unroll
      for (int w = 1; w < NW; ++w) s += ps[w * BJP_BR * RT + idx];
      uint32_t hi, lo;
      bjm_split(s, hi, lo);
      const int d = idx / RT, q = idx - d * RT;
      float *f = reinterpret_cast<float *>(ts + ((d >> 3) * NT8 + (q >> 3)) * 32 + (q & 7) * 4 + (d & 3)) + ((d >> 2) & 1);
      f[0] = __uint_as_float(hi);
      f[2] = __uint_as_float(lo);
    }
    __syncthreads();
  }
  // z through shared memory (coalesced stores; summed over the cluster in rank order)
  __syncthreads();
  float *zs = Xs;  // [RT][n]: RT <= 16 rows of X
#pragma unroll
  for (int c = 0; c < CG; ++c) {
    const int gi = warp + NW * c;
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int q = 0; q < NT8; ++q)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int col = 32 * gi + 4 * (lane >> 2) + 2 * j + (i >> 1), rr = 8 * q + 2 * (lane & 3) + (i & 1);
          if (col < n) zs[rr * n + col] = z[c][j][q][i];
        }
  }
  if (cs == 1) {
    __syncthreads();
    for (int idx = tid; idx < n * RT; idx += NTH) {
      const int rr = idx / n, k = idx - rr * n;
      if (r0 + rr < A.n_rhs) out[(int64_t)(r0 + rr) * A.ndof + vb + k] = zs[idx];
    }
  } else {
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
    const uint32_t zl = bjp_saddr(zs);
    for (int idx = tid + NTH * rank; idx < n * RT; idx += NTH * cs) {
      float s = 0.f, v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        v[q] = 0.f;
        if (q < cs) v[q] = bjp_peer(zl + (uint32_t)(idx * sizeof(float)), q, 0.f);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) s += v[q];
      const int rr = idx / n, k = idx - rr * n;
      if (r0 + rr < A.n_rhs) out[(int64_t)(r0 + rr) * A.ndof + vb + k] = s;
    }
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
  }
  if (tid == 0 && s_bad) bj_flag(A.err);
}

template <int NT8, int NW, int CG, bool PRE = true>
static cudaError_t bjm_launch(const BjArgs &a, const float *X, const float *r, float *z, cudaStream_t s) {
  typedef BjmLayout<NT8, NW, PRE> L;
  const void *fn = (const void *)k_bj_mma<NT8, NW, CG, PRE>;
  // two stages unless one leaves room for a second CTA on the SM (or two do not fit)
  const int stages = L::bytes(a.n, 2) <= 225 * 1024 && (L::bytes(a.n, 1) > 112 * 1024 || L::bytes(a.n, 2) <= 75 * 1024)
                         ? 2
                         : 1;
  const size_t smem = L::bytes(a.n, stages);
  cudaError_t ce = bjp_raise_smem(fn, smem);
  if (ce != cudaSuccess) return ce;
  const int tiles = (a.n_rhs + L::RT - 1) / L::RT;
  const int occ = (int)std::min<size_t>(NW >= 16 ? 1 : 16 / NW, 227 * 1024 / (smem + 1024));
  const int cs = bjp_cluster(a.n, (int64_t)a.n_group * tiles, occ < 1 ? 1 : occ);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.n_group * cs), (unsigned)tiles);
  cfg.blockDim = dim3(32 * NW);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_bj_mma<NT8, NW, CG, PRE>, a, X, r, z, stages, cs);
}

template <int NT8>
static cudaError_t bjm_by_size(const BjArgs &a, const float *X, const float *r, float *z, cudaStream_t s) {
  if (a.n <= 384) return bjm_launch<NT8, 8, 2>(a, X, r, z, s);
  if (a.n <= 512) return bjm_launch<NT8, 16, 1>(a, X, r, z, s);
  // up to 8 right-hand sides two CTAs of 8 warps share an SM
  if (NT8 == 1 && a.n <= 768) return bjm_launch<1, 8, 3>(a, X, r, z, s);
  if (a.n <= 768) return bjm_launch<NT8, 16, 2>(a, X, r, z, s);
  // 16 right-hand sides of r take twice the room in split form: beyond n = 768 they leave
  // none for a second stage (64 blocks of 1000: 110 -> 82 us as FP32 values) or for the first
  // one (64 of 1331: 234 us by 8 right-hand sides per CTA, 162 us so); up to 768 the split at
  // each use costs 5 %
  constexpr bool PRE = NT8 == 1;
  if (a.n <= 1024) return bjm_launch<NT8, 16, 2, PRE>(a, X, r, z, s);
  if (a.n <= 1536) return bjm_launch<NT8, 16, 3, PRE>(a, X, r, z, s);
  return cudaErrorInvalidValue;
}
