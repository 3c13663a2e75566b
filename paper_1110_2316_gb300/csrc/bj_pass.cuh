// bj_pass.cuh -- z = X^T (X r) of the element-block preconditioner in ONE pass
// over the packed factor X (block_precond.cuh): the one-pass variants in FP64,
// and in FP32 for up to 4 right-hand sides and for blocks up to n = 256 at any
// count (bj_mma.cuh takes the others, bj_pass.cu).
//
// The two products of k_bj_tri read X twice and keep a multiply-add per shared
// load; at few right-hand sides the apply is bound by those reads.  Here a CTA
// walks an element's X in blocks of 16 rows, which are contiguous in the packed
// storage and arrive by one bulk copy each: t = X r on the block's rows (they
// need only r), then z += X^T t from the same shared-memory block, so X leaves
// HBM once.  r (all of it), t of the block and the X block live in shared
// memory, z in registers (thread tid: columns tid + NTH c).
//   t: warp w takes MR rows, its lanes the columns; MR x RT sums per lane are
//      reduced over the warp by a transposing butterfly (each level halves them);
//   z: every thread adds x(row, column) t(row); the columns left of the block's
//      diagonal run without a test, fully unrolled over them.
// FP32 runs the right-hand sides two at a time (packed FMA).  With few elements
// a cluster of up to 8 CTAs shares one: row blocks are dealt in turn and the
// partial z summed through distributed shared memory in rank order.
// Bound: FP32 HBM (the factor once: 545 MB for 512 blocks of 729, 80 us; 145 us
// at 1 and 215 us at 4 right-hand sides: latency of the copies, sums and barriers
// at twelve warps per SM, no pipe above 25 %), FP64 its pipe (two
// lanes per clock and SM: 1.73 ms at 4 right-hand sides, 2.42 ms measured).
// Waits on the copies are bounded (bj_pass.h).
#pragma once
#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <utility>

#include "bj_pass.h"

constexpr int BJP_BR = 16;  // rows of X per block

template <typename T>
struct alignas(16) BjpV4 {
  T v[4];
};

// CTAs per element (a cluster that deals the element's row blocks in turn): the
// size with the fewest block times over the waves of the launch, the start and
// end of a CTA counted as three blocks.  items: elements x right-hand-side tiles.
static int bjp_cluster(int n, int64_t items, int per_sm) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return 1;
  const int nblk = (n + BJP_BR - 1) / BJP_BR;
  int best = 1;
  double cost = 1e300;
  for (int cs = 1; cs <= 8 && cs <= nblk; cs *= 2) {
    const double waves = std::ceil((double)items * cs / ((double)sms * per_sm));
    const double c = waves * (3.0 + (double)nblk / cs);
    if (c < cost) {
      cost = c;
      best = cs;
    }
  }
  return best;
}

// dynamic shared-memory limit of a kernel, raised once per device and size
static cudaError_t bjp_raise_smem(const void *fn, size_t bytes) {
  static std::mutex mu;
  static std::map<std::pair<const void *, int>, size_t> done;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  size_t &cur = done[std::make_pair(fn, dev)];
  if (bytes <= cur) return cudaSuccess;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) cur = bytes;
  return e;
}

// shared memory: X stages | r | t
template <typename T, int RT>
struct BjpLayout {
  static constexpr int VR = RT >= 4 ? 4 : 1, G = RT / VR;
  __host__ __device__ static int n32(int n) { return ((n + 31) / 32) * 32; }
  // entries of one X stage: 16 rows of up to n16 entries, the 16-byte slack at both ends
  __host__ __device__ static int stage(int n) {
    const int m = ((n + BJP_BR - 1) / BJP_BR) * BJP_BR;
    return ((BJP_BR * m + 32 / (int)sizeof(T) + 3) / 4) * 4;
  }
  __host__ __device__ static size_t bytes(int n, int stages) {
    return sizeof(T) * ((size_t)stages * stage(n) + (size_t)G * n32(n) * VR + (size_t)BJP_BR * RT);
  }
};

__device__ __forceinline__ uint32_t bjp_saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool bjp_wait(uint32_t bar, uint32_t parity, int polls) {
  for (int it = 0; it < polls; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// value at the same shared-memory address of CTA `rank` of the cluster
__device__ __forceinline__ float bjp_peer(uint32_t addr, int rank, float) {
  uint32_t ra;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(ra) : "memory");
  return v;
}
__device__ __forceinline__ double bjp_peer(uint32_t addr, int rank, double) {
  uint32_t ra;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(ra) : "memory");
  return v;
}

__device__ __forceinline__ int bjp_tri(int i) { return i * (i + 1) / 2; }

// sum of V values per lane over the warp: lane l ends with the sum of value
// bjp_slot<V>(l) (V a power of two up to 32; equal slots hold the same sum)
template <int V, int BIT, typename T>
__device__ __forceinline__ void bjp_reduce(T *v, int lane) {
  if constexpr (BIT > 0) {
    if constexpr (V > 1) {
      const bool up = lane & BIT;
#pragma unroll
      for (int i = 0; i < V / 2; ++i) {
        const T s = up ? v[i] : v[i + V / 2], k = up ? v[i + V / 2] : v[i];
        v[i] = k + __shfl_xor_sync(0xffffffffu, s, BIT);
      }
      bjp_reduce<V / 2, BIT / 2>(v, lane);
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], BIT);
      bjp_reduce<1, BIT / 2>(v, lane);
    }
  }
}

// acc[0..N) += x * b[0..N), FP32 two at a time (packed FMA, each half rounded as fmaf)
template <int N, typename T>
__device__ __forceinline__ void bjp_axpy(T x, const T *b, T *acc) {
  if constexpr (sizeof(T) == 4 && N >= 2) {
    const float2 xx = make_float2(x, x);
#pragma unroll
    for (int q = 0; q < N; q += 2) {
      const float2 a = __ffma2_rn(xx, make_float2(b[q], b[q + 1]), make_float2(acc[q], acc[q + 1]));
      acc[q] = a.x;
      acc[q + 1] = a.y;
    }
  } else {
#pragma unroll
    for (int q = 0; q < N; ++q) acc[q] += x * b[q];
  }
}
// N consecutive right-hand sides of one row of t or r (stride 4-vectors `gs` apart)
template <int N, typename T>
__device__ __forceinline__ void bjp_row(const T *p, int gs, T *b) {
  if constexpr (N >= 4) {
#pragma unroll
    for (int q = 0; q < N / 4; ++q) {
      const BjpV4<T> v = *reinterpret_cast<const BjpV4<T> *>(p + q * gs);
#pragma unroll
      for (int i = 0; i < 4; ++i) b[4 * q + i] = v.v[i];
    }
  } else {
    b[0] = p[0];
  }
}
// z[c] += x(row, tid + NTH c) t(row) for the first CF columns (all left of the diagonal)
template <int CF, int RT, int NTH, typename T>
__device__ __forceinline__ void bjp_back(const T *Xb, const T *ts, int i0, int dn, int tid, T (*z)[RT]) {
  constexpr int U = CF * RT >= 64 ? 2 : 4;
#pragma unroll U
  for (int d = 0; d < dn; ++d) {
    const T *Xr = Xb + d * i0 + d * (d + 1) / 2 + tid;
    T tv[RT], x[CF];
#pragma unroll
    for (int c = 0; c < CF; ++c) x[c] = Xr[NTH * c];
    bjp_row<RT>(ts + d * RT, 4, tv);
#pragma unroll
    for (int c = 0; c < CF; ++c) bjp_axpy<RT>(x[c], tv, z[c]);
  }
}

__host__ __device__ constexpr int bjp_per_sm(size_t size, int nth) { return size == 8 ? (nth >= 256 ? 1 : 256 / nth) : 512 / nth; }

template <typename T, int RT, int NTH, int C>
__global__ void __launch_bounds__(NTH, bjp_per_sm(sizeof(T), NTH))
    k_bj_pass(BjArgs A, const T *X, const T *in, T *out, int stages, int cs) {
  typedef BjpLayout<T, RT> L;
  constexpr int VR = L::VR, G = L::G, NW = NTH / 32;
  constexpr int MR = BJP_BR / NW;                          // rows of a block per warp
  constexpr int RP = MR * RT <= 32 ? RT : 32 / MR;         // right-hand sides per sweep of these rows
  extern __shared__ __align__(16) unsigned char bjp_raw[];
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ int s_bad;
  const int n = A.n, n32 = L::n32(n), stage = L::stage(n);
  T *Xs = reinterpret_cast<T *>(bjp_raw);
  T *rs = Xs + (size_t)stages * stage;  // [G][n32][VR]
  T *ts = rs + (size_t)G * n32 * VR;    // [BR][RT]
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
  constexpr int AL = 16 / (int)sizeof(T);
  auto issue = [&](int b, int st) {
    const int64_t s0 = xb + bjp_tri(b * BJP_BR), s1 = xb + bjp_tri(min(n, (b + 1) * BJP_BR));
    const int64_t a0 = s0 & ~(int64_t)(AL - 1), a1 = (s1 + AL - 1) & ~(int64_t)(AL - 1);
    const uint32_t bytes = (uint32_t)((a1 - a0) * sizeof(T));
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
#pragma unroll 2
  for (int k = tid; k < n32; k += NTH) {
    T v[RT];
#pragma unroll
    for (int q = 0; q < RT; ++q)
      v[q] = (k < n && r0 + q < A.n_rhs) ? in[(int64_t)(r0 + q) * A.ndof + vb + k] : (T)0;
    if constexpr (VR == 4) {
#pragma unroll
      for (int q = 0; q < G; ++q)
        *reinterpret_cast<BjpV4<T> *>(rs + ((size_t)q * n32 + k) * 4) = {v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]};
    } else {
      rs[k] = v[0];
    }
  }
  __syncthreads();

  T z[C][RT];
#pragma unroll
  for (int c = 0; c < C; ++c)
#pragma unroll
    for (int q = 0; q < RT; ++q) z[c][q] = (T)0;
  for (int it = 0; it < mine; ++it) {
    const int b = rank + it * cs, i0 = b * BJP_BR, st = stages == 2 ? (it & 1) : 0;
    if (!bjp_wait(bjp_saddr(&bar[st]), (stages == 2 ? it >> 1 : it) & 1, A.polls)) s_bad = 1;  // gives up after the barrier below
    const int64_t s0 = xb + bjp_tri(i0);
    const T *Xb = Xs + (size_t)st * stage + (s0 & (AL - 1));  // entry (i0, 0)
    const int dn = min(BJP_BR, n - i0);
    // t = X r: warp w takes rows i0 + MR w + m, its lanes the columns.  Of a block of one row
    // block (W = 1) one thread sums a row in turn: over lanes every product of the few terms
    // is rounded by itself (FP32, n = 8: error 7.2e-8, a chain of FMAs 6.2e-8)
    if (C == 1 && n <= BJP_BR) {
      for (int idx = tid; idx < dn * RT; idx += NTH) {
        const int d = idx / RT, q = idx - d * RT;
        const T *rq = rs + (size_t)(q / VR) * n32 * VR + q % VR;
        T s = (T)0;
        for (int k = 0; k <= d; ++k) s += Xb[bjp_tri(d) + k] * rq[k * VR];
        ts[idx] = s;
      }
    } else
#pragma unroll
    for (int q0 = 0; q0 < RT; q0 += RP) {
      T acc[MR * RP];
#pragma unroll
      for (int i = 0; i < MR * RP; ++i) acc[i] = (T)0;
      const int d0 = MR * warp;
      const T *Xr[MR];
#pragma unroll
      for (int m = 0; m < MR; ++m) Xr[m] = Xb + (d0 + m) * i0 + (d0 + m) * (d0 + m + 1) / 2;
      const T *rg = rs + (size_t)(q0 / VR) * n32 * VR;
      const int nfull = (i0 + 1) / 32;  // chunks of 32 columns wholly left of the diagonal
      if (dn == BJP_BR) {
#pragma unroll 2
        for (int k = lane; k < 32 * nfull; k += 32) {
          T rv[RP], x[MR];
#pragma unroll
          for (int m = 0; m < MR; ++m) x[m] = Xr[m][k];
          bjp_row<RP>(rg + k * VR, n32 * VR, rv);
#pragma unroll
          for (int m = 0; m < MR; ++m) bjp_axpy<RP>(x[m], rv, acc + m * RP);
        }
      }
      for (int k = (dn == BJP_BR ? 32 * nfull : 0) + lane; k < i0 + dn; k += 32) {
        T rv[RP];
        bjp_row<RP>(rg + k * VR, n32 * VR, rv);
#pragma unroll
        for (int m = 0; m < MR; ++m) {
          T x = (T)0;
          if (d0 + m < dn && k <= i0 + d0 + m) x = Xr[m][k];
          bjp_axpy<RP>(x, rv, acc + m * RP);
        }
      }
      __syncwarp();
      bjp_reduce<MR * RP, 16>(acc, lane);
      // value index held by this lane, from the top lane bits down
      constexpr int V = MR * RP, LV = V >= 32 ? 5 : (V >= 16 ? 4 : (V >= 8 ? 3 : (V >= 4 ? 2 : (V >= 2 ? 1 : 0))));
      const int slot = lane >> (5 - LV);
      if ((lane & ((1 << (5 - LV)) - 1)) == 0) ts[(d0 + slot / RP) * RT + q0 + slot % RP] = acc[0];
    }
    __syncthreads();
    const bool bad = s_bad != 0;
    // z += X^T t: thread tid holds columns tid + NTH c; cf of the warp's are left of the diagonal, ca reach the block
    const int wmax = i0 - warp * 32 - 31;
    const int cf = wmax >= 0 ? min(C, wmax / NTH + 1) : 0;
    const int ca = (i0 + dn - warp * 32 + NTH - 1) / NTH;
    switch (cf) {
      case 1: bjp_back<1, RT, NTH>(Xb, ts, i0, dn, tid, z); break;
      case 2: if constexpr (C >= 2) bjp_back<2, RT, NTH>(Xb, ts, i0, dn, tid, z); break;
      case 3: if constexpr (C >= 3) bjp_back<3, RT, NTH>(Xb, ts, i0, dn, tid, z); break;
      case 4: if constexpr (C >= 4) bjp_back<4, RT, NTH>(Xb, ts, i0, dn, tid, z); break;
      case 5: if constexpr (C >= 5) bjp_back<5, RT, NTH>(Xb, ts, i0, dn, tid, z); break;
      case 6: if constexpr (C >= 6) bjp_back<6, RT, NTH>(Xb, ts, i0, dn, tid, z); break;
      case 7: if constexpr (C >= 7) bjp_back<7, RT, NTH>(Xb, ts, i0, dn, tid, z); break;
      case 8: if constexpr (C >= 8) bjp_back<8, RT, NTH>(Xb, ts, i0, dn, tid, z); break;
      default: break;
    }
#pragma unroll
    for (int c = 0; c < C; ++c)
      if (c >= cf && c < ca) {
        const int k = tid + NTH * c;
        for (int d = 0; d < dn; ++d)
          if (k <= i0 + d) {
            T tv[RT];
            bjp_row<RT>(ts + d * RT, 4, tv);
            bjp_axpy<RT>(Xb[d * i0 + d * (d + 1) / 2 + k], tv, z[c]);
          }
      }
    __syncthreads();
    if (bad) {
      // the copies in flight land (bounded) before their memory is used again or the CTA ends
      bjp_wait(bjp_saddr(&bar[st]), (stages == 2 ? it >> 1 : it) & 1, BJ_POLLS);
      if (stages == 2 && it + 1 < mine) bjp_wait(bjp_saddr(&bar[st ^ 1]), ((it + 1) >> 1) & 1, BJ_POLLS);
#pragma unroll
      for (int c = 0; c < C; ++c)
#pragma unroll
        for (int q = 0; q < RT; ++q) z[c][q] = (T)__int_as_float(0x7fffffff);
      break;
    }
    if (tid == 0 && it + stages < mine) {
      // the stage's generic reads precede the copy that overwrites it
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(rank + (it + stages) * cs, st);
    }
  }
  if (cs == 1) {
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int k = tid + NTH * c;
      if (k < n)
#pragma unroll
        for (int q = 0; q < RT; ++q)
          if (r0 + q < A.n_rhs) out[(int64_t)(r0 + q) * A.ndof + vb + k] = z[c][q];
    }
  } else {
    // partial z of every CTA of the cluster, summed in rank order by column slices
    T *zs = Xs;  // n x RT values fit one stage (RT <= 16 rows)
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int k = tid + NTH * c;
      if (k < n)
#pragma unroll
        for (int q = 0; q < RT; ++q) zs[q * n + k] = z[c][q];
    }
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
    const uint32_t zl = bjp_saddr(zs);
    for (int idx = tid + NTH * rank; idx < n * RT; idx += NTH * cs) {
      T s = (T)0, v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        v[q] = (T)0;
        if (q < cs) v[q] = bjp_peer(zl + (uint32_t)(idx * sizeof(T)), q, (T)0);
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

template <typename T, int RT, int NTH, int C>
static cudaError_t bjp_launch(const BjArgs &a, const T *X, const T *r, T *z, cudaStream_t s) {
  const void *fn = (const void *)k_bj_pass<T, RT, NTH, C>;
  const int stages = BjpLayout<T, RT>::bytes(a.n, 2) <= 74 * 1024 ? 2 : 1;
  const size_t smem = BjpLayout<T, RT>::bytes(a.n, stages);
  cudaError_t ce = bjp_raise_smem(fn, smem);
  if (ce != cudaSuccess) return ce;
  const int tiles = (a.n_rhs + RT - 1) / RT;
  const int occ = (int)std::min<size_t>(bjp_per_sm(sizeof(T), NTH), 227 * 1024 / (smem + 1024));
  const int cs = bjp_cluster(a.n, (int64_t)a.n_group * tiles, occ < 1 ? 1 : occ);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.n_group * cs), (unsigned)tiles);
  cfg.blockDim = dim3(NTH);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_bj_pass<T, RT, NTH, C>, a, X, r, z, stages, cs);
}

template <typename T, int RT>
static cudaError_t bjp_by_size(const BjArgs &a, const T *X, const T *r, T *z, cudaStream_t s) {
  if (a.n <= 64) return bjp_launch<T, RT, 64, 1>(a, X, r, z, s);
  if (a.n <= 128) return bjp_launch<T, RT, 64, 2>(a, X, r, z, s);
  if constexpr (sizeof(T) == 8) {
    // FP64: one CTA per SM from n = 512 on (the X stage), so eight warps to keep its pipe fed
    if (a.n <= 256) return bjp_launch<T, RT, 128, 2>(a, X, r, z, s);
    if (a.n <= 512) return bjp_launch<T, RT, 256, 2>(a, X, r, z, s);
    if (a.n <= 768) return bjp_launch<T, RT, 256, 3>(a, X, r, z, s);
    if (a.n <= 1024) return bjp_launch<T, RT, 256, 4>(a, X, r, z, s);
  } else {
    if (a.n <= 256) return bjp_launch<T, RT, 64, 4>(a, X, r, z, s);
    if (a.n <= 384) return bjp_launch<T, RT, 128, 3>(a, X, r, z, s);
    if (a.n <= 512) return bjp_launch<T, RT, 128, 4>(a, X, r, z, s);
    if (a.n <= 768) return bjp_launch<T, RT, 128, 6>(a, X, r, z, s);
    if (a.n <= 1024) return bjp_launch<T, RT, 128, 8>(a, X, r, z, s);
  }
  if (a.n <= 1536) return bjp_launch<T, RT, 256, 6>(a, X, r, z, s);
  return cudaErrorInvalidValue;
}
