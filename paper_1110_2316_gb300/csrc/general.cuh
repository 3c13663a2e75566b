// general.cuh -- operator apply for a general second-order operator with
// per-point coefficients, one (REAL, WDEG) instantiation (included after
// kernels.cuh by inst_template.cuh).
//
// On a box element the operator of eq. (2.2), written out as
//   L u = sum_ij A_ij u_{x_i x_j} + sum_i b_i u_{x_i} + c u   (A symmetric),
// is, in the reference coordinates lambda of the element, the ten-term form
// of eq. (5.45):
//   L u = C_11 u_11 + C_22 u_22 + C_33 u_33 + C_12 u_12 + C_23 u_23
//       + C_13 u_13 + C_1 u_1 + C_2 u_2 + C_3 u_3 + C_0 u
// (u_a = du/dlambda_a), with C_aa = A_aa s_a^2, C_ab = 2 A_ab s_a s_b,
// C_a = b_a s_a, C_0 = c, s_a = dlambda_a / dx_a.  The host library stores,
// per volume point, the quadrature weight w_a w_b w_c |J| and the ten C's
// (GEN_NC values per point, the last one padding).
//
// Sum factorisation (Section 5.3) of the ten fields:
//   x-stage:  X_m = B_m along x,              m = 0, 1, 2
//   y-stage:  T_mn = B_n along y of X_m,      (m, n) = 00 01 02 10 11 20
//   z-stage:  u = B0 T00, u_3 = B1 T00, u_33 = B2 T00, u_2 = B0 T01,
//             u_23 = B1 T01, u_22 = B0 T02, u_1 = B0 T10, u_13 = B1 T10,
//             u_12 = B0 T11, u_11 = B0 T20,
// then rho = w |J| (L u) per point and the transposed stages in reverse
// order; the face terms of box meshes (jumps of u and of the physical
// gradient, Dirichlet and Neumann / Robin faces) are those of the Laplacian
// (face_phase of kernels.cuh), since they do not involve the operator.
//
// Design: one CTA per (element, rhs) item with the line stages of k_apply
// (chunks of folded output pairs over whole warps, constant-bank matrix
// entries, FP32 contractions in pairs through the packed FMA).  A z-column
// holds its six folded T lines in registers and forms all ten fields of one
// pair of mirrored points at a time, so that a point's twelve coefficients
// come by three (FP64: six) vector loads and rho goes straight into the
// column's own slots of T00 and T01; the transpose reads rho back from there
// in two sweeps (lines T02, T10, T11, T20, then T00, T01, whose slots rho
// occupies).  Field by field with rho in registers the forward spilled 1.5 KB
// per thread and loaded each coefficient alone at a 48-byte lane stride.
// Bound: FP32 the latency of the coefficient reads from L2 (12, 8 and 12 values
// of a point in the three sweeps: 128 bytes; long-scoreboard 5.4 stalls per
// issue, no pipe above 26 %) at two CTAs per SM, FP64 its pipe.  8^3 elements of W = 8: FP32, 16 rhs
// 2394 -> 895 us; FP64, 2 rhs 2979 -> 2463 us.  (FP64 at W = 1, four lines and nine
// columns, is slower than field by field: 240 items 18.5 -> 20.5 us, 8,192 items
// 225 -> 231; its coefficients kept in registers gave 20.4 and 236.)  Shared memory: su | X[3] | T[6] |
// D copy + face scales | reduction; the T region later holds sy and the face
// scratch.  Instances whose layout exceeds 227 KB (FP64 at W = 10) are not
// built; the host library refuses such meshes.
#pragma once

namespace {

constexpr int GEN_NC = 12;
// resident CTAs asked for: about 20 warps per SM in FP32 (96 registers at W = 8)
constexpr int GEN_MINB = sizeof(real) == 8 ? 1 : (640 / NT < 1 ? 1 : (640 / NT > 4 ? 4 : 640 / NT));

struct GenLayout {
  static constexpr int TS = t_stride(3, 6, GEN_MINB);  // row stride of the T fields
  static constexpr int TF = TS * P;
  static constexpr size_t RED_OFF = red_in_x(3) ? X_OFF : apply_bytes(3, 6, TS) - NT * sizeof(double);
  static constexpr int T_NEED = P3 + 6 * FACE_ARR * P2;
  static constexpr int T_REGION = 6 * TF > T_NEED ? 6 * TF : T_NEED;
  static constexpr size_t BYTES = apply_bytes(3, 6, TS);
  static constexpr bool FITS = BYTES <= 232448;
};

// the twelve coefficients of a point: w |J|, C_11 C_22 C_33 C_12 C_23 C_13 C_1 C_2 C_3 C_0, padding
template <int FROM, int TO>
__device__ __forceinline__ void gen_coef(const real *p, real *c) {
#if defined(HPSE_DOUBLE)
#pragma unroll
  for (int i = FROM; i < TO; i += 2) {
    const double2 v = *reinterpret_cast<const double2 *>(p + i);
    c[i] = v.x;
    c[i + 1] = v.y;
  }
#else
#pragma unroll
  for (int i = FROM; i < TO; i += 4) {
    const float4 v = *reinterpret_cast<const float4 *>(p + i);
    c[i] = v.x;
    c[i + 1] = v.y;
    c[i + 2] = v.z;
    c[i + 3] = v.w;
  }
#endif
}

// forward pair of the odd matrix B1 on two lines: as fwd_pm<1> on both halves
__device__ __forceinline__ void fwd_odd2(const real2 *e, const real2 *o, int q, real2 &pl, real2 &mi) {
#pragma unroll
  for (int j = 0; j < HP; ++j) pl = fma2(c_tab.XO[2][q * HPE + j], o[j], pl);
  if (q < HQ) {
#pragma unroll
    for (int j = 0; j < HPE; ++j) mi = fma2(c_tab.XE[2][q * HPE + j], e[j], mi);
  }
}
// transposed pair of B1: one folded input pair into every output pair / the middle point
__device__ __forceinline__ void rev_pair_odd2(real2 ve, real2 vo, int q, real2 *pl, real2 *mi) {
#pragma unroll
  for (int k = 0; k < HPE; ++k) {
    pl[k] = fma2(c_tab.XE[2][q * HPE + k], vo, pl[k]);
    if (k < HP) mi[k] = fma2(c_tab.XO[2][q * HPE + k], ve, mi[k]);
  }
}
__device__ __forceinline__ void rev_mid_odd2(real2 vm, real2 *mi) {
#pragma unroll
  for (int k = 0; k < HP; ++k) mi[k] = fma2(c_tab.XO[2][HQ * HPE + k], vm, mi[k]);
}
// transposed pair of B1 over a whole folded line into output pair k
__device__ __forceinline__ void rev_line_odd2(const real2 *ve, const real2 *vo, real2 vm, int k, real2 &pl, real2 &mi) {
#pragma unroll
  for (int q = 0; q < HQ; ++q) {
    pl = fma2(c_tab.XE[2][q * HPE + k], vo[q], pl);
    if (k < HP) mi = fma2(c_tab.XO[2][q * HPE + k], ve[q], mi);
  }
  if (k < HP) mi = fma2(c_tab.XO[2][HQ * HPE + k], vm, mi);
}

// y-stage of line (qa, k): T00 T01 T02 from X0, T10 T11 from X1, T20 from X2.
// Pairs: (B0 X0, B2 X0), (B0 X1, B0 X2), (B1 X0, B1 X1).
template <int CI, int NC>
__device__ __forceinline__ void gen_y_fwd(const real2 *de, const real2 *dd, const real2 *we, const real2 *wo, real *T,
                                          bool ok) {
  typedef Range<CI, NC, HQ + 1> R;
  constexpr int TF = GenLayout::TF;
#pragma unroll
  for (int qb = R::B; qb < R::E; ++qb) {
    real2 ap = zero2(), am = zero2(), bp = zero2(), bm = zero2(), cp = zero2(), cm = zero2();
    fwd_pm2<1>(de, dd, qb, ap, am);
    fwd_pm2<0>(we, wo, qb, bp, bm);
    {
      real2 ce[HPE], co[HPE];
#pragma unroll
      for (int j = 0; j < HPE; ++j) {
        ce[j] = mk2(de[j].x, we[j].x);
        co[j] = mk2(dd[j].x, wo[j].x);
      }
      fwd_odd2(ce, co, qb, cp, cm);
    }
    if (ok) {
      put_q(T, Q, qb, ap.x, am.x);
      put_q(T + TF, Q, qb, cp.x, cm.x);
      put_q(T + 2 * TF, Q, qb, ap.y, am.y);
      put_q(T + 3 * TF, Q, qb, bp.x, bm.x);
      put_q(T + 4 * TF, Q, qb, cp.y, cm.y);
      put_q(T + 5 * TF, Q, qb, bp.y, bm.y);
    }
    __syncwarp();  // scheduling fence (register pressure); reached by all 32 lanes
  }
}

// y-stage transpose of line (qa, k), outputs j of a chunk:
//   X0' = B0^T T00' + B1^T T01' + B2^T T02', X1' = B0^T T10' + B1^T T11', X2' = B0^T T20'
// in the pairs (T00', T02') x (B0, B2), (T10', T20') x (B0, B0), (T01', T11') x (B1, B1)
template <int CI, int NC>
__device__ __forceinline__ void gen_y_rev(const real *T, real *X, bool ok) {
  typedef Range<CI, NC, HPE> R;
  constexpr int TF = GenLayout::TF, N = R::E - R::B > 0 ? R::E - R::B : 1;
  real2 ap[N], am[N], bp[N], bm[N];
  {
    real2 ve[HQ], vo[HQ], vm, v[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = mk2(T[q * Q], T[2 * TF + q * Q]);
    fold_q2(v, ve, vo, vm);
#pragma unroll
    for (int j = R::B; j < R::E; ++j) {
      real2 pl = zero2(), mi = zero2();
      rev_line2<1>(ve, vo, vm, j, pl, mi);
      ap[j - R::B] = mk2(pl.x + pl.y, 0);  // X0' so far, X1'
      am[j - R::B] = mk2(mi.x + mi.y, 0);
    }
  }
  __syncwarp();  // scheduling fence (register pressure); reached by all 32 lanes
  {
    real2 ve[HQ], vo[HQ], vm, v[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = mk2(T[3 * TF + q * Q], T[5 * TF + q * Q]);
    fold_q2(v, ve, vo, vm);
#pragma unroll
    for (int j = R::B; j < R::E; ++j) {
      bp[j - R::B] = bm[j - R::B] = zero2();
      rev_line2<0>(ve, vo, vm, j, bp[j - R::B], bm[j - R::B]);
      ap[j - R::B].y = bp[j - R::B].x;
      am[j - R::B].y = bm[j - R::B].x;
    }
  }
  __syncwarp();  // scheduling fence (register pressure); reached by all 32 lanes
  {
    real2 ve[HQ], vo[HQ], vm, v[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = mk2(T[TF + q * Q], T[4 * TF + q * Q]);
    fold_q2(v, ve, vo, vm);
#pragma unroll
    for (int j = R::B; j < R::E; ++j) {
      rev_line_odd2(ve, vo, vm, j, ap[j - R::B], am[j - R::B]);
      if (ok) {
        put_p2(X, X + QP2, Q, j, ap[j - R::B], am[j - R::B]);
        put_p(X + 2 * QP2, Q, j, bp[j - R::B].y, bm[j - R::B].y);
      }
    }
  }
}

template <int MODE>
__global__ void __launch_bounds__(NT, GEN_MINB) k_apply_gen(const ApplyArgs A) {
  typedef GenLayout L;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  real *su = reinterpret_cast<real *>(smem_raw);
  real *sX = su + P3;                 // X0 | X1 | X2, later X0' | X1' | X2'
  real *sT = sX + 3 * QP2;            // T00 T01 T02 T10 T11 T20 (in place -> T')
  real *stab = sT + L::T_REGION;
  double *red = reinterpret_cast<double *>(smem_raw + L::RED_OFF);
  constexpr int TS = L::TS, TF = L::TF;
  real *X0 = sX, *X1 = sX + QP2, *X2 = sX + 2 * QP2;

  const int item = blockIdx.x;
  const int ge = item / A.n_rhs;
  const int r = item - ge * A.n_rhs;
  const int e = A.elems[ge];
  const int64_t base = (int64_t)r * A.ndof + A.dof_off[e];
  const real *geo_e = A.geo + (int64_t)e * 4;
  const int tid = threadIdx.x;
  constexpr int nt = NT;

  for (int t = tid; t < P2; t += nt) stab[t] = c_tab.D[t];
  FaceMeta *fm = face_meta(stab);
  if (MODE != MODE_TRANSPOSE && tid < 6) face_meta_fill<COEF_LAPLACE, MODE>(A, e, r, geo_e, fm, tid);
  if (MODE != MODE_TRANSPOSE) {
    if (MODE == MODE_PCG) {
      const double bt = A.beta[A.prob[e] * A.n_rhs + r];
      for (int t = tid; t < P3; t += nt) {
        const real v = A.z[base + t] + (real)bt * A.u[base + t];
        su[t] = v;
        A.pnew[base + t] = v;
      }
    } else {
      for (int t = tid; t < P3; t += nt) su[t] = A.u[base + t];
    }
    __syncthreads();
    // x-stage: lines (j, k); the stage of -div(a grad u)
    {
      typedef Lines<P2> LS;
      for (int it = tid; it < LS::NC * LS::PADL; it += nt) {
        const int c = it / LS::PADL, lp = it - c * LS::PADL;
        const bool ok = lp < P2;
        const int l = ok ? lp : P2 - 1;
        real v[P], e1[HPE], o1[HPE];
#pragma unroll
        for (int i = 0; i < P; ++i) v[i] = su[l * P + i];
        fold_p(v, e1, o1);
        real2 e2[HPE], o2[HPE];
#pragma unroll
        for (int j = 0; j < HPE; ++j) {
          e2[j] = mk2(e1[j], e1[j]);
          o2[j] = mk2(o1[j], o1[j]);
        }
#define GEN_XF(CI) x_fwd_chunk2<COEF_SCALAR, (CI < LS::NC ? CI : 0), LS::NC>(e2, o2, X0, X1, X2, l, ok)
        HPSE_DISPATCH4(LS::NC, c, GEN_XF);
#undef GEN_XF
      }
    }
    __syncthreads();
    // y-stage: lines (qa, k), six output fields; T[f][k TS + qb Q + qa]
    {
      typedef Lines<QP> LS;
      for (int it = tid; it < LS::NC * LS::PADL; it += nt) {
        const int c = it / LS::PADL, lp = it - c * LS::PADL;
        const bool ok = lp < QP;
        const int l = ok ? lp : QP - 1;
        const int qa = l % Q, k = l / Q;
        real2 de[HPE], dd[HPE], we[HPE], wo[HPE], v[P];
#pragma unroll
        for (int j = 0; j < P; ++j) {
          const real x0 = X0[(k * P + j) * Q + qa];
          v[j] = mk2(x0, x0);
        }
        fold_p2(v, de, dd);
#pragma unroll
        for (int j = 0; j < P; ++j) v[j] = mk2(X1[(k * P + j) * Q + qa], X2[(k * P + j) * Q + qa]);
        fold_p2(v, we, wo);
#define GEN_YF(CI) gen_y_fwd<(CI < LS::NC ? CI : 0), LS::NC>(de, dd, we, wo, sT + k * TS + qa, ok)
        HPSE_DISPATCH4(LS::NC, c, GEN_YF);
#undef GEN_YF
      }
    }
    __syncthreads();
  }

  // z-stage per column (qa, qb).  (The loop runs to whole warps: lanes past the
  // last column read it and store nothing, so that every lane reaches the
  // __syncwarp fences.)
  for (int lp = tid; lp < PAD32(Q2); lp += nt) {
    const bool ok = lp < Q2;
    const int l = ok ? lp : Q2 - 1;
    const int64_t cbase = A.coef_off[e] + l;
    const real *cp = A.coef + GEN_NC * cbase;
    real *T = sT + l;  // rho[q] at T[q TS]: rows of T00, then of T01 (Q <= 2 P)
    if (MODE == MODE_TRANSPOSE) {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const real v = (real)A.rho[(int64_t)r * A.nquad + cbase + (int64_t)q * Q2];
        if (ok) T[q * TS] = v;
      }
    } else {
      // (T00, T01), (T02, T10), (T11, T20)
      real2 ea[HPE], oa[HPE], eb[HPE], ob[HPE], ec[HPE], oc[HPE];
      {
        real2 v[P];
#pragma unroll
        for (int k = 0; k < P; ++k) v[k] = mk2(T[k * TS], T[TF + k * TS]);
        fold_p2(v, ea, oa);
#pragma unroll
        for (int k = 0; k < P; ++k) v[k] = mk2(T[2 * TF + k * TS], T[3 * TF + k * TS]);
        fold_p2(v, eb, ob);
#pragma unroll
        for (int k = 0; k < P; ++k) v[k] = mk2(T[4 * TF + k * TS], T[5 * TF + k * TS]);
        fold_p2(v, ec, oc);
      }
      __syncwarp();  // rho overwrites T00 and T01: every lane has its lines (the last column's are shared)
#pragma unroll
      for (int qc = 0; qc <= HQ; ++qc) {
        real2 ap = zero2(), am = zero2(), bp = zero2(), bm = zero2(), dp = zero2(), dm = zero2(), fp = zero2(),
              fm2 = zero2();
        real p3 = 0, m3 = 0, p13 = 0, m13 = 0;
        fwd_pm2<0>(ea, oa, qc, ap, am);       // u, u_2
        fwd_odd2(ea, oa, qc, dp, dm);         // u_3, u_23
        fwd_pm_h<2, 0>(ea, oa, qc, p3, m3);   // u_33
        fwd_pm2<0>(eb, ob, qc, bp, bm);       // u_22, u_1
        fwd_pm_h<1, 1>(eb, ob, qc, p13, m13); // u_13
        fwd_pm2<0>(ec, oc, qc, fp, fm2);      // u_12, u_11
#pragma unroll
        for (int side = 0; side < (qc < HQ ? 2 : 1); ++side) {
          const int q = side ? Q - 1 - qc : qc;
          const real sg = side ? (real)-1 : (real)1;
          real c[12];
          gen_coef<0, 12>(cp + (int64_t)q * Q2 * GEN_NC, c);
          const real2 a = side ? sub2(ap, am) : add2(ap, am), b = side ? sub2(bp, bm) : add2(bp, bm);
          const real2 d = side ? sub2(dp, dm) : add2(dp, dm), f = side ? sub2(fp, fm2) : add2(fp, fm2);
          real2 s = fma2(mk2(c[10], c[8]), a, mk2(c[3] * (p3 + sg * m3), c[6] * (p13 + sg * m13)));
          s = fma2(mk2(c[9], c[5]), d, s);
          s = fma2(mk2(c[2], c[7]), b, s);
          s = fma2(mk2(c[4], c[1]), f, s);
          if (ok) T[q * TS] = c[0] * (s.x + s.y);
        }
        __syncwarp();  // scheduling fence (register pressure); reached by all 32 lanes
      }
    }
    __syncwarp();
    // transposed, first the lines whose slots hold no rho: (T02', T10') from
    // (C_22, C_1) rho by (B0, B0) and C_13 rho by B1 into T10', (T11', T20') from (C_12, C_11) rho
    {
      real2 pa[HPE], ma[HPE], pb[HPE], mb[HPE];
#pragma unroll
      for (int k = 0; k < HPE; ++k) pa[k] = ma[k] = pb[k] = mb[k] = zero2();
#pragma unroll
      for (int qc = 0; qc <= HQ; ++qc) {
        real2 va[2], vb[2];
        real sd[2];
#pragma unroll
        for (int side = 0; side < (qc < HQ ? 2 : 1); ++side) {
          const int q = side ? Q - 1 - qc : qc;
          const real rq = T[q * TS];
          real c[12];
          gen_coef<0, 8>(cp + (int64_t)q * Q2 * GEN_NC, c);
          va[side] = mk2(c[2] * rq, c[7] * rq);
          vb[side] = mk2(c[4] * rq, c[1] * rq);
          sd[side] = c[6] * rq;
        }
        if (qc < HQ) {
          rev_pair2<0>(add2(va[0], va[1]), sub2(va[0], va[1]), qc, pa, ma);
          rev_pair2<0>(add2(vb[0], vb[1]), sub2(vb[0], vb[1]), qc, pb, mb);
          const real se = sd[0] + sd[1], so = sd[0] - sd[1];
#pragma unroll
          for (int k = 0; k < HPE; ++k) {
            pa[k].y += c_tab.FE[1][qc * HPE + k] * so;
            if (k < HP) ma[k].y += c_tab.FO[1][qc * HPE + k] * se;
          }
        } else {
          rev_mid2<0>(va[0], pa);
          rev_mid2<0>(vb[0], pb);
#pragma unroll
          for (int k = 0; k < HP; ++k) ma[k].y += c_tab.FO[1][HQ * HPE + k] * sd[0];
        }
        __syncwarp();  // scheduling fence (register pressure); reached by all 32 lanes
      }
      if (ok) {
#pragma unroll
        for (int k = 0; k < HPE; ++k) {
          put_p2(T + 2 * TF, T + 3 * TF, TS, k, pa[k], ma[k]);
          put_p2(T + 4 * TF, T + 5 * TF, TS, k, pb[k], mb[k]);
        }
      }
    }
    // then (T00', T01') from (C_0, C_2) rho by (B0, B0), (C_3, C_23) rho by (B1, B1), C_33 rho by B2 into T00'
    {
      real2 pa[HPE], ma[HPE];
#pragma unroll
      for (int k = 0; k < HPE; ++k) pa[k] = ma[k] = zero2();
#pragma unroll
      for (int qc = 0; qc <= HQ; ++qc) {
        real2 va[2], vd[2];
        real s2[2];
#pragma unroll
        for (int side = 0; side < (qc < HQ ? 2 : 1); ++side) {
          const int q = side ? Q - 1 - qc : qc;
          const real rq = T[q * TS];
          real c[12];
          gen_coef<0, 12>(cp + (int64_t)q * Q2 * GEN_NC, c);
          va[side] = mk2(c[10] * rq, c[8] * rq);
          vd[side] = mk2(c[9] * rq, c[5] * rq);
          s2[side] = c[3] * rq;
        }
        if (qc < HQ) {
          rev_pair2<0>(add2(va[0], va[1]), sub2(va[0], va[1]), qc, pa, ma);
          rev_pair_odd2(add2(vd[0], vd[1]), sub2(vd[0], vd[1]), qc, pa, ma);
          const real se = s2[0] + s2[1], so = s2[0] - s2[1];
#pragma unroll
          for (int k = 0; k < HPE; ++k) {
            pa[k].x += c_tab.FE[2][qc * HPE + k] * se;
            if (k < HP) ma[k].x += c_tab.FO[2][qc * HPE + k] * so;
          }
        } else {
          rev_mid2<0>(va[0], pa);
          rev_mid_odd2(vd[0], ma);
#pragma unroll
          for (int k = 0; k < HPE; ++k) pa[k].x += c_tab.FE[2][HQ * HPE + k] * s2[0];
        }
        __syncwarp();  // scheduling fence (register pressure); reached by all 32 lanes
      }
      if (ok) {
#pragma unroll
        for (int k = 0; k < HPE; ++k) put_p2(T, T + TF, TS, k, pa[k], ma[k]);
      }
    }
  }
  __syncthreads();

  // y-stage transpose (lines (qa, k)), outputs j in chunks; X_m'[(k P + j) Q + qa]
  {
    typedef Lines<QP> LS;
    for (int it = tid; it < LS::NC * LS::PADL; it += nt) {
      const int c = it / LS::PADL, lp = it - c * LS::PADL;
      const bool ok = lp < QP;
      const int l = ok ? lp : QP - 1;
      const int qa = l % Q, k = l / Q;
#define GEN_YR(CI) gen_y_rev<(CI < LS::NC ? CI : 0), LS::NC>(sT + k * TS + qa, sX + k * P * Q + qa, ok)
      HPSE_DISPATCH4(LS::NC, c, GEN_YR);
#undef GEN_YR
    }
  }
  __syncthreads();

  // x-stage transpose (lines (j, k)): y = sum_m B_m^T X_m'
  real *sy = sT;  // the T region is free now
  {
    typedef Lines<P2> LS;
    for (int it = tid; it < LS::NC * LS::PADL; it += nt) {
      const int c = it / LS::PADL, lp = it - c * LS::PADL;
      const bool ok = lp < P2;
      const int l = ok ? lp : P2 - 1;
#define GEN_XR(CI) x_rev_chunk2<COEF_SCALAR, (CI < LS::NC ? CI : 0), LS::NC>(X0, X1, X2, sy, l, ok)
      HPSE_DISPATCH4(LS::NC, c, GEN_XR);
#undef GEN_XR
    }
  }
  __syncthreads();

  // faces: those of the Laplacian on box meshes (the operator does not enter)
  if (MODE != MODE_TRANSPOSE && !A.skip_faces)
    face_phase<COEF_LAPLACE, MODE>(A, e, r, su, sy, sT + P3, stab, geo_e, fm);

  double part = 0.0;
  for (int t = tid; t < P3; t += nt) {
    const real v = sy[t];
    A.y[base + t] = v;
    if (MODE == MODE_PCG) part += hpse::widen(v) * hpse::widen(su[t]);
  }
  if (MODE == MODE_PCG) {
    const double s = block_sum(part, red);
    if (tid == 0) A.partial[(int64_t)e * A.n_rhs + r] = s;
  }
}

template <int MODE>
cudaError_t launch_apply_gen(const void *args, int n_items, cudaStream_t s) {
  if constexpr (GenLayout::FITS) {
    k_apply_gen<MODE><<<n_items, NT, GenLayout::BYTES, s>>>(*static_cast<const ApplyArgs *>(args));
    return cudaGetLastError();
  } else {
    (void)args;
    (void)n_items;
    (void)s;
    return cudaErrorInvalidConfiguration;
  }
}

template <int MODE>
cudaError_t set_smem_attr_gen() {
  if constexpr (GenLayout::FITS) {
    cudaError_t e = cudaFuncSetAttribute(k_apply_gen<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)GenLayout::BYTES);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_apply_gen<MODE>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                (int)cudaSharedmemCarveoutMaxShared);
  } else {
    return cudaSuccess;
  }
}

}  // namespace
