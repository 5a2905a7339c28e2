// Reverse (vector-Jacobian) pass of the per-voxel Meric-Cailletaud update (Sec. 3 law,
// Sec. 4 regularised rates, RK4 substeps along the linear strain path): given adjoints of
// the outputs (stress at t_{n+1} and state at t_{n+1}) it returns adjoints of the inputs
// (strain at t_n and t_{n+1}, state at t_n, rotation) and of the material parameters.
// This is the constitutive building block of the adjoint of the load history; with unit
// stress adjoints it gives the rows of the algorithmic tangent d sigma / d eps.
//
// One forward pass per voxel, with the primal's operations (constitutive.cuh), leaves a record
// of every RK4 stage (VjpStage): its rates and their derivatives, hardening exponentials and
// plastic rate sums (in blocks for more than 8 substeps, see vjp_sweeps).  A reverse sweep reads
// the records and solves nothing.  The regularised
// rate rho(a, P) solving rho = P ((a - eta rho)/K)^n is differentiated implicitly: with
// z = (a - eta rho)/K and D = K + eta P n z^(n-1),
//   d rho / d a = P n z^(n-1) / D,   d rho / d P = K z^n / D   (0 where rho = 0).
// The sweeps are bound by the FP64 pipe in double and by local memory in float.  Rebuilding every
// stage from its state in every sweep (exponentials, three divisions a system, products with zero
// Schmid coefficients, rotations as nested sums) took 1750 FP64 instructions a stage; a sweep of
// the tangent (k_adj_tangent runs seven over one forward pass) now takes about 240.  20^3 FP64
// history gradient 39.5 -> 29.1 ms; 100003 float points 0.936 -> 0.898 ms.
#pragma once

#include "constitutive.cuh"

namespace rve {

// Adjoints of the material parameters (order of the C ABI's param_bar rows).
constexpr int kParamBar = 9;  // r0_ord, r0_sup, r0_twin, Q_s, Q_b, b_s, b_b, c, d

template <typename T>
__device__ __forceinline__ void state_axpy(MPState<T>& y, T w, const MPState<T>& x) {
  #pragma unroll
  for (int c = 0; c < 6; ++c) y.ep[c] += w * x.ep[c];
  #pragma unroll
  for (int c = 0; c < 16; ++c) y.v[c] += w * x.v[c];
  #pragma unroll
  for (int c = 0; c < 12; ++c) y.al[c] += w * x.al[c];
}
template <typename T>
__device__ __forceinline__ void state_zero(MPState<T>& y) {
  #pragma unroll
  for (int c = 0; c < 6; ++c) y.ep[c] = T(0);
  #pragma unroll
  for (int c = 0; c < 16; ++c) y.v[c] = T(0);
  #pragma unroll
  for (int c = 0; c < 12; ++c) y.al[c] = T(0);
}

// What the reverse of one RK4 stage needs of its forward evaluation.  A system of which no
// voxel of the warp flows has no part in the reverse (its rate and derivative are 0); its bit
// 16 + q of `bits` is 0 and its da and dP are left unset.
template <typename T>
struct VjpStage {
  T rho[16];     // rates
  T da[16];      // d rho / d a
  T dP[4];       // d rho / d P of the twins
  T ex[16];      // exp(-b v)
  T al[12];      // kinematic variables of the stage's state
  T du[6];       // sum_s gdot_s (n x l) of the slip systems, unscaled
  T ftot;        // sum f
  unsigned bits;  // bit q < 12: the slip system's driving stress is negative; bit 16 + q: flows
};

// d rho / d a and d rho / d P at a solved root (rho, a, P; exponent n, K, eta).
template <typename T>
__device__ __forceinline__ void root_partials(T rho, T a, T P, T Kn, T n, T eta, T* d_a, T* d_P) {
  *d_a = *d_P = T(0);
  if (!(rho > T(0)) || !(P > T(0))) return;
  const T z = (a - eta * rho) / Kn;
  if (!(z > T(0))) return;
  const T zn = rho / P;              // z^n
  const T pnz = P * n * (zn / z);    // P n z^(n-1)
  const T D = Kn + eta * pnz;
  *d_a = pnz / D;
  *d_P = Kn * zn / D;
}

// Forward stage (the operations of rk_stage, one system at a time; the float primal runs
// pairs of systems on packed instructions, which may round the last bit differently): rates k
// of state Y at path point s and the stage's record.  Systems in which no voxel of the warp
// flows cost their driving force only.
template <typename T, int NP>
__device__ __forceinline__ void vjp_stage(const MatDev<T>& M, const T* e0, const T* de, T s, const MPState<T>& Y,
                                          const T* tab, VjpStage<T>& V, MPState<T>& k) {
  constexpr double kLog2e = 1.44269504088896340736;
  const unsigned lanes = __activemask();
  T ex[16], Es = T(0), Et = T(0), vtw = T(0);
  const T cb_s = -M.b_s * T(kLog2e), cb_t = -M.b_b * T(kLog2e);
#pragma unroll
  for (int q = 0; q < 12; ++q) {
    ex[q] = hard_exp2<T, NP>(M, cb_s * Y.v[q], tab);
    Es += ex[q];
    V.ex[q] = ex[q];
    V.al[q] = Y.al[q];
  }
#pragma unroll
  for (int q = 12; q < 16; ++q) {
    ex[q] = hard_exp2<T, NP>(M, cb_t * Y.v[q], tab);
    Et += ex[q];
    vtw += Y.v[q];
    V.ex[q] = ex[q];
  }
  const T ftot = T(1.41421356237309504880) * vtw;
  T fm_left = M.fm - ftot;
  fm_left = fm_left > T(0) ? fm_left : T(0);
  const T Ptw = (M.Kc * T(0.70710678118654752440)) * fm_left;
  const T dq = M.h_diag - M.h_off;
  const T Qdq_s = M.Q_s * dq, Qdq_t = M.Q_b * dq;
  const T Rb_s = M.Q_s * (M.h_off * (T(12) - Es) + dq), Rb_t = M.Q_b * (M.h_off * (T(4) - Et) + dq);
  const T rb_sup = M.r0[0] + Rb_s, rb_ord = M.r0[2] + Rb_s, rb_tw = M.r0[12] + Rb_t;
  RootCoef<T> qs, qt;
  T lg_Ptw = T(0), s_tw = T(0), is_tw = T(0);
  bool scaled = false;
  if constexpr (NP != kDirect) lg_Ptw = fast_log2<T>(Ptw > T(0) ? Ptw : T(1));
  if constexpr (NP != 0 && NP != kDirect) {
    qs = root_coef<T>(T(1), M.K, M.n, M.inv_n, M.lg_K, M.eta, M.lg_eta, T(0));
    qt = root_coef<T>(Ptw, M.Kt, M.nt, M.inv_nt, M.lg_Kt, M.eta, M.lg_eta, lg_Ptw);
  }
  // slip-scaled stress C : e / sqrt6
  T ss[6];
  {
    T e[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) e[c] = e0[c] + s * de[c] - Y.ep[c];
    ss[0] = M.C11s * e[0] + M.C12s * e[1] + M.C13s * e[2];
    ss[1] = M.C12s * e[0] + M.C11s * e[1] + M.C13s * e[2];
    ss[2] = M.C13s * (e[0] + e[1]) + M.C33s * e[2];
    ss[3] = M.C44s2 * e[3];
    ss[4] = M.C44s2 * e[4];
    ss[5] = M.C66s2 * e[5];
  }
  unsigned bits = 0;
  T du[6] = {T(0), T(0), T(0), T(0), T(0), T(0)}, G = T(0), H[3] = {T(0), T(0), T(0)};
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    T S[3], D[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int i = 0; i < 3; ++i) S[i] = plane_sig(p, i) > 0 ? ss[i] + ss[i + 3] : ss[i] - ss[i + 3];
#pragma unroll
    for (int q = 3 * p; q < 3 * p + 3; ++q) {
      const T al = Y.al[q];
      const T tk = plane_sum<T>(q, S) - M.c * al;
      const T a = fabs(tk) - ((q % 3 == 2 ? rb_ord : rb_sup) - Qdq_s * ex[q]);
      k.v[q] = k.al[q] = T(0);
      if (__any_sync(lanes, a > T(0))) {
        const T rho = stage_rate<T, NP>(M, qs, a, T(1), false, T(0), tab);
        T d_a, d_P;
        root_partials<T>(rho, a, T(1), M.K, M.n, M.eta, &d_a, &d_P);
        const T gd = copysign(rho, tk);
        bits |= (tk < T(0) ? 1u : 0u) << q | 1u << (16 + q);
        V.da[q] = d_a;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          if (diag_k(q, i) == 1) D[i] += gd;
          else if (diag_k(q, i) == -1) D[i] -= gd;
        }
        k.v[q] = rho;
        k.al[q] = gd - M.d * rho * al;
      }
      V.rho[q] = k.v[q];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      du[i] += D[i];
      if (plane_sig(p, i) > 0) du[i + 3] += D[i];
      else du[i + 3] -= D[i];
    }
    const int q = 12 + p;
    // 1/(|n||l|) of a twin is (1/sqrt3) times the slip systems' scale in ss
    const T a = T(0.57735026918962576451) * plane_sum<T>(q, S) - (rb_tw - Qdq_t * ex[q]);
    k.v[q] = T(0);
    if (__any_sync(lanes, a > T(0) && Ptw > T(0))) {
      T rho;
      if constexpr (NP == kDirect) {
        if (!scaled) {
          const T l = fast_log2<T>(Ptw > T(0) ? Ptw : T(1)) * M.inv_ntm1;
          s_tw = Ptw > T(0) ? hard_exp2<T, NP>(M, l, tab) : T(0);
          is_tw = Ptw > T(0) ? hard_exp2<T, NP>(M, -l, tab) : T(0);
          scaled = true;
        }
        rho = rate_root<T>(M, a * s_tw, true, tab) * is_tw;
      } else {
        rho = stage_rate<T, NP>(M, qt, a, Ptw, true, lg_Ptw, tab);
      }
      T d_a, d_P;
      root_partials<T>(rho, a, Ptw, M.Kt, M.nt, M.eta, &d_a, &d_P);
      bits |= 1u << (16 + q);
      V.da[q] = d_a;
      V.dP[p] = d_P;
      G += rho;
#pragma unroll
      for (int i = 0; i < 3; ++i) H[i] += plane_sig(p, i) > 0 ? rho : -rho;
      k.v[q] = rho;
    }
    V.rho[q] = k.v[q];
  }
  const T fs = (T(1) - ftot) * sys_scale<T>(0), tsc = sys_scale<T>(12);
  const T dt6[6] = {G, G, T(-2) * G, H[0], H[1], T(-2) * H[2]};
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    V.du[c] = du[c];
    k.ep[c] = (c < 3 ? T(1) : T(0.5)) * (fs * du[c] + tsc * dt6[c]);
  }
  V.ftot = ftot;
  V.bits = bits;
}

// Reverse of one stage (record V) of a substep y' = y + h/6 (k1 + 2 k2 + 2 k3 + k4): the
// adjoint of its rates is kb = cw yend + cY Yb, with yend the adjoint of y' and Yb that of the
// next stage's state (in); Yb (out) is the adjoint of this stage's state and is added to yb.
// e0b and deb receive the strain path's adjoint (s: the stage's path point).  With `full` the
// parameters' adjoints are added to pb (v: the stage's slips are v[q] + cv vr[q]).
// The Schmid sums go through the plane sums (plane_sum); systems that do not flow are skipped.
template <typename T>
__device__ __forceinline__ void vjp_stage_reverse(const MatDev<T>& M, const VjpStage<T>& V, T s,
                                                  const MPState<T>& yend, T cw, T cY, MPState<T>& Yb, MPState<T>& yb,
                                                  T* e0b, T* deb, T* pb, bool full, const T* v, T cv, const T* vr) {
  const unsigned bits = V.bits;
  if (!(bits >> 16)) {  // no flow: the rates do not depend on anything
    state_zero<T>(Yb);
    return;
  }
  const T dq = M.h_diag - M.h_off;
  const T ssc = sys_scale<T>(0), tsc = sys_scale<T>(12);
  const T ftot = V.ftot, w = (T(1) - ftot) * ssc;
  // eps_p rate: k.ep[c] = wc (wslip ssc du[c] + tsc du_t[c])
  T kbe[6], wslipb = T(0);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    kbe[c] = (c < 3 ? T(1) : T(0.5)) * (cw * yend.ep[c] + cY * Yb.ep[c]);
    wslipb += kbe[c] * V.du[c];
  }
  wslipb *= ssc;
  T sgs[6] = {T(0), T(0), T(0), T(0), T(0), T(0)}, G = T(0), H[3] = {T(0), T(0), T(0)};
  T As = T(0), At = T(0), Ptwb = T(0);  // sums of the overstress adjoints, adjoint of P
  T hs = T(0), ht = T(0);
  if (full) {  // hardening sums of Q_s and Q_b
    T Es = T(0), Et = T(0);
#pragma unroll
    for (int q = 0; q < 12; ++q) Es += V.ex[q];
#pragma unroll
    for (int q = 12; q < 16; ++q) Et += V.ex[q];
    hs = M.h_off * (T(12) - Es) + dq;
    ht = M.h_off * (T(4) - Et) + dq;
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    T B[3], D[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int i = 0; i < 3; ++i) B[i] = plane_sig(p, i) > 0 ? kbe[i] + kbe[i + 3] : kbe[i] - kbe[i + 3];
#pragma unroll
    for (int q = 3 * p; q < 3 * p + 3; ++q) {
      T exb = T(0), alb = T(0);
      if (bits >> (16 + q) & 1u) {
        const bool neg = bits >> q & 1u;
        const T rho = V.rho[q], al = V.al[q];
        const T kal = cw * yend.al[q] + cY * Yb.al[q], kv = cw * yend.v[q] + cY * Yb.v[q];
        const T gdb = kal + w * plane_sum<T>(q, B);
        // gd enters the plastic rate and k.al = gd - d rho al
        const T akb = (kv + (neg ? -gdb : gdb) - M.d * al * kal) * V.da[q];
        // a = |tek| - ((r0 + Rb_s) - Qdq_s ex), tek = ssc sum K sg - c al
        const T tekb = neg ? -akb : akb;
        As += akb;
        exb = akb * (M.Q_s * dq);
        alb = -M.d * rho * kal - M.c * tekb;
        yb.al[q] += alb;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          if (diag_k(q, i) == 1) D[i] += tekb;
          else if (diag_k(q, i) == -1) D[i] -= tekb;
        }
        if (full) {
          pb[q % 3 == 2 ? 0 : 1] -= akb;            // r0: ordinary systems, superdislocations
          pb[3] -= akb * (hs - dq * V.ex[q]);       // Q_s
          pb[7] -= al * tekb;                       // c
          pb[8] -= rho * al * kal;                  // d
        }
      }
      Yb.al[q] = alb;
      Yb.v[q] = exb;  // the exponential's adjoint for now
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      sgs[i] += D[i];
      if (plane_sig(p, i) > 0) sgs[i + 3] += D[i];
      else sgs[i + 3] -= D[i];
    }
    const int q = 12 + p;
    T exb = T(0);
    if (bits >> (16 + q) & 1u) {
      const T rhob = cw * yend.v[q] + cY * Yb.v[q] + tsc * plane_sum<T>(q, B);
      const T akb = rhob * V.da[q];
      Ptwb += rhob * V.dP[p];
      At += akb;
      exb = akb * (M.Q_b * dq);
      G += akb;
#pragma unroll
      for (int i = 0; i < 3; ++i) H[i] += plane_sig(p, i) > 0 ? akb : -akb;
      if (full) {
        pb[2] -= akb;                          // r0_twin
        pb[4] -= akb * (ht - dq * V.ex[q]);    // Q_b
      }
    }
    Yb.v[q] = exb;
  }
  // Ptw = Kc/sqrt2 max(fm - ftot, 0); wslip = 1 - ftot; ftot = sqrt2 sum v_twin
  T ftotb = -wslipb;
  if (M.fm - ftot > T(0)) ftotb -= Ptwb * (M.Kc * T(0.70710678118654752440));
  const T vtwb = T(1.41421356237309504880) * ftotb;
  // ex = exp(-b v)
  const T Esb = As * (M.Q_s * M.h_off), Etb = At * (M.Q_b * M.h_off);
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const T exb = Yb.v[q] + (q < 12 ? Esb : Etb);
    const T t = exb * V.ex[q];
    Yb.v[q] = q < 12 ? -M.b_s * t : vtwb - M.b_b * t;
    yb.v[q] += Yb.v[q];
    if (full) pb[q < 12 ? 5 : 6] -= t * (v[q] + cv * vr[q]);  // b_s, b_b
  }
  // stress = C : e, e = e0 + s de - ep
  const T sgt[6] = {G, G, T(-2) * G, H[0], H[1], T(-2) * H[2]};
  T sgb[6], eb[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) sgb[c] = ssc * sgs[c] + tsc * sgt[c];
  hooke<T>(M, sgb, eb);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    e0b[c] += eb[c];
    deb[c] += s * eb[c];
    Yb.ep[c] = -eb[c];
    yb.ep[c] -= eb[c];
  }
}

// Symmetric 3x3 from 6 components (11 22 33 23 13 12) and back.
template <typename T>
__device__ __forceinline__ void sym33(const T* v, T A[3][3]) {
  A[0][0] = v[0]; A[1][1] = v[1]; A[2][2] = v[2];
  A[1][2] = A[2][1] = v[3];
  A[0][2] = A[2][0] = v[4];
  A[0][1] = A[1][0] = v[5];
}
// adjoint of `sym33` for a symmetric tensor adjoint G: off-diagonal components appear twice
template <typename T>
__device__ __forceinline__ void sym33_adj(const T G[3][3], T* vb) {
  vb[0] = G[0][0]; vb[1] = G[1][1]; vb[2] = G[2][2];
  vb[3] = G[1][2] + G[2][1];
  vb[4] = G[0][2] + G[2][0];
  vb[5] = G[0][1] + G[1][0];
}
// tensor adjoint of a 6-component output taken from a symmetric tensor (one entry each)
template <typename T>
__device__ __forceinline__ void out6_adj(const T* ob, T G[3][3]) {
  G[0][0] = ob[0]; G[1][1] = ob[1]; G[2][2] = ob[2];
  G[1][2] = G[2][1] = T(0.5) * ob[3];
  G[0][2] = G[2][0] = T(0.5) * ob[4];
  G[0][1] = G[1][0] = T(0.5) * ob[5];
}

// C = A B (3x3).
template <typename T>
__device__ __forceinline__ void mul33(const T A[3][3], const T B[3][3], T C[3][3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[i][j] = A[i][0] * B[0][j] + A[i][1] * B[1][j] + A[i][2] * B[2][j];
}
template <typename T>
__device__ __forceinline__ void rows33(const T* R, T A[3][3], bool transpose) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) A[i][j] = transpose ? R[j * 3 + i] : R[i * 3 + j];
}

// out = R^T E R (to_crystal): given out_b, adds E_b (6) and, with `full`, R_b (9).
// With A = R G: E_b = A R^T, R_b = 2 E A.
template <typename T>
__device__ __forceinline__ void to_crystal_vjp(const T* R, const T* e, const T* ob, T* eb, T* Rb, bool full) {
  T G[3][3], Q[3][3], A[3][3], Eb[3][3], eb6[6];
  out6_adj<T>(ob, G);
  rows33<T>(R, Q, false);
  mul33<T>(Q, G, A);
  rows33<T>(R, Q, true);
  mul33<T>(A, Q, Eb);
  sym33_adj<T>(Eb, eb6);
#pragma unroll
  for (int c = 0; c < 6; ++c) eb[c] += eb6[c];
  if (!full) return;
  T E[3][3], X[3][3];
  sym33<T>(e, E);
  mul33<T>(E, A, X);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) Rb[i * 3 + j] += T(2) * X[i][j];
}

// out = R S R^T (to_sample): given out_b, adds S_b (6) and, with `full`, R_b (9).
// With A = G R: S_b = R^T A, R_b = 2 A S.
template <typename T>
__device__ __forceinline__ void to_sample_vjp(const T* R, const T* s, const T* ob, T* sb, T* Rb, bool full) {
  T G[3][3], Q[3][3], A[3][3], Sb[3][3], sb6[6];
  out6_adj<T>(ob, G);
  rows33<T>(R, Q, false);
  mul33<T>(G, Q, A);
  rows33<T>(R, Q, true);
  mul33<T>(Q, A, Sb);
  sym33_adj<T>(Sb, sb6);
#pragma unroll
  for (int c = 0; c < 6; ++c) sb[c] += sb6[c];
  if (!full) return;
  T S[3][3], X[3][3];
  sym33<T>(s, S);
  mul33<T>(A, S, X);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) Rb[i * 3 + j] += T(2) * X[i][j];
}

// Per-voxel inputs of the reverse kernels: rotation, strains (sample frame), strain at t_{n+1}
// in the crystal frame, plastic strain at t_{n+1}, and the records of one block of at most NS
// substeps: the slips at the start of each substep and the record of each stage.
template <typename T, int NS>
struct VjpVoxel {
  T r[9], en[6], e[6], e1[6], epN[6];
  T vs[NS][16];
  VjpStage<T> st[4 * NS];
  bool quiet;
};

// Substeps m0 .. m1 - 1 of mc_voxel from the state y (classical RK4, weights 1 2 2 1, stage inputs
// y + h/2 k1, y + h/2 k2, y + h k3), which leave the records that the reverse sweeps need.
template <typename T, int NP, int NS>
__device__ __forceinline__ void mc_forward_store(const MatDev<T>& M, const T* e0, const T* de, T dt, int nsub, int m0,
                                                 int m1, const T* tab, MPState<T>& y, VjpVoxel<T, NS>& P) {
  const T h = dt / T(nsub);
  const T inv = T(1) / T(nsub);
#pragma unroll 1
  for (int m = m0; m < m1; ++m) {
    MPState<T> k, Y = y, acc;
    state_zero<T>(acc);
#pragma unroll
    for (int q = 0; q < 16; ++q) P.vs[m - m0][q] = y.v[q];
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
      const T s = j == 0 ? T(m) * inv : (j == 3 ? (T(m) + T(1)) * inv : (T(m) + T(0.5)) * inv);
      vjp_stage<T, NP>(M, e0, de, s, Y, tab, P.st[4 * (m - m0) + j], k);
      state_axpy<T>(acc, j == 0 || j == 3 ? T(1) : T(2), k);
      if (j < 3) {
        Y = y;
        state_axpy<T>(Y, j == 2 ? h : T(0.5) * h, k);
      }
    }
    state_axpy<T>(y, h / T(6), acc);
  }
}

// A reverse sweep of mc_voxel over the records of its forward pass: the state adjoint yb (at
// t_{n+1}, at the end of the sweep at t_n) and the adjoints of the strain path (crystal frame:
// e0, its step and e1).
template <typename T>
struct VjpSeed {
  MPState<T> yb;
  T e0b[6], deb[6], e1b[6];
};

// Start of a sweep: the stress sigma = R sc R^T, sc = C (e1 - ep_N), with adjoint sigma_b.
template <typename T, int NS>
__device__ __forceinline__ void reverse_stress(const MatDev<T>& M, const VjpVoxel<T, NS>& P, const T* sigma_b,
                                               VjpSeed<T>& S, T* Rb, bool full) {
  T ee[6], sc[6], scb[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
#pragma unroll
  for (int c = 0; c < 6; ++c) ee[c] = P.e1[c] - P.epN[c];
  hooke<T>(M, ee, sc);
  to_sample_vjp<T>(P.r, sc, sigma_b, scb, Rb, full);
  hooke<T>(M, scb, S.e1b);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    S.yb.ep[c] -= S.e1b[c];
    S.e0b[c] = T(0);
    S.deb[c] = T(0);
  }
}

// The substeps m0 .. m1 - 1, whose records are in P; with `full` also pb (kParamBar, added).
template <typename T, int NS>
__device__ __forceinline__ void reverse_substeps(const MatDev<T>& M, const VjpVoxel<T, NS>& P, T dt, int nsub, int m0,
                                                 int m1, VjpSeed<T>& S, T* pb, bool full) {
  const T h = dt / T(nsub);
  const T inv = T(1) / T(nsub);
#pragma unroll 1
  for (int m = m1 - 1; m >= m0; --m) {
    // k4 feeds y' alone, k3 also Y4 = y + h k3, k2 Y3 = y + h/2 k2, k1 Y2 = y + h/2 k1
    const MPState<T> yend = S.yb;
    MPState<T> Yb;
    state_zero<T>(Yb);
    const VjpStage<T>* st = &P.st[4 * (m - m0)];
#pragma unroll 1
    for (int j = 3; j >= 0; --j) {
      const T s = j == 0 ? T(m) * inv : (j == 3 ? (T(m) + T(1)) * inv : (T(m) + T(0.5)) * inv);
      const T cw = j == 0 || j == 3 ? h / T(6) : h / T(3);
      const T cY = j == 3 ? T(0) : (j == 2 ? h : T(0.5) * h);
      const T cv = j == 0 ? T(0) : (j == 3 ? h : T(0.5) * h);
      vjp_stage_reverse<T>(M, st[j], s, yend, cw, cY, Yb, S.yb, S.e0b, S.deb, pb, full, P.vs[m - m0], cv,
                           st[j > 0 ? j - 1 : 0].rho);
    }
  }
}

// End of a sweep: de = e1 - e0; e0 = R^T eps_n R; e1 = R^T eps R.  Adds to epsb and, with `full`,
// to eps_nb and Rb.
template <typename T, int NS>
__device__ __forceinline__ void reverse_strains(const VjpVoxel<T, NS>& P, VjpSeed<T>& S, T* eps_nb, T* epsb, T* Rb,
                                                bool full) {
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    S.e1b[c] += S.deb[c];
    S.e0b[c] -= S.deb[c];
  }
  if (full) to_crystal_vjp<T>(P.r, P.en, S.e0b, eps_nb, Rb, true);
  to_crystal_vjp<T>(P.r, P.e, S.e1b, epsb, Rb, full);
}

template <typename T>
__device__ __forceinline__ void load_state34(const T* __restrict__ src, long long i, size_t n, MPState<T>& y) {
#pragma unroll
  for (int c = 0; c < 6; ++c) y.ep[c] = src[c * n + i];
#pragma unroll
  for (int c = 0; c < 16; ++c) y.v[c] = src[(6 + c) * n + i];
#pragma unroll
  for (int c = 0; c < 12; ++c) y.al[c] = src[(22 + c) * n + i];
}
template <typename T>
__device__ __forceinline__ void store_state34(T* __restrict__ dst, long long i, size_t n, const MPState<T>& y) {
#pragma unroll
  for (int c = 0; c < 6; ++c) dst[c * n + i] = y.ep[c];
#pragma unroll
  for (int c = 0; c < 16; ++c) dst[(6 + c) * n + i] = y.v[c];
#pragma unroll
  for (int c = 0; c < 12; ++c) dst[(22 + c) * n + i] = y.al[c];
}

// Loads a voxel: its state at t_n into y, its strain path in the crystal frame into e0 (at t_n)
// and de (its step).
template <typename T, int NS>
__device__ __forceinline__ void vjp_load(const MatDev<T>& M, long long i, size_t n, const T* __restrict__ R,
                                         const T* __restrict__ eps_n, const T* __restrict__ eps,
                                         const T* __restrict__ state, T* e0, T* de, MPState<T>& y, VjpVoxel<T, NS>& P) {
#pragma unroll
  for (int k = 0; k < 9; ++k) P.r[k] = R[(size_t)i * 9 + k];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    P.en[c] = eps_n[c * n + i];
    P.e[c] = eps[c * n + i];
  }
  load_state34<T>(state, i, n, y);
  to_crystal<T>(P.r, P.en, e0);
  to_crystal<T>(P.r, P.e, P.e1);
#pragma unroll
  for (int c = 0; c < 6; ++c) de[c] = P.e1[c] - e0[c];
  P.quiet = elastic_increment<T>(M, e0, de, y);
}

// The sweeps of SEEDS seeds of a voxel.  seed(k, S, sigma_b) fills seed k's state and stress
// adjoint; take(k, S, ...) receives its results; `full` belongs to the last seed.
// NB = 1: one forward pass leaves the records of all substeps, then each seed is swept in turn.
// NB > 1: the records of one block at a time.  The forward pass runs block after block and keeps
// the state at each block's start; the last block's records are there at its end, those of the
// one before are made again on the way back, and all seeds pass a block before the next.
// CUDA reserves a kernel's local memory for every thread the chip can hold: records of all 16
// substeps, 39.9 KB a thread in double, made the context grow by 12.4 GB in a call with more than
// 4 substeps.  Two blocks of 8 take 24.0 KB (7.5 GB), one of 8 20.4 KB, and kernels
// without records took 24.4 KB.  What the second making of records costs: 20011 points in double
// with 16 substeps 7.0 -> 10.0 ms, 100003 in float 2.4 -> 3.5 ms; up to 8 substeps nothing.
template <typename T, int NP, int NS, int NB, int SEEDS, typename Seed, typename Take>
__device__ __forceinline__ void vjp_sweeps(const MatDev<T>& M, const T* e0, const T* de, T dt, int nsub,
                                           const T* tab, MPState<T>& y, VjpVoxel<T, NS>& P, Seed seed, Take take) {
  T pb[kParamBar], rb[9] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
#pragma unroll
  for (int k = 0; k < kParamBar; ++k) pb[k] = T(0);
  auto finish = [&](int k, VjpSeed<T>& S) {
    T enb[6] = {T(0), T(0), T(0), T(0), T(0), T(0)}, eb[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
    reverse_strains<T, NS>(P, S, enb, eb, rb, k == SEEDS - 1);
    take(k, S.yb, eb, enb, rb, pb);
  };
  if constexpr (NB == 1) {
    if (!P.quiet) mc_forward_store<T, NP, NS>(M, e0, de, dt, nsub, 0, nsub, tab, y, P);
#pragma unroll
    for (int c = 0; c < 6; ++c) P.epN[c] = y.ep[c];
#pragma unroll 1
    for (int k = 0; k < SEEDS; ++k) {
      VjpSeed<T> S;
      T sb[6];
      seed(k, S.yb, sb);
      reverse_stress<T, NS>(M, P, sb, S, rb, k == SEEDS - 1);
      if (!P.quiet) reverse_substeps<T, NS>(M, P, dt, nsub, 0, nsub, S, pb, k == SEEDS - 1);
      finish(k, S);
    }
  } else {
    VjpSeed<T> S[SEEDS];
    MPState<T> start[NB];  // the state at each block's start
    // the first block takes the remainder: its records are made twice
    const int nb = P.quiet ? 1 : (nsub + NS - 1) / NS, n0 = nsub - (nb - 1) * NS;
    // blocks 0 .. nb-1 forward, then nb-2 .. 0 again, each followed by its reverse
#pragma unroll 1
    for (int t = 0; t < 2 * nb - 1; ++t) {
      const int b = t < nb ? t : 2 * nb - 2 - t, m1 = n0 + b * NS, m0 = b > 0 ? m1 - NS : 0;
      if (!P.quiet) {
        if (t < nb) start[b] = y;
        else y = start[b];
        mc_forward_store<T, NP, NS>(M, e0, de, dt, nsub, m0, m1, tab, y, P);
      }
      if (t + 1 < nb) continue;
      if (t + 1 == nb) {
#pragma unroll
        for (int c = 0; c < 6; ++c) P.epN[c] = y.ep[c];
      }
#pragma unroll 1
      for (int k = 0; k < SEEDS; ++k) {
        if (t + 1 == nb) {
          T sb[6];
          seed(k, S[k].yb, sb);
          reverse_stress<T, NS>(M, P, sb, S[k], rb, k == SEEDS - 1);
        }
        if (!P.quiet) reverse_substeps<T, NS>(M, P, dt, nsub, m0, m1, S[k], pb, k == SEEDS - 1);
      }
    }
#pragma unroll 1
    for (int k = 0; k < SEEDS; ++k) finish(k, S[k]);
  }
}

// One thread per voxel; arrays component-major (component * nvox + voxel) as in the
// forward material-point kernel.  state_b: in, adjoint of the state at t_{n+1}; out, adjoint
// of the state at t_n.  R_b (9 x nvox) and param_b (kParamBar x nvox) are per voxel.
template <typename T, int NP, int NS, int NB>
__global__ void k_material_point_vjp(const MatDev<T> M, long long nvox, const T* __restrict__ R,
                                     const T* __restrict__ eps_n, const T* __restrict__ eps,
                                     const T* __restrict__ state, T dt, int nsub, const T* __restrict__ sigma_b,
                                     T* state_b, T* eps_b, T* eps_n_b, T* R_b, T* param_b,
                                     const T* __restrict__ root_tab) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tab = reinterpret_cast<T*>(smem_raw);
  stage_tables<T>(tab, root_tab, table_len<T, NP>(M));
  stage_wait();
  __syncthreads();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nvox) return;
  const size_t n = (size_t)nvox;
  VjpVoxel<T, NS> P;
  MPState<T> y;
  T e0[6], de[6];
  vjp_load<T, NS>(M, i, n, R, eps_n, eps, state, e0, de, y, P);
  vjp_sweeps<T, NP, NS, NB, 1>(
      M, e0, de, dt, nsub, tab, y, P,
      [&](int, MPState<T>& yb, T* sb) {
#pragma unroll
        for (int c = 0; c < 6; ++c) sb[c] = sigma_b[c * n + i];
        load_state34<T>(state_b, i, n, yb);
      },
      [&](int, const MPState<T>& yb, const T* eb, const T* enb, const T* rb, const T* pb) {
        store_state34<T>(state_b, i, n, yb);
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          eps_b[c * n + i] = eb[c];
          eps_n_b[c * n + i] = enb[c];
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) R_b[k * n + i] = rb[k];
#pragma unroll
        for (int k = 0; k < kParamBar; ++k) param_b[k * n + i] = pb[k];
      });
}

// The reverse work of one increment of the history adjoint before its fixed point, over one
// stored forward pass per voxel: the six rows J(k, .) = d sigma_k / d eps of the algorithmic
// tangent (unit stress adjoints, no state adjoint; written to J at (k * 6 + c) * nvox + voxel)
// and the direct part (uniform stress adjoint sd, state adjoint state_b at t_{n+1}, which is
// overwritten with the adjoint at t_n), whose eps, eps_n, rotation and parameter adjoints go
// to eps_b, eps_n_b, R_b and param_b.
template <typename T, int NP, int NS, int NB>
__global__ void k_adj_tangent(const MatDev<T> M, long long nvox, const T* __restrict__ R,
                              const T* __restrict__ eps_n, const T* __restrict__ eps,
                              const T* __restrict__ state, T dt, int nsub, T sd0, T sd1, T sd2, T sd3, T sd4, T sd5,
                              T* state_b, T* J, T* eps_b, T* eps_n_b, T* R_b, T* param_b,
                              const T* __restrict__ root_tab) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tab = reinterpret_cast<T*>(smem_raw);
  stage_tables<T>(tab, root_tab, table_len<T, NP>(M));
  stage_wait();
  __syncthreads();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nvox) return;
  const size_t n = (size_t)nvox;
  VjpVoxel<T, NS> P;
  MPState<T> y;
  T e0[6], de[6];
  vjp_load<T, NS>(M, i, n, R, eps_n, eps, state, e0, de, y, P);
  vjp_sweeps<T, NP, NS, NB, 7>(
      M, e0, de, dt, nsub, tab, y, P,
      [&](int row, MPState<T>& yb, T* sb) {
        if (row < 6) {
#pragma unroll
          for (int c = 0; c < 6; ++c) sb[c] = c == row ? T(1) : T(0);
          state_zero<T>(yb);
        } else {
          sb[0] = sd0; sb[1] = sd1; sb[2] = sd2; sb[3] = sd3; sb[4] = sd4; sb[5] = sd5;
          load_state34<T>(state_b, i, n, yb);
        }
      },
      [&](int row, const MPState<T>& yb, const T* eb, const T* enb, const T* rb, const T* pb) {
        if (row < 6) {
#pragma unroll
          for (int c = 0; c < 6; ++c) J[((size_t)row * 6 + c) * n + i] = eb[c];
          return;
        }
        store_state34<T>(state_b, i, n, yb);
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          eps_b[c * n + i] = eb[c];
          eps_n_b[c * n + i] = enb[c];
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) R_b[k * n + i] = rb[k];
#pragma unroll
        for (int k = 0; k < kParamBar; ++k) param_b[k * n + i] = pb[k];
      });
}

}  // namespace rve
