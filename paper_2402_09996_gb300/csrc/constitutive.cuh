// Per-voxel Meric-Cailletaud crystal plasticity (arXiv 2402.09996, Sec. 3 and 4).
//
// State (crystal frame): plastic strain eps_p (6 tensor components, order 11 22 33 23
// 13 12), accumulated slip v (12 slip systems then 4 twin systems; the twin volume
// fraction is f = sqrt(2) v), kinematic variables alpha of the 12 slip systems.
//
// Rates at strain eps (Sec. 3):
//   sigma   = C : (eps - eps_p)                                 (tetragonal C, c || z)
//   tau     = sigma : m,  m = (n x l + l x n)/2                 (Table 1 systems)
//   r       = r0 + Q sum_s' q_ss' (1 - exp(-b v_s'))            (q = h_diag / h_off)
//   slip:   a = |tau - c alpha| - r,  gdot = sign(tau - c alpha) rho,
//           rho = < (a - eta rho) / K >^n                       (Sec. 4, Eq. (regu))
//           alpha_dot = gdot - d |gdot| alpha
//   twin:   rho = (Kc/sqrt2) <fm - sum f> < (tau - r - eta rho) / Kt >^nt, gdot = rho
//   eps_p_dot = (1 - sum f) sum_s gdot_s m_s + sum_b gdot_b m_b,  v_dot = |gdot|.
// Integration: n_sub classical RK4 steps along the linear strain path of the
// increment (Sec. 3, "explicit ... Runge-Kutta 4th order").
//
// Template parameter NP selects how the regularised rates are solved:
//   NP = kDirect  eta > 0 and both laws tabulated directly (rate_table.cuh): no solve;
//   NP = -1       eta > 0, any real n, nt >= 1 (powers as 2^(p log2 z)): table start,
//                 branch-free;
//   NP = 0        eta = 0, and arguments outside the direct tables: generic per-system solve.
#pragma once

#include <type_traits>

#include "rate_table.cuh"
#include "rve_common.cuh"

namespace rve {

// Table 1 (system 9 read as (1 -1 1)[1 1 0]); crystal frame with c/a = 1.
__host__ __device__ __forceinline__ constexpr int sys_n(int s, int c) {
  constexpr int t[16][3] = {{1, 1, -1}, {1, 1, -1}, {1, 1, -1}, {-1, 1, 1}, {-1, 1, 1}, {-1, 1, 1},
                            {1, -1, 1}, {1, -1, 1}, {1, -1, 1}, {1, 1, 1},  {1, 1, 1},  {1, 1, 1},
                            {1, 1, -1}, {-1, 1, 1}, {1, -1, 1}, {1, 1, 1}};
  return t[s][c];
}
__host__ __device__ __forceinline__ constexpr int sys_l(int s, int c) {
  constexpr int t[16][3] = {{0, 1, 1},  {1, 0, 1},  {1, -1, 0},  {0, -1, 1}, {-1, 0, -1}, {-1, -1, 0},
                            {0, 1, 1},  {1, 0, -1}, {1, 1, 0},   {0, 1, -1}, {1, 0, -1},  {1, -1, 0},
                            {1, 1, 2},  {-1, 1, -2}, {1, -1, -2}, {1, 1, -2}};
  return t[s][c];
}

// 1 / (|n| |l|): sqrt(3) sqrt(2) for slip, sqrt(3) sqrt(6) for twins.
template <typename T>
__device__ __forceinline__ T sys_scale(int s) {
  return s < 12 ? T(0.40824829046386301637) : T(0.23570226039551584147);
}

template <typename T>
struct MPState {
  T ep[6];
  T v[16];
  T al[12];
};

template <typename T>
__device__ __forceinline__ void hooke(const MatDev<T>& M, const T* e, T* s) {
  s[0] = M.C11 * e[0] + M.C12 * e[1] + M.C13 * e[2];
  s[1] = M.C12 * e[0] + M.C11 * e[1] + M.C13 * e[2];
  s[2] = M.C13 * (e[0] + e[1]) + M.C33 * e[2];
  s[3] = T(2) * M.C44 * e[3];
  s[4] = T(2) * M.C44 * e[4];
  s[5] = T(2) * M.C66 * e[5];
}

// Integer Schmid coefficients of system s on the six components (11, 22, 33, 23, 13, 12):
// n . x . l = sum_c schmid_k(s, c) x_c for a symmetric x, with schmid_k = n_i l_i on the
// diagonal and n_i l_j + n_j l_i on the shear components.
__host__ __device__ __forceinline__ constexpr int schmid_k(int s, int c) {
  return c == 0   ? sys_n(s, 0) * sys_l(s, 0)
         : c == 1 ? sys_n(s, 1) * sys_l(s, 1)
         : c == 2 ? sys_n(s, 2) * sys_l(s, 2)
         : c == 3 ? sys_n(s, 1) * sys_l(s, 2) + sys_n(s, 2) * sys_l(s, 1)
         : c == 4 ? sys_n(s, 0) * sys_l(s, 2) + sys_n(s, 2) * sys_l(s, 0)
                  : sys_n(s, 0) * sys_l(s, 1) + sys_n(s, 1) * sys_l(s, 0);
}

// sum_c schmid_k(s, c) x_c.  With s a constant (unrolled loops) the zero coefficients
// drop out and unit ones become additions (a product with 0.0 would not fold under IEEE
// rules).
template <typename T>
__device__ __forceinline__ T schmid_sum(int s, const T* x) {
  T r = T(0);
  bool any = false;
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const int k = schmid_k(s, c);
    if (k != 0) {
      const T term = k == 1 ? x[c] : (k == -1 ? -x[c] : T(k) * x[c]);
      r = any ? r + term : term;
      any = true;
    }
  }
  return r;
}

// tau = sigma : m_s = (n . sigma . l) / (|n||l|)
template <typename T>
__device__ __forceinline__ T resolved(int s, const T* g) {
  return sys_scale<T>(s) * schmid_sum<T>(s, g);
}

// Schmid algebra by slip plane.  Every system of Table 1 has a {111} normal n with
// components +-1; systems 3p, 3p+1, 3p+2 and the twin 12+p share plane p.  For such an n and
// any l with n . l = 0 the shear coefficients of schmid_k are the diagonal ones times a sign
// of the plane: n2 l3 + n3 l2 = -n2 n3 (n1 l1), n1 l3 + n3 l1 = -n1 n3 (n2 l2),
// n1 l2 + n2 l1 = -n1 n2 (n3 l3) (from n . l = 0 and n_i^2 = 1).  Hence
//   sum_c schmid_k(s, c) x_c = sum_i (n_i l_i) S_i,  S_i = x_i + sig_i x_(i+3)  (plane sums),
// and sum_s g_s schmid_k(s, c) puts D_i = sum_s (n_i l_i) g_s on component i and sig_i D_i
// on component i + 3.  A slip system has one zero n_i l_i, so its resolved stress is one
// addition of plane sums and a plane's three systems add 3 + 6 terms to a rate sum
// instead of 12; the twins all have n_i l_i = (1, 1, -2).
__host__ __device__ __forceinline__ constexpr int diag_k(int s, int i) { return sys_n(s, i) * sys_l(s, i); }
__host__ __device__ __forceinline__ constexpr int plane_sig(int p, int i) {
  return -sys_n(3 * p, (i + 1) % 3) * sys_n(3 * p, (i + 2) % 3);
}
// s is the first slip system of its plane with a non-zero n_i l_i
__host__ __device__ __forceinline__ constexpr bool first_in_plane(int s, int i) {
  return diag_k(s, i) != 0 && (s % 3 == 0 || (diag_k(s - 1, i) == 0 && (s % 3 == 1 || diag_k(s - 2, i) == 0)));
}
__host__ __device__ constexpr bool schmid_by_plane_holds() {
  for (int s = 0; s < 16; ++s) {
    const int p = s < 12 ? s / 3 : s - 12;
    for (int i = 0; i < 3; ++i)
      if (schmid_k(s, i + 3) != plane_sig(p, i) * diag_k(s, i) || sys_n(s, i) != sys_n(3 * p, i)) return false;
  }
  for (int t = 12; t < 16; ++t)
    if (diag_k(t, 0) != 1 || diag_k(t, 1) != 1 || diag_k(t, 2) != -2) return false;
  return true;
}
static_assert(schmid_by_plane_holds(), "Table 1 systems: plane factorisation of the Schmid sums");

// sum_i diag_k(s, i) S_i (zero coefficients drop out, unit ones are additions)
template <typename T>
__device__ __forceinline__ T plane_sum(int s, const T* S) {
  T r = T(0);
  bool any = false;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int k = diag_k(s, i);
    if (k != 0) {
      const T term = k == 1 ? S[i] : (k == -1 ? -S[i] : T(k) * S[i]);
      r = any ? r + term : term;
      any = true;
    }
  }
  return r;
}

// Adds the rate g of slip system s to its plane's sums D; after the plane's last system
// adds D to du (the first plane assigns).
template <typename T>
__device__ __forceinline__ void plane_add(int s, T g, T* D, T* du) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int k = diag_k(s, i);
    if (k != 0) {
      const T term = k == 1 ? g : (k == -1 ? -g : T(k) * g);
      if (first_in_plane(s, i)) D[i] = term;
      else D[i] = D[i] + term;
    }
  }
  if (s % 3 == 2) {
    const int p = s / 3;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const T hi = plane_sig(p, i) > 0 ? D[i] : -D[i];
      if (p == 0) {
        du[i] = D[i];
        du[i + 3] = hi;
      } else {
        du[i] = du[i] + D[i];
        du[i + 3] = du[i + 3] + hi;
      }
    }
  }
}

// ---------------------------------------------------------------- powers -------------
// z^n for a small positive integer known at run time (loop).
template <typename T>
__device__ __forceinline__ T ipow(T z, int n) {
  T r = T(1), b = z;
  while (n) {
    if (n & 1) r *= b;
    b *= b;
    n >>= 1;
  }
  return r;
}

template <typename T>
__device__ __forceinline__ T powT(T z, T n, int n_int) {
  return n_int > 0 ? ipow<T>(z, n_int) : pow(z, n);
}

template <typename T> __device__ __forceinline__ T fast_log2(T x);
template <> __device__ __forceinline__ float fast_log2<float>(float x) { return __log2f(x); }
template <> __device__ __forceinline__ double fast_log2<double>(double x) { return log2(x); }
template <typename T> __device__ __forceinline__ T fast_exp2(T x);
// Float: the hardware approximation (relative error below 2^-22, subnormal results
// flushed to zero), used for Newton starting values and the hardening terms
// exp(-b v) = 2^(-b v log2 e) in (0, 1].
template <> __device__ __forceinline__ float fast_exp2<float>(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
template <> __device__ __forceinline__ double fast_exp2<double>(double x) { return exp2(x); }
// e^x for the hardening terms (x = -b v in [-b v_max, 0]): the float intrinsic is within
// a few ulp there.
template <typename T> __device__ __forceinline__ T fast_exp(T x);
template <> __device__ __forceinline__ float fast_exp<float>(float x) { return __expf(x); }
template <> __device__ __forceinline__ double fast_exp<double>(double x) { return exp(x); }
// 2^x for the hardening terms: in double from the table kept with the direct rate tables (tab).
template <typename T, int NP>
__device__ __forceinline__ T hard_exp2(const MatDev<T>& M, T x, const T* tab) {
  if constexpr (NP == kDirect && std::is_same<T, double>::value) return exp2_tab(x, tab + (M.rate_len - kExpTab<double>));
  else return fast_exp2<T>(x);
}
template <typename T> __device__ __forceinline__ T fast_div(T a, T b);
template <> __device__ __forceinline__ float fast_div<float>(float a, float b) { return __fdividef(a, b); }
template <> __device__ __forceinline__ double fast_div<double>(double a, double b) { return a / b; }
// 1/x for the last Newton correction, which needs only a few correct digits in float
template <typename T> __device__ __forceinline__ T fast_rcp(T x);
template <> __device__ __forceinline__ float fast_rcp<float>(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
template <> __device__ __forceinline__ double fast_rcp<double>(double x) { return 1.0 / x; }

// ---------------------------------------------------------------- rate roots ---------
// The regularised rate rho >= 0 solves rho = P < (a - eta rho) / Kn >^n  (Sec. 4), and
// rho = 0 when a <= 0 or P <= 0.  With z = (a - eta rho)/Kn the root solves
// phi(z) = c z^n + Kn z - a = 0, c = eta P, and rho = P z^n.  Scaling z = zB u with
// zB = (a/c)^(1/n) leaves u^n + beta u - 1 = 0, beta = Kn zB / a, whose root u*(beta)
// depends on x = log2(beta) alone.  log2 u*(x) is tabulated per exponent as kRootIv
// linear pieces over [-kRootSpan, kRootSpan] (the kink of its asymptotes min(0, -x) sits
// on a node); outside that range the end pieces continue along the asymptotes.  The
// interpolated start is within 3e-5 of the root, so a fixed number of Newton steps
// reaches round-off (1 in float, 3 in double) and the solve has no data-dependent
// branch.  Logarithms are base 2.

template <typename T> struct TabNewton;
template <> struct TabNewton<float> { static constexpr int value = 1; };
template <> struct TabNewton<double> { static constexpr int value = 3; };

// Coefficients of the branch-free solve for one class of systems at one RK stage: the
// slip systems (P = 1), or the twins at the stage's prefactor P.  With la = log2 a:
// log2 zB = a1 la + b1, and the table coordinate of x = log2 beta is
// t = (x + kRootSpan) kRootPerUnit - 1/2 = a2 la + b2.  P <= 0 is solved as P = 1 (finite
// dummy arithmetic) and the rate is scaled by Pout = 0.
template <typename T>
struct RootCoef {
  T Pout, c, cn, Kn, Kn_n, a1, b1, a2, b2, nm1;
};

template <typename T>
__device__ __forceinline__ RootCoef<T> root_coef(T P, T Kn, T n, T inv_n, T lg_Kn, T eta, T lg_eta, T lg_P) {
  RootCoef<T> q;
  const bool pos = P > T(0);
  q.Pout = pos ? P : T(0);
  q.c = eta * (pos ? P : T(1));
  q.cn = n * q.c;
  q.Kn = Kn;
  q.Kn_n = Kn * inv_n;
  q.a1 = inv_n;
  q.b1 = -(lg_eta + (pos ? lg_P : T(0))) * inv_n;
  q.a2 = (inv_n - T(1)) * T(kRootPerUnit);
  q.b2 = (lg_Kn + q.b1 + T(kRootSpan)) * T(kRootPerUnit) - T(0.5);
  q.nm1 = n - T(1);
  return q;
}

// z^(n-1) for the table-started Newton steps (z > 0), 2^((n-1) log2 z) (in float the hardware
// log2 / exp2, whose relative error stays far below the 2e-4 the float path is held to).
template <typename T>
__device__ __forceinline__ T root_zn1(T z, const RootCoef<T>& q) {
  return fast_exp2<T>(q.nm1 * fast_log2<T>(z));
}

// Table interval of the coordinate t: floor(t + 1/2) clamped to [0, kRootIv - 1] (any t,
// NaN included, gives an index inside the table).  In float the rounding happens at the
// 1.5 * 2^23 binade, where the spacing is 1, keeping it off the conversion pipe.
template <typename T> __device__ __forceinline__ int root_interval(T t);
template <> __device__ __forceinline__ int root_interval<float>(float t) {
  const float m = t + 12582912.0f;
  const int i = __float_as_int(m) - 0x4B400000;
  return min(max(i, 0), kRootIv - 1);
}
template <> __device__ __forceinline__ int root_interval<double>(double t) {
  double u = t + 0.5;
  u = u > 0.0 ? u : 0.0;
  u = u < double(kRootIv - 1) ? u : double(kRootIv - 1);
  return (int)u;
}

template <typename T> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };

// Newton steps from z and the rate.  All but the last step are full; the last one is
// folded into the power: with dz = -phi/phi', phi = z (c z^(n-1) + Kn) - a and
// phi' = n (c z^(n-1) + Kn/n), rho = P (z + dz)^n = P z^(n-1) (z + n dz) + O(dz^2);
// |dz/z| < 3e-5 from the table start, so the dropped term n(n-1)/2 (dz/z)^2 < 4e-8 (n = 10)
// is below float round-off (in double two full steps come first).
template <typename T>
__device__ __forceinline__ T root_newton(T z, T aa, const RootCoef<T>& q) {
#pragma unroll
  for (int it = 0; it + 1 < TabNewton<T>::value; ++it) {
    const T zn1 = root_zn1<T>(z, q);
    const T phi = (q.c * zn1) * z + (q.Kn * z - aa);
    z = z - fast_div<T>(phi, q.cn * zn1 + q.Kn);
  }
  const T zn1 = root_zn1<T>(z, q);
  const T phi = z * (q.c * zn1 + q.Kn) - aa;
  const T r = fast_rcp<T>(q.c * zn1 + q.Kn_n);  // = n / phi'
  return q.Pout * (zn1 * (z - phi * r));
}

// Branch-free solve (eta > 0): inactive systems run the same arithmetic
// on a dummy positive argument and return 0, so all systems of a stage form one basic
// block the compiler can interleave.  tab: kRootIv (a_i, b_i) pairs, log2 u* = a_i + b_i t.
template <typename T>
__device__ __forceinline__ T reg_rate_tab(T a, const RootCoef<T>& q, const T* tab) {
  const bool on = a > T(0);
  const T aa = on ? a : T(1);
  const T la = fast_log2<T>(aa);
  const T lzB = la * q.a1 + q.b1;
  const T t = la * q.a2 + q.b2;
  const auto ab = reinterpret_cast<const typename Vec2<T>::type*>(tab)[root_interval<T>(t)];
  const T z = fast_exp2<T>(lzB + (ab.x + ab.y * t));
  const T rho = root_newton<T>(z, aa, q);
  return on ? rho : T(0);
}

// The same for the slip systems, whose coefficients do not depend on the stage (P = 1):
// their table holds log2 z0 = alpha_i + beta_i la directly (alpha_i = b1 + a_i + b_i b2,
// beta_i = a1 + b_i a2, built on the host for the material's K, n and eta).
template <typename T>
__device__ __forceinline__ T reg_rate_slip(T a, const RootCoef<T>& q, const T* tab) {
  const bool on = a > T(0);
  const T aa = on ? a : T(1);
  const T la = fast_log2<T>(aa);
  const T t = la * q.a2 + q.b2;
  const auto ab = reinterpret_cast<const typename Vec2<T>::type*>(tab)[root_interval<T>(t)];
  const T z = fast_exp2<T>(ab.x + ab.y * la);
  const T rho = root_newton<T>(z, aa, q);
  return on ? rho : T(0);
}

// The float solves of two systems of one class at once, on packed two-lane FP32
// arithmetic (one issue slot per pair of FMAs or products).  Each lane performs the
// operations of reg_rate_slip / reg_rate_tab in the same order and rounding; the
// logarithms, exponentials and reciprocals stay per lane.
__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }

__device__ __forceinline__ float2 root_zn1_2(float2 z, const RootCoef<float>& q) {
  const float2 l = __fmul2_rn(f2(q.nm1), make_float2(fast_log2<float>(z.x), fast_log2<float>(z.y)));
  return make_float2(fast_exp2<float>(l.x), fast_exp2<float>(l.y));
}

// UNIT_P: the slip systems' prefactor P = 1 (no final scaling).
template <bool UNIT_P = false>
__device__ __forceinline__ float2 root_newton2(float2 z, float2 aa, const RootCoef<float>& q) {
  const float2 zn1 = root_zn1_2(z, q);
  const float2 phi = __ffma2_rn(z, __ffma2_rn(f2(q.c), zn1, f2(q.Kn)), make_float2(-aa.x, -aa.y));
  const float2 den = __ffma2_rn(f2(q.c), zn1, f2(q.Kn_n));
  const float2 r = make_float2(fast_rcp<float>(den.x), fast_rcp<float>(den.y));
  const float2 w = __ffma2_rn(make_float2(-phi.x, -phi.y), r, z);
  if constexpr (UNIT_P) return __fmul2_rn(zn1, w);
  else return __fmul2_rn(f2(q.Pout), __fmul2_rn(zn1, w));
}

// Inactive systems (a <= 0, or NaN) are solved at a dummy argument and masked.
__device__ __forceinline__ float2 rate_arg2(float2 a) { return make_float2(a.x > 0.f ? a.x : 1.f, a.y > 0.f ? a.y : 1.f); }
__device__ __forceinline__ float2 rate_out2(float2 a, float2 rho) {
  return make_float2(a.x > 0.f ? rho.x : 0.f, a.y > 0.f ? rho.y : 0.f);
}

__device__ __forceinline__ float2 reg_rate_slip2(float2 a, const RootCoef<float>& q, const float* tab) {
  const float2* tb = reinterpret_cast<const float2*>(tab);
  const float2 aa = rate_arg2(a);
  const float2 la = make_float2(fast_log2<float>(aa.x), fast_log2<float>(aa.y));
  const float2 t = __ffma2_rn(la, f2(q.a2), f2(q.b2));
  const float2 ab0 = tb[root_interval<float>(t.x)], ab1 = tb[root_interval<float>(t.y)];
  // one FMA per lane: the two systems' table entries are not an operand pair
  const float2 ex = make_float2(fmaf(ab0.y, la.x, ab0.x), fmaf(ab1.y, la.y, ab1.x));
  const float2 z = make_float2(fast_exp2<float>(ex.x), fast_exp2<float>(ex.y));
  return rate_out2(a, root_newton2<true>(z, aa, q));
}

__device__ __forceinline__ float2 reg_rate_tab2(float2 a, const RootCoef<float>& q, const float* tab) {
  const float2* tb = reinterpret_cast<const float2*>(tab);
  const float2 aa = rate_arg2(a);
  const float2 la = make_float2(fast_log2<float>(aa.x), fast_log2<float>(aa.y));
  const float2 lzB = __ffma2_rn(la, f2(q.a1), f2(q.b1));
  const float2 t = __ffma2_rn(la, f2(q.a2), f2(q.b2));
  const float2 ab0 = tb[root_interval<float>(t.x)], ab1 = tb[root_interval<float>(t.y)];
  const float2 ex = __fadd2_rn(lzB, make_float2(fmaf(ab0.y, t.x, ab0.x), fmaf(ab1.y, t.y, ab1.x)));
  const float2 z = make_float2(fast_exp2<float>(ex.x), fast_exp2<float>(ex.y));
  return rate_out2(a, root_newton2(z, aa, q));
}

// Generic solve (any eta >= 0 and exponent n >= 1): per-system branch, a smooth-minimum
// start u0 = (1 + beta^m)^(-1/m) of the asymptotes (m makes it exact at beta = 1; within
// 5 % for n >= 1.5) and a fixed Newton count (4 in float, 6 in double).
template <typename T> struct NewtonSteps;
template <> struct NewtonSteps<float> { static constexpr int value = 4; };
template <> struct NewtonSteps<double> { static constexpr int value = 6; };

template <typename T>
__device__ __forceinline__ T reg_rate(T a, T P, T Kn, T n, int n_int, T inv_n, T m, T lg_Kn, T eta, T lg_eta,
                                      T lg_P) {
  if (!(a > T(0)) || !(P > T(0))) return T(0);
  if (!(eta > T(0))) return P * powT<T>(a / Kn, n, n_int);
  const T c = eta * P;
  const T la = fast_log2<T>(a);
  const T lzB = (la - lg_eta - lg_P) * inv_n;
  const T lb = lg_Kn + lzB - la;
  const T L = m * lb;
  const T lu = L > T(0) ? -lb - fast_log2<T>(T(1) + fast_exp2<T>(-L)) / m
                        : -fast_log2<T>(T(1) + fast_exp2<T>(L)) / m;
  T z = fast_exp2<T>(lzB + lu);
#pragma unroll
  for (int it = 0; it < NewtonSteps<T>::value; ++it) {
    const T zn1 = n_int > 0 ? ipow<T>(z, n_int - 1) : pow(z, n - T(1));
    const T phi = c * zn1 * z + Kn * z - a;
    z = z - fast_div<T>(phi, n * c * zn1 + Kn);
  }
  z = z > T(0) ? z : T(0);
  return P * powT<T>(z, n, n_int);
}

// ---------------------------------------------------------------- RK4 stage ----------
// The P = 1 root F(a) by the generic solve, out of line: arguments outside a direct table.
template <typename T>
__device__ __noinline__ T rate_generic(T a, T Kn, T n, int n_int, T inv_n, T m, T lg_Kn, T eta, T lg_eta) {
  return reg_rate<T>(a, T(1), Kn, n, n_int, inv_n, m, lg_Kn, eta, lg_eta, T(0));
}
// F(a) of the slip (twin) law for any a: the table inside its range.
template <typename T>
__device__ __forceinline__ T rate_root(const MatDev<T>& M, T a, bool twin, const T* tab) {
  const RateLaw<T>& L = twin ? M.lt : M.ls;
  if constexpr (std::is_same<T, double>::value) {
    if (!(a > 0.0)) return 0.0;
    if (rate_inside(a, L)) return rate_direct(a, L, tab + L.off);
  } else {
    const T r = rate_direct(a, L, tab + L.off);
    if (r == r) return r;
  }
  return twin ? rate_generic<T>(a, M.Kt, M.nt, M.nt_int, M.inv_nt, M.smt, M.lg_Kt, M.eta, M.lg_eta)
              : rate_generic<T>(a, M.K, M.n, M.n_int, M.inv_n, M.sm, M.lg_K, M.eta, M.lg_eta);
}

// The twins' argument scale s = P^(1/(nt-1)) and its inverse for the direct table (both 0 for
// P = 0: the rate is then 0).
template <typename T>
__device__ __forceinline__ void twin_scale(const MatDev<T>& M, T P, T lg_P, T* s, T* inv_s) {
  const T l = lg_P * M.inv_ntm1;
  *s = P > T(0) ? fast_exp2<T>(l) : T(0);
  *inv_s = P > T(0) ? fast_exp2<T>(-l) : T(0);
}

// One regularised-rate solve: the direct table, a table start, or generic.
template <typename T, int NP>
__device__ __forceinline__ T stage_rate(const MatDev<T>& M, const RootCoef<T>& q, T a, T P, bool twin, T lg_P,
                                        const T* tab) {
  if constexpr (NP == kDirect) {
    if (!twin) return rate_root<T>(M, a, false, tab);
    T sc, isc;
    twin_scale<T>(M, P, lg_P, &sc, &isc);
    return rate_root<T>(M, a * sc, true, tab) * isc;
  } else if constexpr (NP != 0) {
    return twin ? reg_rate_tab<T>(a, q, tab + kRootTabLen) : reg_rate_slip<T>(a, q, tab);
  } else {
    return twin ? reg_rate<T>(a, P, M.Kt, M.nt, M.nt_int, M.inv_nt, M.smt, M.lg_Kt, M.eta, M.lg_eta, lg_P)
                : reg_rate<T>(a, P, M.K, M.n, M.n_int, M.inv_n, M.sm, M.lg_K, M.eta, M.lg_eta, lg_P);
  }
}

// Packed two-lane solves: float with a table-started solve.
template <typename T, int NP>
constexpr bool kPackedSolve = std::is_same<T, float>::value && NP < 0;

// Two values of a pair of systems (or components).  Float: one packed two-lane FP32
// instruction per operation; double: the scalar expressions.
template <typename T> struct PairT;
template <> struct PairT<float> { using type = float2; };
template <> struct PairT<double> { using type = double2; };
template <typename T> using pair_t = typename PairT<T>::type;

template <typename T>
__device__ __forceinline__ pair_t<T> pmk(T a, T b) {
  pair_t<T> r;
  r.x = a;
  r.y = b;
  return r;
}
template <typename T>
__device__ __forceinline__ pair_t<T> pfma(pair_t<T> a, pair_t<T> b, pair_t<T> c) {  // a b + c
  if constexpr (std::is_same<T, float>::value) return __ffma2_rn(a, b, c);
  else return pmk<T>(a.x * b.x + c.x, a.y * b.y + c.y);
}
template <typename T>
__device__ __forceinline__ pair_t<T> pmul(pair_t<T> a, pair_t<T> b) {
  if constexpr (std::is_same<T, float>::value) return __fmul2_rn(a, b);
  else return pmk<T>(a.x * b.x, a.y * b.y);
}
template <typename T>
__device__ __forceinline__ pair_t<T> padd(pair_t<T> a, pair_t<T> b) {
  if constexpr (std::is_same<T, float>::value) return __fadd2_rn(a, b);
  else return pmk<T>(a.x + b.x, a.y + b.y);
}

// The strain path (e0, de: 12 floats) of a thread in shared memory: read again at every stage
// instead of being held in registers (volatile, so that the loads stay where they are; they
// are ordered among each other but not against ordinary stores, so the writer (store_path)
// puts a compiler barrier on both sides of its stores).  With
// the rotation and the strain read again after the integration this freed the registers that
// made the 168-register x pass spill inside the stages: 128^3 743 -> 627 us per launch.  The
// substep-start kinematic variables in shared memory as well: 650 us.
__device__ __forceinline__ void load_path(float* v, const float* sc) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(sc) + 48u * threadIdx.x;
#pragma unroll
  for (int i = 0; i < 3; ++i)
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[4 * i]), "=f"(v[4 * i + 1]), "=f"(v[4 * i + 2]), "=f"(v[4 * i + 3])
                 : "r"(a + 16u * i));
}
__device__ __forceinline__ void load_path(double*, const double*) {}
__device__ __forceinline__ void store_path(float* sc, const float* e0, const float* de) {
  float4* d = reinterpret_cast<float4*>(sc) + 3 * threadIdx.x;
  asm volatile("" ::: "memory");  // after the loads of the thread's voxel before
  d[0] = make_float4(e0[0], e0[1], e0[2], e0[3]);
  d[1] = make_float4(e0[4], e0[5], de[0], de[1]);
  d[2] = make_float4(de[2], de[3], de[4], de[5]);
  asm volatile("" ::: "memory");  // before the loads of this one
}

// Evaluates the rates at elastic strain e0 + s*de - yt.ep and state yt, adds
// wacc * rates to acc and overwrites yt with y0 + cnext * rates.  FIRST (the first stage of
// a substep, wacc = 1): the input state is y0 and acc is assigned the rates, so neither the
// copy yt = y0 nor the zeroing of acc is needed.
// tab: the rate-root tables (slip systems' at 0, twin exponent's at kRootTabLen), NP != 0 only.
// The systems go in pairs (k, k + 1): both are resolved, solved and folded into acc / yt
// before the next pair (yt.v and yt.al of a pair are read before they are overwritten;
// the hardening terms use the stage's yt.v, computed first).  In float the pair's
// arithmetic runs on packed two-lane instructions.  With NP != 0 the solves are
// branch-free, so the whole stage is one basic block the compiler interleaves; this order
// keeps fewer values live than solving all 16 systems first.
// Rewritten forms (same quantities): with e_k = exp(-b v_k) = 1 - g_k,
//   r_k = r0_k + Q (h_off sum g + (h_diag - h_off) g_k) = (r0_k + Q (h_off (N - sum e) + dq)) - Q dq e_k;
// the slip systems' Schmid scale 1/sqrt6 is folded into the moduli (MatDev C*s, the stress
// itself is not formed), the resolved stresses and the plastic strain rate go through the
// plane sums (plane_sum, plane_add), and the rate sums are scaled once at the end.
template <typename T, int NP, bool FIRST = false, bool SC = false>
__device__ __forceinline__ void rk_stage(const MatDev<T>& M, const T* e0_, const T* de_, T s,
                                         const MPState<T>& y0, MPState<T>& yt, MPState<T>& acc, T wacc,
                                         T cnext, const T* tab) {
  constexpr double kLog2e = 1.44269504088896340736;
  // the stage's input state: y0 in the first stage (so yt needs no copy of it), yt after
  const MPState<T>& yin = FIRST ? y0 : yt;
  // e = e0 + s de - eps_p and the slip-scaled stress ss = C : e / sqrt6 (MatDev's C*s)
  T e[6], ss[6], path[12];
  if constexpr (SC) load_path(path, e0_);
  const T *e0 = SC ? path : e0_, *de = SC ? path + 6 : de_;
  if constexpr (std::is_same<T, float>::value) {
#pragma unroll
    for (int c = 0; c < 6; c += 2) {
      const pair_t<T> ec = pfma<T>(pmk<T>(s, s), pmk<T>(de[c], de[c + 1]), pmk<T>(e0[c], e0[c + 1]));
      e[c] = ec.x - yin.ep[c];
      e[c + 1] = ec.y - yin.ep[c + 1];
    }
    const pair_t<T> s01 = pfma<T>(pmk<T>(M.C13s, M.C13s), pmk<T>(e[2], e[2]),
                                  pfma<T>(pmk<T>(M.C12s, M.C11s), pmk<T>(e[1], e[1]),
                                          pmul<T>(pmk<T>(M.C11s, M.C12s), pmk<T>(e[0], e[0]))));
    const pair_t<T> s45 = pmul<T>(pmk<T>(M.C44s2, M.C66s2), pmk<T>(e[4], e[5]));
    ss[0] = s01.x;
    ss[1] = s01.y;
    ss[2] = M.C13s * (e[0] + e[1]) + M.C33s * e[2];
    ss[3] = M.C44s2 * e[3];
    ss[4] = s45.x;
    ss[5] = s45.y;
  } else {
#pragma unroll
    for (int c = 0; c < 6; ++c) e[c] = e0[c] + s * de[c] - yin.ep[c];
    ss[0] = M.C11s * e[0] + M.C12s * e[1] + M.C13s * e[2];
    ss[1] = M.C12s * e[0] + M.C11s * e[1] + M.C13s * e[2];
    ss[2] = M.C13s * (e[0] + e[1]) + M.C33s * e[2];
    ss[3] = M.C44s2 * e[3];
    ss[4] = M.C44s2 * e[4];
    ss[5] = M.C66s2 * e[5];
  }
  T ex[16];
  const T cb_s = -M.b_s * T(kLog2e), cb_t = -M.b_b * T(kLog2e);
  // sums of the hardening terms and twin slips, even and odd systems in the two lanes
  pair_t<T> es2 = pmk<T>(T(0), T(0)), et2 = pmk<T>(T(0), T(0)), vt2 = pmk<T>(T(0), T(0));
#pragma unroll
  for (int k = 0; k < 12; k += 2) {
    const pair_t<T> p = pmul<T>(pmk<T>(cb_s, cb_s), pmk<T>(yin.v[k], yin.v[k + 1]));
    ex[k] = fast_exp2<T>(p.x);
    ex[k + 1] = fast_exp2<T>(p.y);
    es2 = padd<T>(es2, pmk<T>(ex[k], ex[k + 1]));
  }
#pragma unroll
  for (int k = 12; k < 16; k += 2) {
    const pair_t<T> p = pmul<T>(pmk<T>(cb_t, cb_t), pmk<T>(yin.v[k], yin.v[k + 1]));
    ex[k] = fast_exp2<T>(p.x);
    ex[k + 1] = fast_exp2<T>(p.y);
    et2 = padd<T>(et2, pmk<T>(ex[k], ex[k + 1]));
    vt2 = padd<T>(vt2, pmk<T>(yin.v[k], yin.v[k + 1]));
  }
  const T Es = es2.x + es2.y, Et = et2.x + et2.y, vtw = vt2.x + vt2.y;
  const T ftot = T(1.41421356237309504880) * vtw;
  const T wslip = T(1) - ftot;
  T fm_left = M.fm - ftot;
  fm_left = fm_left > T(0) ? fm_left : T(0);
  const T Ptw = (M.Kc * T(0.70710678118654752440)) * fm_left;
  const T lg_Ptw = fast_log2<T>(Ptw > T(0) ? Ptw : T(1));
  const T dq = M.h_diag - M.h_off;
  const T Qdq_s = M.Q_s * dq, Qdq_t = M.Q_b * dq;
  const T Rb_s = M.Q_s * (M.h_off * (T(12) - Es) + dq);
  const T Rb_t = M.Q_b * (M.h_off * (T(4) - Et) + dq);
  // initial resistance plus the stage's common hardening term per kind of system (Table 1:
  // systems 3, 6, 9 and 12 ordinary, the other slip systems superdislocations; one value for
  // the twins), as the host fills M.r0
  const T rb_sup = M.r0[0] + Rb_s, rb_ord = M.r0[2] + Rb_s, rb_tw = M.r0[12] + Rb_t;
  RootCoef<T> qs, qt;
  if constexpr (NP != 0 && NP != kDirect) {
    qs = root_coef<T>(T(1), M.K, M.n, M.inv_n, M.lg_K, M.eta, M.lg_eta, T(0));
    qt = root_coef<T>(Ptw, M.Kt, M.nt, M.inv_nt, M.lg_Kt, M.eta, M.lg_eta, lg_Ptw);
  }
  T s_tw = T(0), is_tw = T(0);
  const T *tab_s = tab, *tab_t = tab;
  if constexpr (NP == kDirect) {
    twin_scale<T>(M, Ptw, lg_Ptw, &s_tw, &is_tw);
    tab_s = tab + M.ls.off;
    tab_t = tab + M.lt.off;
  }
  // plane sums of the slip-scaled stress (plane_sum)
  T S[4][3];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int i = 0; i < 3; ++i) S[p][i] = plane_sig(p, i) > 0 ? ss[i] + ss[i + 3] : ss[i] - ss[i + 3];
  T du_s[6], D[3];
  // the systems in pairs: both driving forces, both rates (packed solve in float), then
  // each system folded into acc / yt
#pragma unroll
  for (int k = 0; k < 12; k += 2) {
    const pair_t<T> alk = pmk<T>(yin.al[k], yin.al[k + 1]);
    const pair_t<T> tk = pfma<T>(pmk<T>(-M.c, -M.c), alk,
                                 pmk<T>(plane_sum<T>(k, S[k / 3]), plane_sum<T>(k + 1, S[(k + 1) / 3])));
    const pair_t<T> rr = pfma<T>(pmk<T>(-Qdq_s, -Qdq_s), pmk<T>(ex[k], ex[k + 1]),
                                 pmk<T>(k % 3 == 2 ? rb_ord : rb_sup, (k + 1) % 3 == 2 ? rb_ord : rb_sup));
    const T tek0 = tk.x, tek1 = tk.y;
    const T ak0 = fabs(tek0) - rr.x;
    const T ak1 = fabs(tek1) - rr.y;
    T rk2[2];
    if constexpr (NP == kDirect) {
      rk2[0] = rate_direct(ak0, M.ls, tab_s);
      rk2[1] = rate_direct(ak1, M.ls, tab_s);
    } else if constexpr (kPackedSolve<T, NP>) {
      const float2 r = reg_rate_slip2(make_float2(ak0, ak1), qs, tab);
      rk2[0] = r.x;
      rk2[1] = r.y;
    } else {
      rk2[0] = stage_rate<T, NP>(M, qs, ak0, T(1), false, T(0), tab);
      rk2[1] = stage_rate<T, NP>(M, qs, ak1, T(1), false, T(0), tab);
    }
    const T gd0 = copysign(rk2[0], tek0);  // rk = 0 unless |tek| > r > 0
    const T gd1 = copysign(rk2[1], tek1);
    plane_add<T>(k, gd0, D, du_s);
    plane_add<T>(k + 1, gd1, D, du_s);
    const pair_t<T> rk = pmk<T>(rk2[0], rk2[1]);
    const pair_t<T> drk = pmul<T>(pmk<T>(-M.d, -M.d), rk);
    const pair_t<T> ald = pfma<T>(drk, alk, pmk<T>(gd0, gd1));  // gd - d rk alpha
    const pair_t<T> wa = pmk<T>(wacc, wacc), cn = pmk<T>(cnext, cnext);
    const pair_t<T> av = FIRST ? rk : pfma<T>(wa, rk, pmk<T>(acc.v[k], acc.v[k + 1]));
    const pair_t<T> yv = pfma<T>(cn, rk, pmk<T>(y0.v[k], y0.v[k + 1]));
    const pair_t<T> aa = FIRST ? ald : pfma<T>(wa, ald, pmk<T>(acc.al[k], acc.al[k + 1]));
    const pair_t<T> ya = pfma<T>(cn, ald, pmk<T>(y0.al[k], y0.al[k + 1]));
    acc.v[k] = av.x;
    acc.v[k + 1] = av.y;
    yt.v[k] = yv.x;
    yt.v[k + 1] = yv.y;
    acc.al[k] = aa.x;
    acc.al[k + 1] = aa.y;
    yt.al[k] = ya.x;
    yt.al[k + 1] = ya.y;
  }
  // twins: the twin rates g_t enter the diagonal components as (G, G, -2 G), G = sum g_t,
  // and component i + 3 as H_i = sum_t sig_i(plane of t) g_t (times -2 for i = 2)
  T G = T(0), H[3] = {T(0), T(0), T(0)};
#pragma unroll
  for (int k = 12; k < 16; k += 2) {
    const pair_t<T> rr = pfma<T>(pmk<T>(-Qdq_t, -Qdq_t), pmk<T>(ex[k], ex[k + 1]),
                                 pmk<T>(rb_tw, rb_tw));
    // 1/(|n||l|) of a twin is (1/sqrt3) times the slip systems' scale in ss
    constexpr T kTw = T(0.57735026918962576451);
    const T ak0 = kTw * plane_sum<T>(k, S[k - 12]) - rr.x;
    const T ak1 = kTw * plane_sum<T>(k + 1, S[k - 11]) - rr.y;
    T rk2[2];
    if constexpr (NP == kDirect) {
      rk2[0] = rate_direct(ak0 * s_tw, M.lt, tab_t) * is_tw;
      rk2[1] = rate_direct(ak1 * s_tw, M.lt, tab_t) * is_tw;
    } else if constexpr (kPackedSolve<T, NP>) {
      const float2 r = reg_rate_tab2(make_float2(ak0, ak1), qt, tab + kRootTabLen);
      rk2[0] = r.x;
      rk2[1] = r.y;
    } else {
      rk2[0] = stage_rate<T, NP>(M, qt, ak0, Ptw, true, lg_Ptw, tab);
      rk2[1] = stage_rate<T, NP>(M, qt, ak1, Ptw, true, lg_Ptw, tab);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int p = k - 12 + j;
      const T g = rk2[j];
      G = p == 0 ? g : G + g;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const T hg = plane_sig(p, i) > 0 ? g : -g;
        H[i] = p == 0 ? hg : H[i] + hg;
      }
    }
    const pair_t<T> rk = pmk<T>(rk2[0], rk2[1]);
    const pair_t<T> av = FIRST ? rk : pfma<T>(pmk<T>(wacc, wacc), rk, pmk<T>(acc.v[k], acc.v[k + 1]));
    const pair_t<T> yv = pfma<T>(pmk<T>(cnext, cnext), rk, pmk<T>(y0.v[k], y0.v[k + 1]));
    acc.v[k] = av.x;
    acc.v[k + 1] = av.y;
    yt.v[k] = yv.x;
    yt.v[k + 1] = yv.y;
  }
  // eps_p rate = (1 - sum f) sum_s gdot_s m_s + sum_b gdot_b m_b, m = scale sym(n x l)
  const T fs = wslip * sys_scale<T>(0);
  const T fsh = T(0.5) * fs;
  const T tsc = sys_scale<T>(12), tsh = T(0.5) * sys_scale<T>(12);
  const T du_t[6] = {G, G, T(-2) * G, H[0], H[1], T(-2) * H[2]};
#pragma unroll
  for (int c = 0; c < 6; c += 2) {
    const pair_t<T> dep = pfma<T>(pmk<T>(c < 3 ? fs : fsh, c + 1 < 3 ? fs : fsh), pmk<T>(du_s[c], du_s[c + 1]),
                                  pmul<T>(pmk<T>(c < 3 ? tsc : tsh, c + 1 < 3 ? tsc : tsh),
                                          pmk<T>(du_t[c], du_t[c + 1])));
    const pair_t<T> ae = FIRST ? dep : pfma<T>(pmk<T>(wacc, wacc), dep, pmk<T>(acc.ep[c], acc.ep[c + 1]));
    const pair_t<T> ye = pfma<T>(pmk<T>(cnext, cnext), dep, pmk<T>(y0.ep[c], y0.ep[c + 1]));
    acc.ep[c] = ae.x;
    acc.ep[c + 1] = ae.y;
    yt.ep[c] = ye.x;
    yt.ep[c + 1] = ye.y;
  }
}

// True when no system can be active anywhere on the increment's strain path with the
// state frozen at t_n: |tau - x| - r (slip) and tau - r (twin) are convex in the path
// parameter, so checking both ends suffices; the exact solution is then "no flow".
template <typename T>
__device__ __forceinline__ bool elastic_increment(const MatDev<T>& M, const T* e0, const T* de,
                                                  const MPState<T>& y) {
  T ea[6], eb[6], sa[6], sb[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    ea[c] = e0[c] - y.ep[c];
    eb[c] = e0[c] + de[c] - y.ep[c];
  }
  hooke<T>(M, ea, sa);
  hooke<T>(M, eb, sb);
  T g[16];
  T Sslip = T(0), Stw = T(0), vtw = T(0);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    g[k] = T(1) - fast_exp<T>(-M.b_s * y.v[k]);
    Sslip += g[k];
  }
#pragma unroll
  for (int k = 12; k < 16; ++k) {
    g[k] = T(1) - fast_exp<T>(-M.b_b * y.v[k]);
    Stw += g[k];
    vtw += y.v[k];
  }
  const T dq = M.h_diag - M.h_off;
  bool quiet = true;
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const T x = M.c * y.al[k];
    const T r = M.r0[k] + M.Q_s * (M.h_off * Sslip + dq * g[k]);
    const T a0 = fabs(resolved<T>(k, sa) - x) - r;
    const T a1 = fabs(resolved<T>(k, sb) - x) - r;
    quiet = quiet && !(a0 > T(0)) && !(a1 > T(0));
  }
  const T ftot = T(1.41421356237309504880) * vtw;
  if (M.fm - ftot > T(0)) {
#pragma unroll
    for (int k = 12; k < 16; ++k) {
      const T r = M.r0[k] + M.Q_b * (M.h_off * Stw + dq * g[k]);
      const T a0 = resolved<T>(k, sa) - r;
      const T a1 = resolved<T>(k, sb) - r;
      quiet = quiet && !(a0 > T(0)) && !(a1 > T(0));
    }
  }
  return quiet;
}

// eps_c = R^T eps R for a symmetric tensor in 6-component storage; R row-major.
template <typename T>
__device__ __forceinline__ void to_crystal(const T* R, const T* e, T* out) {
  const T E[3][3] = {{e[0], e[5], e[4]}, {e[5], e[1], e[3]}, {e[4], e[3], e[2]}};
  T A[3][3];  // E R
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) A[i][j] = E[i][0] * R[0 * 3 + j] + E[i][1] * R[1 * 3 + j] + E[i][2] * R[2 * 3 + j];
  // out_ij = sum_k R_ki A_kj
  out[0] = R[0] * A[0][0] + R[3] * A[1][0] + R[6] * A[2][0];
  out[1] = R[1] * A[0][1] + R[4] * A[1][1] + R[7] * A[2][1];
  out[2] = R[2] * A[0][2] + R[5] * A[1][2] + R[8] * A[2][2];
  out[3] = R[1] * A[0][2] + R[4] * A[1][2] + R[7] * A[2][2];
  out[4] = R[0] * A[0][2] + R[3] * A[1][2] + R[6] * A[2][2];
  out[5] = R[0] * A[0][1] + R[3] * A[1][1] + R[6] * A[2][1];
}

// sigma = R sigma_c R^T
template <typename T>
__device__ __forceinline__ void to_sample(const T* R, const T* s, T* out) {
  const T S[3][3] = {{s[0], s[5], s[4]}, {s[5], s[1], s[3]}, {s[4], s[3], s[2]}};
  T B[3][3];  // S R^T : B_ij = sum_k S_ik R_jk
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) B[i][j] = S[i][0] * R[j * 3 + 0] + S[i][1] * R[j * 3 + 1] + S[i][2] * R[j * 3 + 2];
  // out_ij = sum_k R_ik B_kj
  out[0] = R[0] * B[0][0] + R[1] * B[1][0] + R[2] * B[2][0];
  out[1] = R[3] * B[0][1] + R[4] * B[1][1] + R[5] * B[2][1];
  out[2] = R[6] * B[0][2] + R[7] * B[1][2] + R[8] * B[2][2];
  out[3] = R[3] * B[0][2] + R[4] * B[1][2] + R[5] * B[2][2];
  out[4] = R[0] * B[0][2] + R[1] * B[1][2] + R[2] * B[2][2];
  out[5] = R[0] * B[0][1] + R[1] * B[1][1] + R[2] * B[2][1];
}

// The RK4 substeps of an increment in double with the direct rate tables: the stages of
// rk_stage, one system at a time.  GB300's FP64 pipe takes 16 cycles per warp instruction and
// SM, so the update is bound by its count of FP64 instructions, and everything a warp can
// leave out is:
//  - a rate is 10 FP64 instructions (rate_direct) and a hardening exponential 9 (exp2_tab),
//    against about 100 and 18 with three Newton steps and the library's exp2;
//  - a system in which no lane of the warp flows costs its driving force only: its rate is
//    exactly 0, which leaves its slip, kinematic variable and sums as they are;
//  - exponentials and their sums are kept while the slips they belong to do not change
//    (dirty: systems whose slip in yt changed since ex was formed).
// Skips are decided per warp but do not change any lane's values.  48^3, increments at 0.3 %
// strain: x pass 11.7 -> 3.46 ms per launch.
__device__ __forceinline__ void rk4_fp64(const MatDev<double>& M, const double* e0, const double* de,
                                         MPState<double>& y, double dt, int nsub, const double* tab) {
  constexpr double kLog2e = 1.44269504088896340736;
  const unsigned lanes = __activemask();
  const double* tab_e = tab + (M.rate_len - kExpTab<double>);
  const double h = dt / (double)nsub, inv = 1.0 / (double)nsub;
  const double cb_s = -M.b_s * kLog2e, cb_t = -M.b_b * kLog2e;
  const double dq = M.h_diag - M.h_off, Qdq_s = M.Q_s * dq, Qdq_t = M.Q_b * dq;
  MPState<double> yt = y, acc;
  double ex[16];
  double Es = 0.0, Et = 0.0, ftot = 0.0, s_tw = 0.0, is_tw = 0.0;
  bool scaled = false;        // s_tw, is_tw belong to ftot
  unsigned dirty = 0xffffu;   // systems whose yt.v changed since ex was formed
  unsigned moved = 0;         // systems whose yt.v and yt.al differ from y's
#pragma unroll 1
  for (int m = 0; m < nsub; ++m) {
#pragma unroll
    for (int c = 0; c < 6; ++c) acc.ep[c] = 0.0;
#pragma unroll
    for (int c = 0; c < 16; ++c) acc.v[c] = 0.0;
#pragma unroll
    for (int c = 0; c < 12; ++c) acc.al[c] = 0.0;
    unsigned ever = 0;  // systems that flowed in some stage of the substep
#pragma unroll 1
    for (int stg = 0; stg < 4; ++stg) {
      const double s = ((double)m + 0.5 * (double)((stg + 1) >> 1)) * inv;
      const double wacc = stg == 0 || stg == 3 ? 1.0 : 2.0;
      const double cn = stg == 2 ? h : 0.5 * h;
      const bool step = stg < 3;  // the last stage forms no further state
      if (dirty & 0xfffu) {
        double q0 = 0.0, q1 = 0.0;
#pragma unroll
        for (int k = 0; k < 12; k += 2) {
          if (dirty >> k & 1u) ex[k] = exp2_tab(cb_s * yt.v[k], tab_e);
          if (dirty >> (k + 1) & 1u) ex[k + 1] = exp2_tab(cb_s * yt.v[k + 1], tab_e);
          q0 += ex[k];
          q1 += ex[k + 1];
        }
        Es = q0 + q1;
      }
      if (dirty >> 12) {
#pragma unroll
        for (int k = 12; k < 16; ++k)
          if (dirty >> k & 1u) ex[k] = exp2_tab(cb_t * yt.v[k], tab_e);
        Et = (ex[12] + ex[14]) + (ex[13] + ex[15]);
        ftot = 1.41421356237309504880 * ((yt.v[12] + yt.v[14]) + (yt.v[13] + yt.v[15]));
        scaled = false;
      }
      double fm_left = M.fm - ftot;
      fm_left = fm_left > 0.0 ? fm_left : 0.0;
      const double Rb_s = M.Q_s * (M.h_off * (12.0 - Es) + dq), Rb_t = M.Q_b * (M.h_off * (4.0 - Et) + dq);
      const double rb_sup = M.r0[0] + Rb_s, rb_ord = M.r0[2] + Rb_s, rb_tw = M.r0[12] + Rb_t;
      double ss[6];
      {
        double e[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) e[c] = e0[c] + s * de[c] - yt.ep[c];
        ss[0] = M.C11s * e[0] + M.C12s * e[1] + M.C13s * e[2];
        ss[1] = M.C12s * e[0] + M.C11s * e[1] + M.C13s * e[2];
        ss[2] = M.C13s * (e[0] + e[1]) + M.C33s * e[2];
        ss[3] = M.C44s2 * e[3];
        ss[4] = M.C44s2 * e[4];
        ss[5] = M.C66s2 * e[5];
      }
      unsigned act = 0;
      double du[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0}, G = 0.0, H[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        double S[3], D[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int i = 0; i < 3; ++i) S[i] = plane_sig(p, i) > 0 ? ss[i] + ss[i + 3] : ss[i] - ss[i + 3];
#pragma unroll
        for (int k = 3 * p; k < 3 * p + 3; ++k) {
          const double al = yt.al[k];
          const double tk = plane_sum<double>(k, S) - M.c * al;
          const double a = fabs(tk) - ((k % 3 == 2 ? rb_ord : rb_sup) - Qdq_s * ex[k]);
          if (__any_sync(lanes, a > 0.0)) {
            const double rho = rate_root<double>(M, a, false, tab);
            const double gd = copysign(rho, tk);
            act |= 1u << k;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              if (diag_k(k, i) == 1) D[i] += gd;
              else if (diag_k(k, i) == -1) D[i] -= gd;
            }
            const double ald = gd - M.d * rho * al;
            acc.v[k] += wacc * rho;
            acc.al[k] += wacc * ald;
            if (step) {
              yt.v[k] = y.v[k] + cn * rho;
              yt.al[k] = y.al[k] + cn * ald;
            }
          } else if (step && (moved >> k & 1u)) {
            yt.v[k] = y.v[k];
            yt.al[k] = y.al[k];
          }
        }
        if (act >> (3 * p) & 7u) {
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            du[i] += D[i];
            if (plane_sig(p, i) > 0) du[i + 3] += D[i];
            else du[i + 3] -= D[i];
          }
        }
        const int k = 12 + p;
        // 1/(|n||l|) of a twin is (1/sqrt3) times the slip systems' scale in ss
        const double at = 0.57735026918962576451 * plane_sum<double>(k, S) - (rb_tw - Qdq_t * ex[k]);
        if (__any_sync(lanes, at > 0.0 && fm_left > 0.0)) {
          if (!scaled) {
            const double P = (M.Kc * 0.70710678118654752440) * fm_left;
            const double l = log2(P > 0.0 ? P : 1.0) * M.inv_ntm1;
            s_tw = P > 0.0 ? exp2_tab(l, tab_e) : 0.0;
            is_tw = P > 0.0 ? exp2_tab(-l, tab_e) : 0.0;
            scaled = true;
          }
          const double g = rate_root<double>(M, at * s_tw, true, tab) * is_tw;
          act |= 1u << k;
          G += g;
#pragma unroll
          for (int i = 0; i < 3; ++i) H[i] += plane_sig(p, i) > 0 ? g : -g;
          acc.v[k] += wacc * g;
          if (step) yt.v[k] = y.v[k] + cn * g;
        } else if (step && (moved >> k & 1u)) {
          yt.v[k] = y.v[k];
        }
      }
      if (act | moved) {
        // eps_p rate = (1 - sum f) sum_s gdot_s m_s + sum_b gdot_b m_b, m = scale sym(n x l)
        const double fs = (1.0 - ftot) * sys_scale<double>(0), tsc = sys_scale<double>(12);
        const double dt6[6] = {G, G, -2.0 * G, H[0], H[1], -2.0 * H[2]};
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          const double dep = c < 3 ? fs * du[c] + tsc * dt6[c] : 0.5 * fs * du[c] + 0.5 * tsc * dt6[c];
          acc.ep[c] += wacc * dep;
          if (step) yt.ep[c] = y.ep[c] + cn * dep;
        }
      }
      ever |= act;
      dirty = step ? act | moved : 0u;
      if (step) moved = act;
    }
    if (ever) {
      const double w = h / 6.0;
#pragma unroll
      for (int c = 0; c < 6; ++c) yt.ep[c] = y.ep[c] = y.ep[c] + w * acc.ep[c];
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if (ever >> c & 1u) yt.v[c] = y.v[c] = y.v[c] + w * acc.v[c];
#pragma unroll
      for (int c = 0; c < 12; ++c)
        if (ever >> c & 1u) yt.al[c] = y.al[c] = y.al[c] + w * acc.al[c];
    }
    dirty = ever;
    moved = 0;
  }
}

// A voxel's update in double by four neighbouring lanes, one slip plane each (its three slip
// systems and its twin), for grids with fewer warps of voxels than the chip has schedulers: an
// update is one serial chain of FP64 instructions per warp, and the plane split shortens it (the
// plastic strain and the stress are formed in all four lanes).  16^3, increments of 24
// iterations and 8 substeps: 23.9 -> 11.4 ms; x_geometry has the rule.  In plane terms the systems of all planes are alike: with n . l = 0
// and the signs below, n_i l_i = f (0, 1, -1), (1, 0, -1), (1, -1, 0) and (1, 1, -2).
struct QuadState {
  double ep[6], v[4], al[3];
};
struct QuadLane {
  double sig[3];   // plane_sig of the lane's plane
  double f;        // sign of its first system
  unsigned mask;   // the voxel's four lanes
};
__host__ __device__ constexpr bool quad_sig_minus(int p, int i) { return p == 3 || p == (i == 0 ? 1 : (i == 1 ? 2 : 0)); }
__host__ __device__ constexpr bool quad_f_minus(int p) { return p == 1 || p == 2; }
__host__ __device__ constexpr bool quad_planes_hold() {
  for (int p = 0; p < 4; ++p) {
    const int f = quad_f_minus(p) ? -1 : 1;
    const int d[3][3] = {{0, f, -f}, {1, 0, -1}, {1, -1, 0}};
    for (int i = 0; i < 3; ++i) {
      if (plane_sig(p, i) != (quad_sig_minus(p, i) ? -1 : 1)) return false;
      for (int j = 0; j < 3; ++j)
        if (diag_k(3 * p + j, i) != d[j][i]) return false;
    }
  }
  return true;
}
static_assert(quad_planes_hold(), "Table 1 systems: signs of the planes");

__device__ __forceinline__ QuadLane quad_lane() {
  const int p = threadIdx.x & 3;
  QuadLane q;
#pragma unroll
  for (int i = 0; i < 3; ++i) q.sig[i] = quad_sig_minus(p, i) ? -1.0 : 1.0;
  q.f = quad_f_minus(p) ? -1.0 : 1.0;
  q.mask = 0xfu << (threadIdx.x & 28);
  return q;
}
// Sum over the four lanes, the same bits in each.
__device__ __forceinline__ double quad_sum(unsigned mask, double x) {
  x += __shfl_xor_sync(mask, x, 1);
  return x + __shfl_xor_sync(mask, x, 2);
}
// Plane sums of the slip-scaled stress at elastic strain e.
__device__ __forceinline__ void quad_stress(const MatDev<double>& M, const QuadLane& q, const double* e, double* S) {
  S[0] = M.C11s * e[0] + M.C12s * e[1] + M.C13s * e[2] + q.sig[0] * (M.C44s2 * e[3]);
  S[1] = M.C12s * e[0] + M.C11s * e[1] + M.C13s * e[2] + q.sig[1] * (M.C44s2 * e[4]);
  S[2] = M.C13s * (e[0] + e[1]) + M.C33s * e[2] + q.sig[2] * (M.C66s2 * e[5]);
}
// Resolved stress of the plane's slip system j.
__device__ __forceinline__ double quad_resolved(const QuadLane& q, int j, const double* S) {
  return j == 0 ? q.f * (S[1] - S[2]) : (j == 1 ? S[0] - S[2] : S[0] - S[1]);
}
__device__ __forceinline__ double quad_twin(const double* S) {
  return 0.57735026918962576451 * (S[0] + S[1] - 2.0 * S[2]);
}

// elastic_increment for the four lanes of a voxel.
__device__ __forceinline__ bool quad_elastic(const MatDev<double>& M, const QuadLane& q, const double* e0,
                                             const double* de, const QuadState& y, const double* tab) {
  constexpr double kLog2e = 1.44269504088896340736;
  const double* tab_e = tab + (M.rate_len - kExpTab<double>);
  double ea[6], eb[6], Sa[3], Sb[3], ex[4];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    ea[c] = e0[c] - y.ep[c];
    eb[c] = e0[c] + de[c] - y.ep[c];
  }
  quad_stress(M, q, ea, Sa);
  quad_stress(M, q, eb, Sb);
#pragma unroll
  for (int j = 0; j < 4; ++j) ex[j] = exp2_tab((j < 3 ? -M.b_s : -M.b_b) * kLog2e * y.v[j], tab_e);
  const double Es = quad_sum(q.mask, ex[0] + ex[1] + ex[2]), Et = quad_sum(q.mask, ex[3]);
  const double ftot = 1.41421356237309504880 * quad_sum(q.mask, y.v[3]);
  const double dq = M.h_diag - M.h_off;
  const double Rb_s = M.Q_s * (M.h_off * (12.0 - Es) + dq), Rb_t = M.Q_b * (M.h_off * (4.0 - Et) + dq);
  bool quiet = true;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const double x = M.c * y.al[j], r = (j == 2 ? M.r0[2] : M.r0[0]) + Rb_s - M.Q_s * dq * ex[j];
    quiet = quiet && !(fabs(quad_resolved(q, j, Sa) - x) - r > 0.0) && !(fabs(quad_resolved(q, j, Sb) - x) - r > 0.0);
  }
  if (M.fm - ftot > 0.0) {
    const double r = M.r0[12] + Rb_t - M.Q_b * dq * ex[3];
    quiet = quiet && !(quad_twin(Sa) - r > 0.0) && !(quad_twin(Sb) - r > 0.0);
  }
  return __all_sync(q.mask, quiet);
}

// The substeps of rk4_fp64 for the four lanes of a voxel (bit j < 3 of the masks: the lanes' slip
// systems j, bit 3 the twins).  lanes: the lanes of the warp that call it, whole voxels; the
// masks are formed over them, so a voxel's lanes take the same exchanges.
__device__ __forceinline__ void rk4_quad(const MatDev<double>& M, const QuadLane& q, unsigned lanes, const double* e0,
                                         const double* de, QuadState& y, double dt, int nsub, const double* tab) {
  constexpr double kLog2e = 1.44269504088896340736;
  const double* tab_e = tab + (M.rate_len - kExpTab<double>);
  const double h = dt / (double)nsub, inv = 1.0 / (double)nsub;
  const double dq = M.h_diag - M.h_off, Qdq_s = M.Q_s * dq, Qdq_t = M.Q_b * dq;
  QuadState yt = y, acc;
  double ex[4];
  double Es = 0.0, Et = 0.0, ftot = 0.0, s_tw = 0.0, is_tw = 0.0;
  bool scaled = false;
  unsigned dirty = 0xfu, moved = 0;
#pragma unroll 1
  for (int m = 0; m < nsub; ++m) {
#pragma unroll
    for (int c = 0; c < 6; ++c) acc.ep[c] = 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c) acc.v[c] = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) acc.al[c] = 0.0;
    unsigned ever = 0;
#pragma unroll 1
    for (int stg = 0; stg < 4; ++stg) {
      const double s = ((double)m + 0.5 * (double)((stg + 1) >> 1)) * inv;
      const double wacc = stg == 0 || stg == 3 ? 1.0 : 2.0;
      const double cn = stg == 2 ? h : 0.5 * h;
      const bool step = stg < 3;
      if (dirty & 7u) {
#pragma unroll
        for (int j = 0; j < 3; ++j)
          if (dirty >> j & 1u) ex[j] = exp2_tab(-M.b_s * kLog2e * yt.v[j], tab_e);
        Es = quad_sum(q.mask, ex[0] + ex[1] + ex[2]);
      }
      if (dirty & 8u) {
        ex[3] = exp2_tab(-M.b_b * kLog2e * yt.v[3], tab_e);
        Et = quad_sum(q.mask, ex[3]);
        ftot = 1.41421356237309504880 * quad_sum(q.mask, yt.v[3]);
        scaled = false;
      }
      double fm_left = M.fm - ftot;
      fm_left = fm_left > 0.0 ? fm_left : 0.0;
      const double Rb_s = M.Q_s * (M.h_off * (12.0 - Es) + dq), Rb_t = M.Q_b * (M.h_off * (4.0 - Et) + dq);
      double S[3];
      {
        double e[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) e[c] = e0[c] + s * de[c] - yt.ep[c];
        quad_stress(M, q, e, S);
      }
      unsigned act = 0;
      double g[3] = {0.0, 0.0, 0.0}, gt = 0.0;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const double al = yt.al[j];
        const double tk = quad_resolved(q, j, S) - M.c * al;
        const double a = fabs(tk) - ((j == 2 ? M.r0[2] : M.r0[0]) + Rb_s - Qdq_s * ex[j]);
        if (__any_sync(lanes, a > 0.0)) {
          const double rho = rate_root<double>(M, a, false, tab);
          g[j] = copysign(rho, tk);
          act |= 1u << j;
          const double ald = g[j] - M.d * rho * al;
          acc.v[j] += wacc * rho;
          acc.al[j] += wacc * ald;
          if (step) {
            yt.v[j] = y.v[j] + cn * rho;
            yt.al[j] = y.al[j] + cn * ald;
          }
        } else if (step && (moved >> j & 1u)) {
          yt.v[j] = y.v[j];
          yt.al[j] = y.al[j];
        }
      }
      const double at = quad_twin(S) - (M.r0[12] + Rb_t - Qdq_t * ex[3]);
      if (__any_sync(lanes, at > 0.0 && fm_left > 0.0)) {
        if (!scaled) {
          const double P = (M.Kc * 0.70710678118654752440) * fm_left;
          const double l = log2(P > 0.0 ? P : 1.0) * M.inv_ntm1;
          s_tw = P > 0.0 ? exp2_tab(l, tab_e) : 0.0;
          is_tw = P > 0.0 ? exp2_tab(-l, tab_e) : 0.0;
          scaled = true;
        }
        gt = rate_root<double>(M, at * s_tw, true, tab) * is_tw;
        act |= 8u;
        acc.v[3] += wacc * gt;
        if (step) yt.v[3] = y.v[3] + cn * gt;
      } else if (step && (moved & 8u)) {
        yt.v[3] = y.v[3];
      }
      if (act) {
        // the plane's part x of the normal components of the rate; sig x / 2 that of the shears
        const double fs = (1.0 - ftot) * sys_scale<double>(0), tg = sys_scale<double>(12) * gt;
        const double x[3] = {fs * (g[1] + g[2]) + tg, fs * (q.f * g[0] - g[2]) + tg,
                             fs * (-q.f * g[0] - g[1]) - 2.0 * tg};
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const double dn = quad_sum(q.mask, x[i]), ds = 0.5 * quad_sum(q.mask, q.sig[i] * x[i]);
          acc.ep[i] += wacc * dn;
          acc.ep[i + 3] += wacc * ds;
          if (step) {
            yt.ep[i] = y.ep[i] + cn * dn;
            yt.ep[i + 3] = y.ep[i + 3] + cn * ds;
          }
        }
      } else if (step && moved) {
#pragma unroll
        for (int c = 0; c < 6; ++c) yt.ep[c] = y.ep[c];
      }
      ever |= act;
      dirty = step ? act | moved : 0u;
      if (step) moved = act;
    }
    if (ever) {
      const double w = h / 6.0;
#pragma unroll
      for (int c = 0; c < 6; ++c) yt.ep[c] = y.ep[c] = y.ep[c] + w * acc.ep[c];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (ever >> j & 1u) yt.v[j] = y.v[j] = y.v[j] + w * acc.v[j];
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (ever >> j & 1u) yt.al[j] = y.al[j] = y.al[j] + w * acc.al[j];
    }
    dirty = ever;
    moved = 0;
  }
}

// mc_voxel for the four lanes of a voxel (lanes: the lanes of the warp that call it); the stress
// is formed in all of them.
__device__ __forceinline__ void mc_voxel_quad(const MatDev<double>& M, const QuadLane& q, unsigned lanes,
                                              const double* R,
                                              const double* eps_n, const double* eps, QuadState& y, double dt,
                                              int nsub, double* sig, const double* tab) {
  double e0[6], e1[6], de[6];
  to_crystal<double>(R, eps_n, e0);
  to_crystal<double>(R, eps, e1);
#pragma unroll
  for (int c = 0; c < 6; ++c) de[c] = e1[c] - e0[c];
  const bool flows = !quad_elastic(M, q, e0, de, y, tab);
  const unsigned flowing = __ballot_sync(lanes, flows);
  if (flows) rk4_quad(M, q, flowing, e0, de, y, dt, nsub, tab);
  double ee[6], sgc[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) ee[c] = e1[c] - y.ep[c];
  hooke<double>(M, ee, sgc);
  to_sample<double>(R, sgc, sig);
}

// Integrates one voxel over the increment [t_n, t_n + dt] (strain eps_n -> eps, sample
// frame) and returns the sample-frame stress at t_n + dt; y is updated in place.
// check: test first whether the increment is elastic and skip the integration if so.  The
// test is a shortcut only: with every rate exactly 0 (inactive systems return 0 in every
// rate-solve variant) the RK4 substeps leave the state bit for bit unchanged, so results do
// not depend on it.  Returns false when the test ran and found the increment elastic.
template <typename T, int NP, bool SC = false>
__device__ __forceinline__ bool mc_voxel(const MatDev<T>& M, const T* R, const T* eps_n, const T* eps,
                                         MPState<T>& y, T dt, int nsub, T* sig, const T* tab, bool check = true,
                                         T* sc = nullptr) {
  T e0[6], e1[6], de[6];
  to_crystal<T>(R, eps_n, e0);
  to_crystal<T>(R, eps, e1);
#pragma unroll
  for (int c = 0; c < 6; ++c) de[c] = e1[c] - e0[c];
  const bool flows = !(check && elastic_increment<T>(M, e0, de, y));
  if constexpr (SC) store_path(sc, e0, de);
  if (flows) {
    if constexpr (NP == kDirect && std::is_same<T, double>::value) {
      rk4_fp64(M, e0, de, y, dt, nsub, tab);
    } else
    for (int m = 0; m < nsub; ++m) {
      const T h = dt / T(nsub);
      const T inv = T(1) / T(nsub);
      const T s0 = T(m) * inv, sh = (T(m) + T(0.5)) * inv, s1 = (T(m) + T(1)) * inv;
      MPState<T> yt, acc;
      // classical RK4: stages at s0, sh, sh, s1 with weights 1, 2, 2, 1.  The first stage
      // reads y and assigns acc and yt; the other three share one copy of the stage body
      // (not unrolled, which keeps the code compact)
      rk_stage<T, NP, true, SC>(M, SC ? sc : e0, de, s0, y, yt, acc, T(1), T(0.5) * h, tab);
#pragma unroll 1
      for (int stg = 1; stg < 4; ++stg) {
        const T s = stg == 3 ? s1 : sh;
        const T wacc = stg == 3 ? T(1) : T(2);
        const T cnext = stg == 1 ? T(0.5) * h : (stg == 2 ? h : T(0));
        rk_stage<T, NP, false, SC>(M, SC ? sc : e0, de, s, y, yt, acc, wacc, cnext, tab);
      }
      const T w = h / T(6);
#pragma unroll
      for (int c = 0; c < 6; ++c) y.ep[c] += w * acc.ep[c];
#pragma unroll
      for (int c = 0; c < 16; ++c) y.v[c] += w * acc.v[c];
#pragma unroll
      for (int c = 0; c < 12; ++c) y.al[c] += w * acc.al[c];
    }
  }
  T ee[6], sgc[6];
  if constexpr (SC) {
    // the path and (behind the compiler barrier) the rotation are read again
    asm volatile("" ::: "memory");
    T path[12];
    load_path(path, sc);
#pragma unroll
    for (int c = 0; c < 6; ++c) ee[c] = path[c] + path[6 + c] - y.ep[c];
  } else {
#pragma unroll
    for (int c = 0; c < 6; ++c) ee[c] = e1[c] - y.ep[c];
  }
  hooke<T>(M, ee, sgc);
  to_sample<T>(R, sgc, sig);
  return flows;
}

// The whole update by the generic solve, out of line: voxels with an overstress beyond the
// direct tables (their stress is NaN after mc_voxel<T, kDirect>), from the state at t_n.
template <typename T>
__device__ __noinline__ bool mc_voxel_generic(const MatDev<T>& M, const T* R, const T* eps_n, const T* eps,
                                              MPState<T>& y, T dt, int nsub, T* sig) {
  return mc_voxel<T, 0>(M, R, eps_n, eps, y, dt, nsub, sig, nullptr);
}

// Loads a voxel's state (component-major arrays of n voxels): eps_p, v, alpha.
template <typename T>
__device__ __forceinline__ void load_voxel(const T* ep, const T* v, const T* al, size_t n, size_t i, MPState<T>& y) {
#pragma unroll
  for (int c = 0; c < 6; ++c) y.ep[c] = ep[c * n + i];
#pragma unroll
  for (int c = 0; c < 16; ++c) y.v[c] = v[c * n + i];
#pragma unroll
  for (int c = 0; c < 12; ++c) y.al[c] = al[c * n + i];
}

// Integrates a voxel again by the generic solve if its stress is NaN after
// mc_voxel<T, kDirect> in float (an overstress beyond the tables): its state at t_n is at
// (ep, v, al), eps_n and eps have the stride n and ne.  The copies keep the arrays of the
// common path in registers.
template <typename T, int NP>
__device__ __forceinline__ void mc_recover(const MatDev<T>& M, const T* R, const T* eps_n, const T* eps, size_t ne,
                                           MPState<T>& y, T dt, int nsub, T* sig, const T* ep, const T* v,
                                           const T* al, size_t n, size_t i) {
  if constexpr (NP == kDirect && std::is_same<T, float>::value) {
    if (sig[0] != sig[0]) {
      T r2[9], a2[6], b2[6], s2[6];
      MPState<T> y2;
      load_voxel<T>(ep, v, al, n, i, y2);
#pragma unroll
      for (int c = 0; c < 9; ++c) r2[c] = R[c];
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        a2[c] = eps_n[c * n + i];
        b2[c] = eps[c * ne];
      }
      mc_voxel_generic<T>(M, r2, a2, b2, y2, dt, nsub, s2);
      y = y2;
#pragma unroll
      for (int c = 0; c < 6; ++c) sig[c] = s2[c];
    }
  }
}

// Starts the copy of the rate tables (16-byte aligned, a multiple of 16 bytes) to shared memory;
// stage_wait and a barrier complete it.
template <typename T>
__device__ __forceinline__ void stage_tables(T* tab, const T* src, int len) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(tab);
  const int n = (int)((size_t)len * sizeof(T) / 16);
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16u * i),
                 "l"(reinterpret_cast<const char*>(src) + 16 * (size_t)i)
                 : "memory");
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// values of the tables that a constitutive kernel of variant NP keeps in shared memory
template <typename T, int NP>
__host__ __device__ inline int table_len(const MatDev<T>& M) {
  return NP == 0 || NP == kLinearLaw ? 0 : (NP == kDirect ? M.rate_len : kRootTabs);
}

template <typename T>
__device__ __forceinline__ T von_mises6(const T* s) {
  const T p = (s[0] + s[1] + s[2]) / T(3);
  const T a = s[0] - p, b = s[1] - p, c = s[2] - p;
  return sqrt(T(1.5) * (a * a + b * b + c * c + T(2) * (s[3] * s[3] + s[4] * s[4] + s[5] * s[5])));
}

}  // namespace rve
