// Direct tables of the regularised rate (Sec. 4): the root rho = F(a) of
//   rho = < (a - eta rho) / K >^n
// as piecewise polynomials in a.
//
// One function of one variable serves all systems of a law (K, n, eta).  A prefactor P (the
// twins' Kc/sqrt2 <fm - sum f>) only rescales it: with s = P^(1/(n-1)), rho = r / s and
// a = A / s the equation rho = P ((a - eta rho)/K)^n becomes r = ((A - eta r)/K)^n, so
//   rho_P(a) = F(s a) / s.
//
// Segments: each octave of a is cut into 2^S equal segments, so the segment index is the
// exponent and the leading S mantissa bits of a and the distance d to its midpoint is exact.
// Per segment a polynomial in d:
//   float   degree 3 (4 coefficients, one 16-byte load), 22 * 2^6 = 1408 segments (22 KB);
//   double  degree 9 (10 coefficients, 80 bytes),        22 * 2^5 =  704 segments (55 KB).
// S and the octaves below K follow from n (rate_law_fit): the table starts where F falls below
// 2^-100 and takes the finest S that leaves at least 5 octaves above K.  For 2 <= n <= 10.2
// the relative error against the exact root is then below 2.1e-7 in float and 2.4e-16 in
// double for all F >= 2^-100 in the table, rounding included; the power law needs finer segments
// for larger n and more octaves for smaller n (those laws take the Newton variants).  The
// cubic's last coefficient is about n^3/6 F/a^3: in float it is subnormal, and lost, at small
// rates of a large K (relative errors of 2.8e-7 at K = 1e8, 3e-3 at 1e12, against 2.1e-7 at 3e7),
// so float tables end at K = 1e7.
// Below the table the float rate is 0 (< 2^-100 per second); above it the last segment
// holds NaN, which reaches the voxel's stress, and the voxel is integrated again by the
// generic solve.  Double solves generically outside the table.
#pragma once

#include "rve_common.cuh"

namespace rve {

template <typename T> struct RateFmt;
template <> struct RateFmt<float> {
  static constexpr int kDeg = 3, kSeries = 8, kSegs = 1408, kFine = 6;
  static constexpr int kRow = kDeg + 1;
  static constexpr int kLen = (kSegs + 2) * kRow;  // zero segment, polynomials, NaN segment
  static constexpr double kKmax = 1e7;
};
template <> struct RateFmt<double> {
  static constexpr int kDeg = 9, kSeries = 16, kSegs = 704, kFine = 5;
  static constexpr int kRow = kDeg + 1;
  static constexpr int kLen = kSegs * kRow;
  static constexpr double kKmax = 1e12;
};

// 2^(j/64), j = 0 .. 63, follow the law tables in double (exp2_tab)
template <typename T> constexpr int kExpTab = sizeof(T) == 8 ? 64 : 0;
// values of a material's tables: one law (slip and twins alike) or two, then the exponential's
template <typename T>
constexpr int rate_tab_len(bool two) { return (two ? 2 : 1) * RateFmt<T>::kLen + kExpTab<T>; }

// Grid of a law's table: S subdivision bits, first octave 2^e0 .. 2^(e0+1).
struct RateGrid {
  int S, e0;
};

// Host: the table grid of a law, or false where no table is built.
inline bool rate_law_fit(double K, double n, double eta, int segs, int fine, double K_max, RateGrid* g) {
  if (!(eta > 0.0) || !(n >= 2.0 && n <= 10.2) || !(K >= 1e-6 && K <= K_max)) return false;
  int below = 1;
  while (below * n < 100.0) ++below;
  for (int S = fine; S > fine - 3; --S) {
    if ((segs >> S) - below < 5) continue;
    int e = 0;
    double p = 1.0;
    while (p > K) { p *= 0.5; --e; }
    while (2.0 * p <= K) { p *= 2.0; ++e; }
    g->S = S;
    g->e0 = e - below;
    return true;
  }
  return false;
}

template <typename T>
inline bool rate_law_fit_t(double K, double n, double eta, RateGrid* g) {
  return rate_law_fit(K, n, eta, RateFmt<T>::kSegs, RateFmt<T>::kFine, RateFmt<T>::kKmax, g);
}

inline RateLaw<float> rate_law_f(const RateGrid& g, int off) {
  RateLaw<float> L;
  L.shift = 23 - g.S;
  L.base = ((g.e0 + 127) << g.S) - 1;  // the zero segment just below the first octave
  L.last = L.base + RateFmt<float>::kSegs + 1;
  L.mask = ~((1 << L.shift) - 1);
  L.half = 1 << (L.shift - 1);
  const int bits = L.base << L.shift;
  __builtin_memcpy(&L.lo, &bits, sizeof(bits));
  L.off = off;
  return L;
}
inline RateLaw<double> rate_law_d(const RateGrid& g, int off) {
  RateLaw<double> L;
  L.shift = 20 - g.S;
  L.base = (g.e0 + 1023) << g.S;
  L.last = L.base + RateFmt<double>::kSegs - 1;
  L.mask = ~((1 << L.shift) - 1);
  L.half = 1 << (L.shift - 1);
  L.lo = 0.0;
  L.off = off;
  return L;
}
template <typename T>
inline RateLaw<T> rate_law(const RateGrid& g, int off) {
  if constexpr (sizeof(T) == 4) return rate_law_f(g, off);
  else return rate_law_d(g, off);
}

// ---------------------------------------------------------------- evaluation ---------
// F(a), tab: the law's table.  a at or below the floor (inactive systems, NaN) gives 0,
// a beyond the table NaN.
__device__ __forceinline__ float rate_direct(float a, const RateLaw<float>& L, const float* tab) {
  const float aa = fmaxf(a, L.lo);
  const int b = __float_as_int(aa);
  // the row's shared-memory address from the argument's bits: the base is folded into the
  // table's address once, one integer instruction less per rate (128^3 increment 40.9 -> 40.2 ms)
  const unsigned row0 = (unsigned)__cvta_generic_to_shared(tab) - 16u * (unsigned)L.base;
  const unsigned at = row0 + 16u * (unsigned)min(b >> L.shift, L.last);
  const float d = aa - __int_as_float((b & L.mask) | L.half);
  const float4 c = *reinterpret_cast<const float4*>(__cvta_shared_to_generic(at));
  return fmaf(d, fmaf(d, fmaf(d, c.w, c.z), c.y), c.x);
}

// F(a) for a inside the table (rate_inside).
__device__ __forceinline__ bool rate_inside(double a, const RateLaw<double>& L) {
  const int k = __double2hiint(a) >> L.shift;  // negative for a < 0
  return k >= L.base && k <= L.last;
}
__device__ __forceinline__ double rate_direct(double a, const RateLaw<double>& L, const double* tab) {
  const int hi = __double2hiint(a);
  const int i = (hi >> L.shift) - L.base;
  const double d = a - __hiloint2double((hi & L.mask) | L.half, 0);
  const double2* row = reinterpret_cast<const double2*>(tab + i * RateFmt<double>::kRow);
  double2 c = row[4];
  double r = fma(d, c.y, c.x);
#pragma unroll
  for (int k = 3; k >= 0; --k) {
    c = row[k];
    r = fma(d, fma(d, r, c.y), c.x);
  }
  return r;
}

// 2^x beyond exp2_tab's range, out of line.
static __device__ __noinline__ double exp2_far(double x) { return exp2(x); }

// 2^x in double from the 64-entry table of 2^(j/64) (tab) and the Taylor polynomial of 2^r,
// |r| <= 1/128, degree 5 (its remainder is below 2^-54): 9 FP64 instructions.  |x| >= 1000 and
// NaN take the library function.
__device__ __forceinline__ double exp2_tab(double x, const double* tab) {
  if (!((__double2hiint(x) & 0x7fffffff) < 0x408f4000)) return exp2_far(x);
  const double M = 105553116266496.0;  // 1.5 * 2^46: the sum is x rounded to a multiple of 1/64
  const double t = x + M;
  const double r = x - (t - M);
  const int k = __double2loint(t);
  double q = fma(r, 0.0013333558146428443423, 0.0096181291076284771619);
  q = fma(r, q, 0.055504108664821579953);
  q = fma(r, q, 0.24022650695910071233);
  q = fma(r, q, 0.69314718055994530942);
  q = q * r;
  const double T = tab[k & 63];
  const double v = fma(T, q, T);
  return __hiloint2double(__double2hiint(v) + ((k >> 6) << 20), __double2loint(v));
}

// ---------------------------------------------------------------- construction -------
// One thread per segment (and per entry of the exponential's table).  The root at the
// segment's midpoint a0: Newton on c z^n + K z = a0 from above in float, then in double; the
// Taylor series of z and w = z^n in t = (a - a0)/h (h the half width) by z w' = n z' w with
// c w_k + K z_k = 0 (k >= 2) or h (k = 1); economised from degree kSeries to kDeg by
// subtracting multiples of the Chebyshev polynomials.  Bound by the latency of its FP64
// chain; both laws' segments run at once.
template <typename T>
__global__ void k_rate_table(T* out, int two, RateGrid g0, RateGrid g1, double K0, double n0, double K1, double n1,
                             double eta) {
  using Fmt = RateFmt<T>;
  constexpr int N = Fmt::kSegs, M = Fmt::kSeries, D = Fmt::kDeg;
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  const int laws = two ? 2 : 1;
  if (id >= laws * N) {
    const int j = id - laws * N;
    if constexpr (kExpTab<T> > 0) {
      if (j < kExpTab<T>) out[laws * Fmt::kLen + j] = (T)exp2((double)j / 64.0);
    } else if (j < laws) {  // the zero and NaN segments of law j
      T* t = out + j * Fmt::kLen;
      for (int k = 0; k <= D; ++k) {
        t[k] = T(0);
        t[(N + 1) * Fmt::kRow + k] = (T)nan("");
      }
    }
    return;
  }
  const int law = id / N, seg = id - law * N;
  const RateGrid g = law ? g1 : g0;
  const double K = law ? K1 : K0, n = law ? n1 : n0;
  const double h = ldexp(1.0, g.e0 + (seg >> g.S) - g.S - 1);
  const double a0 = ldexp(1.0 + ((seg & ((1 << g.S) - 1)) + 0.5) / (double)(1 << g.S), g.e0 + (seg >> g.S));
  // Newton decreases monotonically from the upper bound min(a/K, (a/eta)^(1/n)); in float
  // on the scaled root u = z / zB, u^n + beta u = 1 (zB = (a/eta)^(1/n), beta = K zB / a)
  const double lzB = log2(a0 / eta) / n;
  const double zB = exp2(lzB), beta = K * zB / a0;
  const float bf = (float)fmin(beta, 1e30), nf = (float)n;
  float u = fminf(1.0f, 1.0f / bf);
  for (int it = 0; it < 12; ++it) {
    const float un1 = powf(u, nf - 1.0f);
    u = u - ((un1 + bf) * u - 1.0f) / (nf * un1 + bf);
  }
  double z = beta < 1e30 ? zB * (double)u : a0 / K;
  for (int it = 0; it < 2; ++it) {
    const double c1 = eta * pow(z, n - 1.0);
    z = z - ((c1 + K) * z - a0) / (n * c1 + K);
  }
  // the root's residual corrects w to the accuracy of pow (a rounding of z alone would enter
  // w = z^n n-fold)
  double Z[M + 1], W[M + 1];
  Z[0] = z;
  const double w = pow(z, n), e = fma(K, z, -a0);
  const double dz = -(eta * w + e) / (n * eta * w / z + K);
  W[0] = eta * w > K * z ? -(e + K * dz) / eta : fma(w, n * dz / z, w);
  const double nw = n * W[0] / z, den = 1.0 / (eta * nw + K);
  for (int k = 1; k <= M; ++k) {
    double R = 0.0;
    for (int j = 1; j < k; ++j) R += (n * j - (k - j)) * Z[j] * W[k - j];
    R /= k * z;
    Z[k] = ((k == 1 ? h : 0.0) - eta * R) * den;
    W[k] = nw * Z[k] + R;
  }
  for (int k = M; k > D; --k) {
    // W -= W_k 2^(1-k) T_k, T_k = sum_j t_j x^(k-2j), t_0 = 2^(k-1)
    double t = W[k];
    for (int j = 0, p = k; p >= 0; ++j, p -= 2) {
      W[p] -= t;
      if (p >= 2) t *= -(double)(p * (p - 1)) / (4.0 * (j + 1) * (k - j - 1));
    }
  }
  T* row = out + law * Fmt::kLen + (size_t)(seg + (kExpTab<T> > 0 ? 0 : 1)) * Fmt::kRow;
  double hk = 1.0;
  for (int k = 0; k <= D; ++k) {
    row[k] = (T)(W[k] * hk);
    hk /= h;
  }
}

}  // namespace rve
