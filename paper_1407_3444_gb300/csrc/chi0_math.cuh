// chi0_math.cuh -- device arithmetic of the doubly carved linear tetrahedron method.
//
// Sec. II of Heil et al. (arXiv:1407.3444): the integrand of Eqs. 1-2 is restricted to
// the region where Th(eF - e^m_k) Th(e^n_{k+q} - eF) = 1 (Eq. 4) by cutting every
// tetrahedron twice, first by a = e^m_k - eF < 0, then by b = e^n_{k+q} - eF > 0.  On
// each final tetrahedron S (volume V, vertex values d_j = b_j - a_j >= 0 of
// D = e^n_{k+q} - e^m_k and f_j of |M|^2) the integrals are exact for the linear
// interpolants (Hermite-Genocchi):
//   (1/V) int_S lambda_j / (D - x)   = g[d_1-x, .., d_4-x, d_j-x],  g(t) = t^3 ln|t|
//   (1/V) int_S lambda_j delta(w - D) = M(w; d_1..d_4, d_j) / 4     (cubic B-spline density)
// with g[...] the fourth divided difference (knot d_j repeated).  The paper does not print
// its formulas; these are the closed forms for linear integrands on a simplex.
//
// Evaluation strategy (GPU-first; all branches exact up to rounding):
//  * knots clustered away from 0 (spread <= RHO * |nearest|): one Taylor series about
//    the mean for all four j at once (h_k complete homogeneous polynomials);
//  * otherwise the divided-difference table of the sorted knots, each entry by the
//    difference recursion or, where its own knots cluster, by its Taylor series;
//  * mixed precision: the table in FP32 only when every gap between sorted knots is at
//    least tau * max|knot|; below that (the near-degenerate, cancellation-prone case)
//    the table is evaluated in FP64.
#pragma once

#ifdef __CUDACC__
#include <cuda_runtime.h>
#endif
#include <math.h>
#include <stdint.h>

#include <type_traits>

namespace chi0dev {

constexpr double kRho = 0.25;                     // Taylor branch threshold
constexpr double kFloor = 9.313225746154785e-10;  // 2^-30: >= 3 exactly-zero knots

template <typename T> struct Num;
template <> struct Num<double> {
  static __device__ __forceinline__ double lg(double x) { return log(x); }
  static constexpr double tol = 1e-17;
  static constexpr double kappa = 0.25;  // series branch: (x3 - x0) <= kappa (x3 + x0)
  static constexpr int kmax = 80;
};
template <> struct Num<float> {
  static __device__ __forceinline__ float lg(float x) { return logf(x); }
  static constexpr float tol = 2e-8f;
  static constexpr float kappa = 0.5f;       // series branch inside the carving loop
  static constexpr float kappa_long = 0.7f;  // series branch of queued pieces (evaluated together)
  static constexpr float kappa_far = 0.5f;   // far-field expansion of the dynamic PV terms
  static constexpr int kmax = 64;
};

template <typename T> __device__ __forceinline__ T tabs(T x) { return x < T(0) ? -x : x; }

// Reciprocal and quotient of the weight kernels.  FP64: IEEE division.  FP32: the hardware
// reciprocal approximation refined by one Newton-Raphson step, r' = r + r (1 - x r), within
// about 1 ulp of 1/x for normal x (0 and denormals are never divided by: ties and zero knots
// take their own branches), and the fast quotient (at most 2 ulp from a / b for the cut
// fractions, |b| < 2^126); both far below the FP32 path's 1e-6 target.  The correctly rounded
// intrinsics carry slow paths for special operands that made the weight kernels' hot code
// several times larger (instruction-cache misses).
__device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
__device__ __forceinline__ float rcp(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return fmaf(r, fmaf(-x, r, 1.0f), r);
#else
  return __frcp_rn(x);
#endif
}
// FP64 reciprocal of the weight kernels' hot paths: the hardware seed and two Newton-Raphson steps (four
// multiply-adds on the FP64 pipe, about 1 ulp; IEEE division takes more than twice that).  For
// 2^-1022 <= |x| < 2^1022; a NaN at 0, below 2^-1022 and at infinity, which callers keep away from it.
__device__ __forceinline__ double rcp_nr(double x) {
#ifdef __CUDA_ARCH__
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
#else
  return 1.0 / x;
#endif
}
__device__ __forceinline__ float rcp_nr(float x) { return rcp(x); }
// a - b with no product of the operands contracted into it (FP32)
__device__ __forceinline__ float sub_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fsub_rn(a, b);
#else
  return a - b;
#endif
}
__device__ __forceinline__ double sub_rn(double a, double b) { return a - b; }
__device__ __forceinline__ double quot(double a, double b) { return a / b; }
__device__ __forceinline__ float quot(float a, float b) { return __fdividef(a, b); }

template <typename T> __device__ __forceinline__ void cswap(T &x, T &y, T &fx, T &fy) {
  if (y < x) {
    T t = x; x = y; y = t;
    t = fx; fx = fy; fy = t;
  }
}

// ascending sort of 4 knots carrying their weights (5-comparator network)
template <typename T> __device__ __forceinline__ void sort4(T d[4], T f[4]) {
  cswap(d[0], d[1], f[0], f[1]);
  cswap(d[2], d[3], f[2], f[3]);
  cswap(d[0], d[2], f[0], f[2]);
  cswap(d[1], d[3], f[1], f[3]);
  cswap(d[1], d[2], f[1], f[2]);
}

// g(t) = t^3 ln|t|, g(0) = 0
template <typename T> __device__ __forceinline__ T g0(T t) {
  return t == T(0) ? T(0) : t * t * t * Num<T>::lg(tabs(t));
}

// g^(k)(c)/k! for k = 1..3 (c != 0)
template <typename T> __device__ __forceinline__ T glow(int k, T c, T L) {
  if (k == 1) return T(3) * c * c * L + c * c;
  if (k == 2) return (T(6) * c * L + T(5) * c) * T(0.5);
  return (T(6) * L + T(11)) * T(1.0 / 6.0);
}

// 6 (-1)^m / ((m+4)(m+3)(m+2)(m+1)): coefficients of the Taylor series below (k = m + 4)
template <typename T, int N> struct TaylorCoef {
  T v[N];
  constexpr TaylorCoef() : v() {
    for (int m = 0; m < N; ++m) {
      const T c = T(6) / (T(m + 4) * T(m + 3) * T(m + 2) * T(m + 1));
      v[m] = (m & 1) ? -c : c;
    }
  }
};
__constant__ constexpr TaylorCoef<float, Num<float>::kmax + 4> kTayF{};
__constant__ constexpr TaylorCoef<double, Num<double>::kmax + 4> kTayD{};
template <typename T> __device__ __forceinline__ T taylor_coef(int m);
template <> __device__ __forceinline__ float taylor_coef<float>(int m) { return kTayF.v[m]; }
template <> __device__ __forceinline__ double taylor_coef<double>(int m) { return kTayD.v[m]; }

// Taylor series of the divided difference g[t_i..t_j] (n = j - i) of knots clustered about
// their mean c != 0, in the scaled offsets e = (t - c)/c (no powers of 1/c that could
// overflow):  g[t_i..t_j] = sum_{k=n}^{3} g^(k)(c)/k! c^(k-n) h_{k-n}(e)
//                        + c^(3-n) sum_{k>=4} 6 (-1)^(k-4) / (k(k-1)(k-2)(k-3)) h_{k-n}(e)
// with h_m the complete homogeneous symmetric polynomials.
template <typename T> __device__ __noinline__ T dd_taylor(const T t[5], int i, int j) {
  const int n = j - i;
  T c = T(0);
#pragma unroll
  for (int l = 0; l < 5; ++l) c += (l >= i && l <= j) ? t[l] : T(0);
  c = c / T(n + 1);
  const T ci = rcp(c);
  T e[5], h[5];
#pragma unroll
  for (int l = 0; l < 5; ++l) {
    e[l] = (l >= i && l <= j) ? (t[l] - c) * ci : T(0);  // padding variables are 0: no effect on h
    h[l] = T(1);
  }
  const T L = Num<T>::lg(tabs(c));
  T low = T(0), cp = T(1);  // cp = c^(k-n)
  for (int k = n; k < 4; ++k) {
    if (k > n) {
      h[0] = e[0] * h[0];
#pragma unroll
      for (int l = 1; l < 5; ++l) h[l] = h[l - 1] + e[l] * h[l];
      cp *= c;
    }
    low += (k == 0 ? g0(c) : glow(k, c, L)) * cp * h[4];
  }
  T high = T(0), prev = T(0), big = T(0);
  for (int k = 4; k < n + Num<T>::kmax; ++k) {
    if (k > n) {
      h[0] = e[0] * h[0];
#pragma unroll
      for (int l = 1; l < 5; ++l) h[l] = h[l - 1] + e[l] * h[l];
    }
    const T coef = taylor_coef<T>(k - 4);  // 6 (-1)^(k-4) / (k (k-1) (k-2) (k-3))
    const T term = coef * h[4];
    high += term;
    big = tabs(term) > big ? tabs(term) : big;
    if (k >= 5 && k - n >= 2 &&
        tabs(term) + tabs(prev) <= Num<T>::tol * (tabs(high) > big ? tabs(high) : big))
      break;
    prev = term;
  }
  T scale = T(1);  // c^(3-n)
  if (n == 4) scale = ci;
  else if (n == 2) scale = c;
  else if (n == 1) scale = c * c;
  return low + scale * high;
}

// Fourth divided difference g[t0..t4] of sorted knots (no 4 equal zeros).
template <typename T> __device__ T dd5(const T t[5]) {
  const T rho = T(kRho);
  T v[5];
#pragma unroll
  for (int l = 0; l < 5; ++l) v[l] = g0(t[l]);
#pragma unroll
  for (int n = 1; n <= 4; ++n) {
#pragma unroll
    for (int i = 0; i + n <= 4; ++i) {
      const int j = i + n;
      const T ti = t[i], tj = t[j];
      T r;
      if (ti == tj) {
        // all knots equal: g^(n)(t)/n!; at t = 0: 0 for n <= 2
        r = (ti == T(0)) ? T(0) : glow(n < 4 ? n : 3, ti, Num<T>::lg(tabs(ti)));
        if (n == 4) r = (ti == T(0)) ? T(0) : T(0.25) / ti;
      } else if ((ti > T(0) && tj - ti <= rho * ti) || (tj < T(0) && tj - ti <= rho * (-tj))) {
        r = dd_taylor(t, i, j);
      } else {
        r = (v[i + 1] - v[i]) / (tj - ti);
      }
      v[i] = r;
    }
  }
  return v[0];
}

// (-1)^k 6 k!/(k+4)! = (-1)^k 6/((k+1)(k+2)(k+3)(k+4)), the series coefficients below
template <typename T, int N> struct SeriesCoef {
  T v[N];
  constexpr SeriesCoef() : v() {
    for (int k = 0; k < N; ++k) {
      const T c = T(6) / (T(k + 1) * T(k + 2) * T(k + 3) * T(k + 4));
      v[k] = (k & 1) ? -c : c;
    }
  }
};
__constant__ constexpr SeriesCoef<float, Num<float>::kmax> kCoefF{};
__constant__ constexpr SeriesCoef<double, Num<double>::kmax> kCoefD{};
template <typename T> __device__ __forceinline__ T series_coef(int k);
template <> __device__ __forceinline__ float series_coef<float>(int k) { return kCoefF.v[k]; }
template <> __device__ __forceinline__ double series_coef<double>(int k) { return kCoefD.v[k]; }

// sum_j f_j (1/V) int_S lambda_j / X for sorted knots x of one sign with
// |x_i - c| <= kappa |c| about the midpoint c = (x_0 + x_3)/2:
// 1/(c (1 + lambda.e)), e = (x - c)/c, expanded in lambda.e:
//   (1/V) int lambda_j / X = (1/c) sum_k (-1)^k 6 k!/(k+4)! h_k(e_1..e_4, e_j)
template <typename T> __device__ T series_sum(const T x[4], const T f[4]) {
  const T c = (x[0] + x[3]) * T(0.5);
  const T ci = rcp(c);
  T e[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) e[l] = (x[l] - c) * ci;
  T H[4] = {T(1), T(1), T(1), T(1)};  // H_k over the first l+1 variables
  T P[4] = {T(1), T(1), T(1), T(1)};  // h_k(e, e_j)
  T sum = T(0.25) * (f[0] + f[1] + f[2] + f[3]);  // k = 0: 6/24 sum_j f_j
  T prev = T(0), big = tabs(sum);
  for (int k = 1; k < Num<T>::kmax; ++k) {
    H[0] = e[0] * H[0];
#pragma unroll
    for (int l = 1; l < 4; ++l) H[l] = H[l - 1] + e[l] * H[l];
    T s = T(0);
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      P[jj] = H[3] + e[jj] * P[jj];
      s += f[jj] * P[jj];
    }
    const T term = series_coef<T>(k) * s;
    sum += term;
    big = tabs(term) > big ? tabs(term) : big;
    if (k >= 2 && tabs(term) + tabs(prev) <= Num<T>::tol * (tabs(sum) > big ? tabs(sum) : big)) break;
    prev = term;
  }
  return sum * ci;
}

// ------------------------------------------------------------------------------------
// The same integral by a polynomial of fixed length about the MEAN of the knots (FP64 static
// weights).  With c = mean(x), e = (x - c)/c and |e_j| <= R < 1, 1/(1 + t) is replaced on
// [-R, R] by the degree K - 1 polynomial p(t) = sum_k p_k t^k, and
//   sum_j f_j (1/V) int_S lambda_j / X = (1/c) sum_k a_k s_k,   a_k = p_k 6 k!/(k+4)!,
//   s_k = sum_j f_j h_k(e_1..e_4, e_j) = [z^k] N(z)/Q(z)^2,
//   Q(z) = prod_i (1 - e_i z) = 1 + E2 z^2 - E3 z^3 + E4 z^4   (E1 = sum e = 0 about the mean),
//   N(z) = sum_j f_j Q(z)/(1 - e_j z) = N0 + N1 z + N2 z^2 + N3 z^3.
// Dividing by Q is a three-term recurrence, so the sum is taken backward (Clenshaw's scheme,
// applied once per factor Q): y_k = a_k - E2 y_{k+2} + E3 y_{k+3} - E4 y_{k+4}, the same from
// y to z, and sum_k a_k s_k = N0 z_0 + N1 z_1 + N2 z_2 + N3 z_3 (Q/(1 - e_j z) = 1 + e_j z +
// (E2 + e_j^2) z^2 + (E2 e_j - E3 + e_j^3) z^3).  Six multiply-adds per term
// and no convergence test, against about twenty operations of the forward series_sum above;
// the knots need not be sorted; E1 = 0 is what drops a fourth multiply-add per factor.
// p is the Chebyshev series of 1/(1 + t) on [-R, R] cut after K terms (q = R/(1 + sqrt(1-R^2)),
// error at most 2 q^K / ((1 - q) sqrt(1 - R^2))), which reaches R ~ 2 tol^(1/K) where the
// Taylor series ends at tol^(1/K): 16 terms where Taylor takes 22 (R = 0.16).
// One tier per K = 4, 8, 12, ...: its largest R, and its a_k in a table.
constexpr double kMeanTolD = 1.0e-17;  // truncation (below one rounding)
constexpr int kMeanTiersD = 14;
constexpr double kMeanRD[kMeanTiersD] = {0.00009, 0.01373, 0.07195, 0.16362, 0.26542, 0.36291, 0.44985,
                                         0.52463, 0.58785, 0.64092, 0.68541, 0.72278, 0.75431, 0.78103};
constexpr double mean_sqrt(double x) {  // Newton's iteration (compile time, 0 < x <= 1)
  double r = 1.0;
  for (int i = 0; i < 60; ++i) r = 0.5 * (r + x / r);
  return r;
}
constexpr double mean_err(double R, int K) {  // the Chebyshev truncation bound above
  const double s = mean_sqrt(1.0 - R * R), q = R / (1.0 + s);
  double t = 2.0 / ((1.0 - q) * s);
  for (int i = 0; i < K; ++i) t *= q;
  return t;
}
// the polynomial for radius R: p_0 .. p_{K-1}, and a_0 .. a_{K-1} in T
template <typename T, int K> struct ChebInv {
  T v[K];
  double p_[K];
  constexpr explicit ChebInv(double R) : v(), p_() {
    // sum_n c_n T_n(t/R), c_0 = 1/s, c_n = 2 (-q)^n / s, collected in powers of u = t/R
    const double s = mean_sqrt(1.0 - R * R), q = R / (1.0 + s);
    double p[K + 1] = {}, t0[K + 1] = {}, t1[K + 1] = {};
    t0[0] = 1.0;
    t1[1] = 1.0;
    double c = 1.0 / s;
    p[0] = c;
    c *= -2.0 * q;
    for (int n = 1; n < K; ++n) {
      for (int k = 0; k <= n; ++k) p[k] += c * t1[k];
      c *= -q;
      double t2[K + 1] = {};
      for (int k = 0; k <= n; ++k) t2[k + 1] = 2.0 * t1[k];
      for (int k = 0; k <= n; ++k) {
        t2[k] -= t0[k];
        t0[k] = t1[k];
      }
      for (int k = 0; k <= K; ++k) t1[k] = t2[k];
    }
    double rk = 1.0;
    for (int k = 0; k < K; ++k) {
      // p_k differs from Taylor's (-1)^k by the truncation; a difference of a few roundings is
      // this computation's own and is dropped (it would be a bias common to all pieces)
      const double one = (k & 1) ? -1.0 : 1.0, dp = p[k] / rk - one;
      const double pk = dp < 1e-15 && dp > -1e-15 ? one : p[k] / rk;
      p_[k] = pk;
      v[k] = (T)(pk * 6.0 / ((k + 1.0) * (k + 2.0) * (k + 3.0) * (k + 4.0)));  // a_k
      rk *= R;
    }
  }
};
constexpr int mean_off(int tier) { return 2 * tier * (tier + 1); }  // a tier's first coefficient
// threshold on the high word of max|e| (FP32: its bits): bits <= thr implies max|e| <= R
constexpr int mean_bits(double x, bool dbl) {
  int e = 0;
  while (x < 1.0) {
    x *= 2.0;
    --e;
  }
  return dbl ? (((1023 + e) << 20) | (int)((x - 1.0) * 1048576.0)) - 1
             : (((127 + e) << 23) | (int)((x - 1.0) * 8388608.0));
}
template <typename T, int NT> struct MeanTab {
  T a[2 * NT * (NT + 1)];
  int thr[NT];
  template <int I> constexpr void tier(const double (&R)[NT]) {
    if constexpr (I < NT) {
      const ChebInv<T, 4 * (I + 1)> c(R[I]);
      for (int k = 0; k < 4 * (I + 1); ++k) a[mean_off(I) + k] = c.v[k];
      thr[I] = mean_bits(R[I], sizeof(T) == 8);
      tier<I + 1>(R);
    }
  }
  constexpr explicit MeanTab(const double (&R)[NT]) : a(), thr() { tier<0>(R); }
};
constexpr bool mean_tiers_ok() {
  for (int i = 0; i < kMeanTiersD; ++i)
    if (mean_err(kMeanRD[i], 4 * (i + 1)) > kMeanTolD) return false;
  return true;
}
static_assert(mean_tiers_ok(), "a tier's R is too large for its K");
__constant__ constexpr MeanTab<double, kMeanTiersD> kMeanD{kMeanRD};
template <typename T> struct Mean;
template <> struct Mean<float> {
  static __device__ __forceinline__ int bits(float x) {
#ifdef __CUDA_ARCH__
    return __float_as_int(x) & 0x7fffffff;
#else
    int i;
    memcpy(&i, &x, 4);
    return i & 0x7fffffff;
#endif
  }
};
template <> struct Mean<double> {
  static constexpr int tiers = kMeanTiersD;
  static __device__ __forceinline__ int thr(int i) { return kMeanD.thr[i]; }
  static __device__ __forceinline__ double a(int i) { return kMeanD.a[i]; }
  static __device__ __forceinline__ int bits(double x) {
#ifdef __CUDA_ARCH__
    return __double2hiint(x) & 0x7fffffff;
#else
    long long i;
    memcpy(&i, &x, 8);
    return (int)(i >> 32) & 0x7fffffff;
#endif
  }
};
// offsets e = d ci - 1 (one rounding each; 1/d = ci/(1 + e) holds for ci as it is), ci = 1/mean,
// and the bits of max|e| (a NaN, from knots that are all 0, lies above every threshold)
template <typename T> __device__ __forceinline__ int mean_offsets(const T d[4], T e[4], T &ci) {
  ci = rcp_nr(((d[0] + d[1]) + (d[2] + d[3])) * T(0.25));
  int r = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    e[i] = fma(d[i], ci, T(-1));
    const int b = Mean<T>::bits(e[i]);
    r = b > r ? b : r;
  }
  return r;
}
// the smallest of the first N tiers that holds max|e| of these bits (N: none)
template <typename T, int N> __device__ __forceinline__ int mean_tier(int bits) {
  int t = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) t += bits > Mean<T>::thr(i) ? 1 : 0;
  return t;
}
template <typename T> __device__ __forceinline__ T mean_series(const T e[4], const T f[4], T ci, int tier) {
  const T s = e[0] + e[1], e3 = -(s + e[2]);  // (sum of e = 0)
  const T P = e[0] * e[1], Q = e[2] * e3;
  const T E2 = (P + Q) - s * s, E3 = s * (Q - P), nE4 = -(P * Q), nE2 = -E2;
  const int base = 2 * tier * (tier + 1);  // the tier's first coefficient
  int t = 4 * tier;
  // the last four terms (nothing above them), then four at a time
  T Y3 = Mean<T>::a(base + t + 3), Y2 = Mean<T>::a(base + t + 2);
  T Y1 = nE2 * Y3 + Mean<T>::a(base + t + 1), Y0 = nE2 * Y2 + (E3 * Y3 + Mean<T>::a(base + t));
  T Z3 = Y3, Z2 = Y2, Z1 = nE2 * Z3 + Y1, Z0 = nE2 * Z2 + (E3 * Z3 + Y0);
#pragma unroll 1
  for (t -= 4; t >= 0; t -= 4) {
    const T n3 = nE2 * Y1 + (E3 * Y2 + (nE4 * Y3 + Mean<T>::a(base + t + 3)));
    const T n2 = nE2 * Y0 + (E3 * Y1 + (nE4 * Y2 + Mean<T>::a(base + t + 2)));
    const T n1 = nE2 * n3 + (E3 * Y0 + (nE4 * Y1 + Mean<T>::a(base + t + 1)));
    const T n0 = nE2 * n2 + (E3 * n3 + (nE4 * Y0 + Mean<T>::a(base + t)));
    const T z3 = nE2 * Z1 + (E3 * Z2 + (nE4 * Z3 + n3));
    const T z2 = nE2 * Z0 + (E3 * Z1 + (nE4 * Z2 + n2));
    const T z1 = nE2 * z3 + (E3 * Z0 + (nE4 * Z1 + n1));
    const T z0 = nE2 * z2 + (E3 * z3 + (nE4 * Z0 + n0));
    Y0 = n0, Y1 = n1, Y2 = n2, Y3 = n3;
    Z0 = z0, Z1 = z1, Z2 = z2, Z3 = z3;
  }
  // sum_k N_k z_k = sum_j f_j (A + e_j (B + e_j (z_2 + e_j z_3)))
  const T A = (Z0 - E3 * Z3) + E2 * Z2, B = Z1 + E2 * Z3;
  T sum = f[0] * (A + e[0] * (B + e[0] * (Z2 + e[0] * Z3)));
  sum += f[1] * (A + e[1] * (B + e[1] * (Z2 + e[1] * Z3)));
  sum += f[2] * (A + e[2] * (B + e[2] * (Z2 + e[2] * Z3)));
  sum += f[3] * (A + e3 * (B + e3 * (Z2 + e3 * Z3)));
  return sum * ci;
}

// series_sum's own terms, by a cheaper recurrence (FP32 static weights): the same expansion about
// the midpoint, cut by the same rule (two successive terms at or below tol), so that the sums agree
// to rounding.  s_k = [z^k] N(z) / Q(z)^2 with Q = (1 - r^2 z^2)(1 - e1 z)(1 - e2 z), r = -e0 = e3: two
// divisions by each factor, six multiply-adds per term where the h_k of all four vertices take
// thirteen operations.  N = n0 + n1 z + n2 z^2 + n3 z^3 from the power sums of f e^i.
__device__ __forceinline__ float series_sum_short(const float x[4], const float f[4]) {
  const float c = (x[0] + x[3]) * 0.5f, ci = rcp(c);
  const float r = (x[3] - x[0]) * 0.5f * ci, e1 = fmaf(x[1], ci, -1.0f), e2 = fmaf(x[2], ci, -1.0f);
  const float r2 = r * r;
  // power sums m_i = sum_j f_j e_j^i
  const float fs = f[0] + f[3], fd = (f[3] - f[0]) * r;
  const float g1 = f[1] * e1, g2 = f[2] * e2, h1 = g1 * e1, h2 = g2 * e2;
  const float m0 = fs + (f[1] + f[2]), m1 = fd + (g1 + g2), m2 = fmaf(r2, fs, h1 + h2);
  const float m3 = fmaf(r2, fd, fmaf(h1, e1, h2 * e2));
  // elementary symmetric polynomials of the offsets (-r, e1, e2, r)
  const float E1 = e1 + e2, P = e1 * e2, E2 = P - r2, E3 = -r2 * E1;
  const float n1 = m1 - E1 * m0, n2 = fmaf(E2, m0, m2 - E1 * m1), n3 = fmaf(E2, m1, m3) - fmaf(E3, m0, E1 * m2);
  // stage by stage: x = N/(1 - r2 z2), y = x/(1 - r2 z2), then twice 1/(1 - e1 z), twice 1/(1 - e2 z)
  float xa = m0, xb = n1, ya = m0, yb = n1;  // the last two of x and y (even, odd)
  float v = m0, vv = m0, u = m0, uu = m0;
  auto step = [&](float y) {
    v = fmaf(e1, v, y);
    vv = fmaf(e1, vv, v);
    u = fmaf(e2, u, vv);
    uu = fmaf(e2, uu, u);
    return uu;
  };
  float sum = 0.25f * m0, big = tabs(sum);
  float tp = series_coef<float>(1) * step(yb);
  sum += tp;
  xa = fmaf(r2, xa, n2);
  ya = fmaf(r2, ya, xa);
  float t = series_coef<float>(2) * step(ya);
  sum += t;
  big = fmaxf(fmaxf(big, tabs(sum)), fmaxf(tabs(tp), tabs(t)));
  const float thr = Num<float>::tol * big;  // (the sum moves little after the second term)
  if (tabs(t) + tabs(tp) > thr) {
    xb = fmaf(r2, xb, n3);
#pragma unroll 1
    for (int k = 3; k + 1 < Num<float>::kmax; k += 2) {  // (two coefficients a step)
      yb = fmaf(r2, yb, xb);
      tp = series_coef<float>(k) * step(yb);
      sum += tp;
      if (tabs(t) + tabs(tp) <= thr) break;
      xb *= r2;
      xa *= r2;
      ya = fmaf(r2, ya, xa);
      t = series_coef<float>(k + 1) * step(ya);
      sum += t;
      if (tabs(t) + tabs(tp) <= thr) break;
    }
  }
  return sum * ci;
}

// f_j (1/V) int lambda_j / X for one vertex j (sorted knots, any signs; PV across X = 0)
template <typename T> __device__ T inv_term_table(const T xin[4], const T f[4], int jj) {
  T x[4] = {xin[0], xin[1], xin[2], xin[3]};
  T s = tabs(x[0]) > tabs(x[3]) ? tabs(x[0]) : tabs(x[3]);
  if (s == T(0)) return T(0);
  const int nz = (x[0] == T(0)) + (x[1] == T(0)) + (x[2] == T(0)) + (x[3] == T(0));
  if (nz >= 3) {
#pragma unroll
    for (int l = 0; l < 4; ++l) x[l] = x[l] == T(0) ? T(kFloor) * s : x[l];
    T dummy[4] = {T(0), T(0), T(0), T(0)};
    sort4(x, dummy);
  }
  const T si = T(1) / s;
  T t5[5];
#pragma unroll
  for (int l = 0; l < 5; ++l) {
    const int src = l <= jj ? l : l - 1;
    t5[l] = (src == 0 ? x[0] : src == 1 ? x[1] : src == 2 ? x[2] : x[3]) * si;
  }
  const T fj = jj == 0 ? f[0] : jj == 1 ? f[1] : jj == 2 ? f[2] : f[3];
  return fj * dd5(t5) * si;
}

// sum_j f_j (1/V) int lambda_j / X for sorted knots x (any signs; PV across X = 0)
template <typename T> __device__ T inv_sum_table(const T xin[4], const T f[4]) {
  T x[4] = {xin[0], xin[1], xin[2], xin[3]};
  T s = tabs(x[0]) > tabs(x[3]) ? tabs(x[0]) : tabs(x[3]);
  if (s == T(0)) return T(0);
  const int nz = (x[0] == T(0)) + (x[1] == T(0)) + (x[2] == T(0)) + (x[3] == T(0));
  if (nz >= 3) {
    // a face with X = 0 (log-divergent): exact zeros floored, measure-zero input
#pragma unroll
    for (int l = 0; l < 4; ++l) x[l] = x[l] == T(0) ? T(kFloor) * s : x[l];
    // re-sort (floored zeros stay below the positive knots; negative knots stay first)
    T dummy[4] = {T(0), T(0), T(0), T(0)};
    sort4(x, dummy);
  }
  const T si = T(1) / s;
  T u[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) u[l] = x[l] * si;
  T acc = T(0);
#pragma unroll 1
  for (int jj = 0; jj < 4; ++jj) {
    T t5[5];
    t5[0] = u[0];
#pragma unroll
    for (int l = 1; l < 5; ++l) t5[l] = l <= jj ? u[l] : u[l - 1];
    const T fj = jj == 0 ? f[0] : jj == 1 ? f[1] : jj == 2 ? f[2] : f[3];
    acc += fj * dd5(t5);
  }
  return acc * si;
}

// sum_j f_j (1/V) int lambda_j / X for sorted knots x (PV across X = 0) by one shared
// divided-difference table: with u = x/s (s = max|x|) and g(t) = t^3 ln|t|, the 4-knot entries
// G[p..r] are common to all j, and the entries with knot j doubled follow the same recursion,
//   H_j[p..r] = ((p < j ? H_j[p+1..r] : G[p..r]) - (r > j ? H_j[p..r-1] : G[p..r])) / (u_r - u_p),
//   H_j[j..j] = g'(u_j) = 3 u_j^2 ln|u_j| + u_j^2,
// so all four fourth divided differences g[u, u_j] = H_j[0..3] take four logarithms (FP64: three) and six
// reciprocals (the per-vertex table below takes twenty and forty divisions).  The result is
// sum_j f_j H_j[0..3] / s.
// A pair of adjacent knots a < b of one sign with y = (b - a)/a small (|y| <= 1/8, ties
// included) would cancel in the recursion; its three entries g[a,b], g[a,a,b], g[a,b,b] are
// taken from the Taylor series about a instead (d = b - a):
//   g[a,b]   = g'(a) + d g2(a)/2 + d^2 g3(a)/6 + d sum_{k>=4} T_k
//   g[a,a,b] = g2(a)/2 + d g3(a)/6 + sum_{k>=4} T_k
//   g[a,b,b] = g2(a)/2 + d g3(a)/3 + sum_{k>=4} (k-1) T_k
// with the second and third derivatives g2 = 6t ln|t| + 5t, g3 = 6 ln|t| + 11, the higher ones
// 6 (-1)^k (k-4)!/a^(k-3) (k >= 4), and T_k = (k-th derivative at a) d^(k-2)/k! =
// 6 (-1)^k (k-4)!/k! a y^(k-2), which falls like y^k.  Two knots at 0 give the limits
// g'(0) = g''(0)/2 = 0.  Returns false, leaving the work to the per-vertex table, where two
// adjacent pairs both cluster (three knots together) or three knots are 0.
constexpr double kRhoShared = 0.125;  // adjacent knots this close (relative): series entries
template <typename T> __device__ __forceinline__ bool inv_sum_shared(const T x[4], const T f[4], T &out) {
  const T s = tabs(x[0]) > tabs(x[3]) ? tabs(x[0]) : tabs(x[3]);
  if (s == T(0)) {
    out = T(0);
    return true;
  }
  const T rho = T(kRhoShared);
  const T si = rcp(s);
  T u[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) u[i] = x[i] * si;
  int nz = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) nz += u[i] == T(0);
  if (nz >= 3) return false;
  bool cl[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const T a = u[i], b = u[i + 1];
    cl[i] = (a > T(0) && b - a <= rho * a) || (b < T(0) && b - a <= rho * (-b));
  }
  if ((cl[0] && cl[1]) || (cl[1] && cl[2])) return false;  // three knots together
  T g[4], gp[4], L[4];
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int i = 0; i < 4; ++i) L[i] = u[i] == T(0) ? T(0) : Num<T>::lg(tabs(u[i]));
  } else {  // (the end knot of largest magnitude is +-1 to rounding: no logarithm)
    const bool low = tabs(x[0]) > tabs(x[3]);
    const T o = low ? u[3] : u[0], Lo = o == T(0) ? T(0) : Num<T>::lg(tabs(o));
    L[0] = low ? T(0) : Lo;
    L[3] = low ? Lo : T(0);
#pragma unroll
    for (int i = 1; i < 3; ++i) L[i] = u[i] == T(0) ? T(0) : Num<T>::lg(tabs(u[i]));
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const T t = u[i], t2 = t * t;
    g[i] = t2 * t * L[i];
    gp[i] = T(3) * t2 * L[i] + t2;
  }
  // first-level entries of every adjacent pair: G1 = g[u_p, u_p+1], HL = g[u_p, u_p, u_p+1],
  // HR = g[u_p, u_p+1, u_p+1]
  T G1[3], HL[3], HR[3];
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const T d = u[p + 1] - u[p];
    const bool zero = !(d > T(0));  // two knots at 0 (a tie elsewhere is clustered): the limits
    const T r = rcp(zero ? T(1) : d);  // g'(0) = 0 and g''(0)/2 = 0
    G1[p] = zero ? T(0) : (p == 2 ? sub_rn(g[3], g[2]) : g[p + 1] - g[p]) * r;
    HL[p] = zero ? T(0) : (G1[p] - gp[p]) * r;
    HR[p] = zero ? T(0) : (gp[p + 1] - G1[p]) * r;
  }
  // the clustered pairs, one after the other whichever they are (at most two: the lanes of a warp
  // share the loop, where a series at each of the three places ran in nearly every warp)
  unsigned cm = (cl[0] ? 1u : 0u) | (cl[1] ? 2u : 0u) | (cl[2] ? 4u : 0u);
#pragma unroll 1
  while (cm) {
    const bool c0 = cm & 1u, c1 = (cm & 3u) == 2u;
    const T a = c0 ? u[0] : (c1 ? u[1] : u[2]), b = c0 ? u[1] : (c1 ? u[2] : u[3]);
    const T Lp = c0 ? L[0] : (c1 ? L[1] : L[2]), gpp = c0 ? gp[0] : (c1 ? gp[1] : gp[2]);
    const T d = b - a, y = d * rcp(a);
    const T g2 = T(6) * a * Lp + T(5) * a, g3 = T(6) * Lp + T(11);
    // T_4 = a y^2 / 4; successive terms: T_{k+1} = -T_k (k-3) y / (k+1)
    T t = T(0.25) * a * y * y;
    T s0 = T(0), s1 = T(0);
#pragma unroll 1
    for (int k = 4; k < 4 + Num<T>::kmax; ++k) {
      s0 += t;
      s1 += T(k - 1) * t;
      if (tabs(t) <= Num<T>::tol * (tabs(s0) + tabs(g2) + tabs(g3))) break;
      t *= -T(k - 3) * y / T(k + 1);
    }
    const T hl = T(0.5) * g2 + d * g3 * T(1.0 / 6.0) + s0, hr = T(0.5) * g2 + d * g3 * T(1.0 / 3.0) + s1;
    const T g1 = gpp + d * (T(0.5) * g2 + d * g3 * T(1.0 / 6.0) + s0);
    const bool c2 = !c0 && !c1;
    G1[0] = c0 ? g1 : G1[0], HL[0] = c0 ? hl : HL[0], HR[0] = c0 ? hr : HR[0];
    G1[1] = c1 ? g1 : G1[1], HL[1] = c1 ? hl : HL[1], HR[1] = c1 ? hr : HR[1];
    G1[2] = c2 ? g1 : G1[2], HL[2] = c2 ? hl : HL[2], HR[2] = c2 ? hr : HR[2];
    cm &= cm - 1u;
  }
  const T r02 = rcp(u[2] - u[0]), r13 = rcp(u[3] - u[1]), r03 = rcp(u[3] - u[0]);
  const T G012 = (G1[1] - G1[0]) * r02, G123 = (G1[2] - G1[1]) * r13;
  const T G0123 = (G123 - G012) * r03;
  T R[4];
  {  // j = 0
    const T h02 = (G012 - HL[0]) * r02;
    R[0] = (G0123 - h02) * r03;
  }
  {  // j = 1
    const T h02 = (HL[1] - HR[0]) * r02, h13 = (G123 - HL[1]) * r13;
    R[1] = (h13 - h02) * r03;
  }
  {  // j = 2
    const T h02 = (HR[1] - G012) * r02, h13 = (HL[2] - HR[1]) * r13;
    R[2] = (h13 - h02) * r03;
  }
  {  // j = 3
    const T h13 = (HR[2] - G123) * r13;
    R[3] = (h13 - G0123) * r03;
  }
  out = (f[0] * R[0] + f[1] * R[1] + f[2] * R[2] + f[3] * R[3]) * si;
  return true;
}

// The case inv_sum_shared leaves most often, in FP64: three knots B of one sign together (adjacent
// ones within kRhoShared) and the fourth, A, apart.  With L = ln|c|, c = mean(B), e = (B - c)/c,
//   g[n + 1 knots of B] = c^(3-n) (sum_{k=n..3} G_k h_{k-n}(e) + sum_{k>=4} K_k h_{k-n}(e)),
//   G_1 = 3 L + 1, G_2 = 3 L + 5/2, G_3 = L + 11/6, K_k = 6 (-1)^k / (k (k-1) (k-2) (k-3)),
// so one loop over the degree gives g[B1,B2], g[B1,B2,B3] and g[B1,B2,B3,Bj] for every j, and the
// entries with A follow by the difference recursion, whose gaps to A are wide.  Three logarithms and
// some 20 terms, where the per-vertex tables sum up to six Taylor series for each of four vertices
// (2400 FP64 operations against 500).
__device__ __forceinline__ bool inv_sum_triple(const double x[4], const double f[4], double &out) {
  const double s = tabs(x[0]) > tabs(x[3]) ? tabs(x[0]) : tabs(x[3]);
  if (!(s > 0.0)) return false;
  const double si = rcp_nr(s);
  double u[4];
  bool cl[3];
#pragma unroll
  for (int i = 0; i < 4; ++i) u[i] = x[i] * si;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double a = u[i], b = u[i + 1];
    cl[i] = (a > 0.0 && b - a <= kRhoShared * a) || (b < 0.0 && b - a <= kRhoShared * (-b));
  }
  if (!cl[1] || cl[0] == cl[2]) return false;
  const bool low = cl[0];  // the lower three are together
  const double A = low ? u[3] : u[0], fA = low ? f[3] : f[0];
  const double B[3] = {low ? u[0] : u[1], low ? u[1] : u[2], low ? u[2] : u[3]};
  const double fB[3] = {low ? f[0] : f[1], low ? f[1] : f[2], low ? f[2] : f[3]};
  const double c = (B[0] + B[1] + B[2]) * (1.0 / 3.0), ci = rcp_nr(c);
  double e[3];
  float em = 0.0f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    e[i] = fma(B[i], ci, -1.0);
    em = fmaxf(em, fabsf((float)e[i]));
  }
  const double L = log(tabs(c));
  // terms: e^n at 2^-58 (the kernel's unit roundoff with the growth of h_m on top)
  int n = 2;
  if (em > 1e-17f) n += (int)(-58.0f / __log2f(em < 0.5f ? em : 0.5f));
  double h1 = 1.0, h2 = 1.0, h3 = 1.0, p0 = 1.0, p1 = 1.0, p2 = 1.0;  // h_m of e1; e1,e2; e1..e3; and of e1..e3, ej
  double s1 = 3.0 * L + 1.0, s2 = 3.0 * L + 2.5, s30 = L + 11.0 / 6.0, s31 = s30, s32 = s30;
  for (int m = 1; m <= n; ++m) {
    h1 = e[0] * h1;
    h2 = h1 + e[1] * h2;
    h3 = h2 + e[2] * h3;
    p0 = h3 + e[0] * p0;
    p1 = h3 + e[1] * p1;
    p2 = h3 + e[2] * p2;
    // K_k = taylor_coef(k - 4)
    const double k3 = taylor_coef<double>(m - 1);
    const double k2 = m == 1 ? L + 11.0 / 6.0 : taylor_coef<double>(m - 2 < 0 ? 0 : m - 2);
    const double k1 = m == 1 ? 3.0 * L + 2.5 : (m == 2 ? L + 11.0 / 6.0 : taylor_coef<double>(m - 3 < 0 ? 0 : m - 3));
    s1 += k1 * h2;
    s2 += k2 * h3;
    s30 += k3 * p0;
    s31 += k3 * p1;
    s32 += k3 * p2;
  }
  const double g1 = c * c * s1, g2 = c * s2;
  const double r1 = rcp_nr(B[0] - A), r2 = rcp_nr(B[1] - A), r3 = rcp_nr(B[2] - A);
  const double LA = A == 0.0 ? 0.0 : log(tabs(A)), A2 = A * A;
  const double a1 = (g0(B[0]) - A2 * A * LA) * r1, a2 = (g1 - a1) * r2, a3 = (g2 - a2) * r3;
  const double d1 = (a1 - (3.0 * A2 * LA + A2)) * r1, d2 = (a2 - d1) * r2, d3 = (a3 - d2) * r3;
  out = (fA * d3 + fB[0] * ((s30 - a3) * r1) + fB[1] * ((s31 - a3) * r2) + fB[2] * ((s32 - a3) * r3)) * si;
  return true;
}

// The same case in FP32, entry by entry as the per-vertex table has it (same expansions, same
// differences, so the same roundings: in FP32 the closed form above has 1.5
// times the table's error).  The three knots B lie within kRho and A beyond it, so the table's entries
// inside B are Taylor series and those with A differences; each is formed once, where the four
// vertices of the table repeat them: seven series instead of eighteen, and no search for which entry
// is which (10^6 entries: 0.1 ms, the table 0.55).
// M entries of N + 1 knots each in one loop (independent chains: the kernels are bound by dependent
// latency), until all have converged.
template <int N, int M> __device__ __forceinline__ void dd_series(float (&e)[M][N + 1], float (&out)[M]) {
  float c[M], L[M], h[M][N + 1] = {}, low[M], high[M], prev[M], big[M];
  auto up = [&](int m) {
    h[m][0] = e[m][0] * h[m][0];
#pragma unroll
    for (int l = 1; l <= N; ++l) h[m][l] = h[m][l - 1] + e[m][l] * h[m][l];
  };
#pragma unroll
  for (int m = 0; m < M; ++m) {
    c[m] = e[m][0];
#pragma unroll
    for (int l = 1; l <= N; ++l) c[m] += e[m][l];
    c[m] = c[m] / float(N + 1);
    const float ci = rcp(c[m]);
#pragma unroll
    for (int l = 0; l <= N; ++l) {
      e[m][l] = (e[m][l] - c[m]) * ci;
      h[m][l] = 1.0f;
    }
    L[m] = Num<float>::lg(tabs(c[m]));
    low[m] = high[m] = prev[m] = big[m] = 0.0f;
    float cp = 1.0f;
#pragma unroll
    for (int k = N; k < 4; ++k) {
      if (k > N) {
        up(m);
        cp *= c[m];
      }
      low[m] += glow(k, c[m], L[m]) * cp * h[m][N];
    }
  }
#pragma unroll 1
  for (int k = 4; k < N + Num<float>::kmax; ++k) {
    const float coef = taylor_coef<float>(k - 4);
    bool more = k < 5 || k - N < 2;
#pragma unroll
    for (int m = 0; m < M; ++m) {
      up(m);
      const float term = coef * h[m][N];
      high[m] += term;
      big[m] = tabs(term) > big[m] ? tabs(term) : big[m];
      more = more || tabs(term) + tabs(prev[m]) > Num<float>::tol * (tabs(high[m]) > big[m] ? tabs(high[m]) : big[m]);
      prev[m] = term;
    }
    if (!more) break;
  }
#pragma unroll
  for (int m = 0; m < M; ++m) out[m] = low[m] + (N == 1 ? c[m] * c[m] : (N == 2 ? c[m] : 1.0f)) * high[m];
}
__device__ __forceinline__ bool within_rho(float a, float b) {
  const float rho = float(kRho);
  return (a > 0.0f && b - a <= rho * a) || (b < 0.0f && b - a <= rho * (-b));
}
__device__ __forceinline__ bool inv_sum_triple_table(const float x[4], const float f[4], float &out) {
  const float s = tabs(x[0]) > tabs(x[3]) ? tabs(x[0]) : tabs(x[3]);
  if (!(s > 0.0f)) return false;
  const float si = 1.0f / s;
  float u[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) u[i] = x[i] * si;
  const bool low = within_rho(u[0], u[2]);  // the lower three are together
  if (low == within_rho(u[1], u[3]) || within_rho(u[low ? 2 : 0], u[low ? 3 : 1])) return false;
  const float A = low ? u[3] : u[0];
  const float B0 = low ? u[0] : u[1], B1 = low ? u[1] : u[2], B2 = low ? u[2] : u[3];
  // C: the knots of B, the one next to A last
  const float C0 = low ? B0 : B2, C2 = low ? B2 : B0;
  const float lo = low ? B1 : B0, hi = low ? B2 : B1;  // C1 and C2 ascending
  float e1[1][2] = {{lo, hi}}, p1[1];                  // g[C1, C2]
  dd_series<1, 1>(e1, p1);
  float e2[3][3] = {{B0, B1, B2}, {lo, B1, hi}, {lo, C2, hi}}, p2[3];  // g[B], g[C1, C1, C2], g[C1, C2, C2]
  dd_series<2, 3>(e2, p2);
  float e3[3][4] = {{B0, B0, B1, B2}, {B0, B1, B1, B2}, {B0, B1, B2, B2}}, p3[3];
  dd_series<3, 3>(e3, p3);
  const float p = p1[0], t = p2[0], d1 = p2[1], d2 = p2[2], v0 = p3[0], v1 = p3[1], v2 = p3[2];
  const float dc = glow(1, C2, Num<float>::lg(tabs(C2)));
  const float da = A == 0.0f ? 0.0f : glow(1, A, Num<float>::lg(tabs(A)));
  const float a0 = A - C0, a1 = A - B1, a2 = A - C2;
  const float q1 = sub_rn(g0(A), g0(C2)) / a2;            // g[C2, A]
  const float q2 = sub_rn(q1, p) / a1;                    // g[C1, C2, A]
  const float q3 = sub_rn(q2, t) / a0;                    // g[C0, C1, C2, A]
  const float r0 = sub_rn(q3, low ? v0 : v2) / a0;        // C0 twice
  const float r1 = sub_rn(sub_rn(q2, d1) / a1, v1) / a0;  // C1 twice
  const float r2 = sub_rn(sub_rn(sub_rn(q1, dc) / a2, d2) / a1, low ? v2 : v0) / a0;  // C2 twice
  const float ra = sub_rn(sub_rn(sub_rn(da, q1) / a2, q2) / a1, q3) / a0;  // A twice
  float acc = f[0] * (low ? r0 : ra);
  acc += f[1] * (low ? r1 : r2);
  acc += f[2] * (low ? r2 : r1);
  acc += f[3] * (low ? ra : r0);
  out = acc * si;
  return true;
}

// series branch: sorted knots of one sign with (x3 - x0) <= kappa |x0 + x3|
template <typename T> __device__ __forceinline__ bool series_ok(const T x[4], T kappa) {
  return (x[0] > T(0) || x[3] < T(0)) && (x[3] - x[0]) <= kappa * tabs(x[0] + x[3]);
}

// Mixed precision, knots of a final tetrahedron that missed the short series: the D = 0
// value of a vertex on both cut planes, interpolated in FP32 along different edges, comes
// out at the FP32 noise level of the corner energies instead of 0, so knots below 2^-20 of
// the largest are set to exactly 0 (the piece's integral moves by ~1e-5 relative; such
// pieces are a few in 10^4).  Returns true when the sorted knots keep an inner gap below
// tau times their scale (the near-degenerate case evaluated in FP64).
constexpr float kZeroSnap = 9.5367431640625e-07f;  // 2^-20
__device__ __forceinline__ bool mixed_knots(float x[4], const float d[4], float tau) {
  const float s = fmaxf(fabsf(d[0]), fabsf(d[3]));
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = fabsf(d[i]) < kZeroSnap * s ? 0.0f : d[i];
  float g = s;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float gi = x[i + 1] - x[i];
    if (gi > 0.0f) g = fminf(g, gi);  // exact ties (e.g. two D = 0 vertices) are exact in FP32
  }
  return g < tau * s;
}

// Far-field moments of a final tetrahedron (sorted knots d >= 0, midpoint c > 0):
//   a_k = (-1)^k 6 k!/(k+4)! sum_j f_j h_k(e_1..e_4, e_j),  e = (d - c)/c,
// so that for any frequency w with rho = max|d - c| / |c - w| < 1
//   (1/V) sum_j f_j int_S lambda_j / (D - w) = (1/(c - w)) sum_k a_k z^k,  z = c / (c - w)
// (expansion of 1/(D - w) about c; at w = 0 this is the static series).  Writes a_0..a_{K-1}
// and returns K, the count after which |a_k| (times the largest z used, kappa c / max|d-c|)
// falls below tol.
template <typename T, int KMAX> __device__ int far_moments(const T d[4], const T f[4], T *a) {
  const T c = (d[0] + d[3]) * T(0.5);
  const T ci = rcp(c);
  T e[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) e[l] = (d[l] - c) * ci;
  const T rmax = (d[3] - d[0]) * T(0.5) * ci;           // max|e|
  const T zmax = rmax > T(0) ? T(Num<T>::kappa_far) / rmax : T(1);  // largest |z| that uses them
  T H[4] = {T(1), T(1), T(1), T(1)};
  T P[4] = {T(1), T(1), T(1), T(1)};
  a[0] = T(0.25) * (f[0] + f[1] + f[2] + f[3]);
  const T ref = tabs(a[0]);
  T zk = T(1), prev = ref;
  int k = 1;
  for (; k < KMAX; ++k) {
    H[0] = e[0] * H[0];
#pragma unroll
    for (int l = 1; l < 4; ++l) H[l] = H[l - 1] + e[l] * H[l];
    T sj = T(0);
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      P[jj] = H[3] + e[jj] * P[jj];
      sj += f[jj] * P[jj];
    }
    a[k] = series_coef<T>(k) * sj;
    zk *= zmax;
    const T mag = tabs(a[k]) * zk;
    if (k >= 2 && mag + prev <= Num<T>::tol * ref) {
      ++k;
      break;
    }
    prev = mag;
  }
  return k;
}

// (1/(c - w)) sum_{k<kk} a_k z^k, z = c/(c - w), as two half-length Horner chains (even and
// odd powers: the weight kernels are bound by dependent latency); on the device, FP32
// coefficients are read in aligned pairs (a + k - 1 even: the caller's stride is even)
template <typename T> __device__ __forceinline__ T far_eval_k(const T *a, int kk, T c, T w) {
  const T den = c - w, rd = rcp(den);
  const T z = c * rd, z2 = z * z;
  T e = T(0), o = T(0);
  int k = kk - 1;
  if (k >= 0 && (k & 1) == 0) e = a[k--];
#pragma unroll 2
  for (; k >= 1; k -= 2) {
    T lo_, hi_;
#ifdef __CUDA_ARCH__
    if constexpr (sizeof(T) == 4) {
      const float2 pr = *reinterpret_cast<const float2 *>(a + k - 1);
      lo_ = pr.x;
      hi_ = pr.y;
    } else {
      lo_ = a[k - 1];
      hi_ = a[k];
    }
#else
    lo_ = a[k - 1];
    hi_ = a[k];
#endif
    o = o * z2 + hi_;
    e = e * z2 + lo_;
  }
  return (e + z * o) * rd;
}

// sum_j f_j (1/V) int_S lambda_j delta(X) = (1/4) sum_j f_j M(0; x, x_j) for sorted knots x, M the cubic
// B-spline density with knot j doubled, with the reciprocals rs of the knot spans 01, 12, 23, 02, 13, 03
// given (of the unshifted knots): the de Boor-Cox recursion per vertex, multiplying by the reciprocal
// spans instead of dividing.  (The B-spline recursion combines nonnegative terms, so spans from the
// unshifted knots cost no accuracy; the divided-difference table of the principal value keeps the
// differences of its own rounded knots.)
template <typename T> __device__ __forceinline__ T delta_sum_pre(const T x[4], const T f[4], const T rs[6]) {
  if (!(x[0] < T(0) && x[3] > T(0))) return T(0);
  // reciprocal span of original knots a <= b (0 for a == b)
  auto R = [&](int a, int b) -> T {
    if (a == b) return T(0);
    const int k = b - a;
    return k == 1 ? rs[a] : (k == 2 ? rs[3 + a] : rs[5]);
  };
  T acc = T(0);
#pragma unroll
  for (int jj = 0; jj < 4; ++jj) {
    int id[5];
    T t[5];
#pragma unroll
    for (int l = 0; l < 5; ++l) {
      id[l] = l <= jj ? l : l - 1;
      t[l] = x[id[l]];
    }
    T M[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) M[i] = (t[i] <= T(0) && T(0) < t[i + 1]) ? R(id[i], id[i + 1]) : T(0);
#pragma unroll
    for (int k = 2; k <= 4; ++k) {
#pragma unroll
      for (int i = 0; i + k <= 4; ++i) {
        const T den = t[i + k] - t[i];
        M[i] = den > T(0) ? (T(k) / T(k - 1)) * ((-t[i]) * M[i] + t[i + k] * M[i + 1]) * R(id[i], id[i + k]) : T(0);
      }
    }
    acc += f[jj] * M[0];
  }
  return T(0.25) * acc;
}

// sum_j f_j (1/V) int_S lambda_j delta(X) for sorted knots x with x_0 < 0 < x_3, spans e_j - e_i from
// the unshifted knots e: the plane X = 0 cuts S in a triangle around vertex 0 (x_1 >= 0) or 3
// (x_2 <= 0), or in a quadrilateral, split by the diagonal between edges 03 and 12; f is linear,
// so each triangle contributes its share of the density (the nonnegative terms of the quadratic
// B-spline's recursion) times the mean of f at its three vertices.  A quarter of the operations of
// the per-vertex cubic recursions of delta_sum_pre.
template <typename T> __device__ __forceinline__ T delta_section(const T x[4], const T e[4], const T f[4]) {
  const T r30 = rcp_nr(e[3] - e[0]);
  const T f03 = f[0] - x[0] * r30 * (f[3] - f[0]);  // f on edge 03 (fraction (0 - x_0)/(x_3 - x_0))
  if (x[1] < T(0) && x[2] > T(0)) {
    const T r20 = rcp_nr(e[2] - e[0]), r21 = rcp_nr(e[2] - e[1]), r31 = rcp_nr(e[3] - e[1]);
    const T f02 = f[0] - x[0] * r20 * (f[2] - f[0]), f12 = f[1] - x[1] * r21 * (f[2] - f[1]);
    const T f13 = f[1] - x[1] * r31 * (f[3] - f[1]);
    const T a = -x[0] * x[2] * r20, b = -x[1] * x[3] * r31, m = f03 + f12;
    return (a * (f02 + m) + b * (f13 + m)) * r21 * r30;
  }
  // around vertex 0 or 3: edges to the other three
  const bool lo = x[1] >= T(0);
  const T p = lo ? x[0] : x[3], fp = lo ? f[0] : f[3], ep = lo ? e[0] : e[3];
  const T u = lo ? e[1] : e[2], fu = lo ? f[1] : f[2], v = lo ? e[2] : e[1], fv = lo ? f[2] : f[1];
  const T ru = rcp_nr(u - ep), rv = rcp_nr(v - ep);
  const T fa = fp - p * ru * (fu - fp), fb = fp - p * rv * (fv - fp);
  return p * ru * p * rv * r30 * (f03 + fa + fb);
}

// Tetrahedron density of states at eF for one band: M(0; a_0..a_3), quadratic B-spline
template <typename T> __device__ __forceinline__ T dos4(T a0, T a1, T a2, T a3) {
  T t[4] = {a0, a1, a2, a3};
  T dm[4] = {T(0), T(0), T(0), T(0)};
  sort4(t, dm);
  if (!(T(0) >= t[0] && T(0) < t[3])) return T(0);
  T M[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) M[i] = (t[i] <= T(0) && T(0) < t[i + 1]) ? T(1) / (t[i + 1] - t[i]) : T(0);
#pragma unroll
  for (int k = 2; k <= 3; ++k) {
#pragma unroll
    for (int i = 0; i + k <= 3; ++i) {
      const T den = t[i + k] - t[i];
      M[i] = den > T(0) ? T(k) * ((T(0) - t[i]) * M[i] + (t[i + k] - T(0)) * M[i + 1]) /
                              (T(k - 1) * den)
                        : T(0);
    }
  }
  return M[0];
}

// ------------------------------------------------------------------------------------
// carving (Sec. II, Fig. 1): the part of a tetrahedron where a key is negative, first key a (occupied
// states), then key -b (empty states at k+q), without branches.  Every piece of a cut has at most three
// vertices on the cut plane, and its volume ratio is the product, over them, of the cut fraction
// t or of 1 - t.  A recipe names them: three slots (i, j, flip) for the point where the key
// vanishes on edge i (key < 0) - j, and the original vertex of the fourth slot; a slot with i = j
// stands for vertex i itself (t = 0, flip: factor 1).  One table of recipes, indexed by the set of
// vertices with key < 0 and the piece number: the lanes of a warp all run the same code, where
// branching on the vertex count runs the one-, two- and three-vertex cases one after the other (ten
// cut points for a piece's three), and the vertices need no sorting (only which side they are on
// matters: FP64; the FP32 callers sort them by key all the same, which keeps the rounding errors of their
// near-degenerate pieces those of a cut of sorted vertices).
// ------------------------------------------------------------------------------------
constexpr unsigned cut_recipe(int mask, int idx) {
  int N[4] = {}, P[4] = {}, nn = 0, np = 0;
  for (int i = 0; i < 4; ++i)
    if ((mask >> i) & 1) N[nn++] = i;
    else P[np++] = i;
  int s[3][3] = {}, last = 0;
  auto set = [&](int k, int i, int j, int flip) {
    s[k][0] = i;
    s[k][1] = j;
    s[k][2] = flip;
  };
  const int a = N[0], b = N[1], c = N[2], p = P[0], q = P[1], r = P[2];
  if (nn == 1) {  // corner tetrahedron
    set(0, a, p, 0);
    set(1, a, q, 0);
    set(2, a, r, 0);
    last = a;
  } else if (nn == 2) {  // prism (a, ap, aq) - (b, bp, bq)
    last = b;
    if (idx == 0) {
      set(0, a, p, 0);
      set(1, a, q, 0);
      set(2, a, a, 1);
    } else if (idx == 1) {
      set(0, a, p, 1);
      set(1, a, q, 0);
      set(2, b, p, 0);
    } else {
      set(0, a, q, 1);
      set(1, b, p, 0);
      set(2, b, q, 0);
    }
  } else if (nn == 3) {  // prism (a, b, c) - (ap, bp, cp)
    last = c;
    set(0, a, p, idx == 0 ? 0 : 1);
    if (idx == 0) set(1, a, a, 1);
    else set(1, b, p, idx == 1 ? 0 : 1);
    if (idx < 2) set(2, b, b, 1);
    else set(2, c, p, 0);
  } else {  // nothing cut
    set(0, 0, 0, 1);
    set(1, 1, 1, 1);
    set(2, 2, 2, 1);
    last = 3;
  }
  unsigned v = 0;
  for (int k = 0; k < 3; ++k) v |= (unsigned)(s[k][0] | (s[k][1] << 2) | (s[k][2] << 4)) << (5 * k);
  return v | ((unsigned)last << 15);
}
struct CutTab {
  unsigned v[64];
  constexpr CutTab() : v() {
    for (int m = 0; m < 16; ++m)
      for (int i = 0; i < 3; ++i) v[m * 4 + i] = cut_recipe(m, i);
  }
};
__constant__ constexpr CutTab kCutTab{};  // (copied to shared memory: lanes index it apart)
// pieces of a cut by the number of vertices kept
__device__ __forceinline__ int cut_count(unsigned mask) {
  const int n = (int)((0x4332322132212110ull >> (4 * mask)) & 7ull);  // bits set
  return n == 0 ? 0 : ((n == 1 || n == 4) ? 1 : 3);
}
template <typename T> __device__ __forceinline__ T sel4(const T v[4], unsigned i) {
  const T a = (i & 1u) ? v[1] : v[0], b = (i & 1u) ? v[3] : v[2];
  return (i & 2u) ? b : a;
}
__device__ __forceinline__ float cut_quot(float a, float b) { return quot(a, b); }
__device__ __forceinline__ double cut_quot(double a, double b) { return a * rcp_nr(b); }
// cut fraction of slot k (0 for an unused slot) and the values at its vertex.  FP64 key differences below
// 2^-1022 have no finite reciprocal.  They are scaled here, exactly; or the caller's keys come scaled
// (SCALED), which costs the FP64 static weights nothing where this test took 1.4% of them.
template <typename T> constexpr T kKeyScale = sizeof(T) == 8 ? T(18446744073709551616.0) : T(1);  // 2^64
template <bool SCALED = false, typename T> __device__ __forceinline__ T cut_frac(unsigned rec, int k, const T key[4]) {
  const unsigned sl = rec >> (5 * k);
  T ki = sel4(key, sl & 3u), den = ki - sel4(key, (sl >> 2) & 3u);
  if constexpr (sizeof(T) == 8 && !SCALED) {
    if (Mean<T>::bits(den) < 0x00100000) {
      ki *= kKeyScale<T>;
      den *= kKeyScale<T>;
    }
  }
  return den != T(0) ? cut_quot(ki, den) : T(0);
}
template <typename T> __device__ __forceinline__ T cut_mix(unsigned rec, int k, const T v[4], T t) {
  const unsigned sl = rec >> (5 * k);
  return (T(1) - t) * sel4(v, sl & 3u) + t * sel4(v, (sl >> 2) & 3u);
}
__device__ __forceinline__ bool cut_used(unsigned rec, int k) {
  const unsigned sl = rec >> (5 * k);
  return (sl & 3u) != ((sl >> 2) & 3u);
}
template <typename T> __device__ __forceinline__ T cut_factor(unsigned rec, int k, T t) {
  return ((rec >> (5 * k + 4)) & 1u) ? T(1) - t : t;
}
// x < 0 (FP64: on the integer pipe; false for -0 and NaN)
__device__ __forceinline__ bool is_neg(float x) { return x < 0.0f; }
__device__ __forceinline__ bool is_neg(double x) {
#ifdef __CUDA_ARCH__
  const long long b = __double_as_longlong(x);
  return b < 0 && ((unsigned long long)b << 1) - 1ull < 0xFFE0000000000000ull;
#else
  return x < 0.0;
#endif
}

// x - y = s + t exactly (Knuth's two-difference; any order of magnitudes)
__device__ __forceinline__ void two_diff(float x, float y, float &s, float &t) {
  s = x - y;
  const float bb = s - x;
  t = (x - (s - bb)) - (y + bb);
}

// ------------------------------------------------------------------------------------
// dynamic weights (chi0_dynamic.cu): moments of a piece, its near pairs and delta term
// ------------------------------------------------------------------------------------
// s_k = [z^k] N(z)/Q(z)^2 of a piece, one after the other (k = 0, 1, ...): Q in the quadratic
// factors of the end and of the middle knots, two divisions by each
template <typename T> struct Moments {
  T A, B, C, D;        // 1 - A z + B z^2 (e_0, e_3), 1 - C z + D z^2 (e_1, e_2)
  T n[4];
  T x1, x2, y1, y2, u1, u2, v1, v2;  // the stages' last two values
  __device__ __forceinline__ Moments(const T e[4], const T f[4]) {
    A = e[0] + e[3];
    B = e[0] * e[3];
    C = e[1] + e[2];
    D = e[1] * e[2];
    const T E1 = A + C, E2 = (B + D) + A * C, E3 = B * C + D * A;
    const T g0 = f[0] * e[0], g1 = f[1] * e[1], g2 = f[2] * e[2], g3 = f[3] * e[3];
    const T h0 = g0 * e[0], h1 = g1 * e[1], h2 = g2 * e[2], h3 = g3 * e[3];
    const T m0 = (f[0] + f[1]) + (f[2] + f[3]), m1 = (g0 + g1) + (g2 + g3), m2 = (h0 + h1) + (h2 + h3);
    const T m3 = (h0 * e[0] + h1 * e[1]) + (h2 * e[2] + h3 * e[3]);
    n[0] = m0;
    n[1] = m1 - E1 * m0;
    n[2] = m2 + (E2 * m0 - E1 * m1);
    n[3] = m3 + (E2 * m1 - E1 * m2) - E3 * m0;
    x1 = x2 = y1 = y2 = u1 = u2 = v1 = v2 = T(0);
  }
  __device__ __forceinline__ T next(T in) {
    const T x = in + (A * x1 - B * x2);
    const T y = x + (A * y1 - B * y2);
    const T u = y + (C * u1 - D * u2);
    const T v = u + (C * v1 - D * v2);
    x2 = x1, x1 = x;
    y2 = y1, y1 = y;
    u2 = u1, u1 = u;
    v2 = v1, v1 = v;
    return v;
  }
};

// The same s_k (k = 1, 2, ...) by the complete homogeneous polynomials h_k(e_1..e_4, e_j) of every
// vertex: the FP32 kernel's form.  Thirteen operations a moment instead of eight, but shorter
// chains and fewer registers: the 64 x 64 x 16 pass takes 6.8 ms with it, 7.4 ms with Moments.
template <typename T> struct MomentsH {
  T e[4], f[4], H[4], P[4];
  __device__ __forceinline__ MomentsH(const T e_[4], const T f_[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      e[i] = e_[i];
      f[i] = f_[i];
      H[i] = P[i] = T(1);
    }
  }
  __device__ __forceinline__ T next() {
    H[0] = e[0] * H[0];
#pragma unroll
    for (int l = 1; l < 4; ++l) H[l] = H[l - 1] + e[l] * H[l];
    T s = T(0);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      P[j] = H[3] + e[j] * P[j];
      s += f[j] * P[j];
    }
    return s;
  }
};

// the delta term of a near pair: FP64 by the plane section; FP32 by the cubic recursion, whose
// rounding (a relative 2.9e-8 common to every piece, from its 4/3) its results have always carried
__device__ __forceinline__ double delta_term(const double x[4], const double e[4], const double f[4]) {
  return delta_section(x, e, f);
}
__device__ __forceinline__ float delta_term(const float x[4], const float e[4], const float f[4]) {
  const float rs[6] = {rcp(e[1] - e[0]), rcp(e[2] - e[1]), rcp(e[3] - e[2]),
                       rcp(e[2] - e[0]), rcp(e[3] - e[1]), rcp(e[3] - e[0])};
  return delta_sum_pre(x, f, rs);
}

// sum_j f_j (1/V) int lambda_j / X for knots x of X near 0: divided-difference table (principal
// value across X = 0); one out-of-line copy
template <bool FP64>
__device__ __noinline__ typename std::conditional<FP64, double, float>::type near_term(
    const typename std::conditional<FP64, double, float>::type *x,
    const typename std::conditional<FP64, double, float>::type *f, float tau, int &nfp64) {
  using T = typename std::conditional<FP64, double, float>::type;
  T xx[4] = {x[0], x[1], x[2], x[3]};
  // (the entries that reach this function are the ones the shared table left: the per-vertex
  // table directly, after the series branches)
  if constexpr (FP64) {
    double v;
    if (series_ok(xx, T(Num<T>::kappa))) return series_sum(xx, f);
    if (inv_sum_triple(xx, f, v)) return v;
    return inv_sum_table(xx, f);
  } else {
    if (series_ok(xx, Num<float>::kappa)) return series_sum(xx, f);
    float y[4];
    if (!mixed_knots(y, xx, tau)) {
      float v;
      if (series_ok(y, Num<float>::kappa_long)) return series_sum(y, f);
      if (inv_sum_triple_table(y, f, v)) return v;
      return inv_sum_table(y, f);
    }
    ++nfp64;
    double yd[4] = {y[0], y[1], y[2], y[3]}, fd[4] = {f[0], f[1], f[2], f[3]}, v;
    if (inv_sum_triple(yd, fd, v)) return (float)v;
    return (float)inv_sum_table(yd, fd);
  }
}

// D0 - w for a frequency near the knots: with D0 = D0h + D0l and w = wh + wl split into
// FP32 parts the difference keeps full relative precision however close D0 is to w
__device__ __forceinline__ float near_shift(float D0h, float D0l, float wh, float wl) {
  float sv, tv;
  two_diff(D0h, wh, sv, tv);
  return sv + (tv + (D0l - wl));
}
__device__ __forceinline__ double near_shift(double D0h, double, double wh, double) { return D0h - wh; }

}  // namespace chi0dev

#ifndef __CUDACC__
#include "chi0_math_host.h"
#endif
