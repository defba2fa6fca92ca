// Host build of what the weight kernels run on one tetrahedron and one band pair, in their own
// sequence: cut recipes in the plain (static) and the offset form (dynamic), the series, the shared
// table and what it leaves, a piece's own moments, the delta term, and the boxes' moments and polynomials.
#include <algorithm>
#include <cmath>
#include <cstring>
using std::max;
using std::min;
#define __device__
#define __forceinline__ inline
#define __noinline__ __attribute__((noinline))
#define __constant__
#define __log2f log2f
#define __frcp_rn(x) (1.0f / (x))
#define __fdividef(a, b) ((a) / (b))
#include "../../paper_1407_3444_gb300/csrc/chi0_math.cuh"

using namespace chi0dev;

namespace {
constexpr float kTau = 9.5367431640625e-07f;  // 2^-20, the library default

template <typename T> unsigned side(const T key[4]) {
  unsigned m = 0u;
  for (int i = 0; i < 4; ++i) m |= (is_neg(key[i]) ? 1u : 0u) << i;
  return m;
}
int corner(unsigned rec, int k) { return (int)((rec >> (5 * k)) & 3u); }

// FP32: the vertices in ascending order of the key
template <typename T> void sort_key(T key[4], T x[4], T y[4]) {
  if (sizeof(T) == 8) return;
  auto sw = [&](int i, int j) {
    if (key[j] < key[i]) {
      std::swap(key[i], key[j]);
      std::swap(x[i], x[j]);
      if (y != x) std::swap(y[i], y[j]);
    }
  };
  sw(0, 1), sw(2, 3), sw(0, 2), sw(1, 3), sw(1, 2);
}

// emit(r, d, f) for every piece: keys a (scaled by S), D = D0 + e with e the attribute that is mixed;
// kb(a or 0, e): the second cut's key
template <bool SCALED, typename T, typename Key, typename Emit>
void pieces(const T a_[4], const T e_[4], const T f_[4], T D0, Key kb, Emit emit) {
  T la[4], le[4];
  for (int i = 0; i < 4; ++i) la[i] = a_[i], le[i] = e_[i];
  sort_key(la, le, le);
  const unsigned m1 = side(la);
  unsigned eb = 0u;
  bool dpos = true;
  for (int i = 0; i < 4; ++i) {
    eb |= (is_neg(kb(la[i], le[i])) ? 1u : 0u) << i;
    dpos = dpos && is_neg(-(D0 + le[i]));
  }
  for (int i1 = 0; i1 < cut_count(m1); ++i1) {
    unsigned rec = kCutTab.v[m1 * 4 + i1], m2 = 0u;
    for (int k = 0; k < 3; ++k) {
      const unsigned own = (eb >> corner(rec, k)) & 1u;
      if (dpos) m2 |= (cut_used(rec, k) ? 1u : own) << k;
      else {
        const T x = D0 + cut_mix(rec, k, le, cut_frac<SCALED>(rec, k, la));
        m2 |= (cut_used(rec, k) ? (is_neg(-x) ? 1u : 0u) : own) << k;
      }
    }
    m2 |= ((eb >> corner(rec, 3)) & 1u) << 3;
    if (sizeof(T) == 4) m2 = (1u << __builtin_popcount(m2)) - 1u;
    for (int i2 = 0; i2 < cut_count(m2); ++i2) {
      T a[4], e[4], f[4], key[4], e1[4], f1[4], d[4], g[4], r = T(1);
      for (int i = 0; i < 4; ++i) a[i] = a_[i], e[i] = e_[i], f[i] = f_[i];
      sort_key(a, e, f);
      rec = kCutTab.v[side(a) * 4 + i1];
      for (int k = 0; k < 3; ++k) {
        const T t = cut_frac<SCALED>(rec, k, a);
        e1[k] = cut_mix(rec, k, e, t);
        f1[k] = cut_mix(rec, k, f, t);
        key[k] = kb(cut_used(rec, k) ? T(0) : sel4(a, (unsigned)corner(rec, k)), e1[k]);
        r *= cut_factor(rec, k, t);
      }
      e1[3] = sel4(e, (unsigned)corner(rec, 3));
      f1[3] = sel4(f, (unsigned)corner(rec, 3));
      key[3] = kb(sel4(a, (unsigned)corner(rec, 3)), e1[3]);
      sort_key(key, e1, f1);
      rec = kCutTab.v[m2 * 4 + i2];
      for (int k = 0; k < 3; ++k) {
        const T t = cut_frac<SCALED>(rec, k, key);
        d[k] = cut_mix(rec, k, e1, t);
        g[k] = cut_mix(rec, k, f1, t);
        r *= cut_factor(rec, k, t);
      }
      d[3] = sel4(e1, (unsigned)corner(rec, 3));
      g[3] = sel4(f1, (unsigned)corner(rec, 3));
      for (int i = 0; i < 4; ++i) d[i] = d[i] > -D0 ? d[i] : -D0;
      if (r > T(0)) emit(r, d, g);
    }
  }
}

double static_piece(double r, double d[4], double f[4]) {
  double e[4], ci, v;
  const int tier = mean_tier<double, Mean<double>::tiers>(mean_offsets(d, e, ci));
  if (tier < Mean<double>::tiers) return r * mean_series(e, f, ci, tier);
  sort4(d, f);
  if (inv_sum_shared(d, f, v) || inv_sum_triple(d, f, v)) return r * v;
  double t = 0.0;
  for (int j = 0; j < 4; ++j) t += inv_term_table(d, f, j);
  return r * t;
}
double static_piece(float r, float d[4], float f[4]) {
  sort4(d, f);
  if (series_ok(d, Num<float>::kappa)) return (double)(r * series_sum_short(d, f));
  float y[4], v;
  double t = 0.0;
  if (!mixed_knots(y, d, kTau)) {
    if (series_ok(y, Num<float>::kappa_long)) return (double)(r * series_sum_short(y, f));
    if (inv_sum_shared(y, f, v)) return (double)(r * v);
    for (int j = 0; j < 4; ++j) t += (double)inv_term_table(y, f, j);
    return (double)r * t;
  }
  const double yd[4] = {y[0], y[1], y[2], y[3]}, fd[4] = {f[0], f[1], f[2], f[3]};
  double vd;
  if (inv_sum_triple(yd, fd, vd)) return (double)r * vd;
  for (int j = 0; j < 4; ++j) t += inv_term_table(yd, fd, j);
  return (double)r * t;
}

template <typename T> double static_tet(const double *a64, const double *b64, const double *f64) {
  constexpr T S = kKeyScale<T>;
  T a[4], D[4], f[4];
  for (int i = 0; i < 4; ++i) {
    D[i] = (T)b64[i] - (T)a64[i];
    a[i] = (T)a64[i] * S;
    f[i] = (T)f64[i];
  }
  double acc = 0.0;
  pieces<true, T>(a, D, f, T(0), [&](T k, T d) { return -(k + S * d); },
                  [&](T r, T d[4], T g[4]) { acc += static_piece(r, d, g); });
  return 2.0 * acc;
}

template <typename T> constexpr int kOwnTerms = sizeof(T) == 8 ? 40 : 32;

template <typename T> void dynamic_tet(const double *a64, const double *b64, const double *f64, int nw, const double *w,
                                       double *re, double *im) {
  constexpr bool FP64 = sizeof(T) == 8;
  constexpr int KO = kOwnTerms<T>;
  static constexpr ChebInv<double, 40> own(1.0 / 1.5);
  const T far = FP64 ? T(1.5) : T(2);
  T a[4], e[4], f[4], D0h = T(0), D0l = T(0);
  for (int i = 0; i < 4; ++i) a[i] = (T)a64[i], f[i] = (T)f64[i];
  if constexpr (FP64) {
    for (int i = 0; i < 4; ++i) e[i] = b64[i] - a64[i];
  } else {
    float al[4], bh[4], bl[4], sv, tv;
    for (int i = 0; i < 4; ++i) {
      al[i] = (float)(a64[i] - (double)a[i]);
      bh[i] = (float)b64[i];
      bl[i] = (float)(b64[i] - (double)bh[i]);
    }
    two_diff(bh[0], a[0], sv, tv);
    const float corr = tv + (bl[0] - al[0]);
    D0h = sv + corr;
    D0l = corr - (D0h - sv);
    e[0] = 0.0f;
    for (int i = 1; i < 4; ++i) {
      float sa, ta, sb, tb;
      two_diff(a[i], a[0], sa, ta);
      two_diff(bh[i], bh[0], sb, tb);
      e[i] = (sb - sa) + ((tb - ta) + ((bl[i] - bl[0]) - (al[i] - al[0])));
    }
  }
  for (int k = 0; k < nw; ++k) re[k] = im[k] = 0.0;
  pieces<false, T>(a, e, f, D0h, [&](T k, T x) { return -((k + D0h) + x); }, [&](T r, T ee[4], T ff[4]) {
    sort4(ee, ff);
    if (!(D0h + ee[3] > T(0))) return;
    const T half = (ee[3] - ee[0]) * T(0.5), mid = (ee[0] + ee[3]) * T(0.5), c = D0h + mid;
    T m[KO];
    int K = KO;
    if constexpr (FP64) {
      const T ri = half > T(0) ? rcp_nr(half) : T(0);
      T x[4];
      for (int i = 0; i < 4; ++i) x[i] = (ee[i] - mid) * ri;
      Moments<T> mm(x, ff);
      for (int k = 0; k < KO; ++k) m[k] = own.v[k] * mm.next(k < 4 ? mm.n[k] : T(0));
    } else {
      T d[4];
      for (int i = 0; i < 4; ++i) d[i] = D0h + ee[i];
      K = far_moments<T, KO>(d, ff, m);
    }
    int nf = 0;
    for (int k = 0; k < nw; ++k) {
      const T wh = (T)w[k], wl = (T)(w[k] - (double)wh);
      const T sh = near_shift(D0h, D0l, wh, wl);
      double v = 0.0;
      for (int plus = 0; plus < 2; ++plus) {
        const T den = plus ? c + wh : c - wh;
        if (tabs(den) > far * half) {
          if constexpr (FP64) {
            const T rd = rcp_nr(den), z = half * rd;
            T s = m[KO - 1];
            for (int j = KO - 2; j >= 0; --j) s = s * z + m[j];
            v += s * rd;
          } else {
            v += far_eval_k(m, K, c, plus ? -wh : wh);
          }
          continue;
        }
        T x[4], t;
        for (int i = 0; i < 4; ++i) x[i] = plus ? (D0h + ee[i]) + wh : sh + ee[i];
        v += inv_sum_shared(x, ff, t) ? t : near_term<FP64>(x, ff, kTau, nf);
      }
      re[k] += (double)r * v;
      T x[4];
      for (int i = 0; i < 4; ++i) x[i] = sh + ee[i];
      if (x[0] < T(0) && x[3] > T(0)) im[k] += (double)(r * delta_term(x, ee, ff)) * 3.141592653589793;
    }
  });
}

// FP32 kernel: MomentsH; FP64 kernel: Moments
template <int K, bool FP64> double box_share(const double e[4], const double f[4], double z, double den, double zmax) {
  const ChebInv<double, K> p(zmax);
  MomentsH<double> h(e, f);
  Moments<double> m(e, f);
  double M[K], s = 0.0;
  for (int k = 0; k < K; ++k)
    M[k] = FP64 ? series_coef<double>(k) * m.next(k < 4 ? m.n[k] : 0.0)
                : (k == 0 ? 0.25 * (f[0] + f[1] + f[2] + f[3]) : series_coef<double>(k) * h.next());
  for (int k = K - 1; k >= 0; --k) s = s * z + ((k & 1) ? -p.p_[k] : p.p_[k]) * M[k];
  return s / den;
}
}  // namespace

// (1/V) int_{a<0<b} 2 f / D over one tetrahedron (a = e_k - eF, b = e_{k+q} - eF)
extern "C" double host_static(const double *a, const double *b, const double *f, int fp64) {
  return fp64 ? static_tet<double>(a, b, f) : static_tet<float>(a, b, f);
}

// (1/V) int f [1/(D - w) + 1/(D + w)] (PV) and pi (1/V) int f delta(w - D), w >= 0
extern "C" void host_dynamic(const double *a, const double *b, const double *f, int fp64, int nw, const double *w,
                             double *re, double *im) {
  if (fp64) dynamic_tet<double>(a, b, f, nw, w, re, im);
  else dynamic_tet<float>(a, b, f, nw, w, re, im);
}

// a piece's share of Re at den = C -+ u by the moments of a box (centre C, radius R), one of the kernels'
// six polynomials
extern "C" double host_box(const double *d, const double *f, double C, double R, double den, int kind) {
  double e[4];
  for (int i = 0; i < 4; ++i) e[i] = (d[i] - C) / R;
  const double z = R / den;
  if (kind == 0) return box_share<20, false>(e, f, z, den, 1.0 / 2.0);
  if (kind == 1) return box_share<12, false>(e, f, z, den, 2.0 / 9.0);
  if (kind == 2) return box_share<20, false>(e, f, z, den, 5.0 / 9.0);
  if (kind == 3) return box_share<40, true>(e, f, z, den, 1.0 / 1.5);
  if (kind == 4) return box_share<18, true>(e, f, z, den, 2.0 / 9.0);
  return box_share<32, true>(e, f, z, den, 5.0 / 9.0);
}
