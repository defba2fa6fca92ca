// Host build of the static weight kernels' arithmetic (chi0_math.cuh) that has forms of its own:
// the cut recipes, the FP64 series about the mean and the FP32 series with the short recurrence,
// each next to the form it stands for.
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
void add(double r, const double D[4], const double f[4], double out[3]) {
  out[0] += r;
  out[1] += r * 0.25 * (f[0] + f[1] + f[2] + f[3]);
  out[2] += r * 0.25 * (D[0] + D[1] + D[2] + D[3]);
}
unsigned side(const double key[4]) {
  unsigned m = 0u;
  for (int i = 0; i < 4; ++i) m |= (is_neg(key[i]) ? 1u : 0u) << i;
  return m;
}
}  // namespace

// volume, int f and int D over the region a < 0 < a + D of one tetrahedron, summed over the pieces
// of the two cuts: by recipes
extern "C" void host_cut_recipes(const double *a, const double *D, const double *f, double *out) {
  out[0] = out[1] = out[2] = 0.0;
  const unsigned m1 = side(a);
  for (int i1 = 0; i1 < cut_count(m1); ++i1) {
    unsigned rec = kCutTab.v[m1 * 4 + i1];
    double key[4], D1[4], f1[4], r1 = 1.0;
    for (int k = 0; k < 3; ++k) {
      const double t = cut_frac(rec, k, a);
      D1[k] = cut_mix(rec, k, D, t);
      f1[k] = cut_mix(rec, k, f, t);
      key[k] = -(cut_used(rec, k) ? D1[k] : sel4(a, (rec >> (5 * k)) & 3u) + D1[k]);
      r1 *= cut_factor(rec, k, t);
    }
    D1[3] = sel4(D, (rec >> 15) & 3u);
    f1[3] = sel4(f, (rec >> 15) & 3u);
    key[3] = -(sel4(a, (rec >> 15) & 3u) + D1[3]);
    const unsigned m2 = side(key);
    for (int i2 = 0; i2 < cut_count(m2); ++i2) {
      rec = kCutTab.v[m2 * 4 + i2];
      double d[4], g[4], r = r1;
      for (int k = 0; k < 3; ++k) {
        const double t = cut_frac(rec, k, key);
        d[k] = cut_mix(rec, k, D1, t);
        g[k] = cut_mix(rec, k, f1, t);
        r *= cut_factor(rec, k, t);
      }
      d[3] = sel4(D1, (rec >> 15) & 3u);
      g[3] = sel4(f1, (rec >> 15) & 3u);
      add(r, d, g, out);
    }
  }
}

// the same by cut_piece
extern "C" void host_cut_pieces(const double *a, const double *D, const double *f, double *out) {
  out[0] = out[1] = out[2] = 0.0;
  Vt<double> V[4];
  for (int i = 0; i < 4; ++i) V[i] = Vt<double>{a[i], D[i], f[i]};
  for (int i1 = 0; i1 < 3; ++i1) {
    Vt<double> P[4];
    double r1 = 0.0;
    if (i1 >= cut_piece<0>(V, i1, P, r1)) break;
    for (int i2 = 0; i2 < 3; ++i2) {
      Vt<double> Q[4];
      double r2 = 0.0;
      if (i2 >= cut_piece<1>(P, i2, Q, r2)) break;
      const double d[4] = {Q[0].D, Q[1].D, Q[2].D, Q[3].D}, g[4] = {Q[0].f, Q[1].f, Q[2].f, Q[3].f};
      add(r1 * r2, d, g, out);
    }
  }
}

// FP64 series about the mean: the tier that holds the knots (-1: none) and the value
extern "C" int host_mean_series(const double *d, const double *f, double *v) {
  double e[4], ci;
  const int tier = mean_tier<double, Mean<double>::tiers>(mean_offsets(d, e, ci));
  if (tier >= Mean<double>::tiers) return -1;
  *v = mean_series(e, f, ci, tier);
  return tier;
}

// FP32 series of sorted knots: short recurrence and series_sum (0: outside the series' range)
extern "C" int host_short_series(const float *d, const float *f, float *v, float *w) {
  if (!series_ok(d, Num<float>::kappa_long)) return 0;
  *v = series_sum_short(d, f);
  *w = series_sum(d, f);
  return 1;
}

// three clustered knots: the shared evaluation (0: not its case) and the per-vertex table
extern "C" int host_triple(const double *x, const double *f, double *v, double *w) {
  *w = inv_sum_table(x, f);
  return inv_sum_triple(x, f, *v) ? 1 : 0;
}
