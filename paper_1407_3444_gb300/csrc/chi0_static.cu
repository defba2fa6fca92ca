// chi0_static.cu -- static weights: chi0(q, w = 0) (Eq. 1, Sec. III) over every final
// tetrahedron of the two carvings of Sec. II.
//
// One launch covers a group of q points.  The work unit is (q, run of 2^tlog tetrahedra);
// persistent warps take units from a launch-wide counter and write one FP64 partial per unit,
// which k_static_reduce adds in unit order: results are bitwise reproducible whatever the
// scheduling and whatever the grouping of the q points.
//
// A unit's (m, n) items split by index alone.  With occf[c] the number of leading bands below
// eF at corner c and empf[c] one past the last band not above eF, a tetrahedron is whole
// (occupied at k and empty at k+q at all four corners: one final tetrahedron with D = b - a)
// exactly for m < min occf and n >= max empf; the rest of its rectangle m < max occ,
// n >= min emp is cut by a Fermi surface.  No energies are read to classify an item, and each
// class runs 32 items at a time, one per lane:
//   whole items   12 loads per item, then the closed form's series;
//   cut items     first the pieces of both carvings are counted from the vertices' sides and
//                 listed (item, piece numbers, second cut's side mask), then the list is
//                 evaluated 32 pieces at a time by cut recipes (chi0_math.cuh): an item has 1 to
//                 9 pieces, 2.5 on average, so walking them inside the item's lane left three
//                 lanes of four idle, and the cut cases ran one after the other.
// FP32: series_sum_short in place; pieces past its range wait in a 64-entry queue of the warp in
// shared memory and are evaluated 32 at a time (table_round).  FP64, where every term costs the
// warp 16 cycles of the FP64 pipe whatever its lanes need: all pieces wait in queues by their
// spread, so that a round of 32 runs mean_series to the length its queue needs (K = 12 for most
// whole tetrahedra of a 24^3 mesh, 28 for the longest of any 32 neighbours).
// table_round: the long tiers of mean_series, then the shared divided-difference table, then (FP64
// form, and near-degenerate knots of the mixed form) its triple-cluster case, and for what is left
// the per-vertex table with four lanes per piece.
// Bound: instruction issue (mixed: 2.2 warp instructions per SM cycle), the FP64 pipe (FP64
// form: busy 75-80%).  Measured per q, weights and reduction, before (classification by loading
// every item's energies, one lane per cut item, a global queue and three more kernels for it,
// FP64 series with a convergence test and a table past knot ratio 5/3) and now: 48^3 x 9 bands
// mixed 708 -> 333 us, 32^3 x 40 bands (windows of 4 to 40) mixed 3.0 -> 1.03 ms, 24^3 x 9 bands
// FP64 8.5 -> 0.62 ms, 16^3 free electron FP64 1.9 ms -> 23 us (32 q in one launch).
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "chi0_grid.cuh"
#include "chi0_internal.h"
#include "chi0_math.cuh"

using namespace chi0dev;

namespace chi0int {
namespace {

using grid::kFull;
using grid::pair_add;
using grid::quick_div;
using grid::tet_corners;
using grid::warp_sum;

constexpr int kQueue = 64;   // pieces per queue of a warp
constexpr int kCodes = 128;  // listed pieces of cut items per warp: < 32 left over + 3 x 32

// queues per warp; the last one holds the pieces of table_round, queue b < bins - 1 those with
// max|e| within a tier of mean_series
template <bool FP64> struct StaticShape;
template <> struct StaticShape<false> {
  static constexpr int bins = 1;
};
template <> struct StaticShape<true> {
  static constexpr int bins = 4;
};
// FP64 series queues: tiers 2, 3 and 5 (K = 12, 16, 24); thresholds on the FP32 estimate of
// max|e| with a margin above its error
constexpr int kBin0 = mean_bits(kMeanRD[2] - 2e-6, false), kBin1 = mean_bits(kMeanRD[3] - 2e-6, false),
              kBin2 = mean_bits(kMeanRD[5] - 2e-6, false);

template <typename T> struct PieceQueue {
  T v[9][kQueue];    // knots d, values f, weight
  int pair[kQueue];  // (m - lo) w + (n - lo)
};

// compensated (Neumaier) accumulator in the kernel's precision
template <typename T> struct Acc {
  T s = T(0), c = T(0);
  __device__ __forceinline__ void add(T x) {
    const T t = s + x;
    const bool big = Mean<T>::bits(s) >= Mean<T>::bits(x);  // (a tie of the high words: either order)
    const T a = big ? s : x, b = big ? x : s;
    c += (a - t) + b;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// n <= 32 queued pieces from entry `at` on, one per lane; returns the lane's sum
template <bool FP64>
__device__ __noinline__ double table_round(const PieceQueue<typename std::conditional<FP64, double, float>::type> &q,
                                           int at, int n, float tau, unsigned long long *pairs, int *nfp64) {
  using T = typename std::conditional<FP64, double, float>::type;
  const int lane = threadIdx.x & 31;
  const bool has = lane < n;
  T d[4], f[4], wv = T(0);
  int pair = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) d[i] = f[i] = T(1);
  if (has) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      d[i] = q.v[i][at + lane];
      f[i] = q.v[4 + i][at + lane];
    }
    wv = q.v[8][at + lane];
    pair = q.pair[at + lane];
  }
  double acc = 0.0;
  bool left = has, fp = false;
  if constexpr (FP64) {  // the long tiers
    T e[4], ci;
    const int rb = mean_offsets(d, e, ci);
    const bool ser = has && rb <= Mean<T>::thr(Mean<T>::tiers - 1);
    if (__any_sync(kFull, ser)) {
      const int tier = mean_tier<T, Mean<T>::tiers>(__reduce_max_sync(kFull, ser ? rb : 0));
      const T v = mean_series(e, f, ci, tier);
      if (ser) acc = (double)(wv * v);
    }
    left = has && !ser;
    sort4(d, f);
  } else {  // (sorted already)
    float y[4];
    fp = mixed_knots(y, d, tau) && left;
#pragma unroll
    for (int i = 0; i < 4; ++i) d[i] = y[i];
    if (left && !fp && series_ok(d, Num<float>::kappa_long)) {
      acc = (double)(wv * series_sum_short(d, f));
      left = false;
    }
  }
  if (left && !fp) {
    T v;
    if (inv_sum_shared(d, f, v)) {
      acc = (double)(wv * v);
      left = false;
    }
  }
  if (FP64 ? left : (left && fp)) {
    const double xd[4] = {(double)d[0], (double)d[1], (double)d[2], (double)d[3]};
    const double fd[4] = {(double)f[0], (double)f[1], (double)f[2], (double)f[3]};
    double v;
    if (inv_sum_triple(xd, fd, v)) {
      acc = (double)wv * v;
      left = false;
    }
  }
  if (has && !left && pairs) pair_add(pairs, pair, acc);
  if (fp) ++*nfp64;
  unsigned lm = __ballot_sync(kFull, left);
  while (lm) {  // warp-uniform: eight pieces a round, four lanes (one vertex each) per piece
    const int g = lane >> 2, j = lane & 3;
    int src = -1;
    unsigned m = lm;
    for (int i = 0; i <= g && m; ++i) {
      src = i == g ? __ffs(m) - 1 : src;
      m &= m - 1u;
    }
    const int from = src < 0 ? 0 : src;
    T x[4], ff[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[i] = __shfl_sync(kFull, d[i], from);
      ff[i] = __shfl_sync(kFull, f[i], from);
    }
    const T pw = __shfl_sync(kFull, wv, from);
    const int pp = __shfl_sync(kFull, pair, from);
    const bool pf = __shfl_sync(kFull, (int)fp, from) != 0;
    double t = 0.0;
    if (src >= 0) {
      if (FP64 || pf) {
        const double xd[4] = {(double)x[0], (double)x[1], (double)x[2], (double)x[3]};
        const double fd[4] = {(double)ff[0], (double)ff[1], (double)ff[2], (double)ff[3]};
        t = inv_term_table(xd, fd, j);
      } else {
        t = (double)inv_term_table(x, ff, j);
      }
    }
    t += __shfl_xor_sync(kFull, t, 1);
    t += __shfl_xor_sync(kFull, t, 2);
    if (src >= 0 && j == 0) {
      const double v = (double)pw * t;
      acc += v;
      if (pairs) pair_add(pairs, pp, v);
    }
    for (int i = 0; i < 8; ++i) lm &= lm - 1u;
  }
  return acc;
}

template <bool FP64, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_static(const __grid_constant__ StaticArgs A) {
  using T = typename std::conditional<FP64, double, float>::type;
  constexpr int W = NT / 32;
  __shared__ int4 s_ck[W][32], s_cq[W][32];
  __shared__ T s_vol[W][32];
  __shared__ int s_pw[W][33], s_pc[W][33];              // prefix sums: whole items, cut items
  __shared__ int s_wm[W][32], s_wn[W][32], s_nn[W][32];  // whole columns m, whole and all rows n
  __shared__ int s_code[W][kCodes];                     // l << 24 | (m - lo) << 12 | (n - lo)
  __shared__ unsigned char s_sub[W][kCodes];            // first-cut piece << 6 | second-cut piece << 4 | mask
  __shared__ PieceQueue<T> s_q[W][StaticShape<FP64>::bins];
  __shared__ unsigned s_rec[64];
  constexpr int NB = StaticShape<FP64>::bins;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const Grid &g = A.g;
  const int nb = g.nb;
  int nfp64 = 0, npieces = 0, nover = 0;
  for (int i = threadIdx.x; i < 64; i += NT) s_rec[i] = kCutTab.v[i];
  __syncthreads();
  for (;;) {
    int u = 0;
    if (lane == 0) u = atomicAdd(A.next, 1);
    u = __shfl_sync(kFull, u, 0);
    if (u >= A.units) break;
    int iq = 0;
    while (iq + 1 < A.nq && u >= A.q[iq + 1].u0) ++iq;  // warp-uniform
    const StaticQ &SQ = A.q[iq];
    const Q &q = SQ.q;
    const int lo = q.lo, w = q.hi - q.lo;
    unsigned long long *pairs = SQ.pairs;
    const void *Ek = A.Ek, *Ekq = SQ.Ekq;
    const T *W2 = (const T *)SQ.W2;
    Acc<T> acc;
    double acc_q = 0.0;
    int qn[NB];  // queued pieces (warp-uniform)
#pragma unroll
    for (int i = 0; i < NB; ++i) qn[i] = 0;
    // one tetrahedron per lane: corners, volume, band rectangle
    const long long t = ((long long)(u - SQ.u0) << SQ.tlog) + lane;
    int cw = 0, cc = 0;
    if (lane < (1 << SQ.tlog) && t < g.ntet) {
      long long c[4], cq[4];
      double vol;
      tet_corners(g, A.tet, q, t, c, cq, vol);
      int mhi = 0, mf = nb, nlo = nb, nf = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        mhi = max(mhi, (int)A.occ[c[i]]);
        mf = min(mf, (int)A.occf[c[i]]);
        nlo = min(nlo, (int)SQ.emp[cq[i]]);
        nf = max(nf, (int)SQ.empf[cq[i]]);
      }
      mhi = min(mhi, q.hi);
      nlo = max(nlo, lo);
      const int nm = mhi - lo, nn = q.hi - nlo;
      if (nm > 0 && nn > 0) {
        const int wm = max(min(mf, mhi) - lo, 0), wn = max(q.hi - max(nf, nlo), 0);
        cw = wm * wn;
        cc = nm * nn - cw;
        s_ck[wib][lane] = make_int4((int)c[0], (int)c[1], (int)c[2], (int)c[3]);
        s_cq[wib][lane] = make_int4((int)cq[0], (int)cq[1], (int)cq[2], (int)cq[3]);
        s_vol[wib][lane] = (T)(2.0 * vol);
        s_wm[wib][lane] = wm;
        s_wn[wib][lane] = wn;
        s_nn[wib][lane] = nn;
      }
    }
    int pw = cw, pc = cc;  // inclusive prefix sums over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int a = __shfl_up_sync(kFull, pw, o), b = __shfl_up_sync(kFull, pc, o);
      if (lane >= o) {
        pw += a;
        pc += b;
      }
    }
    s_pw[wib][lane + 1] = pw;
    s_pc[wib][lane + 1] = pc;
    if (lane == 0) s_pw[wib][0] = s_pc[wib][0] = 0;
    const int total_w = __shfl_sync(kFull, pw, 31), total_c = __shfl_sync(kFull, pc, 31);
    __syncwarp();
    auto push = [&](int bin, int at, const T d[4], const T f[4], T wv, int pair) {
      PieceQueue<T> &p = s_q[wib][bin];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        p.v[i][at] = d[i];
        p.v[4 + i][at] = f[i];
      }
      p.v[8][at] = wv;
      p.pair[at] = pair;
    };
    auto drain_table = [&]() {  // 32 pieces of the last queue, which keeps room for 32 more
      __syncwarp();
      qn[NB - 1] -= 32;
      acc_q += table_round<FP64>(s_q[wib][NB - 1], qn[NB - 1], 32, A.tau, pairs, &nfp64);
      ++nover;
      __syncwarp();
    };
    // FP64: the piece at (bin, at) of each lane by the series, at the length of queue `top`
    auto eval_round = [&](bool has, int bin, int at, int top) {
      if constexpr (FP64) {
        T d[4], f[4];
        const PieceQueue<T> &p = s_q[wib][bin];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          d[i] = has ? p.v[i][at] : T(1);
          f[i] = has ? p.v[4 + i][at] : T(1);
        }
        T e[4], ci;
        mean_offsets(d, e, ci);
        const T v = mean_series(e, f, ci, top + 2 + (top >> 1)) * (has ? p.v[8][at] : T(0));  // tiers 2, 3, 5
        if (has) {
          acc.add(v);
          if (pairs) pair_add(pairs, p.pair[at], v);
        }
      }
    };
    // one final tetrahedron per lane
    auto piece = [&](bool has, T d[4], T f[4], T wv, int pair) {
      npieces += has;
      if constexpr (FP64) {
        // spread from FP32 knots (integer conversions: the FP64 pipe is the bound), with a margin
        float x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = grid::d2f_int(d[i]);
        float e[4], ci;
        const int rb = mean_offsets(x, e, ci);
        int bin = NB - 1;
        bin = rb <= kBin2 ? 2 : bin;
        bin = rb <= kBin1 ? 1 : bin;
        bin = rb <= kBin0 ? 0 : bin;
        unsigned full = 0u;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
          const unsigned bal = __ballot_sync(kFull, has && bin == k);
          if (has && bin == k) push(k, qn[k] + __popc(bal & lt), d, f, wv, pair);
          qn[k] += __popc(bal);
          if (qn[k] >= 32) full |= 1u << k;
        }
        if (full & (1u << (NB - 1))) drain_table();
        full &= (1u << (NB - 1)) - 1u;
        if (full) __syncwarp();
#pragma unroll 1
        while (full) {  // warp-uniform
          const int k = __ffs(full) - 1;
          full &= full - 1u;
          int at = 0;
#pragma unroll
          for (int i = 0; i < NB - 1; ++i)
            if (i == k) at = (qn[i] -= 32);
          eval_round(true, k, at + lane, k);
          __syncwarp();
        }
      } else {
        sort4(d, f);
        const bool ser = has && series_ok(d, Num<float>::kappa);
        if (ser) {
          const T v = wv * series_sum_short(d, f);
          acc.add(v);
          if (pairs) pair_add(pairs, pair, (double)v);
        }
        const unsigned bal = __ballot_sync(kFull, has && !ser);
        if (bal) {  // warp-uniform
          if (has && !ser) push(0, qn[0] + __popc(bal & lt), d, f, wv, pair);
          qn[0] += __popc(bal);
          if (qn[0] >= 32) drain_table();
        }
      }
    };
    auto load_e = [&](const int4 &k4, const int4 &q4, int m, int n, T a[4], T b[4]) {
      const T *em = (const T *)Ek + m, *en = (const T *)Ekq + n;
      const int ck[4] = {k4.x, k4.y, k4.z, k4.w}, cq[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i] = em[(long long)ck[i] * nb];
        b[i] = en[(long long)cq[i] * nb];
      }
    };
    // D = b - a, and the first cut's keys a - eF; FP64 keys carry the factor S = 2^64 (exact, and free
    // in the multiply-add; |E| < 2^959), so that levels as close to eF as the smallest numbers have
    // quotients
    constexpr T S = kKeyScale<T>;
    auto relative = [&](T a[4], const T b[4], T D[4]) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        D[i] = b[i] - a[i];
        if constexpr (FP64) a[i] = fma(a[i], S, -S * g.ef);
      }
    };
    // the second cut's key, -b, at a vertex of key a (0 on the first cut's plane)
    auto key_b = [&](T a, T D) { return FP64 ? -fma(D, S, a) : -(a + D); };
    // FP32: the vertices in ascending order of the key (chi0_math.cuh, recipes)
    auto sort_key = [&](T key[4], T x[4], T y[4]) {
      if constexpr (!FP64) {
        auto sw = [&](int i, int j) {
          if (key[j] < key[i]) {
            T t = key[i];
            key[i] = key[j], key[j] = t;
            t = x[i];
            x[i] = x[j], x[j] = t;
            if (y != x) {
              t = y[i];
              y[i] = y[j], y[j] = t;
            }
          }
        };
        sw(0, 1);
        sw(2, 3);
        sw(0, 2);
        sw(1, 3);
        sw(1, 2);
      }
    };
    auto load_f = [&](const int4 &k4, int pair, T f[4]) {
      const int ck[4] = {k4.x, k4.y, k4.z, k4.w};
      const T *p = W2 + pair;
      const int ww = w * w;
#pragma unroll
      for (int i = 0; i < 4; ++i) f[i] = A.cma ? T(1) : p[(long long)ck[i] * ww];
    };
    // whole items
    int l = 0;
    for (int base = 0; base < total_w; base += 32) {  // warp-uniform
      const int it = base + lane;
      bool has = it < total_w;
      T d[4], f[4], wv = T(0);
      int pair = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] = f[i] = T(1);
      if (has) {
        while (s_pw[wib][l + 1] <= it) ++l;  // the item's tetrahedron: items ascend per lane
        const int wn = s_wn[wib][l];
        int no;
        const int mo = quick_div(it - s_pw[wib][l], wn, no);
        no += w - wn;
        has = !(q.gamma && mo == no);  // intraband at Gamma: replaced by the DOS limit
        pair = mo * w + no;
        wv = s_vol[wib][l];
        const int4 k4 = s_ck[wib][l], q4 = s_cq[wib][l];
        T a[4], b[4];
        load_e(k4, q4, lo + mo, lo + no, a, b);
        load_f(k4, pair, f);
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = b[i] - a[i];
      }
      piece(has, d, f, wv, pair);
    }
    // cut items: list the pieces, evaluate the list
    l = 0;
    int nc = 0;  // listed pieces (warp-uniform)
    for (int base = 0;; base += 32) {  // warp-uniform; the pass after the last items empties the list
      const bool last = base >= total_c;
      const int it = base + lane;
      bool has = it < total_c;
      int code = 0;
      T a[4], D[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = D[i] = T(1);  // nothing occupied
      if (has) {
        while (s_pc[wib][l + 1] <= it) ++l;
        const int wm = s_wm[wib][l], wn = s_wn[wib][l], nn = s_nn[wib][l];
        // rows m < wm hold nn - wn items each, the rows after them nn
        const int loc = it - s_pc[wib][l], first = wm * (nn - wn);
        int mo, no;
        if (loc < first) {
          mo = quick_div(loc, nn - wn, no);
        } else {
          mo = wm + quick_div(loc - first, nn, no);
        }
        no += w - nn;
        has = !(q.gamma && mo == no);
        if (has) {
          code = (l << 24) | (mo << 12) | no;
          T b[4];
          load_e(s_ck[wib][l], s_cq[wib][l], lo + mo, lo + no, a, b);
          relative(a, b, D);
        }
      }
      sort_key(a, D, D);
      // sides of the vertices: occupied (a < 0), empty (a + D > 0); D > 0 everywhere puts every
      // point of the first cut plane (b = D there) on the empty side
      unsigned m1 = 0u, eb = 0u;
      bool dpos = true;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        m1 |= (is_neg(a[i]) ? 1u : 0u) << i;
        eb |= (is_neg(key_b(a[i], D[i])) ? 1u : 0u) << i;
        dpos = dpos && is_neg(-D[i]);
      }
      const int n1 = has ? cut_count(m1) : 0;
      const int n1max = last ? 1 : __reduce_max_sync(kFull, n1);
#pragma unroll 1
      for (int i1 = 0; i1 < n1max; ++i1) {
        unsigned m2 = 0u;
        if (i1 < n1) {
          const unsigned rec = s_rec[m1 * 4 + i1];
          if (dpos) {
#pragma unroll
            for (int k = 0; k < 3; ++k) m2 |= (cut_used(rec, k) ? 1u : (eb >> ((rec >> (5 * k)) & 3u)) & 1u) << k;
          } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const T x = cut_mix(rec, k, D, cut_frac<true>(rec, k, a));
              m2 |= (cut_used(rec, k) ? (is_neg(-x) ? 1u : 0u) : (eb >> ((rec >> (5 * k)) & 3u)) & 1u) << k;
            }
          }
          m2 |= ((eb >> ((rec >> 15) & 3u)) & 1u) << 3;
        }
        if constexpr (!FP64) m2 = (1u << __popc(m2)) - 1u;  // (evaluated in sorted order)
        const int n2 = cut_count(m2);
#pragma unroll
        for (int i2 = 0; i2 < 3; ++i2) {
          const unsigned bal = __ballot_sync(kFull, i2 < n2);
          if (i2 < n2) {
            const int at = nc + __popc(bal & lt);
            s_code[wib][at] = code;
            s_sub[wib][at] = (unsigned char)((i1 << 6) | (i2 << 4) | m2);
          }
          nc += __popc(bal);
        }
        __syncwarp();
#pragma unroll 1
        while (nc >= (last ? 1 : 32)) {  // warp-uniform
          const int take = nc < 32 ? nc : 32;
          nc -= take;
          const bool on = lane < take;
          const unsigned cd = on ? (unsigned)s_code[wib][nc + lane] : 0u;
          const unsigned sub = on ? s_sub[wib][nc + lane] : 0u;
          __syncwarp();
          T d[4], f[4], wv = T(0);
          int pair = 0;
          bool ok = false;
#pragma unroll
          for (int i = 0; i < 4; ++i) d[i] = f[i] = T(1);
          if (on) {
            const int tl = (int)(cd >> 24), mo = (int)((cd >> 12) & 0xFFFu), no = (int)(cd & 0xFFFu);
            const int4 k4 = s_ck[wib][tl];
            T u[4], b[4], x[4], y[4];
            load_e(k4, s_cq[wib][tl], lo + mo, lo + no, u, b);
            pair = mo * w + no;
            load_f(k4, pair, y);
            relative(u, b, x);
            sort_key(u, x, y);
            unsigned m = 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i) m |= (is_neg(u[i]) ? 1u : 0u) << i;
            // first cut: keys b of the piece's vertices (D on the cut plane), D and f
            T key[4], D1[4], f1[4], r = T(1);
            unsigned rec = s_rec[m * 4 + (sub >> 6)];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const T t = cut_frac<true>(rec, k, u);
              D1[k] = cut_mix(rec, k, x, t);
              f1[k] = cut_mix(rec, k, y, t);
              if constexpr (FP64) key[k] = key_b(cut_used(rec, k) ? T(0) : sel4(u, (rec >> (5 * k)) & 3u), D1[k]);
              else key[k] = -(cut_used(rec, k) ? D1[k] : sel4(u, (rec >> (5 * k)) & 3u) + D1[k]);
              r *= cut_factor(rec, k, t);
            }
            D1[3] = sel4(x, (rec >> 15) & 3u);
            f1[3] = sel4(y, (rec >> 15) & 3u);
            key[3] = key_b(sel4(u, (rec >> 15) & 3u), D1[3]);
            // second cut, by the side mask the piece was listed with
            sort_key(key, D1, f1);
            rec = s_rec[(sub & 15u) * 4 + ((sub >> 4) & 3u)];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const T t = cut_frac<true>(rec, k, key);
              d[k] = cut_mix(rec, k, D1, t);
              f[k] = cut_mix(rec, k, f1, t);
              r *= cut_factor(rec, k, t);
            }
            d[3] = sel4(D1, (rec >> 15) & 3u);
            f[3] = sel4(f1, (rec >> 15) & 3u);
            ok = r > T(0);
            wv = s_vol[wib][tl] * r;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              d[i] = is_neg(-d[i]) ? d[i] : T(0);
              if (!ok) d[i] = f[i] = T(1);
            }
          }
          piece(ok, d, f, wv, pair);
        }
      }
      if (last) break;
    }
    __syncwarp();
    if constexpr (FP64) {  // what is left in the series queues, packed
      const int n0 = qn[0], n1 = n0 + qn[1], total = n1 + qn[2];
#pragma unroll 1
      for (int base = 0; base < total; base += 32) {
        const int i = base + lane;
        const int bin = i < n0 ? 0 : (i < n1 ? 1 : 2);
        const int last = min(base + 31, total - 1);  // the longest queue this round holds
        eval_round(i < total, i < total ? bin : 0, i < total ? i - (bin == 0 ? 0 : (bin == 1 ? n0 : n1)) : 0,
                   last < n0 ? 0 : (last < n1 ? 1 : 2));
      }
    }
    if (qn[NB - 1] > 0) acc_q += table_round<FP64>(s_q[wib][NB - 1], 0, qn[NB - 1], A.tau, pairs, &nfp64);  // warp-uniform
    __syncwarp();
    const double v = warp_sum(acc.value() + acc_q);
    if (lane == 0) SQ.partial[u - SQ.u0] = v;
    __syncwarp();
  }
  if (A.counters) {
    unsigned long long a = (unsigned long long)npieces, b = (unsigned long long)nfp64;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(kFull, a, o);
      b += __shfl_xor_sync(kFull, b, o);
    }
    if (lane == 0) {
      atomicAdd(&A.counters[0], a);
      atomicAdd(&A.counters[1], b);
      if (nover) atomicAdd(&A.counters[2], 32ull * (unsigned long long)nover);
    }
  }
}

// chi of one q per block: its units' partials in a fixed order, the Gamma DOS term, scale
constexpr int kRedThreads = 1024;
__global__ void __launch_bounds__(kRedThreads) k_static_reduce(const __grid_constant__ StaticArgs A, double scale,
                                                                int ndos, double *__restrict__ out) {
  const StaticQ &SQ = A.q[blockIdx.x];
  const int n = (blockIdx.x + 1 < A.nq ? A.q[blockIdx.x + 1].u0 : A.units) - SQ.u0;
  const double *p = SQ.partial;
  double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0, sd = 0.0;
  int b = threadIdx.x;
  for (; b + 3 * kRedThreads < n; b += 4 * kRedThreads) {  // independent loads in flight
    s0 += p[b];
    s1 += p[b + kRedThreads];
    s2 += p[b + 2 * kRedThreads];
    s3 += p[b + 3 * kRedThreads];
  }
  for (; b < n; b += kRedThreads) s0 += p[b];
  if (SQ.dos)
    for (int i = threadIdx.x; i < ndos; i += kRedThreads) sd += SQ.dos[i];
  double v = ((s0 + s1) + (s2 + s3)) + sd;
  __shared__ double red[kRedThreads / 32];
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = warp_sum(red[threadIdx.x]);
    if (threadIdx.x == 0) out[blockIdx.x] = scale * v;
  }
}

}  // namespace

// Tetrahedra per unit (as log2), from the mesh and the window alone, so that a q's result does
// not depend on what it is grouped with.  32 where that leaves every warp of the chip several
// units; fewer on small meshes, as long as a unit keeps enough items (about a quarter of the
// window's pairs per tetrahedron) to fill its rounds of 32: a unit is one warp's serial work, and
// on a coarse mesh the slowest unit is the launch.
int static_unit_log2(long long ntet, int w) {
  int t = 5;
  const long long ww = (long long)w * w;
  while (t > 2) {
    const long long units = ntet >> t, items = ww << t;
    if (!((units < 16384 && items > 2048) || (units < 2048 && items > 256) || (units < 1024 && items > 64))) break;
    --t;
  }
  return t;
}

long long static_units(long long ntet, int w) {
  const int t = static_unit_log2(ntet, w);
  return (ntet + (1LL << t) - 1) >> t;
}

int static_max_ctas_per_sm(int fp64, int variant) {
  int nb = 0;
  cudaError_t e;
  if (fp64) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_static<true, 64, 4>, 64, 0);
  else if (variant == 1) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_static<false, 128, 3>, 128, 0);
  else if (variant == 2) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_static<false, 256, 1>, 256, 0);
  else e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_static<false, 256, 2>, 256, 0);
  return (e != cudaSuccess || nb < 1) ? 1 : nb;
}

int static_variants(int fp64) { return fp64 ? 1 : 3; }
int static_variant_threads(int fp64, int variant) { return fp64 ? 64 : (variant == 1 ? 128 : 256); }

int static_persistent_blocks(int fp64) { return static_max_ctas_per_sm(fp64, 0) * device_sms(); }

cudaError_t launch_static(StaticArgs &a, int fp64, int nblocks, cudaStream_t s, int variant) {
  int u0 = 0;
  for (int i = 0; i < a.nq; ++i) {
    const int w = a.q[i].q.hi - a.q[i].q.lo;
    a.q[i].tlog = static_unit_log2(a.g.ntet, w);
    a.q[i].u0 = u0;
    u0 += (int)static_units(a.g.ntet, w);
  }
  a.units = u0;
  cudaError_t e = cudaMemsetAsync(a.next, 0, sizeof(int), s);  // unit counter
  if (e != cudaSuccess) return e;
  const int warps = static_variant_threads(fp64, variant) / 32;
  const int need = (u0 + warps - 1) / warps;
  const int nbk = nblocks < need ? nblocks : need;
  if (fp64) k_static<true, 64, 4><<<nbk, 64, 0, s>>>(a);
  else if (variant == 1) k_static<false, 128, 3><<<nbk, 128, 0, s>>>(a);
  else if (variant == 2) k_static<false, 256, 1><<<nbk, 256, 0, s>>>(a);
  else k_static<false, 256, 2><<<nbk, 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_static_reduce(const StaticArgs &a, double scale, int ndos, double *out, cudaStream_t s) {
  k_static_reduce<<<a.nq, kRedThreads, 0, s>>>(a, scale, ndos, out);
  return cudaGetLastError();
}

}  // namespace chi0int
