// chi0_dynamic.cu -- frequency-resolved weights of the doubly carved tetrahedron method:
// Re chi0 as the principal value of Eq. 1, Im chi0 from the delta function of Eq. 2, odd in w
// (Eq. 3), on every final tetrahedron of the two carvings of Sec. II, for one pass of up to
// 256 frequencies.
//
// Per final tetrahedron S (knots d_j of D, values f_j of |M|^2, weight v = volume fraction):
//   Re(u) += v sum_j f_j (1/V) int_S lambda_j [1/(D - u) + 1/(D + u)],   u = |w|
//   Im(w) += sign(w) pi v sum_j f_j (1/V) int_S lambda_j delta(u - D)
// The delta term is nonzero only for u inside (d_0, d_3) and is always evaluated piece by
// piece.  The principal-value terms are smooth in u away from the knots, so for frequencies
// far from a piece they are gathered per box of D instead of per (piece, frequency):
//
//   box b: centre C_b, radius R_b; every piece assigned to it has |d_j - C_b| <= R_b, and adds
//     its moments  M_k += v a_k s_k,  a_k = (-1)^k 6 k!/(k+4)!,  s_k = sum_j f_j h_k(e_1..e_4, e_j),
//     e = (d - C_b)/R_b (Dirichlet moments of the simplex, h_k the complete homogeneous symmetric
//     polynomials).  With eps = (D - C_b)/R_b and z = R_b/(C_b -+ u),
//     1/(D -+ u) = (1/(C_b -+ u)) / (1 + z eps), and 1/(1 + t) is replaced on |t| <= z_max by a
//     polynomial sum_k p_k t^k (the Chebyshev series of chi0_math.cuh), so the box's share of Re(u)
//     is sum_k (-1)^k p_k M_k z^k/(C_b -+ u), evaluated once per (box, frequency) in FP64 after the
//     moments of all warps are summed.  Against the Taylor series the same accuracy takes 20
//     moments instead of 24 at z = 1/2 (FP32), 40 instead of 90 at z = 2/3 (FP64).
//
// Boxes (rebuilt each pass from u_max = max |w| of the pass):
//   fine boxes, levels l = 0..3 of width w_l = (u_max/32) 2^l: centres (j + 1/2) w_l, radius
//     w_l; a piece of half-width s <= w_l/2 whose centre lies in [j w_l, (j+1) w_l) fits.  The box
//     stands in where |C_b - u| >= F R_b (the - term) or C_b + u >= F R_b (the + term); for the
//     other frequencies its pieces evaluate that term themselves: by their own moments about
//     their midpoint c where |c -+ u| >= F s, by the closed form nearer.  F = 2 (FP32), 1.5 (FP64);
//   past u_max, x = c - u_max in [x_b, 1.25 x_b), x_0 = 5 u_max/32, every frequency of the pass is
//     far and pieces evaluate nothing per frequency: geometric boxes (centre u_max + 1.125 x_b,
//     radius x_b/4, pieces with s <= x_b/8, |z| <= 2/9), and, for pieces without a fine box, wide
//     ones up to s = x_b/2 (radius 0.625 x_b, |z| <= 5/9): on coarse meshes a quarter of all pieces
//     are that wide, and without a box each cost two closed forms at every frequency;
//   pieces wider than any box, or past the last one, are evaluated at every frequency.
// Every (piece, frequency, term) is taken exactly once, either by the piece or by its box.
//
// Work layout.  Frequencies are sorted by |w| once per pass (k_box_setup), so that the
// frequencies a piece evaluates are index ranges.  A warp takes a run of 2^tlog tetrahedra; its
// (m, n) items are whole or cut by band index alone and carved 32 pieces at a time, one final
// tetrahedron per lane, as in the static weights (chi0_static.cu).  Each piece finds its box and
// adds its moments in its lane.  Pieces that evaluate frequencies themselves go to a per-warp ring
// queue that the whole warp drains DC pieces at a time: each lane finds one piece's frequency
// ranges and own moments, then all (piece, frequency, term) pairs of the drain are evaluated packed,
// one per lane, first the own-moment pairs, then the near ones.  Near pairs that the shared
// divided-difference table leaves go to a per-warp fallback buffer in global memory, evaluated in
// full rounds when it fills (FP32: the rest by a kernel of its own, k_dyn_fallback).
// Sums.  FP32 kernel: per-CTA sums in 64-bit fixed point (units of 2^-44) in shared memory, added
// with integer atomics and written once per CTA: integer sums are exact in any order, so the warps
// take units from a launch-wide counter and the results are bitwise reproducible for any launch
// shape.  FP64 kernel: units assigned statically (unit = warp + k * warps); Re and Im in per-warp
// compensated FP64 sums, box moments added to a row of the warp's own in global memory (one
// reduction per moment, in the warp's order; 26 KB of shared memory per warp for them had kept an
// SM at four warps): bitwise reproducible for a given launch shape.
//
// Bound: instruction issue, dependent latency and instruction fetch (FP32: 12 warps per SM), the FP64
// pipe (FP64).  Share of the FP32 kernel's time (32^3, 80 bands; time that goes when a part is left
// out): near pairs 25% and the entries they leave 17%, own pairs 12%, delta terms 5%, own moments 4%,
// carving, boxes and box moments 10%.  Measured per 256-frequency pass, before (one (piece, frequency
// range) at a time, 64-bit float conversions and atomics, batches of 32 tetrahedra, the per-vertex
// table for every left entry) and now: 64 x 64 x 16 mesh, 10 bands FP32 10.5 -> 3.8 ms (k_dyn_fallback
// 0.35 of it), 32^3, 80 bands FP32 836 -> 395 ms; 16 x 16 x 8, 10 bands, 128 frequencies FP64
// 58-100 -> 6.2 ms; Im alone, 32^3, 12 bands FP32 3.3 -> 0.70 ms.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "chi0_grid.cuh"
#include "chi0_internal.h"
#include "chi0_math.cuh"

using namespace chi0dev;

namespace chi0int {
namespace {

using grid::kFull;
using grid::quick_div;
using grid::tet_corners;

constexpr int kNWPass = 256;   // frequencies per dynamic pass
// FP32 kernel: sums in 64-bit fixed point, units of 2^-44 (exact and order-independent; one rounding of
// 2^-45 per term).  Re and Im are sums of v f / energy, so the range (2^19) and the rounding are held
// against the energies: the terms carry a power of two S.  With W_m the largest |E - eF| of band m, S is
// below 1 where every band of the q's window is narrow (the largest W_m < 2^-4: S / W_m in [2^3, 2^4]),
// above 1 where every band is wide (the smallest W_m >= 2^8: S / W_m in [2^-8, 2^-7]), and else 1: core
// levels or placeholder bands at 1e10 do not move the scale of the others.  So W |sum| may reach 2^15 at
// least (80 bands: some 10 with |M|^2, a few 1000 without), W being that largest or smallest W_m, and a
// sum of 10^9 terms rounds by 5e-10 / S, at most 1.3e-7 / W.
constexpr double kFxUnit = 1.0 / 17592186044416.0;
// (least, most: high words of the W_m as doubles; most = 0: none)
__device__ __forceinline__ float fx_scale(unsigned least, unsigned most) {
  if (most == 0u) return 1.0f;
  const int e0 = (int)(least >> 20) - 1023, e1 = (int)(most >> 20) - 1023;  // 2^e <= W < 2^(e + 1)
  return ldexpf(1.0f, max(min(e1 < -4 ? e1 + 4 : (e0 > 7 ? e0 - 7 : 0), 100), -100));
}
constexpr int kQC = 64;        // queue of final tetrahedra that evaluate frequencies themselves
constexpr int kCodes = 128;    // listed pieces of cut items per warp: < 32 left over + 3 x 32

// a near-field entry the shared table leaves: knots x (sorted), values f, weight v, and
// code = frequency index << 1 | term
template <typename T> struct FbEnt {
  T x[4], f[4], v;
  int code;
};

template <bool FP64> struct DynShape {
  static constexpr int threads = FP64 ? 64 : 128;
  static constexpr int warps = threads / 32;
  static constexpr int minb = FP64 ? 4 : 3;
  static constexpr int DC = FP64 ? 16 : 32;  // queued pieces evaluated per round
  static constexpr double far = FP64 ? 1.5 : 2.0;  // a box or a piece's own moments stand in from here on (radii)
  static constexpr int KF = FP64 ? 40 : 20;  // moments of a fine box (z <= 1/far)
  static constexpr int KO = FP64 ? 40 : 32;  // own moments of a queued piece, at most
  static constexpr int KG = FP64 ? 18 : 12;  // moments of a geometric box (z <= 2/9)
  static constexpr int KW = FP64 ? 32 : 20;  // moments of a wide box (z <= 5/9)
  // near-field entries left to the per-vertex table that a warp collects: FP64 flushes them in full
  // rounds when they fill (100 MB for all warps), FP32 leaves the last ones to k_dyn_fallback
  static constexpr int fb = FP64 ? 1024 : 4096;
};
template <bool FP64> constexpr bool poly_ok(double tol) {
  using S = DynShape<FP64>;
  return mean_err(1.0 / S::far, S::KF) <= tol && mean_err(2.0 / 9.0, S::KG) <= tol && mean_err(5.0 / 9.0, S::KW) <= tol;
}
static_assert(poly_ok<false>(2.5e-9) && poly_ok<true>(1e-16), "too few moments");
// The boxes' moments carry Taylor's coefficients (6 k!/(k+4)! with the sign of (-1)^k), and
// p_k (-1)^k is applied in FP64 where the boxes are evaluated: rounding it to FP32 in every moment
// would be a bias common to all pieces.  An FP64 piece's own moments carry the polynomial's.
__constant__ constexpr ChebInv<double, DynShape<true>::KO> kOwn(1.0 / DynShape<true>::far);
template <bool FP64> struct BoxPoly {
  using S = DynShape<FP64>;
  double v[S::KF + S::KG + S::KW];
  constexpr BoxPoly() : v() {
    const ChebInv<double, S::KF> f(1.0 / S::far);
    const ChebInv<double, S::KG> g(2.0 / 9.0);
    const ChebInv<double, S::KW> w(5.0 / 9.0);
    for (int k = 0; k < S::KF; ++k) v[k] = (k & 1) ? -f.p_[k] : f.p_[k];
    for (int k = 0; k < S::KG; ++k) v[S::KF + k] = (k & 1) ? -g.p_[k] : g.p_[k];
    for (int k = 0; k < S::KW; ++k) v[S::KF + S::KG + k] = (k & 1) ? -w.p_[k] : w.p_[k];
  }
};
__constant__ constexpr BoxPoly<false> kBoxPolyF{};
__constant__ constexpr BoxPoly<true> kBoxPolyD{};

// box geometry
constexpr int kBoxL = 4;      // fine levels
constexpr int kBoxJ0 = 32;    // finest boxes across [0, u_max]
constexpr int kBoxExtra = 6;  // fine boxes per level past u_max
constexpr int kBoxG = 40;     // geometric boxes (x_0 1.25^40 = 7500 x_0)
constexpr int kBoxW = 24;     // wide boxes (x_0 1.25^24 = 212 x_0)
constexpr int kMinBoxNw = 8;  // fewer frequencies: every piece evaluates all of them
__host__ __device__ constexpr int box_J(int l) { return (kBoxJ0 >> l) + kBoxExtra; }
constexpr int kBoxFine = box_J(0) + box_J(1) + box_J(2) + box_J(3);
constexpr int kBoxes = kBoxFine + kBoxG + kBoxW;
template <bool FP64> __host__ __device__ constexpr int box_slots() {
  return kBoxFine * DynShape<FP64>::KF + kBoxG * DynShape<FP64>::KG + kBoxW * DynShape<FP64>::KW;
}
template <bool FP64> __host__ __device__ constexpr int box_terms(int b) {
  return b < kBoxFine ? DynShape<FP64>::KF : (b < kBoxFine + kBoxG ? DynShape<FP64>::KG : DynShape<FP64>::KW);
}
template <bool FP64> __host__ __device__ constexpr int slot_base(int b) {
  using S = DynShape<FP64>;
  return b < kBoxFine ? b * S::KF
                      : (b < kBoxFine + kBoxG ? kBoxFine * S::KF + (b - kBoxFine) * S::KG
                                              : kBoxFine * S::KF + kBoxG * S::KG + (b - kBoxFine - kBoxG) * S::KW);
}

// the pass's boxes, and with them its frequencies in ascending |w|, in the kernels' precision
// (written by k_box_setup)
template <typename T> struct BoxGeo {
  T C[kBoxes], R[kBoxes];  // centre and radius
  T lowG[kBoxG + 1];       // lower edges x_b of the geometric boxes (x = c - u_max)
  T W0, x0, umax;
  T S;     // FP32 kernel: factor of the fixed-point sums (1 in FP64)
  int on;
  int nv;  // frequencies that are finite in T: the first nv of the sorted ones
};
template <typename T> struct BoxTab : BoxGeo<T> {
  T om[kNWPass];        // |w| ascending
  T oml[kNWPass];       // |w| - (T)|w|
  short rank[kNWPass];  // place of frequency i in that order
};

template <typename T> __device__ __forceinline__ void kadd_t(T &sum, T &comp, T x) {
  const T t = sum + x;
  const bool big = Mean<T>::bits(sum) >= Mean<T>::bits(x);
  const T a = big ? sum : x, b = big ? x : sum;
  comp += (a - t) + b;
  sum = t;
}

// one block: the sorted frequencies, u_max of the pass and the box table (boxes = 0: none).
// Frequencies that are not finite (NaN, infinite, past T's range) come last and take no part in the
// searches, the boxes or u_max; k_dyn_out gives them their values.
template <typename T>
__global__ void __launch_bounds__(kNWPass) k_box_setup(const double *__restrict__ omega, int nw, int boxes,
                                                       const unsigned long long *__restrict__ erange, int lo, int hi,
                                                       BoxTab<T> *tab) {
  __shared__ double red[8];
  __shared__ unsigned rlo[8], rhi[8];
  __shared__ int cnt[8];
  __shared__ unsigned long long key[kNWPass];
  const int i = threadIdx.x;
  const double a = i < nw ? fabs(omega[i]) : 0.0;
  const bool ok = i < nw && (double)(T)a < (double)INFINITY;
  key[i] = (unsigned long long)__double_as_longlong(a);  // ascends with a; a NaN comes last
  double u = ok ? a : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) u = fmax(u, __shfl_xor_sync(kFull, u, o));
  const unsigned oks = __ballot_sync(kFull, ok);
  unsigned least = ~0u, most = 0u;  // of the bands' W_m (a band at eF throughout, or not finite, has none)
  if constexpr (sizeof(T) == 4) {
    for (int m = lo + i; m < hi; m += kNWPass) {
      const unsigned W = (unsigned)(erange[m] >> 32);
      if (W) least = min(least, W);
      most = max(most, W);
    }
    least = __reduce_min_sync(kFull, least);
    most = __reduce_max_sync(kFull, most);
  }
  if ((i & 31) == 0) {
    red[i >> 5] = u;
    rlo[i >> 5] = least;
    rhi[i >> 5] = most;
    cnt[i >> 5] = __popc(oks);
  }
  __syncthreads();
  if (i < nw) {
    int r = 0;
    for (int j = 0; j < nw; ++j) r += key[j] < key[i] || (key[j] == key[i] && j < i);
    tab->rank[i] = (short)r;
    tab->om[r] = (T)a;
    tab->oml[r] = (T)(a - (double)(T)a);
  }
  double umax = 0.0;
  int nv = 0;
  for (int k = 0; k < kNWPass / 32; ++k) {
    umax = fmax(umax, red[k]);
    nv += cnt[k];
  }
  const T W0 = (T)(umax / kBoxJ0), um = (T)umax, x0 = W0 * T(5);
  const int on = (boxes && nv >= kMinBoxNw && umax > 1e-30 && umax < 1e30 && W0 > T(0)) ? 1 : 0;
  if (i == 0) {
    tab->W0 = W0;
    tab->x0 = x0;
    tab->umax = um;
    tab->on = on;
    tab->nv = nv;
    for (int k = 1; k < kNWPass / 32; ++k) {
      least = min(least, rlo[k]);
      most = max(most, rhi[k]);
    }
    tab->S = sizeof(T) == 4 ? (T)fx_scale(least, most) : T(1);
    double lo = (double)x0;
    for (int b = 0; b <= kBoxG; ++b) {
      tab->lowG[b] = (T)lo;
      lo *= 1.25;
    }
  }
  __syncthreads();
  if (i < kBoxFine) {
    int l = 0, j = i;
    while (j >= box_J(l)) {
      j -= box_J(l);
      ++l;
    }
    const T w = W0 * (T)(1 << l);
    tab->C[i] = ((T)j + T(0.5)) * w;
    tab->R[i] = w;
  } else if (i < kBoxes) {
    const bool wide = i >= kBoxFine + kBoxG;
    const T xb = tab->lowG[i - kBoxFine - (wide ? kBoxG : 0)];
    tab->C[i] = um + xb * T(1.125);
    tab->R[i] = xb * (wide ? T(0.625) : T(0.25));
  }
}

// box of a final tetrahedron with midpoint c and half-width s (-1: none, evaluate directly)
template <typename T> __device__ __forceinline__ int box_of(T c, T s, const BoxGeo<T> &tb) {
  if (!tb.on) return -1;
  const T x = c - tb.umax;
  int wide = -1;
  if (x >= tb.x0) {
    int b = (int)(__log2f(__fdividef((float)x, (float)tb.x0)) * 3.1062837f);  // log base 1.25 (a first guess)
    b = b < 0 ? 0 : (b > kBoxG - 1 ? kBoxG - 1 : b);
    while (b > 0 && x < tb.lowG[b]) --b;
    while (b < kBoxG - 1 && x >= tb.lowG[b + 1]) ++b;
    const T lo = tb.lowG[b];
    if (x >= lo && x < tb.lowG[b + 1]) {
      if (s <= T(0.125) * lo) return kBoxFine + b;
      if (b < kBoxW && s <= T(0.5) * lo) wide = kBoxFine + kBoxG + b;
    }
  }
  T w = tb.W0;
  int off = 0;
#pragma unroll 1
  for (int l = 0; l < kBoxL; ++l) {
    if (s <= T(0.5) * w) {
      const T jf = floor(quot(c, w));
      return jf < (T)box_J(l) ? off + (int)jf : wide;
    }
    off += box_J(l);
    w *= T(2);
  }
  return wide;
}

// v as 64-bit fixed point (units of 2^-44, round to nearest even): the same integer as
// __float2ll_rn(v 2^44), from two 32-bit conversions (the 64-bit conversion runs at the FP64 rate,
// 16 cycles of the SM per warp; these take 4)
__device__ __forceinline__ long long fx_of(float v) {
  const float xs = v * 262144.0f;  // 2^18
  if (!(fabsf(xs) < 1.0e9f)) return __float2ll_rn(v * 17592186044416.0f);
  const int h = __float2int_rn(xs);
  const int l = __float2int_rn((xs - (float)h) * 67108864.0f);  // exact difference, 2^26
  return ((long long)h << 26) + (long long)l;
}
// a 64-bit sum in shared memory as two 32-bit words (native 32-bit atomics; the 64-bit add of shared
// memory took 17 to 42 cycles of the SM per warp, by how many lanes shared an address)
__device__ __forceinline__ void fx_add(unsigned *lo, unsigned *hi, int i, float v) {
  const long long t = fx_of(v);
  if (t == 0) return;
  const unsigned l = (unsigned)t;
  const unsigned old = atomicAdd(&lo[i], l);
  atomicAdd(&hi[i], (unsigned)((unsigned long long)t >> 32) + (old + l < old ? 1u : 0u));
}

// does box b stand in for term (0: 1/(D - u), 1: 1/(D + u)) at frequency u = om?  Fine boxes
// only near themselves; the others always.  Same expression in all kernels.
template <typename T> __device__ __forceinline__ bool box_far(T C, T R, int b, T om, int term) {
  if (b >= kBoxFine) return true;
  const T r2 = R * T(DynShape<sizeof(T) == 8>::far);
  if (term) return !(C + om < r2);
  return !(tabs(C - om) < r2);
}

// first index of the ascending om[0..n) with om[i] > v (strict) or >= v
template <bool STRICT, typename T> __device__ __forceinline__ int first_above(const T *om, int n, T v) {
  int a = 0, z = n;
  while (a < z) {
    const int mid = (a + z) >> 1;
    if (STRICT ? om[mid] > v : om[mid] >= v) z = mid;
    else a = mid + 1;
  }
  return a;
}

// a queued piece's frequency ranges (indices of the sorted frequencies): the - term from f0 to f1,
// its near part n0 to n1; the + term up to p1, its near part up to np; the delta term m0 to m1 (the
// frequencies inside the knots, ends included: the pair's own test decides)
struct Range {
  short f0, n0, n1, f1, np, p1, m0, m1;
};

// IMO: Im only (the delta term of Eq. 2; no principal value, no boxes) for the Kramers-Kronig route
template <bool FP64, bool IMO = false>
__global__ void __launch_bounds__(DynShape<FP64>::threads, DynShape<FP64>::minb)
    k_dynamic(const __grid_constant__ DynArgs A, int nw, int tlog) {
  using T = typename std::conditional<FP64, double, float>::type;
  using S = DynShape<FP64>;
  constexpr int W = S::warps, KO = S::KO, DC = S::DC;
  constexpr int NS = box_slots<FP64>();
  constexpr int SK = KO + 2;  // own moments per queued piece (even: read in aligned pairs)
  static_assert(kQC >= DC + 32, "one carving step adds at most 32 queued pieces");
  constexpr bool FX = !FP64;
  __shared__ int4 s_ck[W][32], s_cq[W][32];
  __shared__ T s_vol[W][32];
  __shared__ int s_pw[W][33], s_pc[W][33];               // prefix sums: whole items, cut items
  __shared__ int s_wm[W][32], s_wn[W][32], s_nn[W][32];  // whole columns m, whole and all rows n
  __shared__ int s_code[W][kCodes];                      // l << 24 | (m - lo) << 12 | (n - lo)
  __shared__ unsigned char s_sub[W][kCodes];             // first-cut piece << 6 | second-cut piece << 4 | mask
  __shared__ unsigned s_rec[64];
  __shared__ __align__(16) T s_mom[IMO ? 1 : W][IMO ? 1 : DC][IMO ? 1 : SK];  // own moments of the drain's pieces
  __shared__ unsigned char s_mk[W][DC];  // their count (FP32)
  // ring queue: offsets e from D0 (sorted), values f, (weight, D0h, D0l), box
  __shared__ __align__(16) T s_qe[W][kQC][4];
  __shared__ __align__(16) T s_qf[W][kQC][4];
  __shared__ T s_qv[W][kQC][3];
  __shared__ short s_qb[W][kQC];
  __shared__ Range s_rg[W][DC];
  __shared__ int s_po[W][DC + 1], s_pn[W][DC + 1], s_pd[W][DC + 1];  // prefix sums: own, near, delta pairs
  // FP64 kernel: per-warp compensated sums; FP32 kernel: per-CTA fixed-point sums (two words)
  constexpr int WA = FX ? 1 : W, NA = FX ? 1 : kNWPass;
  __shared__ T sR[WA][IMO ? 1 : NA], sI[WA][NA];
  __shared__ T cR[WA][IMO ? 1 : NA], cI[WA][NA];  // compensation terms
  __shared__ unsigned s_fxl[FX ? 2 * kNWPass : 1], s_fxh[FX ? 2 * kNWPass : 1];
  __shared__ T s_w[kNWPass];                 // |w| ascending
  __shared__ T s_wl[FP64 ? 1 : kNWPass];     // FP32 path: |w| - (float)|w|
  __shared__ short s_rng[kBoxFine][3];  // frequencies a fine box leaves to its pieces: - term [lo, hi), + term [0, p)
  __shared__ BoxGeo<T> s_tab;
  extern __shared__ __align__(16) unsigned char s_dyn[];  // FP32: box sums, low and high words [NS]
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  unsigned *bl = (unsigned *)s_dyn, *bh = bl + NS;
  const Grid &g = A.g;
  const Q &q = A.q;
  const DynBufs &db = A.db;
  const int lo = q.lo, w = q.hi - q.lo, nb = g.nb;
  const T *W2 = (const T *)A.W2;
  const long long units = (g.ntet + (1LL << tlog) - 1) >> tlog;
  const long long gwarp = (long long)blockIdx.x * W + wib, nwarps = (long long)gridDim.x * W;
  double *gbox = db.box_part + gwarp * NS;  // FP64: the warp's box moments
  FbEnt<T> *gfb = (FbEnt<T> *)db.fb + gwarp * S::fb;
  {
    const BoxTab<T> *src = (const BoxTab<T> *)db.box_tab;
    constexpr int nwords = (int)(sizeof(BoxGeo<T>) / 4);
#pragma unroll 1
    for (int i = threadIdx.x; i < nwords; i += blockDim.x) ((int *)&s_tab)[i] = ((const int *)src)[i];
#pragma unroll 1
    for (int i = threadIdx.x; i < nw; i += blockDim.x) {
      s_w[i] = src->om[i];
      if constexpr (!FP64) s_wl[i] = src->oml[i];
    }
  }
  for (int i = threadIdx.x; i < 64; i += blockDim.x) s_rec[i] = kCutTab.v[i];
  if constexpr (FX) {
    if constexpr (!IMO) {
#pragma unroll 1
      for (int i = threadIdx.x; i < 2 * NS; i += blockDim.x) bl[i] = 0u;
    }
#pragma unroll 1
    for (int i = threadIdx.x; i < 2 * kNWPass; i += blockDim.x) s_fxl[i] = s_fxh[i] = 0u;
  } else {
#pragma unroll 1
    for (int i = lane; i < nw; i += 32) {
      if constexpr (!IMO) sR[wib][i] = cR[wib][i] = T(0);
      sI[wib][i] = cI[wib][i] = T(0);
    }
  }
  __syncthreads();
  if constexpr (!IMO) {
#pragma unroll 1
    for (int b = threadIdx.x; b < kBoxFine; b += blockDim.x) {
      int a = kNWPass, z = 0, p = 0;  // (intervals: |w| ascends)
#pragma unroll 1
      for (int i = 0; i < s_tab.nv; ++i) {
        if (!box_far(s_tab.C[b], s_tab.R[b], b, s_w[i], 0)) {
          a = a < i ? a : i;
          z = i + 1;
        }
        if (!box_far(s_tab.C[b], s_tab.R[b], b, s_w[i], 1)) p = i + 1;
      }
      s_rng[b][0] = (short)(z > a ? a : 0);
      s_rng[b][1] = (short)(z > a ? z : 0);
      s_rng[b][2] = (short)p;
    }
    __syncthreads();
  }
  const bool boxes = !IMO && s_tab.on != 0;
  int nfp64 = 0, npieces = 0, nboxed = 0;
  int qh = 0, qt = 0;  // ring queue head and tail (warp-uniform)
  int nfb = 0;         // entries in the warp's fallback buffer (warp-uniform)
  // one round of per-lane results (iw < 0: nothing).  Fixed point: atomic adds (exact, any
  // order).  FP64: lanes that share a frequency add one at a time in lane order, the others at once.
  auto round_add = [&](int iw, T re, T im) {
    if constexpr (FX) {
      if (iw >= 0) {
        if (!IMO && re != T(0)) fx_add(s_fxl, s_fxh, iw, re);
        if (im != T(0)) fx_add(s_fxl + kNWPass, s_fxh + kNWPass, iw, im);
      }
    } else {
      const unsigned grp = __match_any_sync(kFull, iw >= 0 ? iw : -1 - lane);
      const int rank = __popc(grp & lt);
      const int nr = __reduce_max_sync(kFull, iw >= 0 ? rank : 0);
#pragma unroll 1
      for (int r = 0; r <= nr; ++r) {
        if (iw >= 0 && rank == r) {
          if constexpr (!IMO)
            if (re != T(0)) kadd_t(sR[wib][iw], cR[wib][iw], re);
          if (im != T(0)) kadd_t(sI[wib][iw], cI[wib][iw], im);
        }
        __syncwarp();
      }
    }
  };
  // the fallback buffer: per-vertex table, one entry per lane and round (full rounds: the
  // buffer collects the entries of many pieces, in a fixed order)
  auto fallback_flush = [&]() {
    __syncwarp();
#pragma unroll 1
    for (int base = 0; base < nfb; base += 32) {
      const int k = base + lane;
      T re = T(0);
      int iw = -1;
      if (k < nfb) {
        const FbEnt<T> &o = gfb[k];
        T x[4], ff[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          x[i] = o.x[i];
          ff[i] = o.f[i];
        }
        const T vr = o.v;
        iw = o.code >> 1;
        re = vr * near_term<FP64>(x, ff, A.tau, nfp64);
      }
      round_add(iw, re, T(0));
    }
    nfb = 0;
    __syncwarp();
  };
  // evaluates n <= DC queued pieces: ranges and own moments one piece per lane, then their
  // (piece, frequency, term) pairs packed over the lanes
  auto drain = [&](int n) {
    int no = 0, nn = 0, nd = 0;
    if (lane < n) {
      const int sl = (qh + lane) % kQC, nv = s_tab.nv;
      const T D0h = s_qv[wib][sl][1];
      const T e0 = s_qe[wib][sl][0], e3 = s_qe[wib][sl][3];
      Range r{};
      {
        // frequencies inside the knots, up to the roundings of D0 and |w| to T (ties with either end
        // included, however many); the pair's own test decides
        const T dlo = D0h + e0, dhi = D0h + e3;
        const T eps = FP64 ? T(0) : T(2.384185791015625e-07);  // 2^-22
        const int a = first_above<false>(s_w, nv, dlo - eps * (tabs(D0h) + tabs(dlo)));
        r.m0 = (short)a;
        r.m1 = (short)max(first_above<true>(s_w, nv, dhi + eps * (tabs(D0h) + tabs(dhi))), a);
        nd = r.m1 - r.m0;
      }
      if constexpr (!IMO) {
        const int b = s_qb[wib][sl];
        const T half = (e3 - e0) * T(0.5), c = D0h + (e0 + e3) * T(0.5), near = half * T(S::far);
        const int f0 = b >= 0 ? s_rng[b][0] : 0, f1 = b >= 0 ? s_rng[b][1] : nv, p1 = b >= 0 ? s_rng[b][2] : nv;
        // (closed ends: a frequency at the midpoint of a flat piece, half = 0 or lost in c, is near:
        // the table takes a zero knot, the own moments' 1/(c - w) does not)
        const int a = min(max(first_above<false>(s_w, nv, c - near), f0), f1);
        const int z = max(min(first_above<true>(s_w, nv, c + near), f1), a);
        const int p = p1 > 0 ? min(first_above<true>(s_w, nv, near - c), p1) : 0;
        r.f0 = (short)f0;
        r.n0 = (short)a;
        r.n1 = (short)z;
        r.f1 = (short)f1;
        r.np = (short)p;
        r.p1 = (short)p1;
        nn = (z - a) + p;
        no = (f1 - f0) - (z - a) + (p1 - p);
        if (no > 0) {
          T ff[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) ff[i] = s_qf[wib][sl][i];
          if constexpr (FP64) {  // about the midpoint, offsets in units of the half-width
            // (a half-width below 2^-1000 counts as flat: it has no finite reciprocal below 2^-1022)
            const T ri = half > T(1e-300) ? rcp_nr(half) : T(0), mid = (e0 + e3) * T(0.5), vr = s_qv[wib][sl][0];
            T e[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i] = (s_qe[wib][sl][i] - mid) * ri;
            Moments<T> m(e, ff);
            T *out = s_mom[wib][lane];
#pragma unroll
            for (int k = 0; k < 4; ++k) out[k] = vr * kOwn.v[k] * m.next(m.n[k]);
#pragma unroll 4
            for (int k = 4; k < KO; ++k) out[k] = vr * kOwn.v[k] * m.next(T(0));
          } else {  // in units of the midpoint, as many as the widest ratio needs
            T d[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) d[i] = D0h + s_qe[wib][sl][i];
            s_mk[wib][lane] = far_moments<T, KO>(d, ff, s_mom[wib][lane]);
          }
        }
      }
      s_rg[wib][lane] = r;
    }
    int po = no, pn = nn, pd = nd;  // inclusive prefix sums over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(kFull, po, o), y = __shfl_up_sync(kFull, pn, o), z = __shfl_up_sync(kFull, pd, o);
      if (lane >= o) {
        po += x;
        pn += y;
        pd += z;
      }
    }
    if (lane < n) {
      s_po[wib][lane + 1] = po;
      s_pn[wib][lane + 1] = pn;
      s_pd[wib][lane + 1] = pd;
    }
    if (lane == 0) s_po[wib][0] = s_pn[wib][0] = s_pd[wib][0] = 0;
    const int own = __shfl_sync(kFull, po, 31), near = __shfl_sync(kFull, pn, 31), inside = __shfl_sync(kFull, pd, 31);
    __syncwarp();
    if constexpr (!IMO) {
      int p = 0;
#pragma unroll 1
      for (int base = 0; base < own; base += 32) {  // warp-uniform
        const int it = base + lane;
        T v = T(0);
        int iw = -1;
        if (it < own) {
          while (s_po[wib][p + 1] <= it) ++p;
          const int sl = (qh + p) % kQC;
          const Range r = s_rg[wib][p];
          int k = it - s_po[wib][p];
          const int k1 = r.n0 - r.f0, k2 = k1 + (r.f1 - r.n1);
          const bool plus = k >= k2;
          iw = k < k1 ? r.f0 + k : (plus ? r.np + (k - k2) : r.n1 + (k - k1));
          const T e0 = s_qe[wib][sl][0], e3 = s_qe[wib][sl][3];
          const T om = s_w[iw], c = s_qv[wib][sl][1] + (e0 + e3) * T(0.5);
          const T *m = s_mom[wib][p];
          if constexpr (FP64) {
            const T rd = rcp_nr(plus ? c + om : c - om), z = (e3 - e0) * T(0.5) * rd, z2 = z * z;
            // even and odd powers as two chains (the loop is bound by dependent latency)
            const double2 m0 = *reinterpret_cast<const double2 *>(m + KO - 2);
            T se = m0.x, so = m0.y;
#pragma unroll 4
            for (int j = KO - 4; j >= 0; j -= 2) {
              const double2 mj = *reinterpret_cast<const double2 *>(m + j);
              so = so * z2 + mj.y;
              se = se * z2 + mj.x;
            }
            v = (se + z * so) * rd;
          } else {
            v = s_qv[wib][sl][0] * far_eval_k(m, s_mk[wib][p], c, plus ? -om : om);
          }
        }
        round_add(iw, v, T(0));
      }
    }
    // knots (D0 - |w|) + e of the - term at frequency jw
    auto load_piece = [&](int sl, T ee[4], T ff[4]) {
      if constexpr (FP64) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          ee[i] = s_qe[wib][sl][i];
          ff[i] = s_qf[wib][sl][i];
        }
      } else {  // one 16-byte load each
        const float4 e4 = *reinterpret_cast<const float4 *>(&s_qe[wib][sl][0]);
        const float4 f4 = *reinterpret_cast<const float4 *>(&s_qf[wib][sl][0]);
        ee[0] = e4.x, ee[1] = e4.y, ee[2] = e4.z, ee[3] = e4.w;
        ff[0] = f4.x, ff[1] = f4.y, ff[2] = f4.z, ff[3] = f4.w;
      }
    };
    auto shifted = [&](int sl, int jw, const T ee[4], T x[4]) {
      const T sh = near_shift(s_qv[wib][sl][1], s_qv[wib][sl][2], s_w[jw], FP64 ? T(0) : s_wl[FP64 ? 0 : jw]);
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = sh + ee[i];
    };
    // near pairs: the shared divided-difference table.  Pairs it leaves (three clustered knots, three
    // zero knots) go, knots and all, to the fallback buffer.
    if constexpr (!IMO) {
      int p = 0;
#pragma unroll 1
      for (int base = 0; base < near; base += 32) {  // warp-uniform
        if (nfb > S::fb - 32) fallback_flush();
        const int it = base + lane;
        T re = T(0), x[4], ff[4], vr = T(0);
        int iw = -1, code = 0;
        bool left = false;
        if (it < near) {
          while (s_pn[wib][p + 1] <= it) ++p;
          const int sl = (qh + p) % kQC;
          const Range r = s_rg[wib][p];
          const int k = it - s_pn[wib][p], k1 = r.n1 - r.n0;
          const bool plus = k >= k1;
          const int jw = plus ? k - k1 : r.n0 + k;
          vr = s_qv[wib][sl][0];
          T ee[4], v;
          load_piece(sl, ee, ff);
          if (plus) {  // knots d + |w|
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = (s_qv[wib][sl][1] + ee[i]) + s_w[jw];
          } else {
            shifted(sl, jw, ee, x);
          }
          code = (jw << 1) | (plus ? 1 : 0);
          if (inv_sum_shared(x, ff, v)) {
            iw = jw;
            re = vr * v;
          } else {
            left = true;
          }
        }
        round_add(iw, re, T(0));
        const unsigned bal = __ballot_sync(kFull, left);
        if (bal) {  // warp-uniform
          if (left) {
            FbEnt<T> &o = gfb[nfb + __popc(bal & lt)];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              o.x[i] = x[i];
              o.f[i] = ff[i];
            }
            o.v = vr;
            o.code = code;
          }
          nfb += __popc(bal);
        }
      }
    }
    // the delta term of the frequencies inside the knots
    int p = 0;
#pragma unroll 1
    for (int base = 0; base < inside; base += 32) {  // warp-uniform
      const int it = base + lane;
      T im = T(0);
      int iw = -1;
      if (it < inside) {
        while (s_pd[wib][p + 1] <= it) ++p;
        const int sl = (qh + p) % kQC, jw = s_rg[wib][p].m0 + (it - s_pd[wib][p]);
        T ee[4], ff[4], x[4];
        load_piece(sl, ee, ff);
        shifted(sl, jw, ee, x);
        if (x[0] < T(0) && x[3] > T(0)) {
          iw = jw;
          im = s_qv[wib][sl][0] * delta_term(x, ee, ff) * T(3.141592653589793);
        }
      }
      round_add(iw, T(0), im);
    }
    qh += n;
    __syncwarp();
  };
  // one carving step: at most one final tetrahedron per lane (has).  Its box and moments, and the
  // queue for pieces that evaluate frequencies themselves.  last: the queue is emptied.
  auto piece = [&](bool has, T ee[4], T ff[4], T vr, T D0h, T D0l, bool last) {
    int b = -1;
    if (has) {
      sort4(ee, ff);
      ++npieces;
      has = D0h + ee[3] > T(0);
    }
    if (has && boxes) b = box_of(D0h + (ee[0] + ee[3]) * T(0.5), (ee[3] - ee[0]) * T(0.5), s_tab);
    if constexpr (!IMO) {
      const bool in = has && b >= 0;
      if constexpr (FX) {
        if (in) {
          ++nboxed;
          const T ri = rcp(s_tab.R[b]), base = (D0h - s_tab.C[b]) + D0l;
          T e[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) e[i] = (base + ee[i]) * ri;
          const int K = box_terms<FP64>(b), at = slot_base<FP64>(b);
          fx_add(bl, bh, at, vr * T(0.25) * (ff[0] + ff[1] + ff[2] + ff[3]));
          MomentsH<T> m(e, ff);
#pragma unroll 2
          for (int k = 1; k < K; ++k) fx_add(bl, bh, at + k, vr * series_coef<T>(k) * m.next());
        }
      } else if (__any_sync(kFull, in)) {
        // lanes in the same box add one at a time, in lane order
        const unsigned grp = __match_any_sync(kFull, in ? b : -1 - lane);
        const int rank = __popc(grp & lt), nr = __reduce_max_sync(kFull, in ? rank : 0);
        nboxed += in;
        const int bb = in ? b : 0;
        const T ri = rcp_nr(s_tab.R[bb]), base = D0h - s_tab.C[bb];
        T e[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) e[i] = in ? (base + ee[i]) * ri : T(0);
        const int K = in ? box_terms<FP64>(bb) : 0, Kmax = __reduce_max_sync(kFull, K);
        double *out = gbox + slot_base<FP64>(bb);
        Moments<T> m(e, ff);
        T in4[4] = {m.n[0], m.n[1], m.n[2], m.n[3]};
#pragma unroll 1
        for (int k = 0; k < Kmax; ++k) {
          const T v = m.next(in4[0]);
          in4[0] = in4[1], in4[1] = in4[2], in4[2] = in4[3], in4[3] = T(0);
          const T t = k < K ? vr * series_coef<T>(k) * v : T(0);
#pragma unroll 1
          for (int r = 0; r <= nr; ++r) {
            if (k < K && rank == r) atomicAdd(out + k, t);
            __syncwarp();
          }
        }
      }
    }
    // (Im only: pieces whose knot range meets the pass's frequencies)
    const bool queue = has && (IMO ? s_tab.nv > 0 && D0h + ee[3] > s_w[0] && D0h + ee[0] < s_w[s_tab.nv - 1] : b < kBoxFine);
    const unsigned qm = __ballot_sync(kFull, queue);
    if (queue) {
      const int sl = (qt + __popc(qm & lt)) % kQC;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        s_qe[wib][sl][i] = ee[i];
        s_qf[wib][sl][i] = ff[i];
      }
      s_qv[wib][sl][0] = FX ? vr * s_tab.S : vr;
      s_qv[wib][sl][1] = D0h;
      s_qv[wib][sl][2] = D0l;
      s_qb[wib][sl] = (short)b;
    }
    qt += __popc(qm);
    __syncwarp();
#pragma unroll 1
    while (qt - qh >= (last ? 1 : DC)) drain(qt - qh < DC ? qt - qh : DC);
  };
  // item data: a = e^m_k - eF, D = D0 + e (e_0 = 0) and |M|^2 at the corners.  Mixed path:
  // energies as FP32 hi + lo pairs, so that D0 (hi + lo) and the corner offsets e come out to full
  // FP32 relative precision whatever the size of a, b
  auto load_item = [&](int l, int mo, int no, T a[4], T e[4], T &D0h, T &D0l) {
    const int4 k4 = s_ck[wib][l], q4 = s_cq[wib][l];
    const int ck[4] = {k4.x, k4.y, k4.z, k4.w}, cq[4] = {q4.x, q4.y, q4.z, q4.w};
    D0h = T(0);
    D0l = T(0);
    if constexpr (FP64) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i] = ((const double *)A.Ek)[(long long)ck[i] * nb + lo + mo] - g.ef;
        e[i] = (((const double *)A.Ekq)[(long long)cq[i] * nb + lo + no] - g.ef) - a[i];
      }
    } else {
      float al[4], bh_[4], bl_[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const long long ik = (long long)ck[i] * nb + lo + mo, iq = (long long)cq[i] * nb + lo + no;
        a[i] = ((const float *)A.Ek)[ik];
        al[i] = A.Eklo[ik];
        bh_[i] = ((const float *)A.Ekq)[iq];
        bl_[i] = A.Ekqlo[iq];
      }
      float sv, tv;
      two_diff(bh_[0], a[0], sv, tv);
      const float corr = tv + (bl_[0] - al[0]);
      D0h = sv + corr;
      D0l = corr - (D0h - sv);
      e[0] = 0.0f;
#pragma unroll
      for (int i = 1; i < 4; ++i) {
        float sa, ta, sb, tb;
        two_diff(a[i], a[0], sa, ta);
        two_diff(bh_[i], bh_[0], sb, tb);
        e[i] = (sb - sa) + ((tb - ta) + ((bl_[i] - bl_[0]) - (al[i] - al[0])));
      }
    }
  };
  auto load_f = [&](int l, int mo, int no, T f[4]) {
    const int4 k4 = s_ck[wib][l];
    const int ck[4] = {k4.x, k4.y, k4.z, k4.w};
    const T *pw = W2 + (mo * w + no);
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = A.cma ? T(1) : pw[(long long)ck[i] * w * w];
  };
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
  // a listed piece of a cut item (mask: the second cut's sides): offsets, values, volume ratio
  auto cut_item = [&](unsigned cd, unsigned sub, T ee[4], T ff[4], T &vr, T &D0h, T &D0l) -> bool {
    const int tl = (int)(cd >> 24), mo = (int)((cd >> 12) & 0xFFFu), no = (int)(cd & 0xFFFu);
    T a[4], e[4], fv[4];
    load_item(tl, mo, no, a, e, D0h, D0l);
    load_f(tl, mo, no, fv);
    sort_key(a, e, fv);
    unsigned m = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) m |= (is_neg(a[i]) ? 1u : 0u) << i;
    T key[4], e1[4], f1[4], r = T(1);
    unsigned rec = s_rec[m * 4 + (sub >> 6)];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const T t = cut_frac(rec, k, a);
      e1[k] = cut_mix(rec, k, e, t);
      f1[k] = cut_mix(rec, k, fv, t);
      key[k] = -((cut_used(rec, k) ? D0h : sel4(a, (rec >> (5 * k)) & 3u) + D0h) + e1[k]);
      r *= cut_factor(rec, k, t);
    }
    e1[3] = sel4(e, (rec >> 15) & 3u);
    f1[3] = sel4(fv, (rec >> 15) & 3u);
    key[3] = -((sel4(a, (rec >> 15) & 3u) + D0h) + e1[3]);
    sort_key(key, e1, f1);
    rec = s_rec[(sub & 15u) * 4 + ((sub >> 4) & 3u)];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const T t = cut_frac(rec, k, key);
      ee[k] = cut_mix(rec, k, e1, t);
      ff[k] = cut_mix(rec, k, f1, t);
      r *= cut_factor(rec, k, t);
    }
    ee[3] = sel4(e1, (rec >> 15) & 3u);
    ff[3] = sel4(f1, (rec >> 15) & 3u);
#pragma unroll
    for (int i = 0; i < 4; ++i) ee[i] = ee[i] > -D0h ? ee[i] : -D0h;  // clamped to D >= 0
    vr = s_vol[wib][tl] * r;
    return r > T(0);
  };
  // units: FP64 kernel in a fixed order per warp; FP32 kernel from a launch-wide counter (its sums
  // are exact integers, whatever the order), which balances the warps' loads
  auto next_unit = [&](long long cur) -> long long {
    if constexpr (FX) {
      unsigned long long b = 0ull;
      if (lane == 0) b = atomicAdd(db.ctr, 1ull);
      return (long long)__shfl_sync(kFull, b, 0);
    } else {
      return cur < 0 ? gwarp : cur + nwarps;
    }
  };
  for (long long unit = next_unit(-1);; unit = next_unit(unit)) {
    const bool end = unit >= units;  // (one more turn: empties the queue)
    const long long t = (unit << tlog) + lane;
    int cw = 0, cc = 0;
    if (!end && lane < (1 << tlog) && t < g.ntet) {
      long long c[4], cq[4];
      double vol;
      tet_corners(g, A.tet, q, t, c, cq, vol);
      int mhi = 0, mf = nb, nlo = nb, nf = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        mhi = max(mhi, (int)A.occ[c[i]]);
        mf = min(mf, (int)A.occf[c[i]]);
        nlo = min(nlo, (int)A.emp[cq[i]]);
        nf = max(nf, (int)A.empf[cq[i]]);
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
        s_vol[wib][lane] = (T)vol;
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
    // Rounds of 32 final tetrahedra: first the whole items, then the listed pieces of the cut ones
    // (items are listed 32 at a time whenever fewer than 32 pieces wait); one call site of piece().
    int lw = 0, lc = 0, base_w = 0, base_c = 0, nc = 0, i1 = 0, n1 = 0, n1max = 0;
    unsigned m1 = 0u, eb = 0u;
    int code = 0;
    bool dpos = true;
    T a1[4], e1[4], D1h = T(0);
#pragma unroll
    for (int i = 0; i < 4; ++i) a1[i] = e1[i] = T(0);
#pragma unroll 1
    for (;;) {  // warp-uniform
      T ee[4], ff[4], vr = T(0), D0h = T(0), D0l = T(0);
#pragma unroll
      for (int i = 0; i < 4; ++i) ee[i] = ff[i] = T(0);
      bool has = false, last = false;
      if (base_w < total_w) {
        const int it = base_w + lane;
        base_w += 32;
        has = it < total_w;
        if (has) {
          while (s_pw[wib][lw + 1] <= it) ++lw;  // the item's tetrahedron: items ascend per lane
          const int wn = s_wn[wib][lw];
          int no;
          const int mo = quick_div(it - s_pw[wib][lw], wn, no);
          no += w - wn;
          has = !(q.gamma && mo == no);  // intraband at Gamma: replaced by the DOS limit
          T a[4];
          load_item(lw, mo, no, a, ee, D0h, D0l);
          load_f(lw, mo, no, ff);
          vr = s_vol[wib][lw];
        }
      } else if (nc < 32 && (i1 < n1max || base_c < total_c)) {
        // list pieces: of the current 32 cut items' next first-cut piece, or take the next items
        if (i1 >= n1max) {
          const int it = base_c + lane;
          base_c += 32;
          bool on = it < total_c;
          n1 = 0;
          if (on) {
            while (s_pc[wib][lc + 1] <= it) ++lc;
            const int wm = s_wm[wib][lc], wn = s_wn[wib][lc], nn = s_nn[wib][lc];
            // rows m < wm hold nn - wn items each, the rows after them nn
            const int loc = it - s_pc[wib][lc], first = wm * (nn - wn);
            int mo, no;
            if (loc < first) mo = quick_div(loc, nn - wn, no);
            else mo = wm + quick_div(loc - first, nn, no);
            no += w - nn;
            if (!(q.gamma && mo == no)) {
              code = (lc << 24) | (mo << 12) | no;
              T D1l;
              load_item(lc, mo, no, a1, e1, D1h, D1l);
              sort_key(a1, e1, e1);
              // sides of the vertices: occupied (a < 0), empty (a + D > 0); D > 0 everywhere puts
              // every point of the first cut plane (b = D there) on the empty side
              m1 = eb = 0u;
              dpos = true;
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                m1 |= (is_neg(a1[i]) ? 1u : 0u) << i;
                eb |= (is_neg(-((a1[i] + D1h) + e1[i])) ? 1u : 0u) << i;
                dpos = dpos && is_neg(-(D1h + e1[i]));
              }
              n1 = cut_count(m1);
            }
          }
          i1 = 0;
          n1max = __reduce_max_sync(kFull, n1);
        }
        unsigned m2 = 0u;
        if (i1 < n1) {
          const unsigned rec = s_rec[m1 * 4 + i1];
          if (dpos) {
#pragma unroll
            for (int k = 0; k < 3; ++k) m2 |= (cut_used(rec, k) ? 1u : (eb >> ((rec >> (5 * k)) & 3u)) & 1u) << k;
          } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const T x = D1h + cut_mix(rec, k, e1, cut_frac(rec, k, a1));
              m2 |= (cut_used(rec, k) ? (is_neg(-x) ? 1u : 0u) : (eb >> ((rec >> (5 * k)) & 3u)) & 1u) << k;
            }
          }
          m2 |= ((eb >> ((rec >> 15) & 3u)) & 1u) << 3;
          if constexpr (!FP64) m2 = (1u << __popc(m2)) - 1u;  // (evaluated in sorted order)
        }
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
        ++i1;
        __syncwarp();
        continue;
      } else if (nc > 0) {
        const int take = nc < 32 ? nc : 32;
        nc -= take;
        has = lane < take;
        const unsigned cd = has ? (unsigned)s_code[wib][nc + lane] : 0u;
        const unsigned sub = has ? s_sub[wib][nc + lane] : 0u;
        __syncwarp();
        if (has) has = cut_item(cd, sub, ee, ff, vr, D0h, D0l);
      } else if (end && qt > qh) {
        last = true;
      } else {
        break;
      }
      piece(has, ee, ff, vr, D0h, D0l, last);
    }
    if (end) break;
  }
  if constexpr (FX && !IMO) {
    if (lane == 0) db.fbn[gwarp] = nfb;  // the rest of the buffer: k_dyn_fallback
  } else {
    if (nfb > 0) fallback_flush();  // warp-uniform
  }
  if constexpr (FX) {
    // the CTA's fixed-point sums into its rows
    __syncthreads();
    unsigned long long *row = db.fx + (size_t)blockIdx.x * 2 * kNWPass;
    unsigned long long *brow = (unsigned long long *)db.box_part + (size_t)blockIdx.x * NS;
#pragma unroll 1
    for (int i = threadIdx.x; i < 2 * kNWPass; i += blockDim.x)
      row[i] = ((unsigned long long)s_fxh[i] << 32) | s_fxl[i];
    if constexpr (!IMO) {
#pragma unroll 1
      for (int i = threadIdx.x; i < NS; i += blockDim.x) brow[i] = ((unsigned long long)bh[i] << 32) | bl[i];
    }
  } else {
    __syncwarp();
#pragma unroll 1
    for (int iw = lane; iw < nw; iw += 32) {
      if constexpr (!IMO) db.partR[gwarp * nw + iw] = (double)sR[wib][iw] + (double)cR[wib][iw];
      db.partI[gwarp * nw + iw] = (double)sI[wib][iw] + (double)cI[wib][iw];
    }
  }
  if (A.counters) {
    unsigned long long a = (unsigned long long)npieces, b = (unsigned long long)nfp64,
                       x = (unsigned long long)nboxed;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(kFull, a, o);
      b += __shfl_xor_sync(kFull, b, o);
      x += __shfl_xor_sync(kFull, x, o);
    }
    if (lane == 0) {
      atomicAdd(&A.counters[0], a);  // each lane counted its own pieces
      atomicAdd(&A.counters[1], b);
      atomicAdd(&A.counters[3], x);
    }
  }
}

// FP32 kernel: what is left in the warps' fallback buffers, one entry per thread, into the
// fixed-point rows.  At the end of k_dynamic each warp would walk its last few hundred entries
// (the per-vertex table took up to 50 us a round, most of its lanes in the FP64 branch of
// near-degenerate knots) while finished SMs idle: 30% of the time of a 64 x 64 x 16 pass.
// 64 x 64 x 16, 10 bands: 0.35 ms a pass, 1.05 with the per-vertex table for every entry.
__global__ void __launch_bounds__(128) k_dyn_fallback(DynBufs db, int nbuf, int nrows, float tau,
                                                      unsigned long long *__restrict__ counters) {
  unsigned long long *row = db.fx + (size_t)(blockIdx.x % nrows) * 2 * kNWPass;
  int nfp64 = 0;
  for (int buf = blockIdx.x; buf < nbuf; buf += gridDim.x) {
    const int n = db.fbn[buf];
    const FbEnt<float> *ent = (const FbEnt<float> *)db.fb + (size_t)buf * DynShape<false>::fb;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const FbEnt<float> &o = ent[k];
      float x[4], f[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        x[i] = o.x[i];
        f[i] = o.f[i];
      }
      const float v = o.v * near_term<false>(x, f, tau, nfp64);
      atomicAdd(&row[o.code >> 1], (unsigned long long)fx_of(v));
    }
  }
  if (counters && nfp64) atomicAdd(&counters[1], (unsigned long long)nfp64);
}

// box totals: slot i summed over the rows of the weight launch (FP64 kernel: per-warp FP64
// partials, in warp order; FP32 kernel: per-CTA fixed-point rows, summed exactly)
template <bool FP64>
__global__ void __launch_bounds__(256) k_box_sum(const double *__restrict__ part, int nrows, double *__restrict__ tot) {
  constexpr int NS = box_slots<FP64>();
  // 8 threads per slot, each a contiguous run of rows, added in run order
  __shared__ double red[8][32];
  const int i = blockIdx.x * 32 + (threadIdx.x & 31), run = threadIdx.x >> 5;
  const int per = (nrows + 7) / 8, r0 = run * per, r1 = min(nrows, r0 + per);
  if constexpr (FP64) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    if (i < NS) {
      int r = r0;
      for (; r + 3 < r1; r += 4) {
        s0 += part[(size_t)r * NS + i];
        s1 += part[(size_t)(r + 1) * NS + i];
        s2 += part[(size_t)(r + 2) * NS + i];
        s3 += part[(size_t)(r + 3) * NS + i];
      }
      for (; r < r1; ++r) s0 += part[(size_t)r * NS + i];
    }
    red[run][threadIdx.x & 31] = (s0 + s1) + (s2 + s3);
    __syncthreads();
    if (run == 0 && i < NS) {
      double s = 0.0;
      for (int k = 0; k < 8; ++k) s += red[k][threadIdx.x];
      tot[i] = s;
    }
  } else {
    const unsigned long long *fx = (const unsigned long long *)part;
    unsigned long long a = 0ull;
    if (i < NS) {
#pragma unroll 4
      for (int r = r0; r < r1; ++r) a += fx[(size_t)r * NS + i];
    }
    red[run][threadIdx.x & 31] = __longlong_as_double((long long)a);
    __syncthreads();
    if (run == 0 && i < NS) {
      a = 0ull;
      for (int k = 0; k < 8; ++k) a += (unsigned long long)__double_as_longlong(red[k][threadIdx.x]);
      tot[i] = (double)(long long)a * kFxUnit;
    }
  }
}

// One block per frequency iw (caller's order): the weight launch's sums of its sorted place and the
// boxes' share of Re (FP64 evaluation of the multipoles), normalised, into re[iw] and im[iw].
// FP32 kernel: rows are CTAs' fixed-point sums (added exactly); FP64: per-warp partials.
template <bool FP64>
__global__ void __launch_bounds__(128) k_dyn_out(const double *__restrict__ omega, int nw, const void *__restrict__ tabp,
                                                 const double *__restrict__ tot, DynBufs db, int nrows, double scale,
                                                 const double *__restrict__ dos, int ndos, double *__restrict__ re,
                                                 double *__restrict__ im) {
  using T = typename std::conditional<FP64, double, float>::type;
  using S = DynShape<FP64>;
  const BoxTab<T> &tb = *(const BoxTab<T> *)tabp;
  const int iw = blockIdx.x;
  const double wv = omega[iw], u = fabs(wv);
  const int rk = tb.rank[iw];
  if (rk >= tb.nv) {  // not finite: Re of a NaN is NaN, at infinity everything is 0
    if (threadIdx.x == 0) {
      if (re) re[iw] = wv != wv ? wv : 0.0;
      im[iw] = 0.0;
    }
    return;
  }
  const T om = tb.om[rk];
  double v = 0.0, vi = 0.0;
  unsigned long long ar = 0ull, ai = 0ull;
  if constexpr (FP64) {
    for (int r = threadIdx.x; r < nrows; r += blockDim.x) {
      if (re) v += db.partR[(size_t)r * nw + rk];
      vi += db.partI[(size_t)r * nw + rk];
    }
  } else {
    for (int r = threadIdx.x; r < nrows; r += blockDim.x) {
      ar += db.fx[(size_t)r * 2 * kNWPass + rk];
      ai += db.fx[((size_t)r * 2 + 1) * kNWPass + rk];
    }
  }
  if (re && tb.on) {
    for (int b = threadIdx.x; b < kBoxes; b += blockDim.x) {
      const int K = box_terms<FP64>(b);
      const double *M = tot + slot_base<FP64>(b);
      const double *P = (FP64 ? kBoxPolyD.v : kBoxPolyF.v) +
                        (b < kBoxFine ? 0 : (b < kBoxFine + kBoxG ? S::KF : S::KF + S::KG));
      const double C = (double)tb.C[b], R = (double)tb.R[b];
      for (int term = 0; term < 2; ++term) {
        if (!box_far(tb.C[b], tb.R[b], b, om, term)) continue;
        const double den = term ? C + u : C - u;
        const double z = R / den;
        double s = P[K - 1] * M[K - 1];
        for (int k = K - 2; k >= 0; --k) s = s * z + P[k] * M[k];
        v += s / den;
      }
    }
  }
  if (re && dos && wv == 0.0)
    for (int i = threadIdx.x; i < ndos; i += blockDim.x) v += dos[i];
  __shared__ double red[2][4];
  __shared__ unsigned long long rad[2][4];
  v = grid::warp_sum(v);
  vi = grid::warp_sum(vi);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ar += __shfl_xor_sync(kFull, ar, o);
    ai += __shfl_xor_sync(kFull, ai, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = v;
    red[1][threadIdx.x >> 5] = vi;
    rad[0][threadIdx.x >> 5] = ar;
    rad[1][threadIdx.x >> 5] = ai;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    v = (red[0][0] + red[0][1]) + (red[0][2] + red[0][3]);
    vi = (red[1][0] + red[1][1]) + (red[1][2] + red[1][3]);
    if constexpr (!FP64) {
      const double unit = kFxUnit / (double)tb.S;
      v += (double)(long long)(rad[0][0] + rad[0][1] + rad[0][2] + rad[0][3]) * unit;
      vi = (double)(long long)(rad[1][0] + rad[1][1] + rad[1][2] + rad[1][3]) * unit;
    }
    if (re) re[iw] = scale * v;
    im[iw] = wv < 0.0 ? -scale * vi : scale * vi;
  }
}

template <bool FP64> size_t dyn_smem() { return FP64 ? 0 : (size_t)box_slots<FP64>() * 2 * sizeof(unsigned); }

// Tetrahedra per unit (as log2): 32 at most, fewer on small meshes or wide windows, as long as a
// unit keeps items (about a quarter of the window's pairs per tetrahedron) for full rounds of 32.
// FP64 units are assigned statically: a few per warp even them out.
int dyn_unit_log2(long long ntet, int w, bool fp64) {
  int t = 5;
  const long long ww = (long long)w * w, want = fp64 ? 4864 : 20480, least = fp64 ? 256 : 1024;
  while (t > 0 && (ntet >> t) < want && (ww << t) > least) --t;
  return t;
}

template <bool FP64, bool IMO>
cudaError_t launch_weights(const DynArgs &a, const double *omega, int nw, int nblocks, double scale, const double *dos,
                           int ndos, double *re, double *im, cudaStream_t s) {
  using T = typename std::conditional<FP64, double, float>::type;
  const DynBufs &db = a.db;
  constexpr int NS = box_slots<FP64>();
  const int rows = FP64 ? nblocks * DynShape<FP64>::warps : nblocks;
  cudaError_t e = cudaSuccess;
  if (!FP64) e = cudaMemsetAsync(db.ctr, 0, sizeof(unsigned long long), s);
  else if (!IMO) e = cudaMemsetAsync(db.box_part, 0, sizeof(double) * (size_t)rows * NS, s);
  if (e != cudaSuccess) return e;
  k_box_setup<T><<<1, kNWPass, 0, s>>>(omega, nw, IMO ? 0 : 1, db.erange, a.q.lo, a.q.hi, (BoxTab<T> *)db.box_tab);
  k_dynamic<FP64, IMO><<<nblocks, DynShape<FP64>::threads, IMO ? 0 : dyn_smem<FP64>(), s>>>(
      a, nw, dyn_unit_log2(a.g.ntet, a.q.hi - a.q.lo, FP64));
  if (!FP64 && !IMO) k_dyn_fallback<<<rows * DynShape<FP64>::warps, 128, 0, s>>>(db, rows * DynShape<FP64>::warps, rows, a.tau, a.counters);
  if (!IMO) k_box_sum<FP64><<<(NS + 31) / 32, 256, 0, s>>>(db.box_part, rows, db.box_tot);
  k_dyn_out<FP64><<<nw, 128, 0, s>>>(omega, nw, db.box_tab, db.box_tot, db, rows, scale, dos, ndos, IMO ? nullptr : re, im);
  return cudaGetLastError();
}

}  // namespace

int dynamic_max_nw() { return kNWPass; }
int dynamic_warps_per_cta(int fp64) { return fp64 ? DynShape<true>::warps : DynShape<false>::warps; }
size_t dynamic_box_slots(int fp64) { return fp64 ? box_slots<true>() : box_slots<false>(); }
size_t dynamic_fx_bytes(int nblocks) { return (size_t)nblocks * 2 * kNWPass * sizeof(unsigned long long); }
size_t dynamic_fb_bytes(int fp64) {
  return fp64 ? DynShape<true>::fb * sizeof(FbEnt<double>) : DynShape<false>::fb * sizeof(FbEnt<float>);
}
size_t dynamic_box_tab_bytes() {
  return sizeof(BoxTab<double>) > sizeof(BoxTab<float>) ? sizeof(BoxTab<double>) : sizeof(BoxTab<float>);
}

cudaError_t dynamic_prepare() {
  return cudaFuncSetAttribute(k_dynamic<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn_smem<false>());
}

// Re and Im (im_only: Im alone, for the Kramers-Kronig route) of one q and nw <= dynamic_max_nw()
// frequencies into re[nw], im[nw]
cudaError_t launch_dynamic(const DynArgs &a, int fp64, int im_only, const double *omega, int nw, int nblocks,
                           double scale, const double *dos, int ndos, double *re, double *im, cudaStream_t s) {
  const DynBufs &db = a.db;
  if (nw > kNWPass || nw <= 0 || nblocks <= 0) return cudaErrorInvalidValue;
  if (!fp64 && (!a.Eklo || !a.Ekqlo || !db.erange)) return cudaErrorInvalidValue;
  if (!db.box_tab || !db.box_part || !db.box_tot || !db.fb || !db.fbn || !db.fx || !db.ctr || !db.partR || !db.partI)
    return cudaErrorInvalidValue;
  if (fp64)
    return im_only ? launch_weights<true, true>(a, omega, nw, nblocks, scale, dos, ndos, re, im, s)
                   : launch_weights<true, false>(a, omega, nw, nblocks, scale, dos, ndos, re, im, s);
  return im_only ? launch_weights<false, true>(a, omega, nw, nblocks, scale, dos, ndos, re, im, s)
                 : launch_weights<false, false>(a, omega, nw, nblocks, scale, dos, ndos, re, im, s);
}

int dynamic_max_ctas_per_sm(int fp64) {
  int nb = 0;
  cudaError_t e = fp64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_dynamic<true>, DynShape<true>::threads,
                                                                      dyn_smem<true>())
                       : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_dynamic<false>,
                                                                      DynShape<false>::threads, dyn_smem<false>());
  return (e != cudaSuccess || nb < 1) ? 1 : nb;
}

int dynamic_persistent_blocks(int fp64) { return dynamic_max_ctas_per_sm(fp64) * device_sms(); }

}  // namespace chi0int
