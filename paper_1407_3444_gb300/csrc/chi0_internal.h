// chi0_internal.h -- interface between the C-ABI layer and the kernel translation unit.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace chi0int {

// n / d for 32-bit unsigned n by a multiply-high and shifts (Granlund-Montgomery): no
// integer-division sequence and no int<->float conversions in the index arithmetic.
struct FastDiv {
  unsigned d, m, s;
};
inline FastDiv make_fastdiv(unsigned d) {
  FastDiv f{d, 0u, 0u};
  if (d <= 1) return f;
  unsigned l = 0;
  while ((1ull << l) < d) ++l;                                   // l = ceil(log2 d)
  f.m = (unsigned)((((1ull << l) - d) << 32) / d + 1);           // floor(2^32 (2^l - d)/d) + 1
  f.s = l - 1;
  return f;
}
#ifdef __CUDACC__
__device__ __forceinline__ unsigned fdiv(unsigned n, const FastDiv &f) {
  if (f.d <= 1) return n;
  const unsigned t = __umulhi(n, f.m);
  return (t + ((n - t) >> 1)) >> f.s;
}
#endif

struct Grid {
  int n[3];   // cubes per axis
  int N[3];   // corners per axis
  int periodic;
  int nb, norb;
  long long nc;    // corners (< 2^31, checked when the plan is built)
  long long ntet;  // tetrahedra (< 2^31)
  double ef;
  FastDiv fn1, fn2;  // cube index decode: n1, n2
  FastDiv fN1, fN2;  // corner index decode: N1, N2
};

struct Tet {
  const int4 *corners;  // device [ntet] or nullptr (builtin mesh)
  const double *vol;    // device [ntet] or nullptr
  double vol_builtin;   // 1/(6 n0 n1 n2)
};

// one q point as the kernels see it
struct Q {
  const double *Eq;  // device [nc][nb] explicit energies at k+q, or nullptr (shift)
  const void *Cq;    // device [nc][norb][nb] explicit eigenvectors at k+q, or nullptr
  int shift[3];
  int lo, hi;        // band window
  int gamma;
};

enum { DT_C64 = 1, DT_C128 = 2 };

// q points that one launch may cover: their descriptors travel as a kernel argument (4 KB)
constexpr int kMaxGroup = 32;

// |M_mn|^2 at every k corner for a group of q: W2[iq][c][m-lo][n-lo] (fp64: double, else float);
// the q points are all explicit or all on-grid shifts
struct OverlapArgs {
  Grid g;
  int nq;
  Q q[kMaxGroup];
  void *W2[kMaxGroup];
};
cudaError_t launch_overlap(const OverlapArgs &a, const void *C, int dtype, int fp64, cudaStream_t s, const void *C32,
                           int *launches = nullptr);
// complex128 -> complex64 copy (the k-side eigenvectors of a mixed-precision plan)
cudaError_t launch_c128_to_c64(const void *in, void *out, long long n, cudaStream_t s);

// band bounds per corner: occ[c] (1 + highest occupied band), emp[c] (lowest empty band), occf[c]
// (bands below it are all occupied), empf[c] (bands from it on are all empty)
struct BandBounds {
  short *occ, *emp, *occf, *empf;
};
// Bounds of nq sets of energies E[iq] (set iq's outputs iq * stride_c / stride_e further on);
// E32 (optional) receives (float)(E - ef); E32lo (optional) the remainder
// (float)((E - ef) - E32), so that E32 + E32lo carries E - ef to ~2^-48 relative
struct BandArgs {
  const double *E[kMaxGroup];
  BandBounds out;
  float *E32, *E32lo;
  size_t stride_c, stride_e;
};
cudaError_t launch_bands(const BandArgs &a, int nq, long long nc, int nb, double ef, cudaStream_t s);
// out[band] = bits of the band's largest finite |E - eF| (they give the scale of the FP32 dynamic weights' sums)
cudaError_t launch_energy_range(const double *E, long long nc, int nb, double ef, unsigned long long *out,
                                cudaStream_t s);

// one q of a static launch: k+q energies (FP64 absolute, or FP32 relative to eF) and their band
// bounds, |M|^2, one FP64 partial per unit, the band-pair totals (or none), the Gamma DOS
// partials (or none); u0, tlog: set by launch_static
struct StaticQ {
  Q q;
  const void *Ekq, *W2;
  const short *emp, *empf;
  double *partial;
  unsigned long long *pairs;
  const double *dos;
  int u0, tlog;
};
struct StaticArgs {
  Grid g;
  Tet tet;
  const void *Ek;            // k energies: FP64 absolute, or FP32 relative to eF
  const short *occ, *occf;   // their band bounds
  int cma;
  float tau;
  int *next;                 // unit counter
  unsigned long long *counters;  // profile: pieces, FP64 evaluations, queue overflows (or none)
  int nq, units;
  StaticQ q[kMaxGroup];
};
// static weights of a group of q points, then chi = scale * (sum of partials (+ Gamma DOS))
cudaError_t launch_static(StaticArgs &a, int fp64, int nblocks, cudaStream_t s, int variant = 0);
cudaError_t launch_static_reduce(const StaticArgs &a, double scale, int ndos, double *out, cudaStream_t s);
int static_persistent_blocks(int fp64);
long long static_batches(long long ntet);  // runs of 32 tetrahedra (the no-allocation entry point sizes its array by them)
// partials of one q with a window of w bands (never more with a narrower one)
long long static_units(long long ntet, int w);

// message of the last failed call made without a plan (chi0_last_error(NULL))
void set_global_error(const char *msg);

// Work buffers of the dynamic weights
struct DynBufs {
  double *partR, *partI;    // FP64 kernel: [warps of the launch][nw]
  void *box_tab;            // boxes and sorted frequencies of the pass (dynamic_box_tab_bytes())
  double *box_part;         // box moments: FP64 [warps of the launch][dynamic_box_slots(1)], FP32 int64 per CTA
  double *box_tot;          // [dynamic_box_slots(fp64)]
  void *fb;                 // [warps of the launch][dynamic_fb_bytes(fp64)]: near-field entries
                            // left to the per-vertex table (scratch)
  int *fbn;                 // FP32 kernel: [warps of the launch] entries left at its end
  unsigned long long *fx;   // FP32 kernel: [CTAs of the launch][2][dynamic_max_nw()] fixed-point sums
  unsigned long long *ctr;  // FP32 kernel: unit counter (reset by the launch)
  const unsigned long long *erange;  // FP32 kernel: largest |E - eF| of every band (bits of doubles)
};
// one q of a dynamic launch: energies FP64 absolute, or FP32 relative to eF (hi and lo parts), their
// band bounds, |M|^2
struct DynArgs {
  Grid g;
  Tet tet;
  Q q;
  const void *Ek, *Ekq, *W2;
  const float *Eklo, *Ekqlo;
  const short *occ, *occf, *emp, *empf;
  int cma;
  float tau;
  DynBufs db;
  unsigned long long *counters;  // profile (or none)
};

// dynamic weights of one q and nw <= dynamic_max_nw() frequencies: re[nw], im[nw] = scale times the
// sums (at w = 0 the sum of dos[0..ndos) is added to re); im_only: Im alone (the Kramers-Kronig route)
cudaError_t launch_dynamic(const DynArgs &a, int fp64, int im_only, const double *omega, int nw, int nblocks,
                           double scale, const double *dos, int ndos, double *re, double *im, cudaStream_t s);
size_t dynamic_fx_bytes(int nblocks);
// energies and eigenvectors at k+q (fractional q) by linear interpolation from the periodic
// mesh (chi0_interp.cu): Eq [nc][nb], Cq [nc][norb][nb] (C == nullptr: energies only), c64:
// complex64 vectors, else complex128
cudaError_t launch_interp_kq(const Grid &g, const double *E, const void *C, int c64, const double q[3], double *Eq,
                             void *Cq, cudaStream_t s);
// Re from Im (Kramers-Kronig, chi0_kk.cu): im[0..m) on u_j = j du (im[0] = 0, im = 0 from u_m on),
// re[i] at u_i, i < m, plus scale * (sum of dos[0..ndos)) at u = 0 when dos != NULL
cudaError_t launch_kk(const double *im, int m, double du, double scale, const double *dos, int ndos, double *re,
                      cudaStream_t s);
int dynamic_persistent_blocks(int fp64);
int dynamic_warps_per_cta(int fp64);
size_t dynamic_box_slots(int fp64);
size_t dynamic_box_tab_bytes();
size_t dynamic_fb_bytes(int fp64);
cudaError_t dynamic_prepare();  // kernel attributes (shared memory); call outside stream capture

// Gamma: intraband q -> 0 limit, tetrahedron DOS at eF: partial[nblocks]
cudaError_t launch_dos(const Grid &g, const Tet &tet, const double *E, int lo, int hi, double *partial,
                       int nblocks, cudaStream_t s, unsigned long long *pairs = nullptr);
// band-pair output: out[i] = scale * pairs[i] in FP64 (pairs: fixed-point totals of the static kernels)
cudaError_t launch_pairs_out(const unsigned long long *pairs, int n, double scale, double *out, cudaStream_t s);

int static_blocks();
int dynamic_max_nw();

// |M_mn|^2 on the tensor cores (mixed precision): k side from the plan's complex64 copy C32,
// k+q side from q.Cq (complex64 or complex128, explicit) or C32 at the shifted corner.
// W2[c][m-lo][n-lo] FP32.  budget: clock cycles a bounded wait may take (<= 0: 2^31);
// test_stall: issue no MMA, so that the first wait runs out (error-path test).  A wait that
// runs out sets *err to 1.
enum { TC_TF32 = 0, TC_BF16X3 = 1, TC_BF16X6 = 2 };
constexpr size_t kTcSmemMax = 227 * 1024;
size_t overlap_tc_smem(int w, int norb, int mode);  // bytes of shared memory ((size_t)-1: w > 128)
int overlap_tc_max_corners(int w, int norb, int mode);  // corners per MMA round, untuned
// gcap > 0: at most gcap corners per MMA round (autotuner candidates)
cudaError_t launch_overlap_tc(const Grid &g, const void *C32, int dtype, const Q &q, float *W2, int mode,
                              long long budget, int test_stall, int gcap, int *err, cudaStream_t s);
// tensor-core throughput (TFLOP/s) of `iters` back-to-back MMAs per SM, M = 128, N = 256
cudaError_t tc_peak(int mode, int iters, double *tflops, double *ms);
// resident CTAs per SM of the weight kernels (occupancy limit) and SMs of the device
int static_max_ctas_per_sm(int fp64, int variant);
int static_variants(int fp64);                      // block shapes of the static weight kernel
int static_variant_threads(int fp64, int variant);  // threads per block of a shape
int dynamic_max_ctas_per_sm(int fp64);
int device_sms();

#ifdef __CUDACC__
// corner index with periodic wrap (32-bit: the plan checks that the mesh has fewer than 2^31
// corners), and the corner at integer offset s from corner c
__device__ __forceinline__ int wrap_idx(int i, int N) { return i >= N ? i - N : i; }
__device__ __forceinline__ long long cid(const Grid &g, int i0, int i1, int i2) {
  if (g.periodic) {
    i0 = wrap_idx(i0, g.N[0]);
    i1 = wrap_idx(i1, g.N[1]);
    i2 = wrap_idx(i2, g.N[2]);
  }
  return (long long)(unsigned)((i0 * g.N[1] + i1) * g.N[2] + i2);
}
__device__ __forceinline__ long long shift_corner(const Grid &g, long long c, const int s[3]) {
  const unsigned cu = (unsigned)c;
  const unsigned r = fdiv(cu, g.fN2);
  const int i2 = (int)(cu - r * (unsigned)g.N[2]);
  const unsigned i0 = fdiv(r, g.fN1);
  const int i1 = (int)(r - i0 * (unsigned)g.N[1]);
  return cid(g, (int)i0 + s[0], i1 + s[1], i2 + s[2]);
}
#endif

}  // namespace chi0int
