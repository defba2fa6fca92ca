// chi0_noalloc.cu -- chi0_static_noalloc: static chi0 with every work buffer in one
// file-scope device array instead of cudaMalloc'd memory.
//
// For callers that cannot allocate device memory at the point where they need chi0:
// cudaMalloc and cudaFree can synchronize the whole device and take unbounded time,
// which a real-time loop or a step inside a latency budget cannot afford, and some host
// applications hand all device memory to their own pool allocator, which must account
// for every byte and does not tolerate raw allocations beside it.  Such callers keep
// their inputs and outputs in memory they already own and let this entry point use the
// fixed scratch array below.
//
// The array (CHI0_NOALLOC_SCRATCH_BYTES) is part of the library image: every GPU that
// loads the library holds it until the process exits.  Host code cannot use the array's
// name as a device address; its address is looked up with cudaGetSymbolAddress once per
// device, the first time the entry point runs on that device (with the device current).
// All calls share the array and it keeps the previous call's contents, so everything that
// must start at zero is cleared on the caller's stream; two calls that overlap on the GPU
// (different streams, or different host threads on one device) race on it.
#include <cuda_runtime.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <mutex>

#include "../../include/chi0.h"
#include "chi0_internal.h"

using namespace chi0int;

static __device__ __align__(256) unsigned char g_chi0_scratch[CHI0_NOALLOC_SCRATCH_BYTES];

namespace {

constexpr int kMaxDevices = 64;
// the array's work region per run of 32 tetrahedra: 640 (FP32) or 1280 (FP64) bytes, of which
// the unit partials (at most eight a run, 64 bytes) and the band bounds beyond occ and emp (8 bytes a
// corner) take two fifths at most (FP32, an open 1 x 1 x 5 mesh)
constexpr size_t kNoallocWork32 = 640, kNoallocWork64 = 1280;
unsigned char *g_scratch_ptr[kMaxDevices] = {nullptr};
std::mutex g_scratch_mu;

int err(int code, const char *fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  set_global_error(buf);
  return code;
}

// device address of the scratch array on the current device (looked up once per device)
int scratch_base(unsigned char **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return err(CHI0_ECUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return err(CHI0_ENOTSUP, "device %d beyond %d", dev, kMaxDevices);
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (!g_scratch_ptr[dev]) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_chi0_scratch);
    if (e != cudaSuccess || !p)
      return err(CHI0_ECUDA, "cudaGetSymbolAddress(scratch): %s", cudaGetErrorString(e));
    g_scratch_ptr[dev] = (unsigned char *)p;
  }
  *out = g_scratch_ptr[dev];
  return CHI0_OK;
}

constexpr size_t kSat = ~(size_t)0;  // saturated size: larger than any scratch array

// a * b and a + b rounded up to 256, saturating at kSat instead of wrapping around
size_t mul_sat(size_t a, size_t b) { return (b != 0 && a > kSat / b) ? kSat : a * b; }
size_t align256(size_t x) { return x > kSat - 255 ? kSat : (x + 255) & ~(size_t)255; }

struct Layout {
  size_t bounds, E32, Eq32, C32, W2, next, counters, work, dos, total;
};

Layout layout(const Grid &g, int w, int fp64, int cma, int dtype) {
  Layout L{};
  // every size saturates instead of wrapping, so a mesh too large for the array can never
  // come out small here (total == kSat then fails the size check)
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = align256(bytes > kSat - o ? kSat : o + bytes);
    return at;
  };
  const size_t nc = (size_t)g.nc, nb = (size_t)g.nb, no = (size_t)g.norb, ww = (size_t)w;
  const size_t nbatch = (size_t)static_batches(g.ntet);
  L.bounds = take(mul_sat(sizeof(short), nc));  // occ, emp, and the same at k+q
  take(mul_sat(sizeof(short), nc));
  take(mul_sat(sizeof(short), nc));
  take(mul_sat(sizeof(short), nc));
  L.E32 = take(fp64 ? 0 : mul_sat(mul_sat(sizeof(float), nc), nb));
  L.Eq32 = take(fp64 ? 0 : mul_sat(mul_sat(sizeof(float), nc), nb));
  L.C32 = take((!fp64 && !cma && dtype == CHI0_C128) ? mul_sat(mul_sat(mul_sat(8, nc), no), nb) : 0);
  L.W2 = take(cma ? 0 : mul_sat(mul_sat(mul_sat(fp64 ? 8 : 4, nc), ww), ww));
  L.next = take(sizeof(int));
  L.counters = take(4 * sizeof(unsigned long long));
  L.work = take(mul_sat(fp64 ? kNoallocWork64 : kNoallocWork32, nbatch));
  // not used: with these two the same meshes fit the array as in every version so far
  take(mul_sat(sizeof(int), nbatch));
  take(mul_sat(sizeof(double), mul_sat(2, nbatch)));
  L.dos = take(mul_sat(sizeof(double), (size_t)static_blocks()));
  L.total = o;
  return L;
}

}  // namespace

extern "C" int chi0_static_noalloc(const chi0_kgrid_t *kg, chi0_band_window_t win, const chi0_opts_t *opts,
                                   const chi0_q_t *qs, int nq, double *chi) {
  if (!kg || !opts || !qs || !chi || nq <= 0) return err(CHI0_EINVAL, "NULL argument or nq <= 0");
  const chi0_opts_t &op = *opts;
  if (op.precision != CHI0_PREC_FP64 && op.precision != CHI0_PREC_MIXED)
    return err(CHI0_EINVAL, "precision %d unknown", op.precision);
  if (op.overlap != CHI0_OVL_FP32) return err(CHI0_ENOTSUP, "only the FP32 overlap mode is available here");
  for (int d = 0; d < 3; ++d)
    if (kg->n[d] < 1 || kg->n[d] > (1 << 12)) return err(CHI0_EINVAL, "n[%d] = %d out of range", d, kg->n[d]);
  if (kg->nbands < 1 || kg->nbands > 4096) return err(CHI0_EINVAL, "nbands = %d out of range", kg->nbands);
  if (!kg->energies) return err(CHI0_EINVAL, "energies is NULL");
  if (!op.cma && (!kg->evecs || kg->norb < 1 || (kg->evec_dtype != CHI0_C64 && kg->evec_dtype != CHI0_C128)))
    return err(CHI0_EINVAL, "eigenvectors (norb, dtype) required without CMA");
  if (!op.cma && kg->norb > 65536) return err(CHI0_EINVAL, "norb = %d out of range", kg->norb);
  if (win.lo < 0 || win.hi > kg->nbands || win.lo >= win.hi)
    return err(CHI0_EINVAL, "band window [%d, %d) outside [0, %d)", win.lo, win.hi, kg->nbands);
  const int fp64 = op.precision == CHI0_PREC_FP64;
  Grid g{};
  for (int d = 0; d < 3; ++d) {
    g.n[d] = kg->n[d];
    g.N[d] = kg->periodic ? kg->n[d] : kg->n[d] + 1;
  }
  g.periodic = kg->periodic ? 1 : 0;
  g.nb = kg->nbands;
  g.norb = op.cma ? 0 : kg->norb;
  g.nc = (long long)g.N[0] * g.N[1] * g.N[2];
  g.ntet = 6LL * g.n[0] * g.n[1] * g.n[2];
  g.ef = kg->e_fermi;
  g.fn1 = make_fastdiv((unsigned)g.n[1]);
  g.fn2 = make_fastdiv((unsigned)g.n[2]);
  g.fN1 = make_fastdiv((unsigned)g.N[1]);
  g.fN2 = make_fastdiv((unsigned)g.N[2]);
  if (g.nc >= (1LL << 31) || g.ntet >= (1LL << 31)) return err(CHI0_EINVAL, "mesh too large");
  const int dtype = op.cma ? CHI0_C128 : kg->evec_dtype;
  const int w = win.hi - win.lo;
  const Layout L = layout(g, w, fp64, op.cma, dtype);
  if (L.total > (size_t)CHI0_NOALLOC_SCRATCH_BYTES)
    return err(CHI0_EINVAL, "this mesh needs %zu bytes of scratch; chi0_static_noalloc has %zu", L.total,
               (size_t)CHI0_NOALLOC_SCRATCH_BYTES);
  // q descriptors: windows and shifts (device pointers are the caller's)
  for (int iq = 0; iq < nq; ++iq) {
    const chi0_q_t &qd = qs[iq];
    const int lo = qd.win.lo < 0 ? win.lo : qd.win.lo, hi = qd.win.lo < 0 ? win.hi : qd.win.hi;
    if (lo < win.lo || hi > win.hi || lo >= hi) return err(CHI0_EINVAL, "q %d window outside the window", iq);
    if (qd.e_kq && !op.cma && !qd.c_kq) return err(CHI0_EINVAL, "q %d: e_kq without c_kq", iq);
    if (!qd.e_kq && !g.periodic) return err(CHI0_EINVAL, "q %d: on-grid shift needs a periodic grid", iq);
  }

  unsigned char *base = nullptr;
  int rc = scratch_base(&base);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)op.stream;
  // band bounds: occ, emp (k and k+q) in their own region, occf, empf in the work region
  const size_t cs = align256(sizeof(short) * (size_t)g.nc) / sizeof(short);
  short *bb = (short *)(base + L.bounds), *wb = (short *)(base + L.work);
  const BandBounds kb{bb, bb + cs, wb, wb + g.nc}, qb{bb + 2 * cs, bb + 3 * cs, wb + 2 * g.nc, wb + 3 * g.nc};
  float *E32 = fp64 ? nullptr : (float *)(base + L.E32), *Eq32 = fp64 ? nullptr : (float *)(base + L.Eq32);
  void *C32 = (!fp64 && !op.cma && dtype == CHI0_C128) ? (void *)(base + L.C32) : nullptr;
  void *W2 = op.cma ? nullptr : (void *)(base + L.W2);
  int *next = (int *)(base + L.next);
  double *part = (double *)(base + L.work + ((4 * sizeof(short) * (size_t)g.nc + 7) & ~(size_t)7));
  double *dos = (double *)(base + L.dos);
  Tet tet{nullptr, nullptr, 1.0 / (6.0 * g.n[0] * g.n[1] * g.n[2])};
  const double scale = op.sign == CHI0_SIGN_PAPER ? -2.0 : 2.0;
  cudaError_t e;
#define NA_CK(call)                                                                                  \
  do {                                                                                               \
    if ((e = (call)) != cudaSuccess) return err(CHI0_ECUDA, "%s: %s", #call, cudaGetErrorString(e)); \
  } while (0)
  BandArgs ba{};
  ba.E[0] = kg->energies;
  ba.out = kb;
  ba.E32 = E32;
  NA_CK(launch_bands(ba, 1, g.nc, g.nb, g.ef, s));
  if (C32) NA_CK(launch_c128_to_c64(kg->evecs, C32, g.nc * (long long)g.norb * g.nb, s));
  const int grid = static_persistent_blocks(fp64);
  for (int iq = 0; iq < nq; ++iq) {
    const chi0_q_t &qd = qs[iq];
    Q q{};
    q.lo = qd.win.lo < 0 ? win.lo : qd.win.lo;
    q.hi = qd.win.lo < 0 ? win.hi : qd.win.hi;
    q.gamma = qd.gamma ? 1 : 0;
    bool zero = true;
    if (qd.e_kq) {
      q.Eq = qd.e_kq;
      q.Cq = qd.c_kq;
    } else {
      for (int d = 0; d < 3; ++d) {
        int v = qd.shift[d] % g.N[d];
        if (v < 0) v += g.N[d];
        q.shift[d] = v;
        zero = zero && v == 0;
      }
      if (zero) q.gamma = 1;
    }
    if (!op.cma) {
      OverlapArgs oa{};
      oa.g = g;
      oa.nq = 1;
      oa.q[0] = q;
      oa.W2[0] = W2;
      NA_CK(launch_overlap(oa, kg->evecs, dtype, fp64, s, C32));
    }
    if (q.gamma) NA_CK(launch_dos(g, tet, kg->energies, q.lo, q.hi, dos, static_blocks(), s));
    if (q.Eq) {
      BandArgs bq{};
      bq.E[0] = q.Eq;
      bq.out = qb;
      bq.E32 = Eq32;
      NA_CK(launch_bands(bq, 1, g.nc, g.nb, g.ef, s));
    }
    StaticArgs a{};
    a.g = g;
    a.tet = tet;
    a.Ek = fp64 ? (const void *)kg->energies : (const void *)E32;
    a.occ = kb.occ;
    a.occf = kb.occf;
    a.cma = op.cma;
    a.tau = (float)op.tau;
    a.next = next;
    a.nq = 1;
    StaticQ &d = a.q[0];
    d.q = q;
    d.Ekq = !q.Eq ? a.Ek : (fp64 ? (const void *)q.Eq : (const void *)Eq32);
    d.W2 = W2;
    d.emp = q.Eq ? qb.emp : kb.emp;
    d.empf = q.Eq ? qb.empf : kb.empf;
    d.partial = part;
    d.dos = q.gamma ? dos : nullptr;
    NA_CK(launch_static(a, fp64, grid, s));
    NA_CK(launch_static_reduce(a, scale, static_blocks(), chi + iq, s));
  }
#undef NA_CK
  return CHI0_OK;
}
