// chi0_kernels.cu -- sm_103a kernels of the doubly carved tetrahedron method.
//
//  k_overlap_small / k_overlap  (Eq. 1 matrix elements, tight-binding form of the Sec. III
//             footnote) on the CUDA cores: W2[c][m][n] = |sum_o conj(C_k[o][m]) C_{k+q}[o][n]|^2
//             at every k corner (the tensor-core form is in chi0_overlap_tc.cu).
//  k_bands    E - eF in FP32 (hi, and lo for the dynamic kernel) and the occupied / empty band
//             bounds of every corner.
//  (the static weights, Eq. 1 at w = 0, are in chi0_static.cu)
//  (the dynamic weights, Eqs. 1-3, are in chi0_dynamic.cu)
//  k_dos      Gamma: the intraband q -> 0 limit, tetrahedron DOS at eF (Sec. III).
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "chi0_grid.cuh"
#include "chi0_internal.h"
#include "chi0_math.cuh"

using namespace chi0dev;

namespace chi0int {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kSMs = 152;                 // default when the device cannot be queried
constexpr int kStaticBlocks = kSMs * 8;   // fixed grid of the DOS kernel (its partials)
using grid::kPairScale;
using grid::pair_add;
using grid::tet_corners;
using grid::warp_sum;

using grid::d2f_int;
template <typename T> __device__ __forceinline__ T cvt(double x) { return (T)x; }
template <> __device__ __forceinline__ float cvt<float>(double x) { return d2f_int(x); }
template <typename T> __device__ __forceinline__ T cvt(float x) { return (T)x; }

__device__ __forceinline__ void block_sum_store(double v, double *out) {
  __shared__ double red[kWarps];
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  if (lane == 0) red[wib] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < kWarps; ++i) s += red[i];
    *out = s;
  }
}

// ---------------------------------------------------------------- overlap
// Thread per output (m, n) at a corner: general sizes.
template <typename CT, typename T>
__global__ void __launch_bounds__(kThreads) k_overlap(const __grid_constant__ OverlapArgs A, const CT *__restrict__ C) {
  const Grid &g = A.g;
  const Q &q = A.q[blockIdx.y];
  const CT *Cqx = (const CT *)q.Cq;
  T *W2 = (T *)A.W2[blockIdx.y];
  const int w = q.hi - q.lo;
  const long long total = g.nc * (long long)w * w;
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const long long c = idx / ((long long)w * w);
    const int r = (int)(idx - c * w * w);
    const int mm = r / w, nn = r - (r / w) * w;
    const long long ck = Cqx ? c : shift_corner(g, c, q.shift);
    const CT *Cb = Cqx ? Cqx : C;
    T re = T(0), im = T(0);
    for (int o = 0; o < g.norb; ++o) {
      const CT x = C[(c * g.norb + o) * g.nb + q.lo + mm];
      const CT y = Cb[(ck * g.norb + o) * g.nb + q.lo + nn];
      const T xr = (T)x.x, xi = (T)x.y, yr = (T)y.x, yi = (T)y.y;
      re += xr * yr + xi * yi;  // conj(x) * y
      im += xr * yi - xi * yr;
    }
    W2[idx] = re * re + im * im;
  }
}

// Small blocks (norb * w <= kOvlSmall): a warp takes a run of corners, as many as its lanes hold
// 3 x 3 tiles of (m, n) for (three corners at w = 9, two at w = 10, 12; past 25 tiles one, whose
// tiles the lanes share out).  The eigenvector blocks C_k[:, lo:hi] and C_{k+q}[:, lo:hi] are read
// once, coalesced, into shared memory in the arithmetic precision; a lane then reads six complex
// numbers per orbital for its nine products, where one output per lane and step reads eighteen; and
// the blocks leave through shared memory, coalesced.
// Bound: FP32 memory and the shared-memory traffic of the tiles; FP64 the FP64 pipe (four FMAs per
// product; written as re += xr * yr + xi * yi they were six operations).  One output per lane, one
// corner at a time: 48^3 corners x 9 bands FP32 113 us, now 87; FP64, by the general form (one
// output per thread, operands from the caches): 24^3 x 9 bands 114 us, now 85.
constexpr int kOvlSmall = 256;
constexpr int kOvlBuf = 320;  // complex numbers staged a side: two corners of 12 x 12
template <typename T> constexpr int kOvlThreads = sizeof(T) == 8 ? 128 : 256;
__device__ __forceinline__ void conj_mul_add(float &re, float &im, float2 x, float2 y) {
  re += x.x * y.x + x.y * y.y;
  im += x.x * y.y - x.y * y.x;
}
__device__ __forceinline__ void conj_mul_add(double &re, double &im, double2 x, double2 y) {
  re = fma(x.x, y.x, re);
  im = fma(x.x, y.y, im);
  re = fma(x.y, y.y, re);
  im = fma(-x.y, y.x, im);
}
template <typename CT, typename CTq, typename T>
__global__ void __launch_bounds__(kOvlThreads<T>, 4) k_overlap_small(const __grid_constant__ OverlapArgs A,
                                                                  const CT *__restrict__ C, int explicit_q) {
  using V = typename std::conditional<sizeof(T) == 8, double2, float2>::type;
  constexpr int kW = kOvlThreads<T> / 32;
  const Grid &g = A.g;
  const Q &q = A.q[blockIdx.y];
  const CTq *Cb = explicit_q ? (const CTq *)q.Cq : (const CTq *)C;
  T *W2 = (T *)A.W2[blockIdx.y];
  __shared__ V sm[kW][2][kOvlBuf];  // both sides; then the outputs
  __shared__ long long s_ck[kW][32];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  V *sA = sm[wib][0], *sB = sm[wib][1];
  const int w = q.hi - q.lo, no = g.norb, nel = no * w, ww = w * w;
  const int tr = (w + 2) / 3, nt = tr * tr;  // tiles a side, tiles a corner
  int cpw = nt >= 32 ? 1 : 32 / nt;          // corners a step
  cpw = min(cpw, kOvlBuf / nel);
  const bool through = nt <= 32 && cpw * ww <= 2 * kOvlBuf;  // one round of tiles, and the outputs fit the buffers
  const int st_o = 32 / w, st_m = 32 - st_o * w, o0 = lane / w, m0 = lane - o0 * w;  // staging steps
  const int myj = nt >= 32 ? 0 : lane / nt, mytile = nt >= 32 ? lane : lane - myj * nt;
  for (long long c0 = ((long long)blockIdx.x * kW + wib) * cpw; c0 < g.nc; c0 += (long long)gridDim.x * kW * cpw) {
    const int nj = (int)(g.nc - c0 < cpw ? g.nc - c0 : cpw);
    if (lane < nj) s_ck[wib][lane] = explicit_q ? c0 + lane : shift_corner(g, c0 + lane, q.shift);
    __syncwarp();
    {
      // element i = (corner j, orbital o, band mm), i = lane, lane + 32, ...
      int j = 0, o = o0, mm = m0;
      while (o >= no) {
        o -= no;
        ++j;
      }
      const CT *Ck = C + c0 * no * g.nb + q.lo;
      for (int i = lane; i < nj * nel; i += 32) {
        const CT x = Ck[(j * no + o) * g.nb + mm];
        const CTq y = Cb[(s_ck[wib][j] * no + o) * g.nb + q.lo + mm];
        V a, b;
        a.x = cvt<T>(x.x);
        a.y = cvt<T>(x.y);
        b.x = cvt<T>(y.x);
        b.y = cvt<T>(y.y);
        sA[i] = a;
        sB[i] = b;
        mm += st_m;
        o += st_o;
        if (mm >= w) {
          mm -= w;
          ++o;
        }
        while (o >= no) {
          o -= no;
          ++j;
        }
      }
    }
    __syncwarp();
    for (int base = 0; base < (nt >= 32 ? nt : 1); base += 32) {  // warp-uniform
      const int t = base + mytile;
      const bool on = myj < nj && t < nt;
      const int ti = on ? t / tr : 0, tj = on ? t - ti * tr : 0;
      int mi[3], ni[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        mi[k] = min(ti * 3 + k, w - 1);
        ni[k] = min(tj * 3 + k, w - 1);
      }
      const V *a = sA + (on ? myj : 0) * nel, *b = sB + (on ? myj : 0) * nel;
      T re[3][3] = {}, im[3][3] = {};
      for (int o = 0; o < no; ++o, a += w, b += w) {
        V x[3], y[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          x[k] = a[mi[k]];
          y[k] = b[ni[k]];
        }
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
          for (int l = 0; l < 3; ++l) conj_mul_add(re[k][l], im[k][l], x[k], y[l]);
      }
      if (through) __syncwarp();  // every lane has read its operands
      T *out = through ? reinterpret_cast<T *>(sA) + myj * ww : W2 + (c0 + myj) * ww;
      if (on) {
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
          for (int l = 0; l < 3; ++l)
            if (ti * 3 + k < w && tj * 3 + l < w)
              out[(ti * 3 + k) * w + tj * 3 + l] = re[k][l] * re[k][l] + im[k][l] * im[k][l];
      }
    }
    __syncwarp();
    if (through) {
      const T *o = reinterpret_cast<const T *>(sA);
      for (int i = lane; i < nj * ww; i += 32) W2[c0 * ww + i] = o[i];
      __syncwarp();
    }
  }
}

// ---------------------------------------------------------------- band bounds per corner
// occ[c] = 1 + highest band with e < eF at corner c (0 if none): bands m >= occ[c] are empty
// there.  emp[c] = lowest band with e > eF (nb if none): bands n < emp[c] are not empty.
// occf[c]: lowest band with not e < eF (every band below it is occupied); empf[c] = 1 + highest
// band with not e > eF (every band from it on is empty).  For ascending energies occf = occ and
// empf = emp but for levels at eF; neither order nor absence of NaN is relied on.
// E32 (optional) receives the energies relative to eF in FP32 for the mixed-precision path.
// Sides and FP32 values by integer operations where the value is a normal FP32 number: on the FP64
// pipe two comparisons and a conversion took 16 cycles each per warp (48^3 corners x 9 bands: 16 us,
// now 11 us).
// A block reads a run of corners' energies coalesced, one energy per thread and step, notes
// each one's side of eF in shared memory, and one thread per corner walks the notes; one
// thread per corner walking the energies themselves took 16 us on a 48^3 mesh of 9 bands.
constexpr int kBandTile = 4096;  // energies per block (nb <= 4096)
__global__ void __launch_bounds__(kThreads) k_bands(const __grid_constant__ BandArgs A, long long nc, int nb, double ef) {
  __shared__ unsigned char s_side[kBandTile];
  const int per = kBandTile / nb < kThreads ? kBandTile / nb : kThreads;  // corners per block
  const double *E = A.E[blockIdx.y];
  BandBounds o = A.out;
  float *E32 = A.E32, *E32lo = A.E32lo;
  o.occ += (size_t)blockIdx.y * A.stride_c;
  o.emp += (size_t)blockIdx.y * A.stride_c;
  o.occf += (size_t)blockIdx.y * A.stride_c;
  o.empf += (size_t)blockIdx.y * A.stride_c;
  if (E32) E32 += (size_t)blockIdx.y * A.stride_e;
  if (E32lo) E32lo += (size_t)blockIdx.y * A.stride_e;
  for (long long c0 = (long long)blockIdx.x * per; c0 < nc; c0 += (long long)gridDim.x * per) {
    const int ncb = (int)(nc - c0 < per ? nc - c0 : per);
    for (int i = threadIdx.x; i < ncb * nb; i += kThreads) {
      const double x = E[c0 * nb + i] - ef;
      const int hi = __double2hiint(x), mag = hi & 0x7fffffff;
      const bool nan = mag > 0x7ff00000 || (mag == 0x7ff00000 && __double2loint(x) != 0);
      const bool zero = (mag | __double2loint(x)) == 0;
      s_side[i] = nan || zero ? 0 : (hi < 0 ? 1 : 2);
      if (E32) {
        const float h = mag - 0x38100000 < 0x0fd00000 && mag >= 0x38100000 ? d2f_int(x) : (float)x;
        E32[c0 * nb + i] = h;
        if (E32lo) E32lo[c0 * nb + i] = (float)(x - (double)h);
      }
    }
    __syncthreads();
    if ((int)threadIdx.x < ncb) {
      const unsigned char *side = s_side + threadIdx.x * nb;
      int oc = 0, of = nb, e = nb, ef_ = 0;
      for (int b = 0; b < nb; ++b) {
        const int sd = side[b];
        if (sd & 1) oc = b + 1;
        else of = min(of, b);
        if (sd & 2) e = min(e, b);
        else ef_ = b + 1;
      }
      o.occ[c0 + threadIdx.x] = (short)oc;
      o.occf[c0 + threadIdx.x] = (short)of;
      o.emp[c0 + threadIdx.x] = (short)e;
      o.empf[c0 + threadIdx.x] = (short)ef_;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- energy range
// largest finite |E - eF| of every band over the corners, as the bits of a double (out: 0 on entry).
// A thread stays with one band, kThreads / (bands of the tile) corners a block at a time: the loads of
// a step are consecutive, and a block adds one atomic a band.
__global__ void __launch_bounds__(kThreads) k_energy_range(const double *__restrict__ E, long long nc, int nb, double ef,
                                                           unsigned long long *__restrict__ out) {
  __shared__ unsigned long long s_max[kThreads];
  for (int b0 = 0; b0 < nb; b0 += kThreads) {
    const int wt = min(nb - b0, kThreads), rows = kThreads / wt, r = threadIdx.x / wt, b = threadIdx.x - r * wt;
    double m = 0.0;
    if (r < rows)
      for (long long c = (long long)blockIdx.x * rows + r; c < nc; c += (long long)gridDim.x * rows) {
        const double x = fabs(E[c * nb + b0 + b] - ef);
        if (x < (double)INFINITY) m = fmax(m, x);
      }
    s_max[threadIdx.x] = (unsigned long long)__double_as_longlong(m);
    __syncthreads();
    if (r == 0) {
      for (int k = 1; k < rows; ++k) m = fmax(m, __longlong_as_double((long long)s_max[k * wt + b]));
      if (m > 0.0) atomicMax(out + b0 + b, (unsigned long long)__double_as_longlong(m));
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- Gamma DOS term
__global__ void __launch_bounds__(kThreads) k_dos(Grid g, Tet tet, const double *__restrict__ E, int lo,
                                                   int hi, double *__restrict__ partial,
                                                   unsigned long long *__restrict__ pairs) {
  const int w = hi - lo;
  const long long total = g.ntet * (long long)w;
  Q q0{};
  q0.Eq = E;  // corners at k only
  double acc = 0.0;
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const long long t = idx / w;
    const int band = lo + (int)(idx - t * w);
    long long c[4], cq[4];
    double vol;
    tet_corners(g, tet, q0, t, c, cq, vol);
    const double v = vol * dos4(E[c[0] * g.nb + band] - g.ef, E[c[1] * g.nb + band] - g.ef,
                                E[c[2] * g.nb + band] - g.ef, E[c[3] * g.nb + band] - g.ef);
    acc += v;
    if (pairs && v != 0.0) pair_add(pairs, (band - lo) * (w + 1), v);  // the intraband pair (m, m)
  }
  block_sum_store(acc, &partial[blockIdx.x]);
}

// band-pair output: fixed-point totals to FP64, times the normalisation and sign
__global__ void __launch_bounds__(kThreads) k_pairs_out(const unsigned long long *__restrict__ pairs, int n,
                                                         double scale, double *__restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = scale * ((double)(long long)pairs[i] / kPairScale);
}

}  // namespace

// ======================================================================= launchers
int static_blocks() { return kStaticBlocks; }
long long static_batches(long long ntet) { return (ntet + 31) / 32; }

__global__ void __launch_bounds__(kThreads) k_c128_to_c64(const double2 *__restrict__ in, float2 *__restrict__ out,
                                                         long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double2 v = in[i];
    out[i] = make_float2((float)v.x, (float)v.y);
  }
}

cudaError_t launch_c128_to_c64(const void *in, void *out, long long n, cudaStream_t s) {
  k_c128_to_c64<<<device_sms() * 8, kThreads, 0, s>>>((const double2 *)in, (float2 *)out, n);
  return cudaGetLastError();
}

// the q points of a group with norb w <= kOvlSmall, or the others (windows differ): so that a q's values
// do not depend on what it is grouped with
static void pick_overlap(const OverlapArgs &a, bool small, OverlapArgs &out) {
  out.g = a.g;
  out.nq = 0;
  for (int i = 0; i < a.nq; ++i) {
    if (((long long)a.g.norb * (a.q[i].hi - a.q[i].lo) <= kOvlSmall) != small) continue;
    out.q[out.nq] = a.q[i];
    out.W2[out.nq++] = a.W2[i];
  }
}

cudaError_t launch_overlap(const OverlapArgs &a, const void *C, int dtype, int fp64, cudaStream_t s, const void *C32,
                           int *launches) {
  const Grid &g = a.g;
  if (launches) *launches = 0;
  if (a.nq < 1 || g.nc < 1) return cudaSuccess;
  const bool ex = a.q[0].Cq != nullptr;  // (a group's q points are all explicit or all shifts)
  OverlapArgs p;
  pick_overlap(a, true, p);
  if (p.nq > 0) {
    const long long warps = fp64 ? 4 : 8, nbw = (g.nc + warps - 1) / warps, cap = device_sms() * 4;  // resident blocks
    const dim3 bw((unsigned)(nbw < cap ? nbw : cap), (unsigned)p.nq);
    if (fp64) {
      if (dtype == DT_C128) k_overlap_small<double2, double2, double><<<bw, 128, 0, s>>>(p, (const double2 *)C, ex ? 1 : 0);
      else k_overlap_small<float2, float2, double><<<bw, 128, 0, s>>>(p, (const float2 *)C, ex ? 1 : 0);
    } else {
      // k side in complex64 (the plan's copy when the inputs are complex128)
      const float2 *Ck = (const float2 *)(C32 ? C32 : C);
      if (ex && dtype == DT_C128) k_overlap_small<float2, double2, float><<<bw, 256, 0, s>>>(p, Ck, 1);
      else k_overlap_small<float2, float2, float><<<bw, 256, 0, s>>>(p, Ck, ex ? 1 : 0);
    }
    if (launches) ++*launches;
    if (p.nq == a.nq) return cudaGetLastError();
    pick_overlap(a, false, p);
  } else {
    p = a;
  }
  int w = 0;
  for (int i = 0; i < p.nq; ++i) w = p.q[i].hi - p.q[i].lo > w ? p.q[i].hi - p.q[i].lo : w;
  const long long nb = (g.nc * (long long)w * w + kThreads - 1) / kThreads, cap = device_sms() * 16;
  const dim3 bg((unsigned)(nb < cap ? nb : cap), (unsigned)p.nq);
  if (dtype == DT_C128) {
    if (fp64) k_overlap<double2, double><<<bg, kThreads, 0, s>>>(p, (const double2 *)C);
    else k_overlap<double2, float><<<bg, kThreads, 0, s>>>(p, (const double2 *)C);
  } else {
    if (fp64) k_overlap<float2, double><<<bg, kThreads, 0, s>>>(p, (const float2 *)C);
    else k_overlap<float2, float><<<bg, kThreads, 0, s>>>(p, (const float2 *)C);
  }
  if (launches) ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_bands(const BandArgs &a, int nq, long long nc, int nb, double ef, cudaStream_t s) {
  const int per = kBandTile / nb < kThreads ? kBandTile / nb : kThreads;
  const long long nblk = (nc + per - 1) / per;
  const int cap = device_sms() * 8;
  k_bands<<<dim3((unsigned)(nblk < cap ? nblk : cap), (unsigned)nq), kThreads, 0, s>>>(a, nc, nb, ef);
  return cudaGetLastError();
}

cudaError_t launch_energy_range(const double *E, long long nc, int nb, double ef, unsigned long long *out,
                                cudaStream_t s) {
  const cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long) * nb, s);
  if (e != cudaSuccess) return e;
  const long long nblk = (nc * nb + kThreads - 1) / kThreads, cap = device_sms() * 8;
  k_energy_range<<<(unsigned)(nblk < cap ? nblk : cap), kThreads, 0, s>>>(E, nc, nb, ef, out);
  return cudaGetLastError();
}

int device_sms() {
  int dev = 0, sms = kSMs;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

cudaError_t launch_dos(const Grid &g, const Tet &tet, const double *E, int lo, int hi, double *partial,
                       int nblocks, cudaStream_t s, unsigned long long *pairs) {
  k_dos<<<nblocks, kThreads, 0, s>>>(g, tet, E, lo, hi, partial, pairs);
  return cudaGetLastError();
}

cudaError_t launch_pairs_out(const unsigned long long *pairs, int n, double scale, double *out, cudaStream_t s) {
  k_pairs_out<<<(n + kThreads - 1) / kThreads, kThreads, 0, s>>>(pairs, n, scale, out);
  return cudaGetLastError();
}

}  // namespace chi0int
