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
template <typename T> __device__ __forceinline__ T cvt(double x);
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

// Warp per corner for small blocks (norb * w <= kOvlSmall): both eigenvector blocks
// C_k[:, lo:hi] and C_{k+q}[:, lo:hi] are read once, coalesced, into shared memory in
// the arithmetic precision, then the lanes form the w x w |overlap|^2 block.
constexpr int kOvlSmall = 256;
template <typename CT, typename CTq, typename T>
__global__ void __launch_bounds__(kThreads) k_overlap_small(const __grid_constant__ OverlapArgs A,
                                                             const CT *__restrict__ C, int explicit_q) {
  const Grid &g = A.g;
  const Q &q = A.q[blockIdx.y];
  const CTq *Cb = explicit_q ? (const CTq *)q.Cq : (const CTq *)C;
  T *W2 = (T *)A.W2[blockIdx.y];
  __shared__ T sA[kWarps][2][kOvlSmall], sB[kWarps][2][kOvlSmall];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int w = q.hi - q.lo, no = g.norb, nel = no * w;
  for (long long c = (long long)blockIdx.x * kWarps + wib; c < g.nc; c += (long long)gridDim.x * kWarps) {
    const long long ck = explicit_q ? c : shift_corner(g, c, q.shift);
    for (int i = lane; i < nel; i += 32) {
      const int o = i / w, mm = i - o * w;
      const CT x = C[(c * no + o) * g.nb + q.lo + mm];
      const CTq y = Cb[(ck * no + o) * g.nb + q.lo + mm];
      sA[wib][0][i] = cvt<T>(x.x);
      sA[wib][1][i] = cvt<T>(x.y);
      sB[wib][0][i] = cvt<T>(y.x);
      sB[wib][1][i] = cvt<T>(y.y);
    }
    __syncwarp();
    for (int out = lane; out < w * w; out += 32) {
      const int mm = out / w, nn = out - mm * w;
      T re = T(0), im = T(0);
      for (int o = 0; o < no; ++o) {
        const T xr = sA[wib][0][o * w + mm], xi = sA[wib][1][o * w + mm];
        const T yr = sB[wib][0][o * w + nn], yi = sB[wib][1][o * w + nn];
        re += xr * yr + xi * yi;  // conj(x) * y
        im += xr * yi - xi * yr;
      }
      W2[c * w * w + out] = re * re + im * im;
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------- band bounds per corner
// occ[c] = 1 + highest band with e < eF at corner c (0 if none): bands m >= occ[c] are empty
// there.  emp[c] = lowest band with e > eF (nb if none): bands n < emp[c] are not empty.
// occf[c]: lowest band with not e < eF (every band below it is occupied); empf[c] = 1 + highest
// band with not e > eF (every band from it on is empty).  For ascending energies occf = occ and
// empf = emp but for levels at eF; neither order nor absence of NaN is relied on.
// E32 (optional) receives the energies relative to eF in FP32 for the mixed-precision path.
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
      s_side[i] = (x < 0.0 ? 1 : 0) | (x > 0.0 ? 2 : 0);
      if (E32) {
        const float h = (float)x;
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

cudaError_t launch_overlap(const OverlapArgs &a, const void *C, int dtype, int fp64, cudaStream_t s, const void *C32) {
  int w = 0;
  for (int i = 0; i < a.nq; ++i) w = a.q[i].hi - a.q[i].lo > w ? a.q[i].hi - a.q[i].lo : w;
  const Grid &g = a.g;
  const long long total = g.nc * (long long)w * w;
  long long nb = (total + kThreads - 1) / kThreads;
  const int blocks = (int)(nb < device_sms() * 16 ? nb : device_sms() * 16);
  if (blocks <= 0) return cudaSuccess;
  const bool ex = a.q[0].Cq != nullptr;  // (a group's q points are all explicit or all shifts)
  const bool small = (long long)g.norb * w <= kOvlSmall && !fp64;
  if (small) {
    // k side in complex64 (the plan's copy when the inputs are complex128)
    const float2 *Ck = (const float2 *)(C32 ? C32 : C);
    long long nbw = (g.nc + kWarps - 1) / kWarps;
    const dim3 bw((unsigned)(nbw < device_sms() * 8 ? nbw : device_sms() * 8), (unsigned)a.nq);
    if (ex && dtype == DT_C128) k_overlap_small<float2, double2, float><<<bw, kThreads, 0, s>>>(a, Ck, 1);
    else k_overlap_small<float2, float2, float><<<bw, kThreads, 0, s>>>(a, Ck, ex ? 1 : 0);
    return cudaGetLastError();
  }
  const dim3 bg((unsigned)blocks, (unsigned)a.nq);
  if (dtype == DT_C128) {
    if (fp64) k_overlap<double2, double><<<bg, kThreads, 0, s>>>(a, (const double2 *)C);
    else k_overlap<double2, float><<<bg, kThreads, 0, s>>>(a, (const double2 *)C);
  } else {
    if (fp64) k_overlap<float2, double><<<bg, kThreads, 0, s>>>(a, (const float2 *)C);
    else k_overlap<float2, float><<<bg, kThreads, 0, s>>>(a, (const float2 *)C);
  }
  return cudaGetLastError();
}

cudaError_t launch_bands(const BandArgs &a, int nq, long long nc, int nb, double ef, cudaStream_t s) {
  const int per = kBandTile / nb < kThreads ? kBandTile / nb : kThreads;
  const long long nblk = (nc + per - 1) / per;
  const int cap = device_sms() * 8;
  k_bands<<<dim3((unsigned)(nblk < cap ? nblk : cap), (unsigned)nq), kThreads, 0, s>>>(a, nc, nb, ef);
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
