// chi0_interp.cu -- energies and eigenvectors at k+q for q off the k mesh, by linear
// interpolation from the mesh (Sec. II: the data at k+q, which are in general not on the
// tetrahedron mesh, are approximated by linear interpolation, energies and matrix elements on
// equal footing).
//
// For a corner k of the periodic mesh, k+q lies in one cube of the mesh and, within it, in one
// of the cube's six tetrahedra {000, e_p0, e_p0 + e_p1, 111} (the axis order p that sorts the
// local coordinates t descending, t_p0 >= t_p1 >= t_p2).  Its barycentric weights there are
//   (1 - t_p0, t_p0 - t_p1, t_p1 - t_p2, t_p2),
// and every quantity is the weighted sum of its values at those four corners, band by band.
// Eigenvectors carry an arbitrary phase per corner, so before the sum the vectors of corners
// 1..3 are turned onto the phase of corner 0's (multiplied by conj(<v_0|v_i>) / |<v_0|v_i>|),
// and the sum is normalised.  |M_mn|^2 does not depend on the phase left over.
#include <cuda_runtime.h>
#include <math.h>

#include "chi0_internal.h"

namespace chi0int {
namespace {

struct Cd {
  double x, y;
};
__device__ __forceinline__ Cd ld(const void *C, int dtype, long long i) {
  if (dtype == 0) {  // complex64
    const float2 v = ((const float2 *)C)[i];
    return Cd{v.x, v.y};
  }
  const double2 v = ((const double2 *)C)[i];
  return Cd{v.x, v.y};
}
__device__ __forceinline__ void st(void *C, int dtype, long long i, Cd v) {
  if (dtype == 0) ((float2 *)C)[i] = make_float2((float)v.x, (float)v.y);
  else ((double2 *)C)[i] = make_double2(v.x, v.y);
}

// One thread per (corner, band).  Bound: the FP64 pipe (some 30 operations per corner, band and
// orbital).  NO: orbitals at most (0: any number), whose sums then stay in registers between the norm
// and the store; the weights are folded into the phases, and the norms go through one reciprocal
// square root.  33 x 32 x 31 corners, 9 orbitals, complex128: 0.25 ms (0.40 with unfolded weights, the
// sums formed twice, square roots and divisions).  The line at 16: 24^3 corners, complex128, registers
// against the general form: 10 orbitals 135 against 184 us, 16 orbitals 305 against 423 us (64 of the
// registers are sums there; more would leave too few warps).
template <int NO>
__global__ void __launch_bounds__(256) k_interp_kq(Grid g, const double *__restrict__ E, const void *__restrict__ C,
                                                   int dtype, double q0, double q1, double q2,
                                                   double *__restrict__ Eq, void *__restrict__ Cq) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= g.nc * g.nb) return;
  const long long c = idx / g.nb;
  const int b = (int)(idx - c * g.nb);
  const int i2 = (int)(c % g.N[2]), i1 = (int)((c / g.N[2]) % g.N[1]), i0 = (int)(c / ((long long)g.N[2] * g.N[1]));
  const int ii[3] = {i0, i1, i2};
  const double qq[3] = {q0, q1, q2};
  int base[3];
  double t[3];
  for (int d = 0; d < 3; ++d) {
    const double x = ii[d] + qq[d] * g.n[d];
    const double fl = floor(x);
    t[d] = x - fl;
    long long m = (long long)fl % g.n[d];
    if (m < 0) m += g.n[d];
    base[d] = (int)m;
  }
  // axis order sorting t descending (ties: lower axis first)
  int p0 = 0, p1 = 1, p2 = 2;
  if (t[p1] > t[p0]) { const int s = p0; p0 = p1; p1 = s; }
  if (t[p2] > t[p1]) { const int s = p1; p1 = p2; p2 = s; }
  if (t[p1] > t[p0]) { const int s = p0; p0 = p1; p1 = s; }
  const double w[4] = {1.0 - t[p0], t[p0] - t[p1], t[p1] - t[p2], t[p2]};
  long long cc[4];
  int o[3] = {0, 0, 0};
  for (int v = 0; v < 4; ++v) {
    if (v == 1) o[p0] = 1;
    if (v == 2) o[p1] = 1;
    if (v == 3) o[p2] = 1;
    const int j0 = (base[0] + o[0]) % g.n[0], j1 = (base[1] + o[1]) % g.n[1], j2 = (base[2] + o[2]) % g.n[2];
    cc[v] = ((long long)j0 * g.N[1] + j1) * g.N[2] + j2;
  }
  double e = 0.0;
  for (int v = 0; v < 4; ++v) e += w[v] * E[cc[v] * g.nb + b];
  Eq[c * g.nb + b] = e;
  if (!C) return;
  // phases of corners 1..3 relative to corner 0, conj(<v_0|v_i>) / |.|, times the weights
  const long long at = b, st_o = g.nb;
  Cd ph[4] = {{w[0], 0.0}, {w[1], 0.0}, {w[2], 0.0}, {w[3], 0.0}};
  {
    double re[3] = {0.0, 0.0, 0.0}, im[3] = {0.0, 0.0, 0.0};
    for (int o = 0; o < g.norb; ++o) {
      const Cd a = ld(C, dtype, cc[0] * g.norb * st_o + o * st_o + at);
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        const Cd z = ld(C, dtype, (cc[v + 1] * g.norb + o) * st_o + at);
        re[v] += a.x * z.x + a.y * z.y;
        im[v] += a.x * z.y - a.y * z.x;
      }
    }
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      const double m2 = re[v] * re[v] + im[v] * im[v];
      if (m2 > 0.0) {
        const double r = w[v + 1] * rsqrt(m2);
        ph[v + 1] = Cd{re[v] * r, -im[v] * r};
      }
    }
  }
  // the weighted sum, orbital by orbital
  auto mix = [&](int o) {
    const Cd z0 = ld(C, dtype, (cc[0] * g.norb + o) * st_o + at);
    double sx = ph[0].x * z0.x, sy = ph[0].x * z0.y;
#pragma unroll
    for (int v = 1; v < 4; ++v) {
      const Cd z = ld(C, dtype, (cc[v] * g.norb + o) * st_o + at);
      sx += z.x * ph[v].x - z.y * ph[v].y;
      sy += z.x * ph[v].y + z.y * ph[v].x;
    }
    return Cd{sx, sy};
  };
  double nrm = 0.0;
  if (NO > 0) {  // at most NO orbitals: kept in registers until the norm is known
    Cd s[NO > 0 ? NO : 1];
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      s[o] = o < g.norb ? mix(o) : Cd{0.0, 0.0};
      nrm += s[o].x * s[o].x + s[o].y * s[o].y;
    }
    const double sc = nrm > 0.0 ? rsqrt(nrm) : 0.0;
#pragma unroll
    for (int o = 0; o < NO; ++o)
      if (o < g.norb) st(Cq, dtype, (c * g.norb + o) * st_o + at, Cd{s[o].x * sc, s[o].y * sc});
  } else {
    for (int o = 0; o < g.norb; ++o) {
      const Cd s = mix(o);
      nrm += s.x * s.x + s.y * s.y;
    }
    const double sc = nrm > 0.0 ? rsqrt(nrm) : 0.0;
    for (int o = 0; o < g.norb; ++o) {
      const Cd s = mix(o);
      st(Cq, dtype, (c * g.norb + o) * st_o + at, Cd{s.x * sc, s.y * sc});
    }
  }
}

}  // namespace

cudaError_t launch_interp_kq(const Grid &g, const double *E, const void *C, int c64, const double q[3], double *Eq,
                             void *Cq, cudaStream_t s) {
  const long long n = g.nc * g.nb;
  const unsigned blocks = (unsigned)((n + 255) / 256);
  const int dt = c64 ? 0 : 1;
  if (g.norb <= 10) k_interp_kq<10><<<blocks, 256, 0, s>>>(g, E, C, dt, q[0], q[1], q[2], Eq, Cq);
  else if (g.norb <= 16) k_interp_kq<16><<<blocks, 256, 0, s>>>(g, E, C, dt, q[0], q[1], q[2], Eq, Cq);
  else k_interp_kq<0><<<blocks, 256, 0, s>>>(g, E, C, dt, q[0], q[1], q[2], Eq, Cq);
  return cudaGetLastError();
}

}  // namespace chi0int
