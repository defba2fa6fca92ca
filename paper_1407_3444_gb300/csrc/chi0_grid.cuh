// chi0_grid.cuh -- device helpers shared by the weight kernels: tetrahedron corners of the
// k mesh (Sec. II: the integration domain split into tetrahedra) at k and at k+q, small
// quotients without a division sequence, band-pair sums and warp sums.
#pragma once

#include <cuda_runtime.h>

#include "chi0_internal.h"

namespace chi0int {
namespace grid {

constexpr unsigned kFull = 0xffffffffu;

// x / d for x < 2^24, d < 2^13 (and the remainder), without a division sequence
__device__ __forceinline__ int quick_div(int x, int d, int &rem) {
  int k = (int)__fdividef((float)x + 0.5f, (float)d);
  rem = x - k * d;
  if (rem < 0) {
    --k;
    rem += d;
  } else if (rem >= d) {
    ++k;
    rem -= d;
  }
  return k;
}

// Corners of tetrahedron t at k and at k+q, and its fractional volume.  Builtin mesh:
// tetrahedron 6*cube + p = {000, e_a, e_a + e_b, 111} for the p-th axis order (a, b, .)
// of the lexicographically ordered permutations of (0, 1, 2).
__device__ __forceinline__ void tet_corners(const Grid &g, const Tet &tet, const Q &q, long long t,
                                            long long c[4], long long cq[4], double &vol) {
  if (tet.corners) {
    const int4 v = tet.corners[t];
    c[0] = v.x; c[1] = v.y; c[2] = v.z; c[3] = v.w;
    vol = tet.vol[t];
    for (int i = 0; i < 4; ++i) cq[i] = q.Eq ? c[i] : shift_corner(g, c[i], q.shift);
    return;
  }
  const unsigned tu = (unsigned)t;
  const unsigned cube = tu / 6u;
  const int p = (int)(tu - cube * 6u);
  const unsigned r = fdiv(cube, g.fn2);
  const int i2 = (int)(cube - r * (unsigned)g.n[2]);
  const unsigned i0u = fdiv(r, g.fn1);
  const int i1 = (int)(r - i0u * (unsigned)g.n[1]);
  const int i0 = (int)i0u;
  const int ax = p >> 1;                                // first axis: 0,0,1,1,2,2
  const int bx = (p == 0) ? 1 : (p == 1) ? 2 : (p == 2) ? 0 : (p == 3) ? 2 : (p == 4) ? 0 : 1;
  int o1[3] = {0, 0, 0}, o2[3] = {0, 0, 0};
  o1[ax] = 1;
  o2[ax] = 1;
  o2[bx] = 1;
  const int *s = q.shift;
  const bool ex = q.Eq != nullptr;
  c[0] = cid(g, i0, i1, i2);
  c[1] = cid(g, i0 + o1[0], i1 + o1[1], i2 + o1[2]);
  c[2] = cid(g, i0 + o2[0], i1 + o2[1], i2 + o2[2]);
  c[3] = cid(g, i0 + 1, i1 + 1, i2 + 1);
  if (ex) {
    for (int i = 0; i < 4; ++i) cq[i] = c[i];
  } else {
    cq[0] = cid(g, i0 + s[0], i1 + s[1], i2 + s[2]);
    cq[1] = cid(g, i0 + o1[0] + s[0], i1 + o1[1] + s[1], i2 + o1[2] + s[2]);
    cq[2] = cid(g, i0 + o2[0] + s[0], i1 + o2[1] + s[1], i2 + o2[2] + s[2]);
    cq[3] = cid(g, i0 + 1 + s[0], i1 + 1 + s[1], i2 + 1 + s[2]);
  }
  vol = tet.vol_builtin;
}

// double -> float rounded to nearest even by integer operations (keeps the conversion of
// complex128 inputs off the FP64 pipe); magnitudes below 2^-126 flush to zero
__device__ __forceinline__ float d2f_int(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned hi = (unsigned)(u >> 32);
  const unsigned sign = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7ffu) - 1023 + 127;
  if (e <= 0) return __uint_as_float(sign);
  if (e >= 255) return __uint_as_float(sign | 0x7f800000u | (((u << 12) != 0ull && e > 1000) ? 0x400000u : 0u));
  const unsigned long long mant = u & 0xFFFFFFFFFFFFFull;
  unsigned m = (unsigned)(mant >> 29);
  const unsigned rem = (unsigned)(mant & 0x1FFFFFFFull);
  m += (rem > 0x10000000u) | ((rem == 0x10000000u) & (m & 1u));
  return __uint_as_float(sign | (((unsigned)e << 23) + m));  // a mantissa carry rounds into the exponent
}

// band-pair output: 64-bit fixed point in units of 2^-50 (|pair totals| < 2^13; one rounding
// of 2^-51 per term)
constexpr double kPairScale = 1125899906842624.0;  // 2^50
__device__ __forceinline__ void pair_add(unsigned long long *pairs, int idx, double v) {
  atomicAdd(&pairs[idx], (unsigned long long)__double2ll_rn(v * kPairScale));
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

}  // namespace grid
}  // namespace chi0int
