// Host build of the FP32 entries of three clustered knots (inv_sum_triple_table), next to the
// per-vertex table in FP64.
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

// returns 1 where the FP32 form takes the knots; out: its value and the table's
extern "C" int host_triple_table(const float *x, const float *f, double *out) {
  float v = 0.0f;
  const int took = chi0dev::inv_sum_triple_table(x, f, v) ? 1 : 0;
  double xd[4], fd[4];
  for (int i = 0; i < 4; ++i) xd[i] = x[i], fd[i] = f[i];
  out[0] = v;
  out[1] = chi0dev::inv_sum_table(xd, fd);
  return took;
}
