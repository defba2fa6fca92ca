// Host build of the weight kernels' series for knots and values on which no convergence test ends them:
// compiled with array bounds checked, every coefficient index must lie in its table.  Prints the sums.
#include <algorithm>
#include <cmath>
#include <cstdio>
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

int main() {
  // values whose first moments vanish against the knots' offsets: the terms start at rounding level and
  // grow, so the rule (relative to the first terms) is never met
  const float d[4] = {0.3f, 0.75f, 1.25f, 1.7f};
  float e[4], f[4];
  for (int i = 0; i < 4; ++i) e[i] = d[i] - 1.0f;
  for (int i = 0; i < 4; ++i) {  // weights of the third divided difference
    f[i] = 1.0f;
    for (int j = 0; j < 4; ++j)
      if (j != i) f[i] /= e[i] - e[j];
  }
  const float z[4] = {0.0f, 0.0f, 0.0f, 0.0f}, u[4] = {NAN, NAN, NAN, NAN};
  std::printf("%g %g %g %g %g %g\n", series_sum_short(d, f), series_sum(d, f), series_sum_short(d, z), series_sum(d, z),
              series_sum_short(d, u), series_sum(d, u));
  return 0;
}
