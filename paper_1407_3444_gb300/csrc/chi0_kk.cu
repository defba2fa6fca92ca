// chi0_kk.cu -- Re chi0 from Im chi0 by the Kramers-Kronig relation (the route the paper calls
// the usual one, Sec. II below Eqs. 1-3), the alternative to the principal value of Eq. 1.
//
// With Im odd in w (Eq. 3) and the positive-sign convention of this library,
//   Re(w) = (1/pi) PV int_0^inf Im(u) [1/(u - w) + 1/(u + w)] du.
// Im is known on a uniform grid u_j = j du, j < m (Im(0) = 0, Im = 0 from u_m on: the grid
// must cover the spectrum, the caveat of Sec. IV), and is taken piecewise linear between the
// nodes.  The hat function of node j integrates against 1/(u - w) to the second difference of
// G(x) = x ln|x| (G'' = 1/x, G(0) = 0):
//   int hat_j(u) / (u - w) du = [G(u_{j+1} - w) - 2 G(u_j - w) + G(u_{j-1} - w)] / du,
// finite also where w is a node.  Summing by parts over the nodes,
//   Re(w) = (1 / (pi du)) sum_{k=0..m} [G(u_k - w) + G(u_k + w)] (Im_{k-1} - 2 Im_k + Im_{k+1}),
// with Im_j = 0 for j <= 0 and j >= m.  FP64, O(m) per output node.
#include <cuda_runtime.h>
#include <math.h>

#include "chi0_grid.cuh"
#include "chi0_internal.h"

namespace chi0int {
namespace {

__device__ __forceinline__ double gxl(double x) { return x == 0.0 ? 0.0 : x * log(fabs(x)); }

// One block per output node, its threads over the nodes k (pairwise sums in a fixed order): one thread
// per output node left a 400-node transform on two blocks, 1.9 ms of serial logarithms.
constexpr int kKKThreads = 128;
__global__ void __launch_bounds__(kKKThreads) k_kk(const double *__restrict__ im, int m, double du, double scale,
                                                   const double *__restrict__ dos, int ndos, double *__restrict__ re) {
  const int i = blockIdx.x;
  const double w = i * du;
  double s = 0.0, c = 0.0;  // compensated sum
  auto I = [&](int j) { return j >= 1 && j < m ? im[j] : 0.0; };  // Im(0) = 0; 0 past the grid
  for (int k = threadIdx.x; k <= m; k += kKKThreads) {
    const double d2 = I(k - 1) - 2.0 * I(k) + I(k + 1);
    if (d2 == 0.0) continue;
    const double uk = k * du;
    const double t = (gxl(uk - w) + gxl(uk + w)) * d2;
    const double y = s + t;
    c += fabs(s) >= fabs(t) ? (s - y) + t : (t - y) + s;
    s = y;
  }
  double sd = 0.0;  // the q -> 0 intraband limit at w = 0 (Sec. III), as the direct route adds it
  if (dos && i == 0)
    for (int k = threadIdx.x; k < ndos; k += kKKThreads) sd += dos[k];
  __shared__ double red[2][kKKThreads / 32];
  const double v = grid::warp_sum(s + c);
  sd = grid::warp_sum(sd);
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = v;
    red[1][threadIdx.x >> 5] = sd;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    re[i] = ((red[0][0] + red[0][1]) + (red[0][2] + red[0][3])) / (3.141592653589793 * du) +
            scale * ((red[1][0] + red[1][1]) + (red[1][2] + red[1][3]));
}

}  // namespace

cudaError_t launch_kk(const double *im, int m, double du, double scale, const double *dos, int ndos, double *re,
                      cudaStream_t s) {
  if (m <= 1 || !(du > 0.0)) return cudaErrorInvalidValue;
  k_kk<<<m, kKKThreads, 0, s>>>(im, m, du, scale, dos, ndos, re);
  return cudaGetLastError();
}

}  // namespace chi0int
