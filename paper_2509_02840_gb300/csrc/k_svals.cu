// Singular values of the upper bidiagonal Bd (d, e) on the device, by
// multisection with Sturm counts.
//
// The singular values of Bd are the nonnegative eigenvalues of the
// Golub-Kahan matrix T (order 2n, zero diagonal, off-diagonal
// b = d_1, e_1, d_2, e_2, ..., d_n), whose spectrum is {+-sigma_i}.  The
// number of eigenvalues of T below x is the number of negative pivots q_i of
// the LDL^T factorization of T - x I, q_i = p_i / p_{i-1} with the leading
// principal minors p_0 = 1, p_1 = -x, p_i = -x p_{i-1} - b_{i-1}^2 p_{i-2}: the
// number of sign changes in that sequence (a zero minor counts as opposite to
// the one before it).  For x > 0 the number of singular values below x is that
// count minus n.  Every computed minor satisfies the recurrence with x and
// b_{i-1}^2 perturbed by a few units in their last place, as the computed pivots
// do, and needs two FP64 instructions where a pivot's division takes over a
// dozen (64 cycles each on GB300): 64 values and 64 truncated columns at
// n = 2048 took 21.1 ms with pivots and take 6.7, at the same distance from
// the 64-bit values (2e-15 relative).  The matrix is scaled by a power of two so that its norm bound lies in
// [1, 2), and the pair of minors is brought back near 1 every few steps through
// the exponent fields.
//
// One warp per requested singular value; each iteration its 32 lanes count at
// 32 interior points of the current interval and the interval shrinks to the
// 1/33 that holds the value.  On GB300 a warp's FP64 instruction costs the same
// whatever its active lanes, so the 32 counts cost what one would.
#include "bdu_internal.cuh"

namespace bdu {
namespace {

// x times 2^(d / 2^20) through the exponent field; what would fall below the
// normal range becomes the least normal number of its sign.
__device__ __forceinline__ double shift_exp(double x, int d) {
  const int h = __double2hiint(x), m = (h & 0x7ff00000) + d;
  return m >= 0x00100000 ? __hiloint2double(h + d, __double2loint(x))
                         : __hiloint2double((h & (int)0x80000000) | 0x00100000, 0);
}

// Number of sign changes of the 2n + 1 minors at x > 0 (nx = -x), the pair
// rescaled every STEP steps.
template <int STEP>
__device__ __forceinline__ int count_below(const double *__restrict__ b2, int n, double nx) {
  double p1 = 1.0, p = nx;
  int cnt = 1;
  const int last = 2 * n - 1;  // minors 2 .. 2n, entries b2[0 .. 2n-2]
  double b[STEP];
#pragma unroll
  for (int q = 0; q < STEP; q++) b[q] = q < last ? __ldg(b2 + q) : 0.0;
  for (int i = 0; i < last; i += STEP) {
    double nb[STEP];
#pragma unroll
    for (int q = 0; q < STEP; q++) nb[q] = i + STEP + q < last ? __ldg(b2 + i + STEP + q) : 0.0;
#pragma unroll
    for (int q = 0; q < STEP; q++) {
      if (i + q < last) {
        double pn = fma(nx, p, -(b[q] * p1));
        if (pn == 0.0) pn = shift_exp(-p, -(500 << 20));
        cnt += (unsigned)(__double2hiint(pn) ^ __double2hiint(p)) >> 31;
        p1 = p;
        p = pn;
      }
    }
    const int e = max(__double2hiint(p) & 0x7ff00000, __double2hiint(p1) & 0x7ff00000);
    p = shift_exp(p, 0x3ff00000 - e);
    p1 = shift_exp(p1, 0x3ff00000 - e);
#pragma unroll
    for (int q = 0; q < STEP; q++) b[q] = nb[q];
  }
  return cnt;
}

__global__ void k_bidiag_svals(const double *__restrict__ b2, int n, double hi0, int k, double *__restrict__ sv) {
  const int lane = threadIdx.x & 31;
  const int j = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);  // the (j+1)-th largest value
  if (j >= k) return;  // whole warps exit together
  // #(sigma < x) >= n - j exactly when x lies above sigma_(j+1)
  const int target = n - j;
  double lo = 0.0, hi = hi0;
  for (int it = 0; it < 64; it++) {
    const double w = hi - lo;
    if (!(w > 2.2e-16 * hi)) break;  // uniform across the warp
    const double x = lo + w * (double)(lane + 1) / 33.0;
    // a minor shrinks by at most x (and by cancellation) in a step: four steps
    // between rescalings stay in range for x >= 2^-60, tiny x takes every step
    const int cnt = __all_sync(0xffffffffu, x >= 0x1p-60) ? count_below<4>(b2, n, -x) : count_below<1>(b2, n, -x);
    // #(sigma < x) = cnt - n; the lanes with #(sigma < x) >= target lie above sigma_(j+1)
    const unsigned above = __ballot_sync(0xffffffffu, cnt - n >= target);
    const int first = above ? __ffs(above) - 1 : 32;
    const double nlo = first == 0 ? lo : lo + w * (double)first / 33.0;
    const double nhi = first == 32 ? hi : lo + w * (double)(first + 1) / 33.0;
    lo = nlo;
    hi = nhi;
  }
  if (lane == 0) sv[j] = 0.5 * (lo + hi);
}

}  // namespace

// b2: the 2n-1 squared off-diagonal entries d_1^2, e_1^2, d_2^2, ..., d_n^2 of
// the Golub-Kahan matrix, scaled so that hi, an upper bound of sigma_max, lies
// in [1, 2) (device); sv: the k largest singular values of the scaled matrix,
// descending (device).
cudaError_t launch_bidiag_svals(const double *b2, int n, double hi, int k, double *sv, cudaStream_t s) {
  if (k <= 0) return cudaSuccess;
  const int warps = 4;
  k_bidiag_svals<<<(k + warps - 1) / warps, 32 * warps, 0, s>>>(b2, n, hi, k, sv);
  return cudaGetLastError();
}

}  // namespace bdu
