// edge.cu -- edge-corrected multipoles (Slepian & Eisenstein 2015).
//
// Paper, "Implementation": the estimator includes edge corrections; "Statement
// of need": the harmonic 3PCF after Slepian & Eisenstein.  With the sums
// S_l(b1,b2) = sum over triplets of P_l(mu) of a data-minus-randoms catalogue
// (N) and of its randoms alone (R, weights taken positive), the corrected
// 3PCF zeta(mu) = N(mu) / R(mu) has Legendre coefficients zeta_l that solve,
// per bin pair,
//     n_l / r_0 = sum_l' M_ll' zeta_l',   M_ll' = (2l+1) sum_l'' (l l' l''; 0 0 0)^2 f_l'',
// where n_l = (2l+1)/2 S_l(N), r_l = (2l+1)/2 S_l(R), f_l = r_l / r_0, all
// sums truncated at l_max.  One warp solves one bin pair's system in FP64 by
// Gaussian elimination with partial pivoting.
#include <cmath>
#include <vector>

#include "ctb_internal.cuh"

namespace ctb {

// (a b c; 0 0 0)^2 from the closed form in log-gamma:
// zero unless a+b+c = 2g is even and (a, b, c) a triangle, else
// (2g-2a)!(2g-2b)!(2g-2c)!/(2g+1)! * [g!/((g-a)!(g-b)!(g-c)!)]^2.
static double threej000_sq(int a, int b, int c) {
  if ((a + b + c) & 1) return 0.0;
  if (c < std::abs(a - b) || c > a + b) return 0.0;
  const int g = (a + b + c) / 2;
  auto lf = [](int n) { return std::lgamma((double)n + 1.0); };
  const double lg = lf(2 * g - 2 * a) + lf(2 * g - 2 * b) + lf(2 * g - 2 * c) - lf(2 * g + 1) +
                    2.0 * (lf(g) - lf(g - a) - lf(g - b) - lf(g - c));
  return std::exp(lg);
}

void make_threej_table(int lmax, std::vector<double>& t) {
  const int n = lmax + 1;
  t.assign((size_t)n * n * n, 0.0);
  for (int a = 0; a < n; ++a)
    for (int b = 0; b < n; ++b)
      for (int c = 0; c < n; ++c) t[((size_t)a * n + b) * n + c] = threej000_sq(a, b, c);
}

constexpr int kEdgeN = kLmaxCap + 1;
constexpr int kEdgeStride = kEdgeN + 2;  // doubles per matrix row: the right-hand side in column n, odd
constexpr int kEdgeWarps = 4;

// One warp solves one bin pair's system, the matrix in shared memory: lanes
// take entries while it is built, rows while a pivot is chosen, and columns
// while it is eliminated.  Bound by FP64 (two FMAs a clock and SM; about 110
// warp FMAs a pair at l_max 10, 7 us for 36 x 36 bins) and, at 8 warps per SM,
// by the latency of its steps.  One thread a pair kept
// its matrix in local memory and left most of the chip idle (36 bins, l_max
// 10: 170 us; now 52, cold caches).
__global__ void __launch_bounds__(32 * kEdgeWarps) k_edge_correct(const double* zn, const double* zr,
                                                                  const double* __restrict__ tj, int lmax, int nb,
                                                                  double* out) {
  __shared__ double s_m[kEdgeWarps][kEdgeN * kEdgeStride];
  __shared__ double s_v[kEdgeWarps][kEdgeN + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t = blockIdx.x * kEdgeWarps + warp;
  if (t >= nb * nb) return;  // a whole warp; no block barrier below
  double* m = s_m[warp];
  double* v = s_v[warp];
  const int n = lmax + 1;
  const size_t plane = (size_t)nb * nb;
  const bool row = lane < n;
  const double c = 0.5 * (2.0 * lane + 1.0);
  const double r = row ? c * zr[lane * plane + t] : 0.0;
  const double nn = row ? c * zn[lane * plane + t] : 0.0;
  const double r0 = __shfl_sync(0xffffffffu, r, 0);
  bool ok = r0 != 0.0 && isfinite(r0);
  const double f = ok ? r / r0 : 0.0;
  // a ratio that is not finite enters every row
  ok = ok && __all_sync(0xffffffffu, isfinite(f));
  if (row) {
    v[lane] = f;
    m[lane * kEdgeStride + n] = ok ? nn / r0 : 0.0;
  }
  __syncwarp();
  // M_ll' = (2l+1) sum_l'' (l l' l''; 000)^2 f_l'': l'' of the triangle and parity
  for (int e = lane; e < n * n; e += 32) {
    const int l = e / n, lp = e - l * n;
    double s = 0.0;
    for (int q = l > lp ? l - lp : lp - l; q <= l + lp && q < n; q += 2) s += __ldg(tj + ((size_t)l * n + lp) * n + q) * v[q];
    m[l * kEdgeStride + lp] = (2.0 * l + 1.0) * s;
  }
  __syncwarp();
  // Gaussian elimination with partial pivoting (the first of equal pivots)
  for (int k = 0; k < n && ok; ++k) {
    double best = row && lane >= k ? fabs(m[lane * kEdgeStride + k]) : -1.0;
    const bool bad = isnan(__shfl_sync(0xffffffffu, best, k));
    if (isnan(best)) best = -1.0;
    int piv = lane;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double b2 = __shfl_xor_sync(0xffffffffu, best, o);
      const int p2 = __shfl_xor_sync(0xffffffffu, piv, o);
      if (b2 > best || (b2 == best && p2 < piv)) {
        best = b2;
        piv = p2;
      }
    }
    ok = !bad && best > 0.0;
    if (!ok) break;
    // swap rows k and piv; this lane's column of the pivot row
    const bool col = lane >= k && lane <= n;
    const double pk = col ? m[piv * kEdgeStride + lane] : 0.0;
    if (col && piv != k) {
      m[piv * kEdgeStride + lane] = m[k * kEdgeStride + lane];
      m[k * kEdgeStride + lane] = pk;
    }
    __syncwarp();
    if (row && lane > k) v[lane] = m[lane * kEdgeStride + k] / m[k * kEdgeStride + k];
    __syncwarp();
    if (col)
      for (int i = k + 1; i < n; ++i) m[i * kEdgeStride + lane] -= v[i] * pk;
    __syncwarp();
  }
  // back substitution, a column at a time; lane l ends with zeta_l
  double x = row ? m[lane * kEdgeStride + n] : 0.0;
  for (int k = n - 1; k >= 0 && ok; --k) {
    const double xk = __shfl_sync(0xffffffffu, x, k) / m[k * kEdgeStride + k];
    if (lane == k) x = xk;
    else if (lane < k) x -= m[lane * kEdgeStride + k] * xk;
  }
  if (row) out[lane * plane + t] = ok ? x : NAN;
}

cudaError_t launch_edge_correct(const double* zn, const double* zr, const double* tj, int lmax, int nbins,
                                double* out, cudaStream_t st) {
  const int total = nbins * nbins;
  k_edge_correct<<<(total + kEdgeWarps - 1) / kEdgeWarps, 32 * kEdgeWarps, 0, st>>>(zn, zr, tj, lmax, nbins, out);
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace ctb
