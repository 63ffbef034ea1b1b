// pair_dispatch.cu -- coefficient layout, recurrence constants, and the
// ell_max dispatch of the pair-multipole kernel.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>
#include <vector>

#include "ctb_internal.cuh"

namespace ctb {

// explicit instantiations live in pair_[a-f].cu
template <int L>
cudaError_t launch_alm_L(const AlmArgs&, int, int, int, cudaStream_t);
template <int L>
int alm_occupancy_L(int);

void make_layout(int L, Layout* out) {
  Layout& y = *out;
  y.L = L;
  y.npass = 0;
  int base = 0;
  for (int i = 0; i < (kLmaxCap + 1) * (kLmaxCap + 1); ++i) y.slot[i] = -1;
  for (int m0 = 0; m0 <= L;) {
    int m1 = pass_end(L, m0, pass_cap(L, m0));
    int ncp = round32(coef_count(L, m0, m1));
    y.m0[y.npass] = m0;
    y.m1[y.npass] = m1;
    y.base[y.npass] = base;
    y.ncp[y.npass] = ncp;
    for (int l = m0; l <= L; ++l) {
      int hi = l < m1 ? l : m1;
      for (int m = -hi; m <= hi; ++m) {
        int am = m < 0 ? -m : m;
        if (am < m0) continue;
        y.slot[l * l + l + m] = base + local_slot(L, l, m, m0, m1);
      }
    }
    base += ncp;
    ++y.npass;
    m0 = m1 + 1;
  }
  y.row = base;
}

// a_lm = sqrt((4l^2-1)/(l^2-m^2)),  b_lm = sqrt(((l-1)^2-m^2)/(4(l-1)^2-1)):
// the normalised associated-Legendre recurrence  Pbar_l = a (z Pbar_{l-1} - b Pbar_{l-2}).
static double rec_a(int l, int m) { return std::sqrt((4.0 * l * l - 1.0) / ((double)l * l - (double)m * m)); }
static double rec_b(int l, int m) {
  return std::sqrt((((double)(l - 1) * (l - 1)) - (double)m * m) / (4.0 * (l - 1) * (l - 1) - 1.0));
}

// Normalisation C_lm turning the monic p_l^m times Re/Im (x+iy)^m into the
// real orthonormal Y_l,+-m (Condon-Shortley phase and sqrt 2 for m != 0):
//   C_mm = (-1)^m / sqrt(4 pi) prod_{k=1..m} sqrt((2k+1)/(2k)),
//   C_lm = C_mm prod_{k=m+1..l} a_km.
double norm_lm(int l, int m) {
  int am = m < 0 ? -m : m;
  double c = 1.0 / std::sqrt(4.0 * M_PI);
  for (int k = 1; k <= am; ++k) c *= -std::sqrt((2.0 * k + 1.0) / (2.0 * k));
  for (int k = am + 1; k <= l; ++k) c *= rec_a(k, am);
  if (am != 0) c *= M_SQRT2;
  return c;
}

// T-basis coefficients of the monic recurrence polynomial p_l^m(z) (degree
// l - m): p_m = 1, p_{m+1} = z, p_l = z p_{l-1} - beta_lm p_{l-2}, with
// z T_0 = T_1 and z T_k = (T_{k+1} + T_{k-1}) / 2.
static std::vector<double> monic_in_T(int l, int m) {
  const int n = l - m;
  std::vector<double> p2(n + 2, 0.0), p1(n + 2, 0.0);
  p2[0] = 1.0;  // p_m
  if (n == 0) return std::vector<double>(p2.begin(), p2.begin() + 1);
  p1[1] = 1.0;  // p_{m+1} = z = T_1
  for (int ll = m + 2; ll <= l; ++ll) {
    std::vector<double> zp(n + 2, 0.0);
    for (int k = 0; k <= n; ++k) {
      if (p1[k] == 0.0) continue;
      if (k == 0) {
        zp[1] += p1[0];
      } else {
        zp[k + 1] += 0.5 * p1[k];
        zp[k - 1] += 0.5 * p1[k];
      }
    }
    const double beta = rec_b(ll, m) / rec_a(ll - 1, m);
    for (int k = 0; k <= n; ++k) zp[k] -= beta * p2[k];
    p2 = p1;
    p1 = zp;
  }
  return std::vector<double>(p1.begin(), p1.begin() + n + 1);
}

// T-basis coefficients of the basis of the pass that starts at column m0:
// q_0 = 1, q_1 = c z, q_k = c z q_{k-1} - q_{k-2} with c the device's float
// constant.
static std::vector<std::vector<double>> pass_basis(int n, int m0) {
  const double c = (double)basis_scale(m0);
  std::vector<std::vector<double>> q(n + 1, std::vector<double>(n + 1, 0.0));
  q[0][0] = 1.0;
  for (int k = 1; k <= n; ++k) {
    for (int j = 0; j < k; ++j) {
      if (j == 0) {
        q[k][1] += c * q[k - 1][0];
      } else {
        q[k][j + 1] += 0.5 * c * q[k - 1][j];
        q[k][j - 1] += 0.5 * c * q[k - 1][j];
      }
    }
    if (k >= 2)
      for (int j = 0; j <= k - 2; ++j) q[k][j] -= q[k - 2][j];
  }
  return q;
}

// Coefficients D of p^m_l in that basis: p^m_l = sum_k D_k q_k, by back
// substitution on the T-basis coefficients (q_k has degree k with a nonzero
// T_k coefficient).
static std::vector<double> monic_in_basis(int l, int m, int m0) {
  const int n = l - m;
  const std::vector<std::vector<double>> q = pass_basis(n, m0);
  std::vector<double> r = monic_in_T(l, m), d(n + 1, 0.0);
  for (int k = n; k >= 0; --k) {
    d[k] = r[k] / q[k][k];
    for (int j = 0; j <= k; ++j) r[j] -= d[k] * q[k][j];
  }
  return d;
}

// Each pass accumulates moments S_{m,k} = sum w c_m q_k(z) of its columns in
// slot (m + k, +-m), q_k its basis.  Normalised a_lm = C_lm sum_k D_k S_{m,k},
// D the coefficients of p^m_l in that basis.
bool make_conversion(const Layout& lay, std::vector<uint8_t>& tab) {
  const int L = lay.L;
  struct Ent {
    int src;  // source slot of the even slot of a unit
    float c[2];
  };
  std::vector<std::vector<Ent>> ent(lay.row / 2);  // by unit
  for (int p = 0; p < lay.npass; ++p) {
    const int m0 = lay.m0[p];
    for (int am = m0; am <= lay.m1[p] && am <= L; ++am) {
      for (int l = am; l <= L; ++l) {
        const std::vector<double> d = monic_in_basis(l, am, m0);
        const int s = lay.slot[l * l + l + am];
        std::vector<Ent>& v = ent[s / 2];
        // degrees of the polynomial's parity, from the highest (the others
        // are exactly zero).  Column 0: slots l and l + 1 share a unit, and
        // their e-th entries lie in one unit too.
        for (int k = l - am, e = 0; k >= 0; k -= 2, ++e) {
          const int sl = am + k;
          const int src = lay.slot[sl * sl + sl + am];
          const float c = (float)(norm_lm(l, am) * d[k]);
          if (am > 0) {
            v.push_back({src, {c, (float)(norm_lm(l, -am) * d[k])}});
          } else {
            if ((int)v.size() <= e) v.push_back({src & ~1, {0.f, 0.f}});
            if (v[e].src != (src & ~1) || (src & 1) != (s & 1)) return false;
            v[e].c[s & 1] = c;
          }
        }
      }
    }
  }
  // padded, entry-major per pass; local units
  tab.clear();
  for (int p = 0; p < lay.npass; ++p) {
    const int E = conv_entries(L, lay.m0[p]), U = lay.ncp[p] / 2, base = lay.base[p];
    const size_t t0 = tab.size();
    tab.resize(t0 + (size_t)conv_table_bytes(lay.ncp[p], E), 0);
    for (int u = 0; u < U; ++u) {
      const auto& v = ent[base / 2 + u];
      if ((int)v.size() > conv_round_entries(L, lay.m0[p], lay.m1[p], u / 32)) return false;
      for (int e = 0; e < E; ++e) {
        const size_t k = (size_t)e * U + u;
        const bool in = e < (int)v.size();
        const float c[2] = {in ? v[e].c[0] : 0.f, in ? v[e].c[1] : 0.f};
        std::memcpy(tab.data() + t0 + k * 8, c, 8);
        tab[t0 + (size_t)E * U * 8 + k] = (uint8_t)(in ? (v[e].src - base) / 2 : u);
      }
    }
  }
  return true;
}

int alm_blocks_per_sm(int L, int wpb) {
  switch (L) {
#define CASE(X) \
  case X:       \
    return alm_occupancy_L<X>(wpb);
    CASE(0) CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8) CASE(9) CASE(10)
    CASE(12) CASE(14) CASE(16) CASE(18) CASE(20)
#undef CASE
    default:
      return 0;
  }
}

// A flush costs little more for S lists than for one, but a group of S runs as
// long as its longest list, on 32 / S lanes a list, and the last group does so
// with fewer lists.  Cost of a primary with T neighbours, in hundredths of a
// step of one list (fitted at l_max 10; l_max 4 and 20 lie within 30 %):
//   S 1   100 (T / 32 + nbins / 2)            + 500 nbins
//   S 2   104 (T w2 / 16 + nbins / 2 / 2)     + 460 nbins / 2
//   S 4   104 (T w4 / 8 + nbins / 4 / 2)      + 490 nbins / 4
// w2, w4: the longest lists of the groups as a share of all; numbers of groups
// rounded up.  With many bins that puts the limits near means of 160 and 800
// neighbours a list, where they are held at most; with few they are lower.
// Accumulation with 1 / 2 / 4 lists (8: slower than 4 except at 8 neighbours a
// list, where they tie):
//   mean list 8 (20k uniform points, l_max 10)      0.226 / 0.144 / 0.116 ms
//   28 (200k points, l_max 20)                      24.0 / 16.7 / 14.7
//   80 (24 mock catalogues, l_max 10)               52.3 / 39.4 / 39.4
//   132 (3.1M-pixel sphere, m_max 8)                38.0 / 29.6 / 28.4
//   522 (cut sky of 800k points, l_max 10)          118.1 / 111.1 / 113.2
//   525 (250k primaries of 4M, l_max 20)            134.1 / 132.3 / 145.7
//   1680 (10^6 points, l_max 10)                    221.5 / 243.1 / 274.0
//   100k points from r_min 0, l_max 10: 1 bin of 130  0.247 / 0.299 / 0.448
//     5 bins of 60   0.738 / 0.616 / 0.784;  of 400   1.720 / 2.345 / 4.002
//     10 bins of 16  1.081 / 0.688 / 0.586;  of 130   1.793 / 1.374 / 1.797
// (160 and 800 for any number of bins took up to 1.9 times the best there.)
// A choice by each primary's list lengths, the same costs on its own counts,
// was slower: neighbours in space then differ in S, and three forms running
// at once overflow the instruction cache (7 bins of 60: 0.95 ms).
ListLimits list_limits(const double* share, int nbins) {
  if (nbins < 2) return ListLimits{0, 0};
  double sum = 0, m2 = 0, m4 = 0;
  for (int b = 0; b < nbins; ++b) {
    sum += share[b];
    if (b % 2 == 0) m2 += std::max(share[b], b + 1 < nbins ? share[b + 1] : 0.0);
    if (b % 4 == 0) m4 += *std::max_element(share + b, share + std::min(b + 4, nbins));
  }
  if (!(sum > 0)) sum = m2 = m4 = 1;
  const int g2 = (nbins + 1) / 2, g4 = (nbins + 3) / 4;
  const double a[3] = {100.0 / 32, 104 * m2 / sum / 16, 104 * m4 / sum / 8};  // per neighbour: S 1, 2, 4
  const double f[3] = {550.0 * nbins, 512.0 * g2, 542.0 * g4};                 // per primary
  // neighbours below which form i is cheaper than form j of fewer lists
  auto below = [&](int i, int j) {
    if (f[i] >= f[j]) return 0.0;
    return a[i] > a[j] ? (f[j] - f[i]) / (a[i] - a[j]) : 1e300;
  };
  const double two = std::max(below(1, 0), below(2, 0)), four = std::min(below(2, 1), below(2, 0));
  ListLimits m;
  m.four = (uint32_t)std::min(four, 160.0 * nbins);
  m.two = std::max(m.four, (uint32_t)std::min(two, 800.0 * nbins));
  return m;
}

cudaError_t launch_alm(const AlmArgs& a, int L, int lists, int wpb, int nsm, cudaStream_t st) {
  switch (L) {
#define CASE(X) \
  case X:       \
    return launch_alm_L<X>(a, lists, wpb, nsm, st);
    CASE(0) CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8) CASE(9) CASE(10)
    CASE(12) CASE(14) CASE(16) CASE(18) CASE(20)
#undef CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace ctb
