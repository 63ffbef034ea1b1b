// sphere.cu -- projected (angular) multipoles on the unit sphere.
//
// Paper, "Statement of need": 3PCF multipoles of scalar fields on the sphere
// (weak-lensing convergence, HEALPix pixels) by a harmonic decomposition of
// one angle of the triangle; "Implementation": each pivot's neighbours fill
// the multipole bins, with sin and cos from a Chebyshev recurrence rather
// than trigonometric calls; "Performance": about two operations per
// multipole for that recurrence.
//
// The neighbour lists come from the same grid and enumeration as the 3-D
// path (chord distance, exact integer bin decisions against chord edges
// 2 sin(theta_b / 2)).  Per neighbour j of pivot p: u, v = the separation
// projected on p's east and north unit vectors, cos(phi) = v / |(u, v)|,
// sin(phi) = u / |(u, v)| (phi = 0 when both vanish), and
//     a_m(p, b) += w_j (cos m phi, sin m phi),   m = 0..K,
// with cos m phi and sin m phi from X_m = 2 cos(phi) X_{m-1} - X_{m-2}
// (two FMAs per m; the weight rides along, as the recurrence is linear).
// Row layout per (primary, bin): [Re a_1, Im a_1, ..., Re a_K, Im a_K, a_0],
// padded to a multiple of 32: each (Re, Im) pair on an even slot, so one
// paired FP32 instruction (FFMA2 / FADD2) advances or accumulates both.
#include "pair.cuh"

namespace ctb {

template <int K>
struct StepSphere {
  static constexpr int NCP = round32(2 * K + 1);
  static constexpr bool kFullLaneLoop = true;
  static constexpr bool kPtsInRegs = false;
  static constexpr int kConvE = 0;  // the row holds a_m itself: no conversion
  float ex, ey;      // east unit vector (its z component is zero)
  float nx, ny, nz;  // north unit vector
  __device__ __forceinline__ void operator()(float2* acc, float w, float dx, float dy, float dz) const {
    const float u = fmaf(ex, dx, ey * dy);
    const float v = fmaf(nx, dx, fmaf(ny, dy, nz * dz));
    const float r2 = fmaf(u, u, v * v);
    const bool flat = !(r2 > 0.f);
    const float ir = rsqrtf(flat ? 1.f : r2);
    const float c = flat ? 1.f : v * ir;
    const float s = flat ? 0.f : u * ir;
    slot_ref<2 * K>(acc) += w;
    if constexpr (K >= 1) {
      const float2 c2 = make_float2(c + c, c + c);
      float2 p = make_float2(w, 0.f);          // w (cos, sin) of (m - 2) phi
      float2 q = make_float2(w * c, w * s);    // and of (m - 1) phi
      acc[0] = __fadd2_rn(acc[0], q);
#pragma unroll
      for (int m = 2; m <= K; ++m) {
        const float2 r = __ffma2_rn(c2, q, make_float2(-p.x, -p.y));
        acc[m - 1] = __fadd2_rn(acc[m - 1], r);
        p = q;
        q = r;
      }
    }
  }
};

// East and north unit vectors of the tangent plane at direction (x, y, z):
// e_E = z x n / |z x n|, e_N = n x e_E (n normalised); at a pole e_E = y.
__device__ __forceinline__ StepSphere<0> frame_at(float x, float y, float z) {
  const float il = rsqrtf(fmaf(x, x, fmaf(y, y, z * z)));
  x *= il;
  y *= il;
  z *= il;
  const float rho2 = fmaf(x, x, y * y);
  StepSphere<0> f;
  if (rho2 > 0.f) {
    const float ir = rsqrtf(rho2);
    const float rho = rho2 * ir;
    f.ex = -y * ir;
    f.ey = x * ir;
    f.nx = -z * x * ir;
    f.ny = -z * y * ir;
    f.nz = rho;
  } else {
    f.ex = 0.f;
    f.ey = 1.f;
    f.nx = -z;
    f.ny = 0.f;
    f.nz = x;
  }
  return f;
}

// One warp per primary, one run per group of S (primary, bin) lists (S = 0: the primary's own), as in k_alm.
template <int K, int S>
__global__ void __launch_bounds__(128) k_am(AlmArgs a) {
  extern __shared__ __align__(16) char s_am[];
  constexpr int NCP = StepSphere<K>::NCP;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  // per warp: flush buffers, list offsets, counts
  char* wbase = s_am + (size_t)warp * alm_smem_per_warp(NCP, S);
  float* sbuf = reinterpret_cast<float*>(wbase);
  uint32_t* s_off = reinterpret_cast<uint32_t*>(wbase + (size_t)alm_flush_floats(NCP, S) * sizeof(float));
  uint32_t* s_n = s_off + kNbinsCap;
  while (true) {
    unsigned long long i = 0;
    if (lane == 0) i = atomicAdd(a.work, 1ull);
    i = __shfl_sync(0xffffffffu, i, 0);
    if (i >= (unsigned long long)a.prim_count) break;
    const uint64_t ib = i * (uint64_t)a.nbins;
    load_lists(a, ib, s_off, s_n, true, lane);
    const int64_t gi = a.prim_begin + (int64_t)i;
    const uint32_t sp = a.prim ? __ldg(a.prim + gi) : (uint32_t)gi;
    const uint4 P = __ldg(a.pts + sp);
    const StepSphere<0> f0 = frame_at(fmaf((float)P.x, a.sph_unit, a.sph_origin[0]),
                                      fmaf((float)P.y, a.sph_unit, a.sph_origin[1]),
                                      fmaf((float)P.z, a.sph_unit, a.sph_origin[2]));
    const StepSphere<K> step{f0.ex, f0.ey, f0.nx, f0.ny, f0.nz};
    run_primary<StepSphere<K>, S>(a, step, s_off, s_n, P, a.M + ib * (uint64_t)a.row, nullptr, sbuf, lane);
    __syncwarp();
  }
}

template <int K, int S>
static constexpr size_t am_smem(int wpb) {
  return (size_t)wpb * alm_smem_per_warp(StepSphere<K>::NCP, S);
}

template <int K, int S>
static int am_occupancy_K(int wpb) {
  return resident_blocks((const void*)k_am<K, S>, wpb * 32, am_smem<K, S>(wpb));
}

template <int K, int S>
static cudaError_t launch_am_KS(const AlmArgs& a, int wpb, int nsm, cudaStream_t st) {
  const int bps = am_occupancy_K<K, S>(wpb);
  if (bps < 1) return cudaErrorInvalidConfiguration;
  const cudaError_t e = allow_smem((const void*)k_am<K, S>, am_smem<K, S>(wpb));
  if (e != cudaSuccess) return e;
  k_am<K, S><<<bps * nsm, wpb * 32, am_smem<K, S>(wpb), st>>>(a);
  ++g_launches;
  return cudaGetLastError();
}

template <int K>
static cudaError_t launch_am_K(const AlmArgs& a, int lists, int wpb, int nsm, cudaStream_t st) {
  switch (lists) {
    case 1:
      return launch_am_KS<K, 1>(a, wpb, nsm, st);
    case 2:  // 72 registers against 80 of the mixed kernel: 12.6M pixels 376 ms against 390
      return launch_am_KS<K, 2>(a, wpb, nsm, st);
    case 4:
      return launch_am_KS<K, 4>(a, wpb, nsm, st);
  }
  return launch_am_KS<K, 0>(a, wpb, nsm, st);
}

#define CTB_SPHERE_CASES(X) \
  X(0) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(11) X(12) X(13) X(14) X(15) X(16)

int am_blocks_per_sm(int mmax, int wpb) {
  switch (mmax) {
#define CASE(K) \
  case K:       \
    return am_occupancy_K<K, 1>(wpb);
    CTB_SPHERE_CASES(CASE)
#undef CASE
    default:
      return 0;
  }
}

cudaError_t launch_am(const AlmArgs& a, int mmax, int lists, int wpb, int nsm, cudaStream_t st) {
  switch (mmax) {
#define CASE(K) \
  case K:       \
    return launch_am_K<K>(a, lists, wpb, nsm, st);
    CTB_SPHERE_CASES(CASE)
#undef CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace ctb
