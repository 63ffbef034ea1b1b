// pair.cuh -- harmonic accumulation of the pair multipoles (template;
// instantiated per ell_max in pair_[a-f].cu so they compile in parallel).
//
// Paper, "Implementation": pick a pivot, find all its neighbours inside the
// search range, fill the multipole bins; sin/cos of the angle are replaced by
// a polynomial recurrence because evaluating trigonometric functions is slow.
// "Performance": the time goes into scanning for neighbours and updating the
// histograms, with a per-multipole recurrence cost.
//
// GB300 design.  The neighbour lists of a primary are grouped by bin
// (stream.cu).  One warp owns one primary and takes its (primary, bin) lists
// one at a time (long lists) or two or four side by side, 32, 16 or 8 lanes a
// list (short ones): each lane takes one neighbour per step, evaluates
// polynomial moments of the direction by recurrences in float32 registers and
// accumulates them (one paired FMA per (+m, -m) pair of moments).  Up to
// l_max 10 one kernel holds all coefficients; above, the m columns are split
// into passes of at most kPassCap accumulators, each its own kernel and
// launch (see k_alm).  At the end of the list its lanes' accumulators are
// summed through a shared-memory transpose, mapped to normalised a_lm and
// stored as the (primary, bin) row of M.  The cross-lane reduction happens
// once per list, and the first loads of the next lists are issued while the
// current ones are still being accumulated.
//
// Moments (real Y_lm up to a fixed linear map per (l, m), applied at the flush):
//   (c_m + i s_m) = w (x + i y)^m        one paired FMUL + FFMA per m
//   q_k(z)        = the pass's basis, U_k(z / s): Chebyshev polynomials of the
//                   second kind, scaled (q_0 = 1, q_1 = t, q_k = t q_{k-1} -
//                   q_{k-2}, t = 2 z / s: one FMA per degree)
//   S_{m,k}      += q_k (c_m, s_m)       one paired FFMA per (k, +-m)
// The (1 - z^2)^{m/2} factor of the associated Legendre function is absorbed
// in (x + i y)^m, and it keeps |z| small where m is large: so the pass that
// starts at column m0 takes s < 1 (basis_scale), which makes its polynomials
// nearly orthogonal under that factor.  The flush's map then amplifies
// rounding by at most 11 (rms over z; l_max 10: 9, l_max 20: 6, 11 and 7 in
// the three passes).  T_k(z) for the first pass and the monic recurrence of
// column m0 for the others, the bases before these, amplified by up to 39 at
// l_max 10 and 64 at l_max 20 and took two instructions a degree above m = 2.
// Blackwell's paired FP32 instructions (FFMA2 / FMUL2 / FADD2) update the
// (+m, -m) accumulator pair in one issue slot; a stream of them takes 2.65
// cycles each against 1.65 for a scalar FFMA, 1.25 times the FMA rate.
#pragma once

#include <type_traits>

#include "ctb_internal.cuh"

namespace ctb {

constexpr uint32_t kNone = 0xffffffffu;
// The list words of one primary are one contiguous range; the read position
// is kept this many 128-byte lines ahead of use in L2.  The list buffer is
// allocated with kListSlackBytes past its last entry for prefetches that run
// beyond it.
constexpr uint32_t kListPrefetchLines = 6;

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// accumulator slot S of a float2 array: the even slot is .x, the odd .y
template <int S>
__device__ __forceinline__ float& slot_ref(float2* acc) {
  if constexpr ((S & 1) == 0) return acc[S >> 1].x;
  else return acc[S >> 1].y;
}

// Pair (k, +-M) of column M: acc += q_k (c, s) for k = K..L-M (k = 0: q_0 = 1).
template <int L, int M0, int M1, int M, int K>
__device__ __forceinline__ void column_pairs(float2* acc, const float* Q, float2 cs) {
  if constexpr (K <= L - M) {
    constexpr int i = local_slot(L, M + K, M, M0, M1) >> 1;
    if constexpr (K == 0) acc[i] = __fadd2_rn(acc[i], cs);
    else acc[i] = __ffma2_rn(make_float2(Q[K], Q[K]), cs, acc[i]);
    column_pairs<L, M0, M1, M, K + 1>(acc, Q, cs);
  }
}

// Column 0 (first pass only): acc(k, 0) += w q_k.
template <int L, int M0, int M1, int K>
__device__ __forceinline__ void column_zero(float2* acc, const float* Q, float w) {
  if constexpr (K <= L) {
    float& a = slot_ref<local_slot(L, K, 0, M0, M1)>(acc);
    a = K == 0 ? a + w : fmaf(w, Q[K], a);
    column_zero<L, M0, M1, K + 1>(acc, Q, w);
  }
}

// Columns M..ME with cs = w (x + i y)^M on entry; xy = (x, y), myx = (-y, x),
// so cs (x + i y) = cs.x xy + cs.y myx.
template <int L, int M0, int M1, int M, int ME>
__device__ __forceinline__ void columns(float2* acc, const float* Q, float2 xy, float2 myx, float2 cs) {
  if constexpr (M <= ME) {
    column_pairs<L, M0, M1, M, 0>(acc, Q, cs);
    if constexpr (M + 1 <= ME) {
      const float2 nx = __ffma2_rn(make_float2(cs.x, cs.x), xy, __fmul2_rn(make_float2(cs.y, cs.y), myx));
      columns<L, M0, M1, M + 1, ME>(acc, Q, xy, myx, nx);
    }
  }
}

// q_k, k = K..KMAX: q_k = t q_{k-1} - q_{k-2}.
template <int K, int KMAX>
__device__ __forceinline__ void basis_seq(float* Q, float t) {
  if constexpr (K <= KMAX) {
    Q[K] = fmaf(t, Q[K - 1], -Q[K - 2]);
    basis_seq<K + 1, KMAX>(Q, t);
  }
}

// (x + i y)^E, E >= 1, by repeated squaring: a pass that starts at column
// m0 needs the power m0, in about 4 log2(m0) instructions instead of 4 m0.
template <int E>
__device__ __forceinline__ void cpow(float x, float y, float& r, float& i) {
  if constexpr (E == 1) {
    r = x;
    i = y;
  } else if constexpr (E % 2 == 0) {
    float a, b;
    cpow<E / 2>(x, y, a, b);
    r = fmaf(a, a, -(b * b));
    i = (a + a) * b;
  } else {
    float a, b;
    cpow<E - 1>(x, y, a, b);
    r = fmaf(a, x, -(b * y));
    i = fmaf(a, y, b * x);
  }
}

// Degree-major order for passes of few columns: the powers of all columns
// first, then per degree k the next basis polynomial and the moments of
// every column that reaches degree k.  Only three basis values are live at a
// time (against all L - m0 + 1 in column-major order), which keeps the wide
// passes of l_max 20 within their register budget.
template <int L, int M0, int M1, int K, int KMAX, int MS, int ME>
__device__ __forceinline__ void degrees(float2* acc, const float2* cs, float w, float t, float q2, float q1) {
  if constexpr (K <= KMAX) {
    float q;
    if constexpr (K == 0) q = 1.f;
    else if constexpr (K == 1) q = t;
    else q = fmaf(t, q1, -q2);
    if constexpr (M0 == 0) {
      float& c0 = slot_ref<local_slot(L, K, 0, M0, M1)>(acc);
      c0 = K == 0 ? c0 + w : fmaf(w, q, c0);
    }
#pragma unroll
    for (int m = MS; m <= ME; ++m) {
      if (K <= L - m) {
        const int i = local_slot(L, m + K, m, M0, M1) >> 1;
        if (K == 0) acc[i] = __fadd2_rn(acc[i], cs[m - MS]);
        else acc[i] = __ffma2_rn(make_float2(q, q), cs[m - MS], acc[i]);
      }
    }
    degrees<L, M0, M1, K + 1, KMAX, MS, ME>(acc, cs, w, t, q1, q);
  }
}

// columns of a pass that is accumulated degree-major
__host__ __device__ constexpr bool degree_major(int L, int m0, int m1) {
  return (m1 < L ? m1 : L) - (m0 < 1 ? 1 : m0) + 1 <= 5;
}

// Add one neighbour (weight w, unit direction x, y, z) to the pass's
// accumulators: the pass's basis sequence, the complex powers, and one
// paired FMA per (k, +-m) moment (one FMA per moment of column 0).  The
// caller passes t = basis_scale(M0) z, the only form z appears in.
template <int L, int M0, int M1>
__device__ __forceinline__ void accum_pass(float2* acc, float w, float x, float y, float t) {
  constexpr int KMAX = L - M0;  // highest basis degree this pass needs
  constexpr int MS = M0 < 1 ? 1 : M0;
  constexpr int ME = M1 < L ? M1 : L;
  if constexpr (degree_major(L, M0, M1)) {
    constexpr int NC = ME >= MS ? ME - MS + 1 : 1;
    float2 cs[NC];
    if constexpr (MS <= ME) {
      float pr, pi;
      cpow<MS>(x, y, pr, pi);
      cs[0] = make_float2(w * pr, w * pi);
      const float2 xy = make_float2(x, y), myx = make_float2(-y, x);
#pragma unroll
      for (int c = 1; c < NC; ++c)
        cs[c] = __ffma2_rn(make_float2(cs[c - 1].x, cs[c - 1].x), xy, __fmul2_rn(make_float2(cs[c - 1].y, cs[c - 1].y), myx));
    }
    degrees<L, M0, M1, 0, KMAX, MS, ME>(acc, cs, w, t, 0.f, 0.f);
  } else {
    float Q[KMAX + 1 > 2 ? KMAX + 1 : 2];
    Q[0] = 1.f;
    Q[1] = t;
    basis_seq<2, KMAX>(Q, t);
    if constexpr (M0 == 0) column_zero<L, M0, M1, 0>(acc, Q, w);
    if constexpr (MS <= ME) {
      float pr, pi;
      cpow<MS>(x, y, pr, pi);  // (x + i y)^MS by squaring
      columns<L, M0, M1, MS, ME>(acc, Q, make_float2(x, y), make_float2(-y, x), make_float2(w * pr, w * pi));
    }
  }
}

// Cross-lane sum of the accumulators through shared memory, in chunks of
// at most kFlushChunk slots: every lane writes its chunk (stride W + 4 floats,
// so 16-byte stores of 8 consecutive lanes cover all 32 banks), then the G =
// 32 / S lanes of list s sum the chunk's columns over that list's G rows and
// write its totals to tot[s][chunk start + column].  The 32 rows are written
// and read once whatever S, so S lists share the cost of one flush.
constexpr int kFlushChunk = 64;
__host__ __device__ constexpr int flush_buf_floats(int ncp) {
  return 32 * ((ncp < kFlushChunk ? ncp : kFlushChunk) + 4);
}

template <int NCP, int S, int C0>
__device__ __forceinline__ void flush_chunks(const float2* acc, float* buf, float* tot, int lane) {
  if constexpr (C0 < NCP) {
    constexpr int W = NCP - C0 < kFlushChunk ? NCP - C0 : kFlushChunk;
    constexpr int ST = W + 4;
    constexpr int G = 32 / S;
    constexpr int V = W / G;  // columns per lane
    float* row = buf + lane * ST;
#pragma unroll
    for (int i = 0; i < W / 2; i += 2)
      *reinterpret_cast<float4*>(row + 2 * i) =
          make_float4(acc[C0 / 2 + i].x, acc[C0 / 2 + i].y, acc[C0 / 2 + i + 1].x, acc[C0 / 2 + i + 1].y);
    __syncwarp();
    const int sl = lane & (G - 1), s = lane / G;
    const float* rows = buf + s * G * ST;
    float* t = tot + s * NCP + C0;
    if constexpr (V >= 4) {
      // columns h 4 G + 4 sl .. + 3: contiguous over the list's lanes
#pragma unroll
      for (int h = 0; h < V / 4; ++h) {
        const int col = (h * G + sl) * 4;
        float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
#pragma unroll
        for (int r = 0; r < G; r += 2) {
          const float4 u = *reinterpret_cast<const float4*>(rows + r * ST + col);
          const float4 v = *reinterpret_cast<const float4*>(rows + (r + 1) * ST + col);
          s0.x += u.x; s0.y += u.y; s0.z += u.z; s0.w += u.w;
          s1.x += v.x; s1.y += v.y; s1.z += v.z; s1.w += v.w;
        }
        *reinterpret_cast<float4*>(t + col) = make_float4(s0.x + s1.x, s0.y + s1.y, s0.z + s1.z, s0.w + s1.w);
      }
    } else if constexpr (V == 2) {
      float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll
      for (int r = 0; r < G; r += 2) {
        const float2 u = *reinterpret_cast<const float2*>(rows + r * ST + 2 * sl);
        const float2 v = *reinterpret_cast<const float2*>(rows + (r + 1) * ST + 2 * sl);
        s0.x += u.x; s0.y += u.y;
        s1.x += v.x; s1.y += v.y;
      }
      *reinterpret_cast<float2*>(t + 2 * sl) = make_float2(s0.x + s1.x, s0.y + s1.y);
    } else {
      float sm[V];
#pragma unroll
      for (int c = 0; c < V; ++c) sm[c] = 0.f;
#pragma unroll
      for (int r = 0; r < G; ++r)
#pragma unroll
        for (int c = 0; c < V; ++c) sm[c] += rows[r * ST + V * sl + c];
#pragma unroll
      for (int c = 0; c < V; ++c) t[V * sl + c] = sm[c];
    }
    __syncwarp();  // the buffer is rewritten by the next chunk
    flush_chunks<NCP, S, C0 + W>(acc, buf, tot, lane);
  }
}

// Flush conversion of one pass, in units of two slots (2u, 2u + 1): the (+m,
// -m) pair of one (l, m), or the m = 0 slots of l and l + 1.  Entry e of unit
// u, at [e * NCP / 2 + u]: the coefficients of both slots and the unit whose
// totals they multiply (zero coefficients pad the units with fewer entries).
// Lane l maps units l, l + 32, ..: out[u] = sum_e coef * tot[src], one table
// read for the S lists, the loads of every entry independent of each other.
// `tab`: the coefficient pairs, then the source units as bytes.
template <class Step, int S, int I>
__device__ __forceinline__ void flush_store(const float2* tab, const float* tot, float* __restrict__ out, int64_t row,
                                            int nlists, int lane) {
  constexpr int U = Step::NCP / 2;
  if constexpr (32 * I < U) {
    const int u = lane + 32 * I;
    if (32 * I + 32 <= U || u < U) {
      float2 v[S];
      if constexpr (Step::kConvE == 0) {  // the totals are the row itself
#pragma unroll
        for (int s = 0; s < S; ++s) v[s] = *reinterpret_cast<const float2*>(tot + s * Step::NCP + 2 * u);
      } else {
        constexpr int E = Step::conv_round(I);
#pragma unroll
        for (int s = 0; s < S; ++s) v[s] = make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const float2 c = tab[e * U + u];
          const float* t = tot + 2 * reinterpret_cast<const uint8_t*>(tab + U * Step::kConvE)[e * U + u];
#pragma unroll
          for (int s = 0; s < S; ++s) v[s] = __ffma2_rn(c, *reinterpret_cast<const float2*>(t + s * Step::NCP), v[s]);
        }
      }
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (S == 1 || s < nlists) __stcs(reinterpret_cast<float2*>(out + s * row) + u, v[s]);
    }
    flush_store<Step, S, I + 1>(tab, tot, out, row, nlists, lane);
  }
}

// One neighbour list run: records [off, off + n) of the lists buffer.
struct Run {
  uint32_t off, n;
};

// Loads in flight, for steps t, t + 1 and t + 2 of the concatenated runs:
// the neighbours of the next two steps (q0, q1; j0, j1 their record words,
// kNone for a lane without one) and the record word of the step after.
struct Prefetch {
  uint32_t j0, j1, j2;
  uint4 q0, q1;
};

// Record of iteration t of the concatenated runs [cur | nxt] (T = iterations of cur).
__device__ __forceinline__ uint32_t rec_at(const uint32_t* __restrict__ lists, Run cur, Run nxt, uint32_t T,
                                           uint32_t t, int lane) {
  if (t < T) {
    const uint32_t k = t * 32 + lane;
    return k < cur.n ? __ldcs(lists + cur.off + k) : kNone;
  }
  const uint32_t k = (t - T) * 32 + lane;
  return k < nxt.n ? __ldcs(lists + nxt.off + k) : kNone;
}

// The points' base, as a register pair in k_alm.  Its arguments stay in
// constant memory (__grid_constant__), which suits every pointer but this
// one, used once a step to address the gather: against arguments that the
// compiler may copy, at l_max 10 with one list a warp (3.36e10 pairs) 219.5
// ms with this base in registers, 222.2 without, 225.6 with all of them
// copied; two lists a warp (1.51e10 pairs) 108.5, 111.9 and 108.3.
template <class Step>
__device__ __forceinline__ const uint4* points_base(const uint4* p) {
  if constexpr (Step::kPtsInRegs) asm volatile("" : "+l"(p));
  return p;
}

__device__ __forceinline__ uint4 gather(const uint4* __restrict__ pts, uint32_t j, uint4 P) {
  return j != kNone ? __ldg(pts + j) : P;
}

// Loads of the first three iterations of the concatenated runs [r | nxt].
__device__ __forceinline__ Prefetch prefetch_start(const uint32_t* lists, const uint4* pts, Run r, Run nxt,
                                                   uint4 P, int lane) {
  Prefetch pf;
  const uint32_t T = (r.n + 31u) / 32u;
  pf.j0 = rec_at(lists, r, nxt, T, 0, lane);
  pf.j1 = rec_at(lists, r, nxt, T, 1, lane);
  pf.j2 = rec_at(lists, r, nxt, T, 2, lane);
  pf.q0 = gather(pts, pf.j0, P);
  pf.q1 = gather(pts, pf.j1, P);
  return pf;
}

// The per-neighbour work of one m-range pass of the 3-D harmonics: the unit
// direction, then the pass's recurrences and one FMA per coefficient.
template <int L, int M0, int M1>
struct Step3D {
  static constexpr int NCP = round32(coef_count(L, M0, M1));
  // Each launch runs one m-pass, so the full-lane copy of the step and the
  // general one are the only code in the instruction cache.
  static constexpr bool kFullLaneLoop = true;
  static constexpr bool kPtsInRegs = true;
  // flush conversion entries per unit: moment degrees of the same parity, and
  // how many the units of one round of 32 need (they are sorted by degree)
  static constexpr int kConvE = conv_entries(L, M0);
  static constexpr int conv_round(int r) { return conv_round_entries(L, M0, M1, r); }
  __device__ __forceinline__ void operator()(float2* acc, float w, float dx, float dy, float dz) const {
    accum(acc, unit(w, dx, dy, dz));
  }
  // The unit direction (x, y, basis_scale z) and weight of a neighbour, ahead of its
  // accumulation.  The full-lane loop of a single-pass kernel (l_max <= 10)
  // prepares each step's direction one iteration ahead (5 % faster at
  // l_max 10); in the 255-register passes of l_max 20 the extra live state
  // made the pass slower, so they keep the plain step.
  __device__ __forceinline__ float4 prep(uint4 q, uint4 P) const {
    const float dx = __int2float_rn((int)(q.x - P.x));
    const float dy = __int2float_rn((int)(q.y - P.y));
    const float dz = __int2float_rn((int)(q.z - P.z));
    return unit(__uint_as_float(q.w), dx, dy, dz);
  }
  __device__ __forceinline__ float4 unit(float w, float dx, float dy, float dz) const {
    const float ir = rsqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    return make_float4(dx * ir, dy * ir, dz * (ir * basis_scale(M0)), w);
  }
  __device__ __forceinline__ void accum(float2* acc, float4 s) const { accum_pass<L, M0, M1>(acc, s.w, s.x, s.y, s.z); }
  static constexpr bool kPrep = L <= kSinglePassLmax;
};

template <class S, class = void>
struct has_prep : std::false_type {};
template <class S>
struct has_prep<S, std::void_t<decltype(&S::prep)>> : std::true_type {};
template <class S>
__host__ __device__ constexpr bool use_prep() {
  if constexpr (has_prep<S>::value) return S::kPrep;
  else return false;
}

// Totals of the S lists held by the warp, in chunks of at most kFlushChunk
// slots through the transpose buffer, into tot[list][slot]; then every lane
// maps its units' totals to normalised a_lm (moments in the pass's basis ->
// the Legendre values of their column).
template <class Step, int S>
__device__ __forceinline__ void flush(const float2* acc, float* __restrict__ out, int64_t row, int nlists,
                                      const float2* ctab, float* sbuf, int lane) {
  float* tot = sbuf + flush_buf_floats(Step::NCP);
  flush_chunks<Step::NCP, S, 0>(acc, sbuf, tot, lane);
  __syncwarp();
  flush_store<Step, S, 0>(ctab, tot, out, row, nlists, lane);
  __syncwarp();
}

// Accumulate one pass over one run and store it to the row; the loads for
// the first iterations of `nxt` are issued inside the loop, so the next run
// starts without a memory bubble.  `step` adds one neighbour (weight and
// separation in units; a lane without a neighbour passes w = 0) to the
// Step::NCP accumulators.
template <class Step>
__device__ __forceinline__ void run_steps(const AlmArgs& a, const Step& step, Run cur, Run nxt, const uint4 P,
                                          Prefetch& pf, float* __restrict__ out, const float2* ctab, float* sbuf,
                                          int lane, uint32_t pe) {
  constexpr int NCP = Step::NCP;
  const uint32_t* __restrict__ lists = a.lists;
  const uint4* pts = points_base<Step>(a.pts);
  float2 acc[NCP / 2];
#pragma unroll
  for (int i = 0; i < NCP / 2; ++i) acc[i] = make_float2(0.f, 0.f);
  const uint32_t T = (cur.n + 31u) / 32u;
  // Steps 1 and 2 of [cur | nxt]: the previous run looked only one run
  // ahead, so when cur is shorter than that they are taken again here.
  {
    const uint32_t w1 = rec_at(lists, cur, nxt, T, 1, lane);
    if (w1 != pf.j1) {
      pf.j1 = w1;
      pf.q1 = gather(pts, w1, P);
    }
    pf.j2 = rec_at(lists, cur, nxt, T, 2, lane);
  }
  uint32_t t = 0;
  // Steps whose lanes all hold a neighbour and whose look-ahead words are in
  // this run: no validity tests, no run switch.  (The list buffer has slack
  // past its last entry, so the L2 prefetch needs no bound here.)  Two
  // neighbour gathers are in flight and the record word one step before
  // its gather.
  if constexpr (Step::kFullLaneLoop) {
    const uint32_t full = cur.n >> 5;
    if (t + 3u < full) {
      const uint32_t* __restrict__ wp = lists + cur.off + 96u + (uint32_t)lane;
      const uint32_t* pp = lists + cur.off + kListPrefetchLines * 32u;
      const bool lane0 = lane == 0;
      uint4 q0 = pf.q0, q1 = pf.q1;
      uint32_t j2 = pf.j2;
      if constexpr (use_prep<Step>()) {
        // each step's direction is prepared one iteration ahead, so its
        // dependent chain overlaps the previous step's accumulation
        float4 S = step.prep(q0, P);
#pragma unroll 1
        for (; t + 3u < full; ++t) {
          if (lane0) prefetch_l2(pp);
          pp += 32;
          const float4 Sn = step.prep(q1, P);
          q0 = q1;
          q1 = __ldg(pts + j2);
          j2 = __ldcs(wp);
          wp += 32;
          step.accum(acc, S);
          S = Sn;
        }
      } else {
#pragma unroll 1
        for (; t + 3u < full; ++t) {
          if (lane0) prefetch_l2(pp);
          pp += 32;
          const uint4 q = q0;
          q0 = q1;
          q1 = __ldg(pts + j2);
          j2 = __ldcs(wp);
          wp += 32;
          const float dx = __int2float_rn((int)(q.x - P.x));
          const float dy = __int2float_rn((int)(q.y - P.y));
          const float dz = __int2float_rn((int)(q.z - P.z));
          step(acc, __uint_as_float(q.w), dx, dy, dz);
        }
      }
      // t + 1 and t + 2 are full-lane steps of this run
      pf.q0 = q0;
      pf.q1 = q1;
      pf.j0 = 0u;
      pf.j1 = 0u;
      pf.j2 = j2;
    }
  }
  // the last steps of the run: partial lanes, look-ahead into the next run,
  // the same two gathers in flight
  for (; t < T; ++t) {
    const uint32_t pa = cur.off + (t + kListPrefetchLines) * 32u;
    if (lane == 0 && pa < pe) prefetch_l2(lists + pa);
    const uint4 q = pf.q0;
    const bool valid = pf.j0 != kNone;
    pf.q0 = pf.q1;
    pf.j0 = pf.j1;
    pf.q1 = gather(pts, pf.j2, P);
    pf.j1 = pf.j2;
    pf.j2 = rec_at(lists, cur, nxt, T, t + 3, lane);
    float dx = __int2float_rn((int)(q.x - P.x));
    float dy = __int2float_rn((int)(q.y - P.y));
    float dz = __int2float_rn((int)(q.z - P.z));
    float w = __uint_as_float(q.w);
    if (!valid) {
      dx = 1.f;
      dy = 0.f;
      dz = 0.f;
      w = 0.f;
    }
    step(acc, w, dx, dy, dz);
  }
  flush<Step, 1>(acc, out, a.row, 1, ctab, sbuf, lane);
}

// One primary's lists, one after another (S = 1): long lists.
template <class Step>
__device__ __forceinline__ void run_primary1(const AlmArgs& a, const Step& step, const uint32_t* s_off,
                                             const uint32_t* s_n, const uint4 P, float* __restrict__ rows,
                                             const float2* ctab, float* sbuf, int lane) {
  const int nbins = a.nbins;
  int b = 0;
  while (b < nbins && s_n[b] == 0) ++b;
  if (b >= nbins) return;
  int nb = b + 1;
  while (nb < nbins && s_n[nb] == 0) ++nb;
  Run cur{s_off[b], s_n[b]};
  Run nxt = nb < nbins ? Run{s_off[nb], s_n[nb]} : Run{0, 0};
  // end of this primary's list range; its first lines go to L2 now
  const uint32_t pe = s_off[nbins - 1] + s_n[nbins - 1];
  if (lane < (int)kListPrefetchLines && cur.off + (uint32_t)lane * 32u < pe)
    prefetch_l2(a.lists + cur.off + (uint32_t)lane * 32u);
  Prefetch pf = prefetch_start(a.lists, a.pts, cur, nxt, P, lane);
  while (true) {
    run_steps(a, step, cur, nxt, P, pf, rows + (int64_t)b * a.row, ctab, sbuf, lane, pe);
    b = nb;
    if (b >= nbins) return;
    cur = nxt;
    nb = b + 1;
    while (nb < nbins && s_n[nb] == 0) ++nb;
    nxt = nb < nbins ? Run{s_off[nb], s_n[nb]} : Run{0, 0};
  }
}

// One primary's lists S bins at a time, 32 / S lanes a list: short lists.
// The flush costs the same for S lists as for one, and the lanes of a list
// that is not a multiple of 32 are filled by the others'.  A group runs as
// long as its longest list (neighbouring bins are alike in size), lanes past
// the end of theirs adding a zero weight.  The loads run three steps ahead
// of the accumulation on a cursor of their own that walks the primary's
// groups: the record word, a step later its neighbour, a step later its
// direction (where the step prepares it).
template <class Step, int S>
__device__ __forceinline__ void run_groups(const AlmArgs& a, const Step& step, const uint32_t* s_off,
                                           const uint32_t* s_n, const uint4 P, float* __restrict__ rows,
                                           const float2* ctab, float* sbuf, int lane) {
  constexpr uint32_t G = 32 / S;
  const uint4* pts = points_base<Step>(a.pts);
  constexpr int NCP = Step::NCP;
  const int nbins = a.nbins;
  const int ls = lane / (int)G;
  const uint32_t sl = lane & (G - 1);
  // steps of the group at bin b: those of its longest list
  auto iters = [&](int b) {
    uint32_t n = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) n = max(n, s_n[b + s]);
    return (n + G - 1) / G;
  };
  auto skip = [&](int b, uint32_t& T) {  // first group with a neighbour at or after b
    for (T = 0; b < nbins; b += S)
      if ((T = iters(b)) != 0) break;
    return b;
  };
  // a group's list words to L2, while the group before it is read
  auto fetch = [&](int b) {
    if (b >= nbins) return;
    each_list_line(s_off[b], s_off[b + S - 1] + s_n[b + S - 1], (uint32_t)lane,
                   [&](uint32_t w) { prefetch_l2(a.lists + w); });
  };
  uint32_t T;
  int b = skip(0, T);
  if (b >= nbins) return;
  fetch(b);
  // the load cursor: group lb, step lt of lT, this lane's list
  int lb = b;
  uint32_t lT = T, k = sl, n = s_n[b + ls], ln = 0;
  const uint32_t* lp = a.lists + s_off[b + ls];
  fetch(b + S);
  auto word = [&] {
    const uint32_t j = k < n ? __ldcs(lp + k) : kNone;
    k += G;
    if (++ln == lT) {  // the group's last step: on to the next
      lb = skip(lb + S, lT);
      ln = 0;
      k = sl;
      n = lb < nbins ? s_n[lb + ls] : 0u;
      lp = a.lists + (lb < nbins ? s_off[lb + ls] : 0u);
      fetch(lb + S);
    }
    return j;
  };
  uint32_t j0 = word(), j1 = word(), j2 = word();
  uint4 q0 = gather(pts, j0, P), q1 = gather(pts, j1, P);
  auto sep = [&](uint4 q, bool valid, float& w, float& dx, float& dy, float& dz) {
    dx = valid ? __int2float_rn((int)(q.x - P.x)) : 1.f;  // an idle lane holds q = P
    dy = __int2float_rn((int)(q.y - P.y));
    dz = __int2float_rn((int)(q.z - P.z));
    w = valid ? __uint_as_float(q.w) : 0.f;
  };
  float4 D = make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (use_prep<Step>()) {
    float w, dx, dy, dz;
    sep(q0, j0 != kNone, w, dx, dy, dz);
    D = step.unit(w, dx, dy, dz);
  }
  while (b < nbins) {
    float2 acc[NCP / 2];
#pragma unroll
    for (int i = 0; i < NCP / 2; ++i) acc[i] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (uint32_t t = 0; t < T; ++t) {
      float w, dx, dy, dz;
      if constexpr (use_prep<Step>()) {
        sep(q1, j1 != kNone, w, dx, dy, dz);
        const float4 Dn = step.unit(w, dx, dy, dz);
        q1 = gather(pts, j2, P);
        j1 = j2;
        j2 = word();
        step.accum(acc, D);
        D = Dn;
      } else {
        sep(q0, j0 != kNone, w, dx, dy, dz);
        q0 = q1;
        j0 = j1;
        q1 = gather(pts, j2, P);
        j1 = j2;
        j2 = word();
        step(acc, w, dx, dy, dz);
      }
    }
    flush<Step, S>(acc, rows + (int64_t)b * a.row, a.row, nbins - b, ctab, sbuf, lane);
    b = skip(b + S, T);
  }
}

template <class Step, int S>
__device__ __forceinline__ void run_primary(const AlmArgs& a, const Step& step, const uint32_t* s_off,
                                            const uint32_t* s_n, const uint4 P, float* __restrict__ rows,
                                            const float2* ctab, float* sbuf, int lane) {
  if constexpr (S == 0) {
    const uint32_t total = s_off[a.nbins - 1] + s_n[a.nbins - 1] - s_off[0];
    switch (lists_per_warp(total, a.limits)) {
      case 1:
        return run_primary1(a, step, s_off, s_n, P, rows, ctab, sbuf, lane);
      case 2:
        return run_groups<Step, 2>(a, step, s_off, s_n, P, rows, ctab, sbuf, lane);
      default:
        return run_groups<Step, 4>(a, step, s_off, s_n, P, rows, ctab, sbuf, lane);
    }
  } else if constexpr (S == 1) {
    run_primary1(a, step, s_off, s_n, P, rows, ctab, sbuf, lane);
  } else {
    run_groups<Step, S>(a, step, s_off, s_n, P, rows, ctab, sbuf, lane);
  }
}

// number of m-passes of kernel L, and the columns and row offset of pass P
__host__ __device__ constexpr int pass_count(int L) {
  int n = 0;
  for (int m0 = 0; m0 <= L; m0 = pass_end(L, m0, pass_cap(L, m0)) + 1) ++n;
  return n;
}
__host__ __device__ constexpr int pass_m0(int L, int P) {
  int m0 = 0;
  for (int p = 0; p < P; ++p) m0 = pass_end(L, m0, pass_cap(L, m0)) + 1;
  return m0;
}
__host__ __device__ constexpr int pass_m1(int L, int P) { return pass_end(L, pass_m0(L, P), pass_cap(L, pass_m0(L, P))); }
__host__ __device__ constexpr int pass_ncp(int L, int P) { return round32(coef_count(L, pass_m0(L, P), pass_m1(L, P))); }
__host__ __device__ constexpr int pass_base(int L, int P) {
  int b = 0;
  for (int p = 0; p < P; ++p) b += pass_ncp(L, p);
  return b;
}
// bytes of one pass's conversion table ([E][U] coefficient pairs, then [E][U]
// source units), and of the passes before P
__host__ __device__ constexpr size_t conv_bytes(int L, int P) {
  return (size_t)conv_table_bytes(pass_ncp(L, P), conv_entries(L, pass_m0(L, P)));
}
__host__ __device__ constexpr size_t conv_pass_offset(int L, int P) {
  size_t b = 0;
  for (int p = 0; p < P; ++p) b += conv_bytes(L, p);
  return b;
}

// resident blocks of 4 warps the register budget of a pass is sized for
// (each of the SM's four schedulers holds a quarter of the registers: 2
// warps per scheduler allow 255 registers a thread, 3 allow 168, 4 allow 128)
__host__ __device__ constexpr int alm_min_blocks(int ncp) { return ncp <= 32 ? 5 : (ncp <= 64 ? 4 : (ncp <= 136 ? 3 : 2)); }

// per warp: the flush's transpose buffer and the slot totals of S lists (four
// for S = 0), then the primary's list offsets and counts
__host__ __device__ constexpr int alm_flush_floats(int ncp, int S) { return flush_buf_floats(ncp) + (S ? S : 4) * ncp; }
__host__ __device__ constexpr size_t alm_smem_per_warp(int ncp, int S) {
  return (size_t)alm_flush_floats(ncp, S) * sizeof(float) + 2 * kNbinsCap * sizeof(uint32_t);
}

// Counts and offsets of primary i into shared memory (empty lists at the end
// of its range past nbins, so that every group of S bins is whole); with
// `zero`, the rows of its empty bins are cleared (the slots of every pass).
__device__ __forceinline__ void load_lists(const AlmArgs& a, uint64_t ib, uint32_t* s_off, uint32_t* s_n, bool zero,
                                           int lane) {
  for (int b = lane; b < kNbinsCap; b += 32) {
    const bool in = b < a.nbins;
    const uint32_t n = in ? __ldg(a.counts + ib + b) : 0u;
    s_n[b] = n;
    s_off[b] = in ? __ldg(a.offsets + ib + b) : __ldg(a.offsets + ib + a.nbins - 1) + __ldg(a.counts + ib + a.nbins - 1);
    if (zero && in && n == 0) {
      float4* o = reinterpret_cast<float4*>(a.M + (ib + b) * (uint64_t)a.row);
      for (int k = 0; k < a.row / 4; ++k) o[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __syncwarp();
}

// One warp per primary: its (primary, bin) lists are consecutive runs of the
// lists buffer; S of them at a time are accumulated in registers for m-pass P
// of kernel L and flushed once, with the next lists' first loads already in
// flight.  S: lists_per_warp of every primary (1 or 4), or 0 for 2 and where
// they differ: the three forms in one kernel, each primary with its own.  Its code
// is scheduled less well in the longest loops (chosen primaries of 10^6 points
// at l_max 10, all with S = 1: 3.55 ms against 3.50; 3.1M pixels on the
// sphere, all 4: 94.7 against 94.1), and gains where S = 2 is the most
// frequent (250k primaries of 4M, l_max 20: 157.2 against 158.8).
//
// The passes of a kernel with several (l_max > 10) are separate kernels,
// launched one after another.  With all passes in one launch, warps in
// different passes overflowed the instruction cache; as separate kernels
// every warp on the GPU runs the same pass body, and each pass gets its own
// register budget (a pass with fewer accumulators runs more warps per SM).
// The lists are re-read once per pass; the points stay in L2.
template <int L, int P, int S>
__global__ void __launch_bounds__(128, alm_min_blocks(pass_ncp(L, P))) k_alm(const __grid_constant__ AlmArgs a) {
  constexpr int M0 = pass_m0(L, P), M1 = pass_m1(L, P), NCP = pass_ncp(L, P), BASE = pass_base(L, P);
  constexpr int TB = (int)conv_bytes(L, P);
  extern __shared__ __align__(16) char s_alm[];
  // [the pass's conversion table | per warp: flush buffers, list offsets, counts]
  for (int k = threadIdx.x; k < TB / 4; k += blockDim.x)
    reinterpret_cast<uint32_t*>(s_alm)[k] = __ldg(reinterpret_cast<const uint32_t*>(a.conv + conv_pass_offset(L, P)) + k);
  __syncthreads();
  const float2* ctab = reinterpret_cast<const float2*>(s_alm);
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  char* wbase = s_alm + TB + (size_t)warp * alm_smem_per_warp(NCP, S);
  float* sbuf = reinterpret_cast<float*>(wbase);
  uint32_t* s_off = reinterpret_cast<uint32_t*>(wbase + (size_t)alm_flush_floats(NCP, S) * sizeof(float));
  uint32_t* s_n = s_off + kNbinsCap;
  while (true) {
    unsigned long long i = 0;
    if (lane == 0) i = atomicAdd(a.work, 1ull);
    i = __shfl_sync(0xffffffffu, i, 0);
    if (i >= (unsigned long long)a.prim_count) break;
    const uint64_t ib = i * (uint64_t)a.nbins;
    load_lists(a, ib, s_off, s_n, P == 0, lane);
    const int64_t gi = a.prim_begin + (int64_t)i;
    const uint32_t sp = a.prim ? __ldg(a.prim + gi) : (uint32_t)gi;
    const uint4 Pt = __ldg(a.pts + sp);
    run_primary<Step3D<L, M0, M1>, S>(a, Step3D<L, M0, M1>{}, s_off, s_n, Pt, a.M + ib * (uint64_t)a.row + BASE, ctab,
                                      sbuf, lane);
    __syncwarp();  // s_n / s_off are rewritten for the next primary
  }
}

template <int L, int P, int S>
constexpr size_t alm_smem(int wpb) {
  return conv_bytes(L, P) + (size_t)wpb * alm_smem_per_warp(pass_ncp(L, P), S);
}

template <int L, int P, int S>
int alm_occupancy_pass(int wpb) {
  return resident_blocks((const void*)k_alm<L, P, S>, wpb * 32, alm_smem<L, P, S>(wpb));
}

// passes P.. of kernel L: each launch resident-sized from its own occupancy
// and with a work counter of its own (a.work, the next pass's after it)
template <int L, int P, int S>
cudaError_t launch_passes(const AlmArgs& a, int wpb, int nsm, cudaStream_t st) {
  if constexpr (P >= pass_count(L)) {
    return cudaSuccess;
  } else {
    const int bps = alm_occupancy_pass<L, P, S>(wpb);
    if (bps < 1) return cudaErrorInvalidConfiguration;
    cudaError_t e = allow_smem((const void*)k_alm<L, P, S>, alm_smem<L, P, S>(wpb));
    if (e != cudaSuccess) return e;
    k_alm<L, P, S><<<bps * nsm, wpb * 32, alm_smem<L, P, S>(wpb), st>>>(a);
    ++g_launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    AlmArgs next = a;
    ++next.work;
    return launch_passes<L, P + 1, S>(next, wpb, nsm, st);
  }
}

template <int L>
cudaError_t launch_alm_L(const AlmArgs& a, int lists, int wpb, int nsm, cudaStream_t st) {
  switch (lists) {
    case 1:
      return launch_passes<L, 0, 1>(a, wpb, nsm, st);
    case 4:
      return launch_passes<L, 0, 4>(a, wpb, nsm, st);
  }
  return launch_passes<L, 0, 0>(a, wpb, nsm, st);
}

// the smallest occupancy over the passes (0: some pass cannot be resident)
template <int L, int P>
int alm_occupancy_from(int wpb) {
  if constexpr (P >= pass_count(L)) {
    return 1 << 30;
  } else {
    const int o = alm_occupancy_pass<L, P, 1>(wpb);
    const int r = alm_occupancy_from<L, P + 1>(wpb);
    return o < r ? o : r;
  }
}

template <int L>
int alm_occupancy_L(int wpb) {
  return alm_occupancy_from<L, 0>(wpb);
}

}  // namespace ctb
