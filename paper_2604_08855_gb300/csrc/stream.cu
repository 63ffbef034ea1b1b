// stream.cu -- neighbour enumeration on the uniform cell grid.
//
// Paper, "Implementation": for each pivot, find all neighbours by scanning the
// spatial index over the search range.  Here one warp owns one primary and
// walks the x-rows of grid cells that intersect its ball r < r_max: each row
// is one contiguous run of cell-sorted points, read with coalesced 16-byte
// loads, 32 candidates per step.  Rows are split finer along x than across
// (kXSub), so a row's range ends close to the ball; in sphere mode a row is
// also cut to the shell that holds the points.  Every candidate gets its exact radial bin:
// float32 r from the fixed-point separation, and, for the rare candidates
// within float rounding of an edge, the exact integer r^2 against exact
// thresholds.
//
// Two passes per chunk of primaries:
//   count: pairs per (primary, bin)  -> counts (then an exclusive scan on the
//          host stream gives each (primary, bin) list its start); the bin of
//          every candidate is also stored as one byte (kNoBin: not a pair)
//   fill:  walks the same candidate stream, from the segments and bin codes
//          that the count pass stored (no cell rows, points or distances), and
//          writes each pair's neighbour index into its (primary, bin) list
//          (match_any ranks the lanes that share a bin)
//
// The candidate stream.  A row's point ranges (segments) are short where the
// catalogue is sparse or the points lie on a surface: 0.4 points a row in a
// 20k-point box, 15 on a half-degree sphere map.  So segments are collected
// from the row blocks into a list in shared memory (a batch), and the batch is
// walked as one stream, 32 candidates a step, whatever segments they come
// from.  A lane finds its segment from the boundaries that fall into the
// step's window: the 32 lanes hold the next 32 boundaries, one warp
// OR-reduction makes them a bit mask, and the bits at or below the lane count
// the segments passed.  Steps inside one segment skip the search.  Walking
// segment by segment spent a step on every segment however short, and about
// 25 instructions more.
//
// Codes.  Four steps share one 32-bit word per lane (byte k: step k of the
// group of 128 candidates), so the count pass stores every fourth step, and a
// step of the fill pass ranks 32 consecutive candidates.  match_any takes 8
// cycles per distinct value (measured), which bounds the fill: 32 neighbours
// along a row lie in few bins, 32 taken four apart in twice as many.
//
// An idle lane of the count pass looks at the primary itself (r = 0, never a
// pair), and the codes past the stream's end read kNoBin, so neither pass
// tests positions.
//
// A batch in the code buffer: a 16-byte head (segments, candidates), its
// segments (point offset, end position: 8 bytes each, padded to 16), its
// codes.
#include <algorithm>

#include "ctb_internal.cuh"

namespace ctb {

__device__ __forceinline__ float slab_dist(int d, float fr) {
  return d > 0 ? (float)d - fr : (d < 0 ? (float)(-d - 1) + fr : 0.f);
}

// a in [-n, 2 n) wrapped into [0, n): a row window reaches at most half a
// period to either side of its primary's cell
__device__ __forceinline__ int wrap1(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// sqrt to 2^-22: a row's ends carry a slack of 1e-3 cells (g.rcell, and the
// shell's padding)
__device__ __forceinline__ float sqrt_fast(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ float rsqrt_fast(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

constexpr uint8_t kNoBin = 0xff;  // bin code of a candidate that is not a pair
constexpr unsigned long long kNoBatch = ~0ull;  // ends a primary's batches

// Geometry of one primary's row window (count pass).
struct RowWin {
  int W, off0, nrows;
  uint32_t invW;  // ceil(2^32 / W): t / W = umulhi(t, invW) for t < 2^32 / W
  bool fullwin;
  float R2, fx, fry, frz;  // (r_max in cell units)^2; primary's x in x-cell units, y and z fractions
  float xs;                // x-cells per cell (ncx / nc)
  int cxp, cyp, czp;
  uint32_t cbase;
};

// The point ranges of row t of the window (up to two: periodic wrap in x,
// or the two crossings of the sphere's shell); empty ranges have s >= e.
// SHELL (sphere mode): every point lies in the shell of g.shell_r2lo ..
// g.shell_r2hi around the origin, so a row that misses it is skipped without
// a load, and a row that crosses it is cut to its crossings.
template <bool SHELL>
__device__ __forceinline__ void row_ranges(const StreamArgs& a, const Geom& g, const RowWin& rw, int t, uint32_t& s0,
                                           uint32_t& e0, uint32_t& s1, uint32_t& e1) {
  const uint32_t nc = g.nc;
  s0 = e0 = s1 = e1 = 0;
  if (t >= rw.nrows) return;
  const int tz = rw.W == 1 ? t : (int)__umulhi((uint32_t)t, rw.invW);
  const int dy = t - tz * rw.W + rw.off0, dz = tz + rw.off0;
  float gy = slab_dist(dy, rw.fry), gz = slab_dist(dz, rw.frz);
  if (rw.fullwin) {
    gy = fminf(gy, fminf(slab_dist(dy - (int)nc, rw.fry), slab_dist(dy + (int)nc, rw.fry)));
    gz = fminf(gz, fminf(slab_dist(dz - (int)nc, rw.frz), slab_dist(dz + (int)nc, rw.frz)));
  }
  const float rho2 = __fmaf_rn(gy, gy, __fmul_rn(gz, gz));
  int cy = rw.cyp + dy, cz = rw.czp + dz;
  bool ok = rho2 < rw.R2;
  if (g.periodic) {
    cy = wrap1(cy, (int)nc);
    cz = wrap1(cz, (int)nc);
  } else {
    ok = ok && cy >= 0 && cy < (int)nc && cz >= 0 && cz < (int)nc;
  }
  if (!ok) return;
  // the row's x-range in x-cells (a row is split xs times finer along x
  // than across, so its ends overshoot the ball by less)
  const float hw = __fmul_rn(sqrt_fast(__fsub_rn(rw.R2, rho2)), rw.xs);
  const int nx = (int)g.ncx;
  int lo = (int)floorf(__fsub_rn(rw.fx, hw)), hi = (int)floorf(__fadd_rn(rw.fx, hw));
  const uint32_t rb = rw.cbase + ((uint32_t)cz * nc + (uint32_t)cy) * (uint32_t)nx;
  int a0 = 1, b0 = 0, a1 = 1, b1 = 0;
  if constexpr (SHELL) {
    // distance range from the shell's axis to the row's (y, z) cross-section
    const float ly = (float)cy - g.shell_c[1], lz = (float)cz - g.shell_c[2];
    const float ny = ly > 0.f ? ly : (ly + 1.f < 0.f ? -(ly + 1.f) : 0.f);
    const float nz = lz > 0.f ? lz : (lz + 1.f < 0.f ? -(lz + 1.f) : 0.f);
    const float fy = fmaxf(fabsf(ly), fabsf(ly + 1.f)), fz = fmaxf(fabsf(lz), fabsf(lz + 1.f));
    const float d2min = __fmaf_rn(ny, ny, __fmul_rn(nz, nz)), d2max = __fmaf_rn(fy, fy, __fmul_rn(fz, fz));
    if (d2min >= g.shell_r2hi) return;
    // x offsets (x-cells) of the shell along the row: [alo, ahi] either side of the centre
    const float ahi = __fmul_rn(sqrt_fast(__fsub_rn(g.shell_r2hi, d2min)), rw.xs);
    const float alo = g.shell_r2lo > d2max ? __fmul_rn(sqrt_fast(__fsub_rn(g.shell_r2lo, d2max)), rw.xs) : 0.f;
    const float xl = __fsub_rn(rw.fx, hw), xh = __fadd_rn(rw.fx, hw), cx = g.shell_c[0];
    // the ball's x-range meets the upper crossing [cx + alo, cx + ahi] and the lower one
    const float pl = fmaxf(xl, __fadd_rn(cx, alo)), ph = fminf(xh, __fadd_rn(cx, ahi));
    const float ml = fmaxf(xl, __fsub_rn(cx, ahi)), mh = fminf(xh, __fsub_rn(cx, alo));
    int ma = nx, mb = -1, pa = nx, pb = -1;
    if (ml <= mh) {
      ma = max((int)floorf(ml), 0);
      mb = min((int)floorf(mh), nx - 1);
    }
    if (pl <= ph) {
      pa = max((int)floorf(pl), 0);
      pb = min((int)floorf(ph), nx - 1);
    }
    if (ma <= mb && pa <= pb && pa <= mb + 1) {  // touching or overlapping: one range
      a0 = ma;
      b0 = max(mb, pb);
    } else if (ma <= mb) {
      a0 = ma;
      b0 = mb;
      a1 = pa;
      b1 = pb;
    } else {
      a0 = pa;
      b0 = pb;
    }
  } else if (g.periodic) {
    if (hi - lo + 1 >= nx) {
      a0 = 0;
      b0 = nx - 1;
    } else {
      const int lm = wrap1(lo, nx), hm = wrap1(hi, nx);
      a0 = lm;
      if (lm <= hm) {
        b0 = hm;
      } else {
        b0 = nx - 1;
        a1 = 0;
        b1 = hm;
      }
    }
  } else {
    a0 = max(lo, 0);
    b0 = min(hi, nx - 1);
  }
  if (a0 <= b0) {
    s0 = __ldg(a.cell_start + rb + a0);
    e0 = __ldg(a.cell_start + rb + b0 + 1);
  }
  if (a1 <= b1) {
    s1 = __ldg(a.cell_start + rb + a1);
    e1 = __ldg(a.cell_start + rb + b1 + 1);
  }
}

// A batch of segments in shared memory: a row block adds at most 64, and the
// batch is walked once it holds more than kSegCap - 64.
constexpr int kSegCap = 96;

struct WarpSegs {
  uint2 seg[kSegCap + 1];       // point index = seg.x + stream position, below seg.y
  uint32_t incl[kSegCap + 32];  // stream position of the segment's end
};

__device__ __forceinline__ uint32_t batch_head(uint32_t nseg) { return (16u + 8u * nseg + 15u) & ~15u; }

// Segment of this lane's position in the step at k0; f: the segments that end
// before the step, moved past those that end in it.
__device__ __forceinline__ uint32_t find_segment(const WarpSegs& sg, uint32_t k0, uint32_t& f, int lane, unsigned le) {
  const uint32_t d = sg.incl[f + lane] - k0;
  const unsigned ends = __reduce_or_sync(0xffffffffu, d < 32u ? 1u << d : 0u);
  const uint32_t t = f + __popc(ends & le);
  f += __popc(ends);
  return t;
}

// Count pass.  GEN: sphere mode -- bin edges not linear in r (the angle bins)
// and rows cut to the points' shell.  LONG: four steps of a row at a time
// (plan_pairs says when).
//
// Bound by instruction issue (about 60 instructions per 32 candidates; 71 %
// of the issue slots) and, in the fill, by match_any.  Enumeration with the
// walk segment by segment / with this one: 10^6 points 168 / 133 ms, cut sky
// of 800k 121 / 98.7, 3.1M-pixel sphere 90 / 60.5, 24 mock catalogues 35.8 /
// 22.9, 20k uniform points 0.384 / 0.139.  With the fill finding the rows
// again, as the count does, the second numbers rose by 0, -2, 6.4, 2.6 and
// 0.043.  Four blocks of 8 warps per SM (64 registers): five spill in the
// count (sphere 67 ms) and cost the fill its look-ahead (cut sky 106 ms).
template <bool GEN, bool LONG>
__global__ void __launch_bounds__(kStreamThreads, 4) k_count(StreamArgs a) {
  extern __shared__ uint32_t s_cnt_all[];
  __shared__ uint32_t s_classes;  // lists_per_warp of this block's primaries, OR-ed
  __shared__ WarpSegs s_segs[kStreamThreads / 32];
  if (threadIdx.x == 0) s_classes = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const Geom g = a.g;
  const int nbins = g.nbins;
  uint32_t* cnt = s_cnt_all + warp * nbins;  // pairs of each bin
  WarpSegs& sg = s_segs[warp];
  const unsigned lt = (1u << lane) - 1u, le = lt | (1u << lane);
  const uint32_t nc = g.nc;
  RowWin rw;
  rw.R2 = __fmul_rn(g.rcell, g.rcell);
  rw.xs = (float)(g.ncx / nc);
  {
    const RowWindow win = row_window(g);
    rw.W = win.W;
    rw.off0 = win.off0;
    rw.fullwin = win.fullwin;
    rw.invW = 0xffffffffu / (uint32_t)win.W + 1u;
  }
  rw.nrows = rw.W * rw.W;
  const int nrb = (rw.nrows + 31) / 32;
  const uint64_t lowmask = (1ull << g.shift) - 1ull;
  const float frac_scale = 1.0f / (float)(1ull << g.shift);
  unsigned long long my_pairs = 0;
  // the constants of a step, passed through a shuffle so that they
  // stay in registers (the compiler otherwise loads each from the parameter
  // bank in every step)
  auto pin = [](float v) { return __shfl_sync(0xffffffffu, v, 0); };
  const float rlo2 = pin(g.rlo2_u), rhi2 = pin(g.rhi2_u);
  const float inv_dr = pin(g.inv_dr_u), shift = pin(g.bin_shift);
  const float half_bin = pin(g.half_bin);
  // this warp's pool in the code buffer (batches take consecutive
  // ranges of it; a new pool is taken when one does not fit)
  unsigned long long pool = 0, pool_end = 0;

  while (true) {
    unsigned long long i = 0;
    if (lane == 0) i = atomicAdd(a.work, 1ull);
    i = __shfl_sync(0xffffffffu, i, 0);
    if (i >= (unsigned long long)a.prim_count) break;
    const int64_t gi = a.prim_begin + (int64_t)i;
    const uint32_t sp = a.prim ? __ldg(a.prim + gi) : (uint32_t)gi;
    const uint4 P = __ldg(a.pts + sp);
    // batch: the primary's catalogue owns cells [cat * ncells, (cat + 1) * ncells)
    rw.cbase = a.keys ? (__ldg(a.keys + sp) / g.ncells) * g.ncells : 0u;
    if (lane == 0) a.wprim[i] = a.wsub ? __ldg(a.wsub + gi) : __uint_as_float(P.w);
    const uint64_t ib = i * (uint64_t)nbins;
    for (int b = lane; b < nbins; b += 32) cnt[b] = 0u;
    __syncwarp();

    const uint64_t sx = (uint64_t)P.x * g.ncx, sy = (uint64_t)P.y * nc, sz = (uint64_t)P.z * nc;
    rw.cxp = (int)(sx >> g.shift);
    rw.cyp = (int)(sy >> g.shift);
    rw.czp = (int)(sz >> g.shift);
    rw.fry = __fmul_rn((float)(sy & lowmask), frac_scale);
    rw.frz = __fmul_rn((float)(sz & lowmask), frac_scale);
    rw.fx = __fadd_rn((float)rw.cxp, __fmul_rn((float)(sx & lowmask), frac_scale));

    uint32_t nseg = 0, total = 0;  // the batch: its segments and candidates
    unsigned long long* cb = a.code_base + i * (uint64_t)nrb;  // start of each batch, ended by kNoBatch
    for (int t0 = 0; t0 < rw.nrows; t0 += 32) {
      // ---- add a row block's segments
      {
        uint32_t s0, e0, s1, e1;
        row_ranges<GEN>(a, g, rw, t0 + lane, s0, e0, s1, e1);
        const unsigned m0 = __ballot_sync(0xffffffffu, s0 < e0), m1 = __ballot_sync(0xffffffffu, s1 < e1);
        if (m0 | m1) {
          const uint32_t len0 = s0 < e0 ? e0 - s0 : 0u;
          const uint32_t len1 = s1 < e1 ? e1 - s1 : 0u;
          uint32_t incl = len0 + len1;  // inclusive prefix of the lengths over the lanes
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
          }
          const uint32_t end1 = total + incl, end0 = end1 - len1, beg0 = end0 - len0;
          uint32_t k = nseg + __popc(m0 & lt) + __popc(m1 & lt);
          if (s0 < e0) {
            sg.seg[k] = make_uint2(s0 - beg0, e0);
            sg.incl[k] = end0;
            ++k;
          }
          if (s1 < e1) {
            sg.seg[k] = make_uint2(s1 - end0, e1);
            sg.incl[k] = end1;
          }
          nseg += __popc(m0) + __popc(m1);
          total += __shfl_sync(0xffffffffu, incl, 31);
        }
      }
      if (nseg <= (uint32_t)kSegCap - 64u && t0 + 32 < rw.nrows) continue;
      if (nseg == 0) continue;
      // ---- walk the batch
      sg.incl[nseg + lane] = 0xffffffffu;
      if (lane == 0) sg.seg[nseg] = make_uint2(0u, 0u);  // a step's positions past the end
      __syncwarp();
      const uint32_t ngroups = (total + 127u) >> 7;
      {
        const uint32_t head = batch_head(nseg);
        const unsigned long long span = head + 128ull * ngroups;
        if (pool + span > pool_end) {
          const unsigned long long take = span > a.code_pool ? span : a.code_pool;
          if (lane == 0) pool = atomicAdd(a.code_total, take);
          pool = __shfl_sync(0xffffffffu, pool, 0);
          pool_end = pool + take;
        }
        if (lane == 0) *cb = pool;
        // past the buffer: counts stay exact, the codes go to the buffer's
        // start, and the host grows the buffer and counts the chunk again
        const bool codes_ok = pool + span <= a.code_cap;
        if (codes_ok) {
          uint2* hp = reinterpret_cast<uint2*>(a.codes + pool);
          if (lane == 0) *hp = make_uint2(nseg, total);
          for (uint32_t k = lane; k < nseg; k += 32) hp[2 + k] = make_uint2(sg.seg[k].x, sg.incl[k]);
        }
        uint32_t* cp = reinterpret_cast<uint32_t*>(a.codes + (codes_ok ? pool + head : 0ull)) + lane;
        const uint32_t cstep = codes_ok ? 32u : 0u;
        pool += span;
        uint32_t word = 0;  // the codes of the group's steps so far
        auto store = [&] {
          __stcs(cp, word);
          cp += cstep;
        };
        // One candidate per lane: is it in range (inb), its bin b, and whether
        // it lies within float rounding of an edge.
        auto classify = [&](const uint4 q, bool& inb, uint32_t& b) -> bool {
          const float dx = __int2float_rn((int)(q.x - P.x)), dy = __int2float_rn((int)(q.y - P.y)),
                      dz = __int2float_rn((int)(q.z - P.z));
          const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          // rlo2_u > 0 also excludes r = 0 (coincident points)
          inb = r2 >= rlo2 && r2 < rhi2;
          const float r = r2 * rsqrt_fast(r2);
          // th: the bin coordinate minus 1/2.  Rounded to the nearest integer
          // (by adding 1.5 * 2^23) it is the bin, and what is left over is
          // the distance from the bin's middle, within `half` of it unless
          // the pair may lie on an edge.  rlo2 and rhi2 are so close to the
          // first and last edge that a pair past them is within that margin
          // too: b needs no range test (10^6 points: 144 ms with one).
          float th, half;
          if constexpr (GEN) {
            // sphere: the bin of theta = 2 asin(chord / 2).  Its float
            // error stays below 1e-6 theta while chord / 2 <= 0.99 (asin
            // is ill-conditioned towards 1); the guard is ten times that,
            // and larger chords always take the exact test.  Up to
            // chord / 2 = 1/8 (theta 14 degrees) the Maclaurin series of
            // asin to x^7 serves: truncation below 2e-9 theta, float
            // evaluation below 4e-7 theta.
            const float x = r * g.half_unit;
            const float x2 = x * x;
            float ang = 2.f * x * fmaf(x2, fmaf(x2, fmaf(x2, 5.f / 112.f, 3.f / 40.f), 1.f / 6.f), 1.f);
            if (__any_sync(0xffffffffu, inb && x > 0.125f)) ang = x > 0.125f ? 2.f * asinf(fminf(x, 1.f)) : ang;
            th = fmaf(ang, inv_dr, shift);
            half = x > 0.99f ? -1.f : fminf(half_bin, fmaf(ang, -1e-5f * inv_dr, 0.5f - 1e-7f * inv_dr));
          } else {
            th = fmaf(r, inv_dr, shift);
            half = half_bin;
          }
          const float tm = th + 12582912.f;
          b = __float_as_uint(tm) - 0x4b400000u;
          return inb & (fabsf(th - (tm - 12582912.f)) > half);
        };
        // Two candidates of a lane in paired FP32 instructions, the same
        // operations as above in half the issue slots: count and fill of 10^6
        // points in 132.8 ms against 134.9.
        auto classify2 = [&](const uint4 qa, const uint4 qb, bool* in, uint32_t* bin, bool* edge) {
          auto sep = [](uint32_t p, uint32_t u, uint32_t v) {
            return make_float2(__int2float_rn((int)(u - p)), __int2float_rn((int)(v - p)));
          };
          auto both = [](float v) { return make_float2(v, v); };
          const float2 dx = sep(P.x, qa.x, qb.x), dy = sep(P.y, qa.y, qb.y), dz = sep(P.z, qa.z, qb.z);
          const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
          const float2 r = __fmul2_rn(r2, make_float2(rsqrt_fast(r2.x), rsqrt_fast(r2.y)));
          const float2 th = __ffma2_rn(r, both(inv_dr), both(shift));
          const float2 tm = __fadd2_rn(th, both(12582912.f));
          const float2 d = __ffma2_rn(__fadd2_rn(tm, both(-12582912.f)), both(-1.f), th);
          in[0] = r2.x >= rlo2 && r2.x < rhi2;
          in[1] = r2.y >= rlo2 && r2.y < rhi2;
          bin[0] = __float_as_uint(tm.x) - 0x4b400000u;
          bin[1] = __float_as_uint(tm.y) - 0x4b400000u;
          edge[0] = in[0] & (fabsf(d.x) > half_bin);
          edge[1] = in[1] & (fabsf(d.y) > half_bin);
        };
        // on an edge: exact integer r^2 against exact thresholds
        auto exact = [&](const uint4 q, bool& inb, uint32_t& b) {
          const long long ix = (int)(q.x - P.x), iy = (int)(q.y - P.y), iz = (int)(q.z - P.z);
          const unsigned long long e2 = (unsigned long long)(ix * ix + iy * iy + iz * iz);
          if (e2 == 0ull || e2 < __ldg(a.thr) || e2 >= __ldg(a.thr + nbins)) {
            inb = false;
          } else {
            int c = min(max((int)b, 0), nbins - 1);
            while (e2 < __ldg(a.thr + c)) --c;
            while (e2 >= __ldg(a.thr + c + 1)) ++c;
            b = (uint32_t)c;
          }
        };
        // its code into the word, its bin's count
        auto emit = [&](bool inb, uint32_t b) {
          word = __funnelshift_r(word, inb ? b : (uint32_t)kNoBin, 8);
          if (inb) atomicAdd(cnt + b, 1u);
        };
        auto one = [&](const uint4 q) {
          bool inb;
          uint32_t b;
          const bool edge = classify(q, inb, b);
          if (__any_sync(0xffffffffu, edge)) {
            if (edge) exact(q, inb, b);
          }
          emit(inb, b);
        };
        uint32_t f = 0, k0 = 0;
        while (k0 < total) {
          // steps inside one segment: consecutive points (LONG: four steps at a time)
          {
            const uint2 sgm = sg.seg[f];
            const uint32_t uend = sgm.y - sgm.x;
            const uint4* qp = a.pts + (sgm.x + k0 + (uint32_t)lane);
            if constexpr (LONG) {
              const uint32_t last = 3u - ((k0 >> 5) & 3u);  // the step of the four that ends a word
              for (; k0 + 128u <= uend; k0 += 128u, qp += 128) {
                uint4 q[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) q[u] = __ldg(qp + 32 * u);
                bool inb[4], edge[4];
                uint32_t b[4];
#pragma unroll
                for (int u = 0; u < 4; u += 2) classify2(q[u], q[u + 1], inb + u, b + u, edge + u);
                if (__any_sync(0xffffffffu, edge[0] | edge[1] | edge[2] | edge[3])) {
#pragma unroll
                  for (int u = 0; u < 4; ++u)
                    if (edge[u]) exact(q[u], inb[u], b[u]);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  emit(inb[u], b[u]);
                  if (last == (uint32_t)u) __stcs(cp, word);
                }
                cp += cstep;
              }
            }
            for (; k0 + 32u <= uend; qp += 32) {
              one(__ldg(qp));
              k0 += 32u;
              if ((k0 & 127u) == 0u) store();
            }
          }
          if (k0 >= total) break;
          // a step with a boundary
          const uint2 sgm = sg.seg[find_segment(sg, k0, f, lane, le)];
          const uint32_t j = sgm.x + k0 + (uint32_t)lane;
          one(__ldg(a.pts + (j < sgm.y ? j : sp)));
          k0 += 32u;
          if ((k0 & 127u) == 0u) store();
        }
        if (k0 & 127u) {  // the last group: no codes in the steps it lacks
          for (; k0 & 127u; k0 += 32u) word = __funnelshift_r(word, (uint32_t)kNoBin, 8);
          store();
        }
      }
      ++cb;
      nseg = 0;
      total = 0;
      __syncwarp();  // the batch's list is rewritten
    }
    if (lane == 0 && cb < a.code_base + (i + 1) * (uint64_t)nrb) *cb = kNoBatch;
    __syncwarp();
    uint32_t mine = 0;
    for (int b = lane; b < nbins; b += 32) {
      const uint32_t s = cnt[b];
      a.counts[ib + b] = s;
      mine += s;
    }
    my_pairs += mine;
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0 && mine) atomicOr(&s_classes, (uint32_t)lists_per_warp(mine, a.limits));
    __syncwarp();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_pairs += __shfl_xor_sync(0xffffffffu, my_pairs, o);
  if (lane == 0 && my_pairs) atomicAdd(a.total, my_pairs);
  __syncthreads();
  if (threadIdx.x == 0 && s_classes) atomicOr(a.classes, (unsigned long long)s_classes);
}

// Fill pass.
__global__ void __launch_bounds__(kStreamThreads, 4) k_fill(StreamArgs a) {
  extern __shared__ uint32_t s_cnt_all[];
  __shared__ WarpSegs s_segs[kStreamThreads / 32];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int nbins = a.g.nbins;
  uint32_t* cnt = s_cnt_all + warp * nbins;  // next list entry of each bin
  WarpSegs& sg = s_segs[warp];
  const unsigned lt = (1u << lane) - 1u, le = lt | (1u << lane);
  const int nrb = row_blocks(a.g);
  while (true) {
    unsigned long long i = 0;
    if (lane == 0) i = atomicAdd(a.work, 1ull);
    i = __shfl_sync(0xffffffffu, i, 0);
    if (i >= (unsigned long long)a.prim_count) break;
    for (int b = lane; b < nbins; b += 32) cnt[b] = __ldg(a.offsets + i * (uint64_t)nbins + b);
    const unsigned long long* cb = a.code_base + i * (uint64_t)nrb;
    unsigned long long next = __ldg(cb);
    for (int ib = 0; ib < nrb; ++ib) {
      const unsigned long long pos = next;
      if (pos == kNoBatch) break;
      if (ib + 1 < nrb) next = __ldg(cb + ib + 1);
      const uint2* hp = reinterpret_cast<const uint2*>(a.codes + pos);
      const uint2 hd = __ldg(hp);
      const uint32_t nseg = hd.x, ngroups = (hd.y + 127u) >> 7;
      const uint32_t* wp = reinterpret_cast<const uint32_t*>(a.codes + pos + batch_head(nseg)) + lane;
      uint32_t word = __ldcs(wp);
      for (uint32_t k = lane; k < nseg; k += 32) {
        const uint2 v = __ldcs(hp + 2 + k);
        sg.seg[k].x = v.x;
        sg.incl[k] = v.y;
      }
      sg.incl[nseg + lane] = 0xffffffffu;
      if (lane == 0) sg.seg[nseg].x = 0u;
      __syncwarp();
      uint32_t f = 0;
      uint32_t sx = sg.seg[0].x, send = sg.incl[0];  // segment f: steps inside it need no search
      for (uint32_t q = 0; q < ngroups; ++q) {
        const uint32_t wnext = q + 1 < ngroups ? __ldcs(wp + 32u) : 0u;
        wp += 32;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t code = (word >> (8 * k)) & 0xffu;
          const unsigned act = __ballot_sync(0xffffffffu, code != kNoBin);
          const uint32_t k0 = 128u * q + 32u * (uint32_t)k;
          uint32_t j = k0 + (uint32_t)lane;
          if (k0 + 32u <= send) {
            j += sx;
          } else {
            j += sg.seg[find_segment(sg, k0, f, lane, le)].x;
            sx = sg.seg[f].x;
            send = f < nseg ? sg.incl[f] : 0u;
          }
          if (code != kNoBin) {
            const unsigned grp = __match_any_sync(act, code);
            const uint32_t c0 = cnt[code];
            const uint32_t rank = __popc(grp & lt);
            __syncwarp(act);
            __stcs(a.lists + (uint64_t)(c0 + rank), j);
            if (rank == 0) cnt[code] = c0 + __popc(grp);
          }
          __syncwarp();
        }
        word = wnext;
      }
    }
    __syncwarp();  // the cursors are rewritten
  }
}

// the bins' counts or cursors of each warp (at most 2 KB a block)
static size_t stream_smem(int nbins) { return (size_t)(kStreamThreads / 32) * nbins * sizeof(uint32_t); }

static const void* stream_fn(const Geom& g, bool fill) {
  if (fill) return (const void*)k_fill;
  if (g.general) return (const void*)k_count<true, false>;
  return g.long_rows ? (const void*)k_count<false, true> : (const void*)k_count<false, false>;
}

int stream_blocks_per_sm(const Geom& g, bool fill) {
  return resident_blocks(stream_fn(g, fill), kStreamThreads, stream_smem(g.nbins));
}

cudaError_t launch_stream(const StreamArgs& a, bool fill, int nblocks, cudaStream_t st) {
  StreamArgs sa = a;
  void* args[] = {&sa};
  const cudaError_t e = cudaLaunchKernel(stream_fn(a.g, fill), dim3(nblocks), dim3(kStreamThreads), args,
                                         stream_smem(a.g.nbins), st);
  if (e != cudaSuccess) return e;
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace ctb
