// contract.cu -- the zeta contraction on the CUDA cores (plain FP32 form) and
// the FP64 cross-block reduction + normalisation.
//
//   zeta~_l(b1,b2) = sum_p w_p sum_{m=-l..l} a_lm(p,b1) a_lm(p,b2)
//   zeta_l(b1,b2)  = 4 pi / (2l+1) zeta~_l(b1,b2)
// (the estimator the paper's "Implementation" section fills bin by bin; its
// normalisation is the triplet-sum one, so that zeta_0 = sum_p w_p N_p N_p).
#include "ctb_internal.cuh"

namespace ctb {

// Outer-product form.  A thread owns one coefficient slot c of the rows and a
// T x T tile of bin pairs (B1 <= B2), and walks the primaries of the block's
// slice: per primary it reads its slot of the tile's bins (2 T scalar shared
// loads, T on the diagonal) and adds w x y^T in T^2 / 2 paired FMAs.  A
// warp's lanes are 32 consecutive slots of one tile, so the loads are
// conflict-free on the rows as they lie in memory: nothing is transposed, any
// row length will do, and the staging is one asynchronous copy per element.
// The sum over m within a multipole is left to the end, where the slots of
// each l are added in a fixed order.
//
// What bounds it: the issue of paired FMAs and their operands at three warps
// a scheduler (20k rows of 20 bins x 128, l_max 10: 62 us, FMA pipe 42 %, issue
// 54 %, 0.49 of HBM).  The form before this one, 4 x 4 tiles by 16-byte loads
// of transposed rows, spent its time on shared-memory loads and, for the
// 121-float rows of a caller, on transposing them element by element (20k
// such rows, the whole call: 734 us; now 86).  Half tiles of 5 x 10 with twice
// the warps were slower (200k rows: 667 us against 546): more loads and
// address arithmetic per FMA.
//
// Block: CH slots x tiles x PG primary groups (group g takes the stage's
// primaries q = g mod PG).  Rows of more than CH slots are taken in chunks of
// CH, the block walking its slice once per chunk, and where the tiles do not
// fit a block they are split over blockIdx.y: a block reads each element of
// its slice once, so the rows come from HBM once up to 40 bins, twice from 41
// and three times from 61 (less what L2 still holds).
//
// Rounding.  A thread adds a run of primaries in FP32; at its end (flush) the
// slots of a multipole and the groups are added with their rounding errors
// carried along, and one owner thread adds each (l, b1 <= b2) entry to the
// block's FP64 partial row.  So an entry's error is that of the runs alone.
// l = 0 has one slot, nothing averages over it, and its run is the longest
// for its size: a block with one group takes its slice in two runs (the
// length that two blocks per SM would give it), and no run is longer than
// kConFlush.  Rows of eight chunks or more (32 bins from l_max 15) stay at
// one run: they flush once a chunk already, and a second of each took 72 us
// of 5.2 ms at 200k rows, l_max 20.  Float64 output at l = 0 against 64 bits,
// one run / two, relative rms: 20k rows of 20 bins at l_max 10 1.43e-8 /
// 7.0e-9, 100k rows 3.1e-8 / 1.5e-8, 20k of 16 bins 1.36e-8 / 7.0e-9; with
// several groups, plain sums / errors carried: 2000 rows of 10 bins 3.9e-9 /
// 2.2e-9.  The second flush costs 2 us at 20k rows of 20 bins.  (With
// one thread per entry and multipole, whose loads collide in the shared
// memory's banks and whose partial row is read, added to and written in turn,
// a flush took 8 us.)
//
// Copies (16 bytes each where the rows allow it): rows that fit one chunk are
// copied as they lie, one contiguous run per stage (kConLinear; kConLinearAny
// reads at the row's own stride where that is not CH, as for 121-float rows);
// chunks of longer rows are copied row by row (kConRows16, kConRows4).
constexpr int kConFlush = 1024;         // primaries of a group between two flushes
constexpr int kConMaxQ = 64;            // primaries per stage at most
constexpr int kConStageFloats = 11264;  // one staged buffer at most, when more than PG primaries fit it
constexpr int kConStages = 3;           // staged buffers: one in use, one in, one on its way
constexpr int kConMaxTiles = 24;        // tiles per block at most (768 threads / 32)
enum { kConRows4 = 0, kConRows16 = 1, kConLinear = 2, kConLinearAny = 3 };
constexpr size_t kConSmemCap = 220 * 1024;

struct ConShape {
  int T;        // tile side
  int nbt;      // tiles across the bins
  int tiles;    // tiles B1 <= B2 per block
  int ntiles;   // all of them (split over blockIdx.y)
  int ch;       // slots per chunk
  int nchunk;
  int pg;       // primary groups
  int threads;
  int stride;   // staged floats between bins: the row, or CH when the row is chunked
  int Q;        // primaries per stage
  int stage_floats;  // one staged buffer
  int smem_bytes;
};

// threads of a block by tile side: T^2 accumulators and 2 T operands a thread
// (T 6: 80 registers, T 8: 128, T 10: 168)
__host__ __device__ constexpr int con_max_threads(int T) { return T == 6 ? 768 : (T == 8 ? 512 : 384); }

// Work of one slot and primary in issue cycles of an SM sub-partition: paired
// FMAs at 2.65, or four shared loads' time per load where that is more (an SM
// serves one load of a warp per cycle, for four sub-partitions).
static double con_cost(int T, int nb) {
  const int nbt = (nb + T - 1) / T, off = nbt * (nbt - 1) / 2;
  const double fma = 2.65 * (nbt * (T / 2) * (T / 2 + 1) + off * T * T / 2);
  const double lds = 4.0 * (nbt * T + off * 2 * T);
  return fma > lds ? fma + 0.3 * lds : lds + 0.3 * fma;
}

static ConShape con_shape(int nbins, int row) {
  ConShape c{};
  // the tile side with the least work: 10 for 10 and 20 bins, 8 for 16 and
  // 32, 6 for 36 (the side that pads the bins least wins over a larger one)
  c.T = 6;
  for (int T = 8; T <= 10; T += 2)
    if (con_cost(T, nbins) < con_cost(c.T, nbins)) c.T = T;
  const int cap = con_max_threads(c.T);
  c.nbt = (nbins + c.T - 1) / c.T;
  c.ntiles = c.nbt * (c.nbt + 1) / 2;
  c.tiles = c.ntiles * 32 <= cap ? c.ntiles : cap / 32;
  const int rows32 = (row + 31) / 32 * 32;
  c.ch = 32;
  while (c.ch < 128 && 2 * c.ch * c.tiles <= cap && c.ch < rows32) c.ch *= 2;
  c.nchunk = (row + c.ch - 1) / c.ch;
  c.pg = cap / (c.ch * c.tiles);
  if (c.pg > 8) c.pg = 8;
  c.threads = c.ch * c.tiles * c.pg;
  c.stride = c.nchunk == 1 ? row : c.ch;
  // primaries per stage: a multiple of the groups, and of four so that every
  // contiguous run starts on 16 bytes when the base does
  const int unit = c.pg % 4 == 0 ? c.pg : (c.pg % 2 == 0 ? 2 * c.pg : 4 * c.pg);
  int q = kConStageFloats / (nbins * c.stride) / unit * unit;
  if (q > kConMaxQ) q = kConMaxQ / unit * unit;
  if (q < unit) q = unit;
  c.Q = q;
  // a tile wider than the bins and a chunk wider than the row read on past
  // their end: slots and bins that nothing owns
  c.stage_floats = c.Q * nbins * c.stride + (nbins < c.T ? (c.T - nbins) * c.stride : 0) + c.ch;
  c.stage_floats = (c.stage_floats + 3) & ~3;
  const int red = (c.threads + 1) * c.T * c.T;  // the flush buffer aliases the stages (154 KB at most)
  const int body = kConStages * c.stage_floats > red ? kConStages * c.stage_floats : red;
  c.smem_bytes = (body + kConStages * kConMaxQ + kConMaxTiles) * 4;  // 187 KB at most
  return c;
}

__device__ __forceinline__ void con_cp4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void con_cp16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

__device__ __forceinline__ float con_lds(uint32_t p) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(p) : "memory");
  return v;
}

// One primary: S1, S2 the first bin of the tile's sides, ST floats between
// bins (0: st, at run time).  On the diagonal only pairs with a column at or
// right of the row.
template <int T, bool DIAG, int ST>
__device__ __forceinline__ void con_step(float2 (&acc)[T][T / 2], const float* S1, const float* S2, int st, float w) {
  float x[T], y[T];
  if constexpr (ST > 0) {
#pragma unroll
    for (int i = 0; i < T; ++i) x[i] = S1[i * ST];
    if constexpr (!DIAG) {
#pragma unroll
      for (int i = 0; i < T; ++i) y[i] = S2[i * ST];
    }
  } else {
    // the row's own stride: addresses by addition (products take the FMA pipe)
    uint32_t p = (uint32_t)__cvta_generic_to_shared(S1);
#pragma unroll
    for (int i = 0; i < T; ++i, p += 4u * (uint32_t)st) x[i] = con_lds(p);
    if constexpr (!DIAG) {
      p = (uint32_t)__cvta_generic_to_shared(S2);
#pragma unroll
      for (int i = 0; i < T; ++i, p += 4u * (uint32_t)st) y[i] = con_lds(p);
    }
  }
#pragma unroll
  for (int i = 0; i < T; ++i) {
    const float xi = w * x[i];
#pragma unroll
    for (int j = DIAG ? i / 2 : 0; j < T / 2; ++j) {
      const float2 v = DIAG ? make_float2(x[2 * j], x[2 * j + 1]) : make_float2(y[2 * j], y[2 * j + 1]);
      acc[i][j] = __ffma2_rn(make_float2(xi, xi), v, acc[i][j]);
    }
  }
}

template <int T, int CH, int MODE>
__global__ void __launch_bounds__(con_max_threads(T), 1) k_contract_fp32(ContractArgs a, ConShape sh) {
  extern __shared__ __align__(16) float s_dyn[];
  __shared__ int s_coef[(kLmaxCap + 1) * (kLmaxCap + 1)];  // slot of each coefficient | its multipole << 16
  __shared__ int s_ord[CH];                                // the chunk's slots by multipole
  __shared__ int s_l[kLmaxCap + 1], s_l0[kLmaxCap + 2], s_nl;  // its multipoles and where their slots start
  const int nb = a.nbins, L = a.lmax;
  const int nc = a.sphere ? 2 * L + 1 : (L + 1) * (L + 1);  // coefficients per (primary, bin)
  int* s_tile = reinterpret_cast<int*>(s_dyn);              // [kConMaxTiles] B1 | B2 << 8 (-1: none)
  float* s_w = s_dyn + kConMaxTiles;                        // [stages][kConMaxQ]
  float* s_stage = s_w + kConStages * kConMaxQ;             // [stages][Q][nb][stride]
  const int tid = threadIdx.x;
  const int c = tid % CH;
  const int tl = (tid / CH) % sh.tiles, pg = tid / (CH * sh.tiles);
  // Slices and runs of whole multiples of `gran` primaries, so that they start
  // on 16 bytes when the base does; long ones on whole 128-byte lines where
  // four primaries or fewer make one (100k rows of 16 bins x 121: 229 us
  // against 241 where every other run started in the middle of a line).
  const int64_t even = (a.np + gridDim.x - 1) / gridDim.x;
  int gran = 1;
  while (gran < 4 && (gran * nb * a.row) % (even >= 64 ? 32 : 4) != 0) gran *= 2;
  auto whole = [&](int64_t n) { return (n + gran - 1) / gran * gran; };
  const int64_t slice = whole(even);
  const int64_t p0 = (int64_t)blockIdx.x * slice;
  const int64_t p1 = min(a.np, p0 + slice);
  if (p0 >= p1) return;  // uniform for the block
  // primaries between two flushes
  const int runs = sh.pg > 1 || sh.nchunk >= 8 ? 1 : a.runs;
  const int64_t run = min(whole((slice + runs - 1) / runs), (int64_t)kConFlush * sh.pg);
  // tile -> (B1 <= B2); the last tile of a side is moved back so that it ends
  // at the last bin (its bins before B T are computed twice, written once)
  for (int t = tid; t < sh.tiles; t += blockDim.x) {
    int r = blockIdx.y * sh.tiles + t, v = -1;
    if (r < sh.ntiles) {
      int B = 0;
      while (r >= sh.nbt - B) {
        r -= sh.nbt - B;
        ++B;
      }
      v = B | (B + r) << 8;
    }
    s_tile[t] = v;
  }
  for (int k = tid; k < nc; k += blockDim.x) {
    int l = a.sphere ? (k + 1) / 2 : (int)sqrtf((float)k);
    if (!a.sphere) {
      while ((l + 1) * (l + 1) <= k) ++l;
      while (l * l > k) --l;
    }
    s_coef[k] = __ldg(a.slot + k) | l << 16;
  }
  __syncthreads();
  const int tv = s_tile[tl];
  const bool active = tv >= 0;
  const int B1 = active ? tv & 255 : 0, B2 = active ? tv >> 8 : 0;
  auto start = [&](int B) { return max(min(B * T, nb - T), 0); };
  const int stride = MODE == kConLinearAny ? sh.stride : CH;
  const int off1 = start(B1) * stride + c, off2 = start(B2) * stride + c;
  const int qstride = nb * stride;
  double* out = a.partial + (size_t)(a.part0 + blockIdx.x) * (L + 1) * nb * nb;
  float2 acc[T][T / 2];
#pragma unroll
  for (int i = 0; i < T; ++i)
#pragma unroll
    for (int j = 0; j < T / 2; ++j) acc[i][j] = make_float2(0.f, 0.f);

  // the slots of the chunk at c0 by multipole (the coefficients are in that
  // order), and the multipoles that have any: by one warp, while the chunk's
  // first copies are in flight
  auto order_slots = [&](int c0) {
    const int lane = tid & 31;
    const unsigned lt = (1u << lane) - 1u;
    int n = 0, nl = 0, last = -1;  // slots and multipoles so far, and the last of these
    for (int k = lane; k - lane < nc; k += 32) {
      const int v = k < nc ? s_coef[k] : -1;
      const int s = (v & 0xffff) - c0, l = v >> 16;
      const bool in = v >= 0 && s >= 0 && s < CH;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      const int before = __shfl_sync(0xffffffffu, l, 31 - __clz((m & lt) | 1u));
      const bool first = in && l != (m & lt ? before : last);
      const unsigned mf = __ballot_sync(0xffffffffu, first);
      const int at = n + __popc(m & lt);
      if (in) s_ord[at] = s;
      if (first) {
        s_l[nl + __popc(mf & lt)] = l;
        s_l0[nl + __popc(mf & lt)] = at;
      }
      n += __popc(m);
      nl += __popc(mf);
      const int end = __shfl_sync(0xffffffffu, l, 31 - __clz(m | 1u));
      if (m) last = end;
    }
    if (lane == 0) {
      s_nl = nl;
      s_l0[nl] = n;
    }
  };
  for (int ck = 0; ck < sh.nchunk; ++ck) {
    const int c0 = ck * CH;
    // copy of the stage of primaries [pb, pb + cnt)
    auto issue = [&](int64_t pb, int cnt, int st) {
      float* buf = s_stage + st * sh.stage_floats;
      if (tid < cnt) con_cp4(s_w + st * kConMaxQ + tid, a.wprim + pb + tid);
      const float* src = a.M + pb * nb * (int64_t)a.row;
      if constexpr (MODE == kConLinear || MODE == kConLinearAny) {
        const int total = cnt * nb * a.row;
        int k = tid * 4;
        if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
#pragma unroll 4
          for (; k + 4 <= total; k += blockDim.x * 4) con_cp16(buf + k, src + k);
          for (k = (total & ~3) + tid; k < total; k += blockDim.x) con_cp4(buf + k, src + k);
        } else {
#pragma unroll 4
          for (k = tid; k < total; k += blockDim.x) con_cp4(buf + k, src + k);
        }
      } else {
        // thread tid takes one column (four with 16-byte copies) of every
        // (threads / columns)-th row
        constexpr int E = MODE == kConRows16 ? 4 : 1, COLS = CH / E;
        const int col = (tid % COLS) * E, rs = blockDim.x / COLS, r0 = tid / COLS;
        if (c0 + col < a.row) {
          const float* sp = src + c0 + col + (int64_t)r0 * a.row;
          float* dp = buf + r0 * CH + col;
          const int64_t sstep = (int64_t)rs * a.row;
          const int dstep = rs * CH, rows = cnt * nb;
#pragma unroll 4
          for (int r = r0; r < rows; r += rs) {
            if constexpr (E == 4) con_cp16(dp, sp);
            else con_cp4(dp, sp);
            sp += sstep;
            dp += dstep;
          }
        }
      }
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    // the sums over each multipole's slots: all accumulators to shared memory
    // ([entry of the tile][thread], rows padded by one), then a warp takes 32
    // entries of one multipole, every lane the same slots of its entry
    auto flush = [&] {
      float* red = s_stage;
      const int nthr = blockDim.x, ld = nthr + 1;
      __syncthreads();
      const int nl = s_nl;
#pragma unroll
      for (int i = 0; i < T; ++i)
#pragma unroll
        for (int j = 0; j < T / 2; ++j) {
          red[(i * T + 2 * j) * ld + tid] = acc[i][j].x;
          red[(i * T + 2 * j + 1) * ld + tid] = acc[i][j].y;
          acc[i][j] = make_float2(0.f, 0.f);
        }
      __syncthreads();
      const int entries = sh.tiles * T * T;
      const int items = (entries + 31) / 32 * nl;
      for (int o = tid >> 5; o < items; o += nthr >> 5) {
        const int gr = o / nl;
        const int k = (o - gr * nl + gr) % nl;  // rotated, so that every warp gets long and short ones
        const int en = gr * 32 + (tid & 31);
        const int t = en < entries ? en / (T * T) : 0, ij = en < entries ? en - t * T * T : 0;
        const int v2 = s_tile[t];
        const int C1 = v2 & 255, C2 = v2 >> 8;
        const int b1 = start(C1) + ij / T, b2 = start(C2) + ij % T;
        const bool own = en < entries && v2 >= 0 && b1 < nb && b2 < nb && b1 <= b2 && b1 >= C1 * T && b2 >= C2 * T;
        const int q0 = s_l0[k], q1 = s_l0[k + 1];
        float v = 0.f, c = 0.f;  // the sum and the errors of its additions
        for (int g = 0; g < sh.pg; ++g) {
          const float* rg = red + ij * ld + (g * sh.tiles + t) * CH;
#pragma unroll 4
          for (int q = q0; q < q1; ++q) {
            const float x = rg[s_ord[q]], s = v + x, b = s - v;
            c += (v - (s - b)) + (x - b);
            v = s;
          }
        }
        // one thread an entry, one flush after another: the order of the adds is fixed
        if (own)
          atomicAdd(out + ((size_t)s_l[k] * nb + b1) * nb + b2, (double)v + (isfinite(c) ? (double)c : 0.0));  // v may be infinite
      }
      __syncthreads();
    };

    for (int64_t f0 = p0; f0 < p1; f0 += run) {
      const int64_t f1 = min(p1, f0 + run);
      const int nst = (int)((f1 - f0 + sh.Q - 1) / sh.Q);
      auto count = [&](int k) { return (int)min((int64_t)sh.Q, f1 - f0 - (int64_t)k * sh.Q); };
      for (int k = 0; k < kConStages - 1; ++k) {
        if (k < nst) issue(f0 + (int64_t)k * sh.Q, count(k), k);
        commit();
      }
      if (f0 == p0 && tid < 32) order_slots(c0);
      int st = 0, nx = kConStages - 1;
      for (int k = 0; k < nst; ++k) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kConStages - 2) : "memory");
        __syncthreads();  // stage k is in, and every thread is done with stage k - 1
        const int kn = k + kConStages - 1;
        if (kn < nst) issue(f0 + (int64_t)kn * sh.Q, count(kn), nx);
        commit();
        const int cnt = count(k);
        const float* buf = s_stage + st * sh.stage_floats + pg * qstride;
        const float* wq = s_w + st * kConMaxQ;
        if (active) {
          constexpr int ST = MODE == kConLinearAny ? 0 : CH;
          if (B1 == B2) {
            for (int q = pg; q < cnt; q += sh.pg, buf += sh.pg * qstride)
              con_step<T, true, ST>(acc, buf + off1, nullptr, stride, wq[q]);
          } else {
            for (int q = pg; q < cnt; q += sh.pg, buf += sh.pg * qstride)
              con_step<T, false, ST>(acc, buf + off1, buf + off2, stride, wq[q]);
          }
        }
        st = st + 1 == kConStages ? 0 : st + 1;
        nx = nx + 1 == kConStages ? 0 : nx + 1;
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      flush();
    }
  }
}

template <int T, int CH>
static const void* con_fn(int mode) {
  return mode == kConLinear      ? (const void*)k_contract_fp32<T, CH, kConLinear>
         : mode == kConLinearAny ? (const void*)k_contract_fp32<T, CH, kConLinearAny>
         : mode == kConRows16    ? (const void*)k_contract_fp32<T, CH, kConRows16>
                              : (const void*)k_contract_fp32<T, CH, kConRows4>;
}

static const void* con_kernel(const ConShape& sh, int row, bool aligned) {
  const int mode = sh.nchunk == 1 ? (row == sh.ch ? kConLinear : kConLinearAny) : ((row & 3) == 0 && aligned ? kConRows16 : kConRows4);
  switch (sh.T * 1000 + sh.ch) {
    case 6032: return con_fn<6, 32>(mode);
    case 6064: return con_fn<6, 64>(mode);
    case 6128: return con_fn<6, 128>(mode);
    case 8032: return con_fn<8, 32>(mode);
    case 8064: return con_fn<8, 64>(mode);
    case 8128: return con_fn<8, 128>(mode);
    case 10032: return con_fn<10, 32>(mode);
    case 10064: return con_fn<10, 64>(mode);
    default: return con_fn<10, 128>(mode);
  }
}

// Resident blocks per SM of the contraction for this shape (0 if it cannot run).
int contract_fp32_blocks_per_sm(int nbins, int row) {
  const ConShape sh = con_shape(nbins, row);
  if ((size_t)sh.smem_bytes > kConSmemCap) return 0;
  // (the copies of an aligned and of an unaligned base are two kernels)
  const int x = resident_blocks(con_kernel(sh, row, false), sh.threads, sh.smem_bytes);
  const int y = resident_blocks(con_kernel(sh, row, true), sh.threads, sh.smem_bytes);
  return x < y ? x : y;
}

cudaError_t launch_contract_fp32(const ContractArgs& a, int nparts, cudaStream_t st) {
  if (a.np == 0) return cudaSuccess;
  const ConShape sh = con_shape(a.nbins, a.row);
  if ((size_t)sh.smem_bytes > kConSmemCap) return cudaErrorInvalidValue;
  const void* fn = con_kernel(sh, a.row, (reinterpret_cast<uintptr_t>(a.M) & 15) == 0);
  if (allow_smem(fn, sh.smem_bytes) != cudaSuccess) return cudaErrorInvalidConfiguration;
  ContractArgs ca = a;
  ConShape cs = sh;
  void* args[] = {&ca, &cs};
  const cudaError_t e = cudaLaunchKernel(fn, dim3(nparts, (sh.ntiles + sh.tiles - 1) / sh.tiles), dim3(sh.threads), args,
                       (size_t)sh.smem_bytes, st);
  if (e != cudaSuccess) return e;
  ++g_launches;
  return cudaGetLastError();
}

// zeta_l(b1,b2) = f_l * sum_parts partial[part][l][min b][max b]; f_l =
// 4 pi/(2l+1) for the 3-D multipoles, 1 on the sphere.  32 consecutive entries
// per block, eight threads an entry taking every eighth partial row and added
// in a fixed order: one thread an entry walked 152 to 304 rows one latency
// after another (75 us at 4400 entries; 6 us so).  blockIdx.y: the catalogue
// of a batch.
constexpr int kFinGroups = 8;
__global__ void __launch_bounds__(32 * kFinGroups) k_finalize(const double* __restrict__ partial, int nparts, int lmax,
                                                              int nb, int sphere, double* __restrict__ zeta) {
  __shared__ double s[kFinGroups][32];
  const int total = (lmax + 1) * nb * nb;
  const size_t stride = (size_t)total;
  partial += (size_t)blockIdx.y * nparts * stride;
  zeta += (size_t)blockIdx.y * stride;
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int o = blockIdx.x * 32 + lane;
  const int l = o / (nb * nb), r = o - l * nb * nb;
  const int b1 = r / nb, b2 = r - b1 * nb;
  const bool own = o < total && b1 <= b2;
  double v = 0.0;
  if (own) {
#pragma unroll 4
    for (int p = g; p < nparts; p += kFinGroups) v += partial[(size_t)p * stride + o];
  }
  s[g][lane] = v;
  __syncthreads();
  if (own && g == 0) {
#pragma unroll
    for (int k = 1; k < kFinGroups; ++k) v += s[k][lane];
    if (!sphere) v *= 4.0 * 3.14159265358979323846 / (2.0 * l + 1.0);
    zeta[o] = v;
    zeta[((size_t)l * nb + b2) * nb + b1] = v;
  }
}

// Loads every kernel of launch_contract_fp32 and launch_finalize.
cudaError_t load_contract_fp32() {
  cudaFuncAttributes at{};
  cudaError_t e = cudaFuncGetAttributes(&at, k_finalize);
  for (int mode = kConRows4; mode <= kConLinearAny; ++mode)
    for (const void* fn : {con_fn<6, 32>(mode), con_fn<6, 64>(mode), con_fn<6, 128>(mode), con_fn<8, 32>(mode),
                           con_fn<8, 64>(mode), con_fn<8, 128>(mode), con_fn<10, 32>(mode), con_fn<10, 64>(mode),
                           con_fn<10, 128>(mode)})
      if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, fn);
  return e;
}

cudaError_t launch_finalize(const double* partial, int nparts, int lmax, int nbins, double* zeta, bool sphere,
                            int ncat, cudaStream_t st) {
  const int total = (lmax + 1) * nbins * nbins;
  k_finalize<<<dim3((total + 31) / 32, ncat), 32 * kFinGroups, 0, st>>>(partial, nparts, lmax, nbins, sphere ? 1 : 0,
                                                                        zeta);
  ++g_launches;
  return cudaGetLastError();
}

// Weighted pair sums of the two-point function from the same pass:
// sum_p w_p sum_{j in b} w_j = sqrt(4 pi) sum_p w_p a_00(p, b), the a_00 column
// of the M rows (col).  Block bx takes a fixed slice of the primaries; its
// 256 / nbins groups of nbins threads interleave over the slice (each thread
// keeps its bin) and are added in a fixed order to partial[bx][b] (FP64;
// accumulated over the chunks of one compute).
__global__ void __launch_bounds__(256) k_pair_sums(const float* __restrict__ M, const float* __restrict__ w,
                                                   int64_t np, int nbins, int row, int col,
                                                   double* __restrict__ partial) {
  __shared__ double s[256];
  const int64_t nparts = gridDim.x, bx = blockIdx.x;
  const int64_t p0 = np * bx / nparts, p1 = np * (bx + 1) / nparts;
  const int ng = 256 / nbins;
  const int g = threadIdx.x / nbins, b = threadIdx.x - g * nbins;
  double acc = 0.0;
  if (g < ng) {
    const float* m = M + ((p0 + g) * nbins + b) * (int64_t)row + col;
    const int64_t step = (int64_t)ng * nbins * row;
#pragma unroll 8
    for (int64_t p = p0 + g; p < p1; p += ng, m += step) acc += (double)(__ldg(w + p)) * (double)__ldg(m);
  }
  s[threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.x < nbins) {
    double v = 0.0;
    for (int k = 0; k < ng; ++k) v += s[k * nbins + threadIdx.x];
    partial[bx * nbins + threadIdx.x] += v;
  }
}

cudaError_t launch_pair_sums(const float* M, const float* w, int64_t np, int nbins, int row, int col,
                             double* partial, int nparts, cudaStream_t st) {
  k_pair_sums<<<nparts, 256, 0, st>>>(M, w, np, nbins, row, col, partial);
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace ctb
