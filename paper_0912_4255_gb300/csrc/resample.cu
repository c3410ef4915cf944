// Steps 2-5 of Sec. III.A.2.  k_resample, one thread per point of the
// barycentric grid, writes the weighted series w_a, w_b (zero-padded to the
// FFT length) and the block partial sums of A, B, C for fstat_resample (parity
// and debug output).  fstat_compute takes the tiled kernels below
// (launch_resample_t), which leave both series in the first FFT pass's order
// and agree with k_resample to the rounding of single precision.
#include "passes.cuh"
#include "sinc_run.cuh"

namespace fs {

namespace {

constexpr int kResThreads = 256;

template <typename R, int INTERP, int TAPS, typename OutC>
__global__ void __launch_bounds__(kResThreads)
k_resample(PlanConst pc, Chunk c, int ti, const float2* __restrict__ x, const int64_t* __restrict__ gaps,
           const double* __restrict__ wcs, OutC* __restrict__ out_a, OutC* __restrict__ out_b,
           int64_t out_stride, double* __restrict__ abcd, int* status) {
  using Knot = typename KnotOf<R>::T;
  __shared__ double red[96];
  const int t = ti >= 0 ? ti : (int)blockIdx.y;
  const TmplMeta m = c.meta[t];
  const int64_t n = (int64_t)1 << m.log2n;
  const int64_t k = (int64_t)blockIdx.x * kResThreads + threadIdx.x;
  if ((int64_t)blockIdx.x * kResThreads >= n) return;
  OutC* oa = out_a + (ti >= 0 ? 0 : (int64_t)t * out_stride);
  OutC* ob = out_b + (ti >= 0 ? 0 : (int64_t)t * out_stride);
  if (m.status != FSTAT_OK) {
    if (k < n) {
      const float nan = __int_as_float(0x7fc00000);
      oa[k].x = nan; oa[k].y = nan; ob[k].x = nan; ob[k].y = nan;
    }
    if (abcd && k == 0) { abcd[4 * t] = abcd[4 * t + 1] = abcd[4 * t + 2] = abcd[4 * t + 3] = __longlong_as_double(0x7ff8000000000000ll); }
    return;
  }
  const Knot* kn = reinterpret_cast<const Knot*>(c.knots) + (int64_t)t * c.knot_stride;
  cpx<R> va = czero<cpx<R>>(), vb = czero<cpx<R>>();
  R pa = 0, pb = 0, pcc = 0;
  if (k < m.n_b) {
    R aa, bb;
    GapCursor gc = make_cursor(m, gaps);
    if (sample_weights<R, INTERP, TAPS>(pc, kn, (int)k, x, gc, wcs, va, vb, aa, bb)) {
      pa = aa * aa; pb = bb * bb; pcc = aa * bb;
    }
  }
  if (k < n) {
    oa[k].x = va.x; oa[k].y = va.y;
    ob[k].x = vb.x; ob[k].y = vb.y;
  }
  double sA, sB, sC;
  block_sum3((float)pa, (float)pb, (float)pcc, sA, sB, sC, red);
  double* part = c.partials + (int64_t)t * c.part_stride * 3;
  if (threadIdx.x == 0) {
    part[3 * blockIdx.x] = sA; part[3 * blockIdx.x + 1] = sB; part[3 * blockIdx.x + 2] = sC;
  }
  finalize_sums(c.meta + t, part, (int)((n + kResThreads - 1) / kResThreads), c.counters + t, pc.sigma2,
                abcd ? abcd + 4 * t : nullptr, status);
}

template <typename R, typename OutC>
cudaError_t dispatch(const PlanConst& pc, const Chunk& c, int ti, int log2n, const float2* x,
                     const int64_t* gaps, const double* wcs, void* oa, void* ob, int64_t stride,
                     double* abcd, int* status, cudaStream_t s) {
  const int64_t n = (int64_t)1 << log2n;
  dim3 grid((unsigned)((n + kResThreads - 1) / kResThreads), ti >= 0 ? 1u : (unsigned)c.nt);
  OutC* a = reinterpret_cast<OutC*>(oa);
  OutC* b = reinterpret_cast<OutC*>(ob);
  if (pc.interp == FSTAT_NEAREST)
    k_resample<R, FSTAT_NEAREST, 8, OutC><<<grid, kResThreads, 0, s>>>(pc, c, ti, x, gaps, wcs, a, b, stride, abcd, status);
  else if (pc.taps == 8)
    k_resample<R, FSTAT_SINC, 8, OutC><<<grid, kResThreads, 0, s>>>(pc, c, ti, x, gaps, wcs, a, b, stride, abcd, status);
  else
    k_resample<R, FSTAT_SINC, 0, OutC><<<grid, kResThreads, 0, s>>>(pc, c, ti, x, gaps, wcs, a, b, stride, abcd, status);
  return cudaGetLastError();
}

// Tiled form for the unfused path, one warp per tile of 8 rows x 32
// consecutive columns of the N1 x N2 grid (grid point k = k2 + N2 k1).  The
// tile goes through the warp's own shared memory and leaves in the order in
// which the first FFT pass reads its columns, W[k2 / C][k1][k2 % C], as runs
// of 8 C pairs (128 bytes at C = 1): no warp waits for another one.  Tiles are
// numbered by row tile, then column tile; those of the row tiles with a point
// below n_b are done, and the first pass reads every point at k >= n_b as
// zero without loading it.  A warp takes per_warp consecutive tiles and
// adds its part of A, B, C to the template's.
constexpr int kTileRows = 8, kTileCols = 32;
constexpr int kTilePts = kTileRows * kTileCols;
constexpr int kTileWarps = 4;                       // warps per block
constexpr int kTileThreads = 32 * kTileWarps;
constexpr int kMaxPerWarp = 8;

// Position of (row, col) in a warp's tile: rows of 32 pairs, the low three
// bits of the column xored with a key of the row and the column's group of
// eight.  Writes (8 lanes: two rows x four groups, one column each) and reads
// (8 lanes: eight rows of one column) then fall on distinct 16-byte banks.
__device__ __forceinline__ int tile_key(int row, int grp) { return grp ^ ((row >> 1) | ((row & 1) << 2)); }
__device__ __forceinline__ int tile_pos(int row, int col) {
  return row * kTileCols + (col & 24) + ((col & 7) ^ tile_key(row, col >> 3));
}

// The warp's tile from shared memory into W (first column c0, first row r0).
template <typename R>
__device__ __forceinline__ void store_tile(Pair<R>* __restrict__ w_out, const Pair<R>* __restrict__ so, int c0, int r0,
                                           int lc, int64_t gstride, int lane) {
  if (lc == 0) {
    // one column pair per first-pass block: eight lanes a column
    const int row = lane & 7, cl = lane >> 3;
    const Pair<R>* sr = so + row * kTileCols;
    Pair<R>* o = w_out + (int64_t)(c0 + cl) * gstride + r0 + row;
#pragma unroll
    for (int it = 0; it < kTilePts / 32; ++it) {
      const int grp = it >> 1;                      // column 4 it + cl
      stcs(o, sr[8 * grp + ((4 * (it & 1) + cl) ^ tile_key(row, grp))]);
      o += 4 * gstride;
    }
    return;
  }
#pragma unroll
  for (int it = 0; it < kTilePts / 32; ++it) {
    const int e = it * 32 + lane;
    const int g = e >> (3 + lc), w = e & ((8 << lc) - 1);
    const int row = w >> lc, col = (g << lc) + (w & ((1 << lc) - 1));
    stcs(w_out + ((int64_t)(c0 >> lc) + g) * gstride + ((int64_t)r0 << lc) + w, so[tile_pos(row, col)]);
  }
}

// Adds the warp's sums of a^2, b^2, a b to the template's, in units of 2^-36 of
// what one point can add (scale_beams).  One atomic addition per
// warp and sum: partial sums in memory and a kernel to reduce them took 10 us
// of every call, a barrier over the block's warps held them until the slowest
// was done.
__device__ __forceinline__ void add_sums(float pa, float pb, float pcc, TmplMeta* m) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    pa += __shfl_xor_sync(0xffffffffu, pa, o);
    pb += __shfl_xor_sync(0xffffffffu, pb, o);
    pcc += __shfl_xor_sync(0xffffffffu, pcc, o);
  }
  const int lane = threadIdx.x & 31;
  if (lane < 3) {
    const float v = lane == 0 ? pa : (lane == 1 ? pb : pcc);
    atomicAdd(&m->acc[lane], (unsigned long long)__double2ll_rn((double)v * (double)(1ll << kSumBits)));
  }
}

// Other tap counts, FP64 (and knot intervals of fewer than 32 points): one point
// per lane and row (32 consecutive points of a row at a time: one knot record
// for all lanes, taps from one contiguous run of x).  A tile's points start
// below those at which the tile before ended; in a long gap list they are found
// by binary search.  2000 gaps in 8 templates of 1,728,000 samples, FP32 with
// knots 16 apart, took 2406 us when every tile walked the list from its
// beginning, 1100 now.  Lists of up to 16 are walked; a call without longer ones
// takes the form without the search, which costs registers (one template of 2^20
// points, 16 taps, 54 -> 59 us).
constexpr int kGapsWalked = 16;
__device__ __noinline__ void find_gap(GapCursor& gc, int j) { gc.seek(j); }
__device__ __forceinline__ int knot_base(const KnotF& r) { return __ldg(&r.I); }
__device__ __forceinline__ int knot_base(const KnotD& r) { return (int)floor(__ldg(&r.U)); }

template <typename R, int INTERP, int TAPS, bool SEARCH>
__global__ void __launch_bounds__(kTileThreads)
k_resample_t(PlanConst pc, Chunk c, int l2, int lc, int per_warp, const float2* __restrict__ x,
             const int64_t* __restrict__ gaps, const double* __restrict__ wcs) {
  using Cx = cpx<R>;
  using Knot = typename KnotOf<R>::T;
  __shared__ Pair<R> tiles[kTileWarps][kTilePts];
  let_next_start();
  wait_for_previous();
  const int t = blockIdx.y;
  const TmplMeta& m = c.meta[t];
  if (m.status != FSTAT_OK) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_b = (int)m.n_b;
  const int nlive = live_tiles(m.n_b, l2);
  const int wid = (int)blockIdx.x * kTileWarps + warp;
  const int b0 = wid * per_warp;
  if (b0 >= nlive) return;
  const Knot* kn = reinterpret_cast<const Knot*>(c.knots) + (int64_t)t * c.knot_stride;
  Pair<R>* w_out = reinterpret_cast<Pair<R>*>(c.wa) + (int64_t)t * c.z_stride;
  const int64_t gstride = (int64_t)1 << (m.log2n - l2 + lc);   // N1 * C
  Pair<R>* so = tiles[warp];
  float pa = 0.f, pb = 0.f, pcc = 0.f;
#pragma unroll 1
  for (int b = b0; b < b0 + per_warp && b < nlive; ++b) {
    const int c0 = (b & ((1 << (l2 - 5)) - 1)) << 5;
    const int r0 = (b >> (l2 - 5)) * kTileRows;
    const int k0 = c0 + lane + (r0 << l2);
    GapCursor gc = make_cursor(m, gaps);      // the points of a new tile start lower
    // u grows with k: the tile's samples lie above its first knot's, less the taps
    if constexpr (SEARCH) {
      if (gc.n > kGapsWalked && c0 + lane + (r0 << l2) < n_b)
        find_gap(gc, knot_base(kn[(c0 + lane + (r0 << l2)) >> pc.log2h]) - 64);
    }
#pragma unroll 1
    for (int row = 0; row < kTileRows; ++row) {
      const int k = c0 + lane + ((r0 + row) << l2);
      Cx va = czero<Cx>(), vb = czero<Cx>();
      if (k < n_b) {
        R aa, bb;
        if (sample_weights<R, INTERP, TAPS>(pc, kn, k, x, gc, wcs, va, vb, aa, bb)) {
          pa += (float)(aa * aa); pb += (float)(bb * bb); pcc += (float)(aa * bb);
        }
      }
      so[tile_pos(row, lane)] = Pair<R>{va, vb};
    }
    __syncwarp();
    store_tile<R>(w_out, so, c0, r0, lc, gstride, lane);
    __syncwarp();                             // before the next tile overwrites so
  }
  add_sums(pa, pb, pcc, c.meta + t);
}

// One point of a run that cannot take the shared tap run (a slip, a gap or
// span edge, n_b): rare, kept out of line.  The windows of consecutive points
// overlap, so a cursor that one point's last taps moved past a gap would
// misjudge the next point's first taps: every point starts from the cursor
// as the run found it (gap index g).
template <int INTERP>
__device__ __noinline__ void slow_point(const PlanConst& pc, const KnotF* __restrict__ kn, int k, int n_b,
                                        const float2* __restrict__ x, GapCursor gc, int g,
                                        const double* __restrict__ wcs, Pair<float>* dst, float& pa, float& pb,
                                        float& pcc) {
  float2 va = make_float2(0.f, 0.f), vb = make_float2(0.f, 0.f);
  if (k < n_b) {
    float aa, bb;
    gc.g = g;
    gc.load();
    if (sample_weights<float, INTERP, 8>(pc, kn, k, x, gc, wcs, va, vb, aa, bb)) {
      pa += aa * aa; pb += bb * bb; pcc += aa * bb;
    }
  }
  *dst = Pair<float>{va, vb};
}

// FP32, 8-tap windowed sinc or nearest neighbour, in runs of eight points: a lane owns eight
// consecutive grid points of a row, four lanes a row of the tile.  The eight
// points lie in one knot interval, and since u advances by 1 + O(1e-4)
// samples per grid point floor(u) - k is the same for all of them except at
// rare slips, so that their taps are the one run x[n0 - 3 .. n0 + 11],
// n0 = floor(u) at k0, and the gap list is consulted once.  The knot's cubics
// (u, phase, a, b) are taken to second order about the run's centre, the tap
// weights come from one expansion (sinc_run.cuh), and the phase factor is the
// centre's times a rotation, whose sine and cosine serve the two points at
// equal distances from the centre.  A run with a slip, one that meets a gap
// or the span's edge, one that reaches n_b, and one whose u moves too far for
// the expansion are done point by point; a run inside one gap is zero.
// With the Lanczos window a slip of at most e = kRunNarrow needs no care: the
// tap that it drops and the one that it adds sit where the kernel is e^2 / 16.
//
// The samples of a row (44 from the one before its first tap: the last run's first
// tap lies at 28 at most and a run takes 16) are copied as
// 16-byte pieces into the warp's shared memory, a tile ahead (cp.async): read
// straight from memory, the lanes' 64-byte stride cost 16 wavefronts a load.  Instruction issue
// bounds the kernel (60 % of the cycles at 16 warps per SM, 128 registers; 96
// registers spill and measured 1.07 times the time).  64 templates of 1,728,000
// samples: 531 us, 1016 us when a block formed the weights of an 8 x 256 tile
// point by point (240 instructions a point, now about 120); nearest neighbour,
// 128 templates of 86,400: 62 us, 98 us with one point per lane.
constexpr int kRowSamples = 44;
constexpr int kRowUnits = kRowSamples / 2;        // 16-byte pieces of two samples
constexpr float kRunRotation = 0.125f;            // cycles: sincospi_small holds for |2 cycles| <= 1/4

enum { RUN_NEAREST = 0, RUN_LANCZOS = 1, RUN_RECT = 2 };

template <int KIND, bool QUAD>
__global__ void __launch_bounds__(kTileThreads, 4)
k_resample_run(PlanConst pc, Chunk c, int l2, int lc, int per_warp, const float2* __restrict__ x,
               const int64_t* __restrict__ gaps, const double* __restrict__ wcs) {
  __shared__ __align__(128) Pair<float> tiles[kTileWarps][kTilePts];
  __shared__ float4 rows[kTileWarps][2][kTileRows * kRowUnits];
  __shared__ float4 recs[kTileWarps][kTileRows][5];
  let_next_start();
  wait_for_previous();
  const int t = blockIdx.y;
  const TmplMeta& m = c.meta[t];
  if (m.status != FSTAT_OK) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_b = (int)m.n_b;
  const int nlive = live_tiles(m.n_b, l2);
  const int wid = (int)blockIdx.x * kTileWarps + warp;
  const int b0 = wid * per_warp;
  if (b0 >= nlive) return;
  const int b1 = b0 + per_warp < nlive ? b0 + per_warp : nlive;
  const KnotF* kn = reinterpret_cast<const KnotF*>(c.knots) + (int64_t)t * c.knot_stride;
  Pair<float>* w_out = reinterpret_cast<Pair<float>*>(c.wa) + (int64_t)t * c.z_stride;
  const int64_t gstride = (int64_t)1 << (m.log2n - l2 + lc);   // N1 * C
  const int row = lane >> 2, grp = lane & 3;
  Pair<float>* so = tiles[warp];
  const int key = tile_key(row, grp);
  Pair<float>* dw = so + row * kTileCols + 8 * grp;
  const unsigned out0 = (unsigned)__cvta_generic_to_shared(dw) + 16u * key;   // point i goes to out0 ^ 16 i
  // x may start in the middle of a 16-byte piece: samples j with j + odd even
  // start a piece, and samples outside [odd, x_end) lie in no whole piece
  const int odd = (int)(((uintptr_t)x >> 3) & 1);
  const int x_end = (((int)pc.n_data + odd) & ~1) - odd;
  const int hmask = (1 << pc.log2h) - 1;

  // the lane's run in tile b: its first point
  auto first_point = [&](int b) {
    const int c0 = (b & ((1 << (l2 - 5)) - 1)) << 5;
    const int r0 = (b >> (l2 - 5)) * kTileRows;
    return c0 + 8 * grp + ((r0 + row) << l2);
  };
  // The knot records of the tile's eight rows, kept in shared memory: rows are
  // N2 points apart and intervals h, both powers of two, so all rows enter
  // their next interval at the same column.
  float4(*rec)[5] = recs[warp];
  auto load_records = [&](int k) {
    const int kc = k < n_b ? k : n_b - 1;          // a record that exists
    const float4* q = reinterpret_cast<const float4*>(kn + (kc >> pc.log2h));
    __syncwarp();                                  // the last readers are done
    rec[row][grp] = __ldg(q + grp);
    if (grp == 0) rec[row][4] = __ldg(q + 4);
    __syncwarp();
  };
  // floor(u) at the run's first point; f = the fraction at its centre
  // (u = I + sk + i + dev(s + tau), s = sk + 3.5, tau = i - 3.5)
  auto centre = [&](int k, float& s, float& f) {
    const float4 q0 = rec[row][0];
    const float u3 = rec[row][1].x;
    const int sk = k & hmask;                      // a run stays in one knot interval
    s = small_int_to_float(sk) + 3.5f;
    const float dev = fmaf(fmaf(fmaf(u3, s, q0.w), s, q0.z), s, q0.y);
    int fl;
    float flf = round_nearest(dev, &fl);
    if (flf > dev) { flf -= 1.0f; --fl; }
    f = dev - flf;
    return __float_as_int(q0.x) + sk + fl;
  };
  // starts the copy of the row's samples into buffer u; returns the index of
  // the first one
  auto stage = [&](int n0, int u) {
    const int first = __shfl_sync(0xffffffffu, n0, lane & 28) - 4;
    const int base = ((first + odd) & ~1) - odd;
    float4* dst = rows[warp][u] + row * kRowUnits + grp;
    const float2* src = x + base + 2 * grp;
    if (__all_sync(0xffffffffu, base >= odd && base + kRowSamples <= x_end)) {
#pragma unroll
      for (int i = 0; i < (kRowUnits + 3) / 4; ++i)
        if (4 * i + 4 <= kRowUnits || grp < kRowUnits % 4) copy_async16(dst + 4 * i, src + 8 * i, true);
    } else {
#pragma unroll 1
      for (int i = 0; grp + 4 * i < kRowUnits; ++i) {
        const int jx = base + 2 * (grp + 4 * i);
        const bool inside = jx >= odd && jx < x_end;
        copy_async16(dst + 4 * i, inside ? src + 8 * i : x + odd, inside);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    return base;
  };

  GapCursor gc = make_cursor(m, gaps);
  float pa = 0.f, pb = 0.f, pcc = 0.f;
  int k0 = first_point(b0);
  load_records(k0);
  float s, f;
  int n0 = centre(k0, s, f);
  int base = stage(n0, 0);
  if (gc.n > 0) gc.seek(n0 - 64);                    // this warp's points only move forward
#pragma unroll 1
  for (int b = b0; b < b1; ++b) {
    const float4 q0 = rec[row][0], q1 = rec[row][1], q2 = rec[row][2], q3 = rec[row][3], q4 = rec[row][4];
    const float d1 = q0.z + s * (2.0f * q0.w + 3.0f * q1.x * s), d2 = q0.w + 3.0f * q1.x * s;
    const float p1 = q1.z + s * (2.0f * q1.w + 3.0f * q2.x * s), p2 = q1.w + 3.0f * q2.x * s;
    const float pc0 = knot_phase(q1.y, q1.z, q1.w, q2.x, s);
    const float a0 = q2.y + ((q3.x * s + q2.w) * s + q2.z) * s;
    const float a1 = q2.z + s * (2.0f * q2.w + 3.0f * q3.x * s), a2 = q2.w + 3.0f * q3.x * s;
    const float b0f = q3.y + ((q4.x * s + q3.w) * s + q3.z) * s;
    const float b1f = q3.z + s * (2.0f * q3.w + 3.0f * q4.x * s), b2 = q3.w + 3.0f * q4.x * s;
    const float spread = 3.5f * fabsf(d1) + 12.25f * fabsf(d2);
    const int off = n0 - 3 - base;                   // the run's first tap
    // the first gap that ends above the run (a slip may lower a tap by one)
    gc.advance(n0 - 5);
    const bool live = k0 < n_b;
    const bool smooth = spread <= (QUAD ? kRunSpread : kRunNarrow);
    // the nearest sample of every point in one gap: all masked
    const bool masked = smooth && gc.cs < n0 && n0 + 9 < gc.ce;
    // the data samples that the run's points may take: [j0, j1]
    const int j0 = KIND == RUN_NEAREST ? n0 - 1 : n0 - 3, j1 = KIND == RUN_NEAREST ? n0 + 9 : n0 + 11;
    const bool fast = live && smooth && k0 + 7 < n_b && j0 >= base && base + kRowSamples > j0 + 15 && j0 >= odd &&
                      j1 < x_end && j0 >= gc.lo && j1 < gc.hi && j1 < gc.cs &&
                      (KIND == RUN_NEAREST || (KIND == RUN_LANCZOS && !QUAD) ||
                       (f >= spread + 1e-6f && f + spread < 1.0f - 1e-6f));
    // the next tile's samples are on their way while this one is computed
    const int k0n = first_point(b + 1 < b1 ? b + 1 : b);
    if ((((k0n ^ k0) >> pc.log2h) | ((k0n ^ k0) >> l2)) != 0) load_records(k0n);
    float sn_, fn_;
    const int n0n = centre(k0n, sn_, fn_);
    const int basen = stage(n0n, (b + 1 - b0) & 1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
    if (fast) {
      // rotations of the points 3 - h and 4 + h (tau = -+(h + 1/2)) to the
      // phase removed: the centre's factor times exp(-2 pi i (tau p1 + tau^2 p2));
      // the linear part is one sine and cosine for both, the square a first-order turn
      int di;
      const float2 ec = expm2pi(pc0 - round_nearest(pc0, &di));
      float2 rm[4], rp[4];
      if (3.5f * fabsf(p1) <= kRunRotation && 12.25f * fabsf(p2) <= 1e-5f) {
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const float tau = (float)h + 0.5f;
          float sn, cs;
          sincospi_small(2.0f * tau * p1, &sn, &cs);
          const float eps = (6.28318531f * tau * tau) * p2;
          const float ex = fmaf(eps, ec.y, ec.x), ey = fmaf(-eps, ec.x, ec.y);
          const float xc = ex * cs, yc = ey * cs;
          rp[h] = make_float2(fmaf(ey, sn, xc), fmaf(-ex, sn, yc));
          rm[h] = make_float2(fmaf(-ey, sn, xc), fmaf(ex, sn, yc));
        }
      } else {
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const float tau = (float)h + 0.5f;
          const float gp = tau * fmaf(tau, p2, p1), gm = tau * fmaf(tau, p2, -p1);
          rp[h] = cmul(ec, expm2pi(gp - round_nearest(gp, &di)));
          rm[h] = cmul(ec, expm2pi(gm - round_nearest(gm, &di)));
        }
      }
      [[maybe_unused]] float w0[8], w1[8], w2[8];
      [[maybe_unused]] float2 v[16];
      const float4* xr = rows[warp][(b - b0) & 1] + row * kRowUnits;
      if constexpr (KIND != RUN_NEAREST) {
        run_weights<KIND == RUN_LANCZOS>(f - 0.5f, w0, w1, w2);
        if constexpr (!QUAD) {
          // d^2 w2 by its mean over |d| <= spread: what is left, (d^2 -
          // spread^2 / 2) w2, is below 1.7e-7 (1.1e-7 at the Earth's)
          const float hs = 0.5f * spread * spread;
#pragma unroll
          for (int tp = 0; tp < 8; ++tp) w0[tp] = fmaf(hs, w2[tp], w0[tp]);
        }
        const float4* xo = xr + (off >> 1);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float4 p = xo[j];
          v[2 * j] = make_float2(p.x, p.y);
          v[2 * j + 1] = make_float2(p.z, p.w);
        }
        if (off & 1) {
#pragma unroll
          for (int j = 0; j < 15; ++j) v[j] = v[j + 1];
        }
      }
      const int sk = k0 & hmask;
      [[maybe_unused]] const int ibase = __float_as_int(q0.x) + sk - base;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int h = i < 4 ? 3 - i : i - 4;
        const float tau = (float)i - 3.5f, tau2 = tau * tau;
        float2 z;
        if constexpr (KIND == RUN_NEAREST) {
          // the nearest sample is decided point by point: floor(dev + 1/2)
          const float si = small_int_to_float(sk + i);
          const float dv = q0.y + ((q1.x * si + q0.w) * si + q0.z) * si;
          int ji;
          if (round_nearest(dv + 0.5f, &ji) > dv + 0.5f) --ji;
          z = reinterpret_cast<const float2*>(xr)[ibase + i + ji];
        } else {
          const float d = fmaf(tau, d1, tau2 * d2);
          z = make_float2(0.f, 0.f);
#pragma unroll
          for (int tp = 0; tp < 8; ++tp) {
            float w;
            if constexpr (QUAD) w = fmaf(d, fmaf(d, w2[tp], w1[tp]), w0[tp]);
            else w = fmaf(d, w1[tp], w0[tp]);
            z.x = fmaf(w, v[i + tp].x, z.x);
            z.y = fmaf(w, v[i + tp].y, z.y);
          }
        }
        const float2 y = cmul(z, i < 4 ? rm[h] : rp[h]);
        const float a = fmaf(tau, a1, fmaf(tau2, a2, a0));
        const float bb = fmaf(tau, b1f, fmaf(tau2, b2, b0f));
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(out0 ^ (16u * i)), "f"(a * y.x), "f"(a * y.y),
                     "f"(bb * y.x), "f"(bb * y.y) : "memory");
      }
      // sums over the run of a^2, b^2, a b: sum tau^2 = 42, sum tau^4 = 388.5
      pa += fmaf(8.0f * a0, a0, fmaf(42.0f, fmaf(a1, a1, 2.0f * a0 * a2), 388.5f * a2 * a2));
      pb += fmaf(8.0f * b0f, b0f, fmaf(42.0f, fmaf(b1f, b1f, 2.0f * b0f * b2), 388.5f * b2 * b2));
      pcc += fmaf(8.0f * a0, b0f, fmaf(42.0f, fmaf(a1, b1f, fmaf(a0, b2, a2 * b0f)), 388.5f * a2 * b2));
    } else if (!live || masked) {
#pragma unroll
      for (int i = 0; i < 8; ++i) dw[i] = Pair<float>{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    }
    // the other runs, four at a time, eight lanes a run (by its own lane, point
    // after point, one such run held its warp for 10 us)
    unsigned slow = __ballot_sync(0xffffffffu, live && !fast && !masked);
    while (slow) {
      int src = -1;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (lane >> 3 == r) src = __ffs(slow) - 1;
        slow &= slow - 1;
      }
      const int sl = src < 0 ? 0 : src, i = lane & 7;
      const int ks = __shfl_sync(0xffffffffu, k0, sl), gs = __shfl_sync(0xffffffffu, gc.g, sl);
      if (src >= 0)
        slow_point<KIND == RUN_NEAREST ? FSTAT_NEAREST : FSTAT_SINC>(
            pc, kn, ks + i, n_b, x, gc, gs, wcs, so + tile_pos(sl >> 2, 8 * (sl & 3) + i), pa, pb, pcc);
      __syncwarp();
    }
    __syncwarp();
    store_tile<float>(w_out, so, (b & ((1 << (l2 - 5)) - 1)) << 5, (b >> (l2 - 5)) * kTileRows, lc, gstride, lane);
    __syncwarp();                             // before the next tile overwrites so and the rows
    k0 = k0n; n0 = n0n; base = basen; s = sn_; f = fn_;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  add_sums(pa, pb, pcc, c.meta + t);
}

// Upper bound on n_b for every template of the plan: t_b = t + t_m(t) and
// |dt_m/dt| <= (2 pi / year) au / c + (2 pi / sidereal day) R / c, so a span
// of n_data samples maps to at most (n_data - 1)(1 + beta) + 1 grid points.
int64_t nb_bound(const PlanConst& pc, int64_t n_fft) {
  const double beta = pc.beta;
  const double b = (double)(pc.n_data - 1) * (1.0 + 1.01 * beta + 1e-12) + 3.0;
  const int64_t nb = (int64_t)b;
  return nb < n_fft ? nb : n_fft;
}

int log2_cols(const Shape& sh) {
  int lc = 0;
  while ((1 << lc) < sh.cols) ++lc;
  return lc;
}

// Tiles the grid covers per template, and the tiles each warp takes, by the
// rounds of the 16 warps x 152 SMs that hold the kernel at once: up to four
// rounds, as many as make it one round (a warp overlaps its next tile's loads
// with the present one, and a second round would start over: one template of
// 1,728,000 samples 32.5 -> 30.5 us); above, enough for six rounds, so that
// the last one is short, and at most 8.
struct TileGrid { int per_warp, blocks; };
// In FP64 a tile holds the FP64 pipe for tens of microseconds: one tile a warp,
// so that the blocks spread evenly (16 templates of 2^17 points: with three
// tiles a warp, 3.2 blocks an SM, 16 taps 2063 us and 8 taps 638, with one 1400
// and 531; one template of 2^22, 8 taps, 1053 and 1004).
TileGrid tile_grid(const PlanConst& pc, const Shape& sh, int nt) {
  TileGrid g;
  const int covered = resample_covered(pc, sh);
  const int64_t warps = 16 * 152;
  const int64_t rounds = ((int64_t)covered * nt + warps - 1) / warps;
  g.per_warp = (int)(rounds <= 4 ? rounds : rounds / 6 < 2 ? 2 : rounds / 6 > kMaxPerWarp ? kMaxPerWarp : rounds / 6);
  if (g.per_warp < 1 || pc.precision == FSTAT_PREC_FP64) g.per_warp = 1;
  const int per_block = g.per_warp * kTileWarps;
  g.blocks = (covered + per_block - 1) / per_block;
  return g;
}

}  // namespace

cudaError_t launch_resample_t(const PlanConst& pc, const Chunk& c, const Shape& sh, const float2* x,
                              const int64_t* gaps, int64_t n_gaps_total, const double* wcs, cudaStream_t s) {
  const int lc = log2_cols(sh);
  const TileGrid tg = tile_grid(pc, sh, c.nt);
  if (tg.blocks == 0) return cudaSuccess;
  const dim3 grid((unsigned)tg.blocks, (unsigned)c.nt);
  cudaError_t e = cudaSuccess;
  const int64_t points = (int64_t)c.nt << (sh.l1 + sh.l2);
  const bool early = pc.precision == FSTAT_PREC_FP64 ? starts_early<double>(points) : starts_early<float>(points);
  auto go = [&](auto kern) {
    e = launch_after(early, kern, grid, kTileThreads, 0, s, pc, c, sh.l2, lc, tg.per_warp, x, gaps, wcs);
  };
  const auto points_of = [&](auto search) {
    constexpr bool S = decltype(search)::value;
    if (pc.precision == FSTAT_PREC_FP64) {
      if (pc.interp == FSTAT_NEAREST) go(k_resample_t<double, FSTAT_NEAREST, 8, S>);
      else if (pc.taps == 8) go(k_resample_t<double, FSTAT_SINC, 8, S>);
      else go(k_resample_t<double, FSTAT_SINC, 0, S>);
    } else if (pc.interp == FSTAT_NEAREST) {
      go(k_resample_t<float, FSTAT_NEAREST, 8, S>);
    } else if (pc.taps == 8) {
      go(k_resample_t<float, FSTAT_SINC, 8, S>);
    } else {
      go(k_resample_t<float, FSTAT_SINC, 0, S>);
    }
  };
  // point by point: FP64, other tap counts, and knot intervals shorter than a
  // tile's 32 columns
  if (pc.precision == FSTAT_PREC_FP64 || (pc.interp == FSTAT_SINC && pc.taps != 8) || pc.log2h < 5) {
    if (n_gaps_total > kGapsWalked) points_of(std::true_type{});
    else points_of(std::false_type{});
  } else {
    const bool quad = runs_need_square(pc);
    if (pc.interp == FSTAT_NEAREST) {
      go(k_resample_run<RUN_NEAREST, true>);
    } else if (pc.window == FSTAT_WIN_LANCZOS) {
      if (quad) go(k_resample_run<RUN_LANCZOS, true>);
      else go(k_resample_run<RUN_LANCZOS, false>);
    } else {
      if (quad) go(k_resample_run<RUN_RECT, true>);
      else go(k_resample_run<RUN_RECT, false>);
    }
  }
  return e;
}

// Tiles per template that the resampling grid covers.
int resample_covered(const PlanConst& pc, const Shape& sh) {
  return live_tiles(nb_bound(pc, (int64_t)1 << sh.log2n), sh.l2);
}

// out_double: 0 -> complex64 output, 1 -> complex128 output (FP64 internal buffers)
cudaError_t launch_resample_w(const PlanConst& pc, const Chunk& c, int ti, int log2n, const float2* x,
                              const int64_t* gaps, const double* wcs, void* out_a, void* out_b,
                              int64_t out_stride, int out_double, double* abcd, int* status,
                              cudaStream_t s) {
  if (pc.precision == FSTAT_PREC_FP64) {
    if (out_double) return dispatch<double, double2>(pc, c, ti, log2n, x, gaps, wcs, out_a, out_b, out_stride, abcd, status, s);
    return dispatch<double, float2>(pc, c, ti, log2n, x, gaps, wcs, out_a, out_b, out_stride, abcd, status, s);
  }
  return dispatch<float, float2>(pc, c, ti, log2n, x, gaps, wcs, out_a, out_b, out_stride, abcd, status, s);
}

}  // namespace fs
