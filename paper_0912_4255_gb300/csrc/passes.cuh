// The two passes of the four-step FFT that evaluates Eqs. 19-20 for every
// bin.  Steps 2-5 of Sec. III.A.2 are done by the tiled resampler, whose
// output the first pass loads, or in the first pass (persistent mode); Eq. 6
// is fused into the second pass.
//
// N = N1 N2, k = k2 + N2 k1, p = p1 + N1 p2:
//   X[p1 + N1 p2] = sum_k2 W_N2^{p2 k2} W_N^{p1 k2} sum_k1 x[k2 + N2 k1] W_N1^{p1 k1}.
// Both series (w_a, w_b) travel together, a Pair per point, in memory, in
// shared memory and in a thread's registers.
// Pass A (columns): a block owns C consecutive columns k2, produces their
// samples (resampled on the fly, or loaded), runs the N1-point FFTs over k1
// in shared memory, multiplies by W_N^{p1 k2} and stores into Z laid out as
// Z[p1 / RR][k2][p1 % RR].
// Pass B (rows): a block owns the RR consecutive rows p1 of one row block,
// which are one contiguous run of N2 * RR pairs; it runs the N2-point FFTs
// over k2 and writes 2F for every (p1, p2) at the ascending-frequency
// position q = p1 + N1 ((p2 + N2/2) mod N2).
#pragma once

#include "fstat_internal.cuh"

namespace fs {

// Where pass A's samples come from: the tiled resampler's series (SRC_LOAD),
// the same with the result written over it (SRC_INPLACE), or the resampling
// of each point in the pass itself (persistent mode).
enum { SRC_LOAD = 0, SRC_NN = 1, SRC_SINC = 2, SRC_INPLACE = 3 };
__host__ __device__ constexpr bool loads(int src) { return src == SRC_LOAD || src == SRC_INPLACE; }

// Bulk prefetch of [p, p + bytes) into L2 (p 16-byte aligned, bytes a
// multiple of 16): issued by one thread, completes in the background.
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

template <typename R>
struct ColsArgs {
  PlanConst pc;
  Chunk c;
  const float2* x;
  const int64_t* gaps;
  const double* wcs;
  Tw<R> tw;
  int tiles_max; // column tiles of one template
  int covered;   // tiles per template that the resampling grid covered
  int* status;
  int rr, log2rr; // rows of one group of Z (rows_group)
};

template <typename R>
struct RowsArgs {
  PlanConst pc;
  Chunk c;
  Tw<R> tw;
  float* out;
  int cols;      // C of pass A
  int log2cols;
  int blocks_max; // row blocks of one template
  int band;       // the plan's output band is partial (k_rows<..., true>)
};

// --------------------------------------------------------------- shapes

// Points per block (both series), at most 16 columns (rows) per block.
// Pass A, FP32: 8k, so that the longest first pass (N1 = 2^12) is one column
// pair of 68 KB, 256 threads of 16 points of each series, and two
// independent blocks share an SM: one loads or stores while the other
// computes.  Pass B, FP32: 16k (one block of 512 threads per SM), because
// its 2F leaves in runs of R values and R = 8 rows at N = 2^22 fill a 32-byte
// sector (runs of 4 measured 1.25 times the time); at N2 = 2^9, where 8k is
// enough for that, two blocks of 256 threads (12 templates of 2^21: 126 ->
// 110 us).  FP64: 4k, bound by the FP64 pipe at any size.
template <typename R> constexpr int points_a() { return std::is_same<R, float>::value ? 8192 : 4096; }
template <typename R> constexpr int points_b(int L2) { return !std::is_same<R, float>::value ? 4096 : L2 == 9 ? 8192 : 16384; }
template <int P> constexpr int cols_for(int L1) {
  const int c = (P / 2) >> L1;
  return c > 16 ? 16 : (c < 1 ? 1 : c);
}
template <typename R> constexpr int rows_for(int L2) {
  const int c = (points_b<R>(L2) / 2) >> L2;
  return c > 16 ? 16 : (c < 1 ? 1 : c);
}
// Rows of one group of the intermediate, Z[p1 / G][k2][p1 % G]: those of a
// block of pass B, but 16 at N2 = 2^9, two blocks' worth, because pass A writes
// runs of G C pairs (256 bytes instead of 128: 147 us, 160 with 128).
template <typename R> constexpr int rows_group(int L2) {
  return std::is_same<R, float>::value && L2 == 9 ? 16 : rows_for<R>(L2);
}
// one thread per 16 points of both series
template <typename R> constexpr int threads_for(int logn, int count) {
  const int units = (count << logn) / 16;
  return units >= 512 ? 512 : (units < 32 ? 32 : units);
}
// Blocks per SM to compile for: 512 threads of 128 registers (FP64: 256 of
// 255), as far as shared memory allows.
template <typename R> constexpr int min_blocks(int nt, size_t smem) {
  const int by_regs = (std::is_same<R, float>::value ? 512 : 256) / nt;
  const int by_smem = (int)((220 * 1024) / smem);
  const int b = by_regs < by_smem ? by_regs : by_smem;
  return b < 1 ? 1 : b;
}
// Stage plan of pass A: radix 16, a middle stage up to sub-transforms of
// 2^NSL_LAST, then a last stage of radix 2^RBL, its outputs in registers.  Its shared memory: C
// column pairs, the stage twiddle tables, and the two factors of the
// inter-pass twiddle W_N^{p1 k2} = W_N^{j k2} W_N^{q NS k2} (p1 = j + q NS)
// for the block's C columns.
template <int L1> struct PlanA {
  static constexpr int RBL = L1 >= 8 ? 4 : L1 - 4;
  static constexpr int NSL_LAST = L1 - RBL;
  static constexpr int RADL = 1 << RBL;
  static constexpr int NS = (1 << L1) / RADL;
  static constexpr int MID_TW = mid_tw_count(NSL_LAST - 4);
  static constexpr int LAST_TW = last_tw_count<NSL_LAST, RBL>();
};
// Pass B: a first radix-16 stage from global memory, a middle stage, a last
// stage with its outputs in registers: radix 16 at N2 = 2^8 (no middle stage)
// and 2^12, else at most 8.
template <int L2> struct PlanB {
  static constexpr int RB0 = 4;
  static constexpr int RBL = L2 == 8 || L2 == 12 ? 4 : (L2 - RB0 >= 3 ? 3 : L2 - RB0);
  static constexpr int NSL_LAST = L2 - RBL;
  static constexpr int RADL = 1 << RBL;
  static constexpr int NS = (1 << L2) / RADL;
  static constexpr int MID_TW = mid_tw_count(NSL_LAST - RB0);
  static constexpr int LAST_TW = last_tw_count<NSL_LAST, RBL>();
};
template <typename R, int L1, int C> constexpr size_t cols_smem() {
  using P = PlanA<L1>;
  return (size_t)C * FftGeom<L1, C>::STRIDE * sizeof(Pair<R>) +
         (size_t)(P::MID_TW + P::LAST_TW + C * (P::NS + P::RADL)) * sizeof(cpx<R>);
}
template <typename R, int L2, int RR> constexpr size_t rows_smem() {
  using P = PlanB<L2>;
  return (size_t)RR * FftGeom<L2, RR>::STRIDE * sizeof(Pair<R>) + (size_t)(P::MID_TW + P::LAST_TW) * sizeof(cpx<R>);
}

// f(u) for the units u < COUNT of a block of NT threads.
template <int COUNT, int NT, typename F>
__device__ __forceinline__ void each_unit(F&& f) {
  if constexpr (COUNT == NT) {
    f((int)threadIdx.x);
  } else {
#pragma unroll 1
    for (int u = threadIdx.x; u < COUNT; u += NT) f(u);
  }
}

// --------------------------------------------------------------- pass A

// Stage twiddle tables of pass A, the same for every tile of one shape
// (all threads of the block; read after a barrier).
template <typename R, int L1, int C, int NT>
__device__ __forceinline__ void cols_tables(const Tw<R>& tw, Pair<R>* buf) {
  using PA = PlanA<L1>;
  cpx<R>* tws = reinterpret_cast<cpx<R>*>(buf + C * FftGeom<L1, C>::STRIDE);
  build_mid_tw<R, L1, PA::NSL_LAST - 4, NT>(tws, tw.tl[L1]);
  build_last_tw<R, L1, PA::NSL_LAST, PA::RBL, NT>(tws + PA::MID_TW, tw.tl[L1]);
}

// One column tile of pass A for template t (all threads of the block; the
// stage tables from cols_tables).  za: this template's intermediate.
//
// Per point of a series (N1 = 2^12) the three radix-16 stages are about 50
// FP32 instructions; carrying both series in one thread halves what is
// around them: twiddle loads and products, addresses, and the load, store
// and shared-memory instructions (16 bytes each instead of 8).
template <typename R, int L1, int C, int NT, int SRC, int TAPS>
__device__ __forceinline__ void cols_tile(const ColsArgs<R>& a, int t, int tile, Pair<R>* __restrict__ buf,
                                          double* red, Pair<R>* __restrict__ za, int RRr, int lr) {
  using Cx = cpx<R>;
  using Knot = typename KnotOf<R>::T;
  constexpr int N1 = 1 << L1;
  constexpr int STRIDE = FftGeom<L1, C>::STRIDE;
  const TmplMeta& m = a.c.meta[t];
  const int L = m.log2n;
  const int N2 = 1 << (L - L1);
  const int tiles = N2 / C;
  const int c0 = tile * C;
  const int n_b = (int)m.n_b;
  const Knot* kn = reinterpret_cast<const Knot*>(a.c.knots) + (int64_t)t * a.c.knot_stride;
  R pA = 0, pB = 0, pC = 0;
  // twiddle tables (cols_tables); this tile's inter-pass factors are
  // written here and read after the barriers that end the fill
  using PA = PlanA<L1>;
  using F = FftPlan<L1, PA::RBL, C>;
  constexpr int NSL_LAST = PA::NSL_LAST;
  constexpr int RADL = PA::RADL;
  constexpr int NS = PA::NS;
  Cx* tws = reinterpret_cast<Cx*>(buf + C * STRIDE);   // shared-memory stages
  Cx* tlast = tws + PA::MID_TW;           // last stage, rows of powers
  Cx* ta = tlast + PA::LAST_TW;           // [c][j]: W_N^{j (c0 + c)}, j < NS
  Cx* tb = ta + C * NS;                   // [c][q]: W_N^{q NS (c0 + c)}, q < RADL
  auto factors = [&] {
#pragma unroll
    for (int e0 = 0; e0 < C * NS; e0 += NT) {
      const int e = e0 + threadIdx.x;
      if (C * NS % NT == 0 || e < C * NS)
        ta[e] = twiddle<R>(a.tw, L, (uint32_t)(e & (NS - 1)) * (uint32_t)(c0 + e / NS));
    }
    for (int e = threadIdx.x; e < C * RADL; e += NT)
      tb[e] = twiddle<R>(a.tw, L, (uint32_t)((e & (RADL - 1)) * NS) * (uint32_t)(c0 + e / RADL));
  };
  if constexpr (loads(SRC)) {
    // the tiled resampler's order W[k2 / C][k1][k2 % C]: this tile's C * N1
    // pairs are contiguous, pair i = c + C k1 at offset i
    const Pair<R>* w_in = reinterpret_cast<const Pair<R>*>(a.c.wa) + (int64_t)t * a.c.z_stride +
                          (int64_t)tile * (C * N1);
    // first radix-16 stage straight from the resampled series: unit
    // (j, column) with the column fastest, so that the lanes of a
    // warp read consecutive values
    constexpr int Q1 = N1 / 16;
    each_unit<C * Q1, NT>([&](int u) {
      const int c = u & (C - 1);
      const int j = u / C;
      const Pair<R>* src = w_in + c + j * C;
      // points k = c0 + c + (j + r Q1) N2 < n_b: r below nr
      const int step = Q1 * N2;                        // N / 16
      const int left = n_b - (c0 + c + j * N2);
      const int nr = left > 0 ? (left + step - 1) >> (L - 4) : 0;
      Cx va[16], vb[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        Pair<R> v{czero<Cx>(), czero<Cx>()};
        if (r < nr) v = ldcs(src + r * (Q1 * C));
        va[r] = v.a;
        vb[r] = v.b;
      }
      // behind the loads: the table look-ups of the factors wait on memory too
      // (64 search templates 1372 -> 1343 us)
      if (u == (int)threadIdx.x) factors();
      Dft<Cx, 16>::run(va);
      Dft<Cx, 16>::run(vb);
      Pair<R>* dst = buf + c * STRIDE;
#pragma unroll
      for (int r = 0; r < 16; ++r) dst[F::place(r, j)] = Pair<R>{va[r], vb[r]};
    });
  } else {
    factors();
    GapCursor gc = make_cursor(m, a.gaps);
#pragma unroll 2
    for (int i = threadIdx.x; i < C * N1; i += NT) {
      const int c = i & (C - 1);
      const int k1 = i / C;
      const int k = c0 + c + k1 * N2;
      Cx va = czero<Cx>(), vb = czero<Cx>();
      if (k < n_b) {
        R aa, bb;
        if (sample_weights<R, SRC == SRC_NN ? FSTAT_NEAREST : FSTAT_SINC, TAPS>(a.pc, kn, k, a.x, gc, a.wcs,
                                                                              va, vb, aa, bb)) {
          pA += aa * aa; pB += bb * bb; pC += aa * bb;
        }
      }
      buf[c * STRIDE + F::place(k1 / F::SUB, k1 & (F::SUB - 1))] = Pair<R>{va, vb};
    }
  }
  if constexpr (!loads(SRC)) {
    double sA, sB, sC;
    block_sum3((float)pA, (float)pB, (float)pC, sA, sB, sC, red);
    double* part = a.c.partials + (int64_t)t * a.c.part_stride * 3;
    if (threadIdx.x == 0) {
      part[3 * tile] = sA; part[3 * tile + 1] = sB; part[3 * tile + 2] = sC;
    }
    finalize_sums(a.c.meta + t, part, tiles, a.c.counters + t, a.pc.sigma2, nullptr, a.status);
  }
  __syncthreads();
  if constexpr (!loads(SRC)) first_stage<R, L1, PA::RBL, NT, C, STRIDE>(buf);
  mid_stage<R, L1, PA::RBL, NT, C, STRIDE>(buf, tws);
  // last stage: inputs from shared memory, outputs X[p1 = j + q NS] stay in
  // registers, are multiplied by W_N^{p1 k2} and stored into Z.  Of that
  // twiddle the factor W_N^{j k2} is common to a butterfly's outputs, so it
  // joins the stage twiddles of the inputs (t[q] = W_N^{j k2} W_N1^{q j}) and
  // only W_N^{q NS k2} multiplies the outputs.  Lanes run over j mod RR, then
  // the column, then j / RR, so that a warp writes runs of RR * C
  // consecutive pairs of Z.
  each_unit<C * NS, NT>([&](int u) {
    const int jr = u & (RRr - 1);
    const int rest = u >> lr;
    const int c = rest & (C - 1);
    const int j = ((rest / C) << lr) + jr;
    Cx xa[RADL], xb[RADL];
    {
      Cx tq[RADL];
      last_twiddles<R, NSL_LAST, PA::RBL>(tlast + j, ta[c * NS + j], tq);
      const int p0 = j & 15, q1 = j >> 4;
      const Pair<R>* src = buf + c * STRIDE + p0 * F::SUB + q1 * RADL;
      const int key = F::key(p0);
#pragma unroll
      for (int q = 0; q < RADL; ++q) {
        const Pair<R> v = src[q ^ key];
        xa[q] = cmul(v.a, tq[q]);
        xb[q] = cmul(v.b, tq[q]);
      }
    }
    Dft<Cx, RADL>::run(xa);
    Dft<Cx, RADL>::run(xb);
    const int k2 = c0 + c;
    // p1 = j + q NS lands at Z[p1 / R][k2][p1 % R]; NS is a multiple of R, so
    // consecutive q are N / RADL elements apart
    Pair<R>* zq;
    int64_t zstep;
    if constexpr (SRC == SRC_INPLACE) {
      // over the tile's own columns, which were read whole above: [k2 / C][p1][k2 % C]
      zq = za + (int64_t)tile * (C * N1) + j * C + c;
      zstep = NS * C;
    } else {
      zq = za + ((((int64_t)(j >> lr) * N2 + k2) << lr) + (j & (RRr - 1)));
      zstep = ((int64_t)1 << L) / RADL;
    }
#pragma unroll
    for (int q = 0; q < RADL; ++q) {
      const Cx w = tb[c * RADL + q];
      *zq = q == 0 ? Pair<R>{xa[q], xb[q]} : Pair<R>{cmul(xa[q], w), cmul(xb[q], w)};
      zq += zstep;
    }
  });
}

// A, B, C of template t and the coefficients of 2F from the resampler's sums
// (one thread of the block that has the template's first column tile; the
// second pass, which needs them, starts after this one).  A template with
// more tiles below n_b than the resampling grid covered (not expected: the
// grid is sized from a bound on n_b) is reported as FSTAT_ERANGE.
template <typename R>
__device__ __forceinline__ void finish_sums(const ColsArgs<R>& a, int t, int l2) {
  TmplMeta* m = a.c.meta + t;
  if (live_tiles(m->n_b, l2) > a.covered) {
    m->status_2f = FSTAT_ERANGE;
    set_status(a.status, FSTAT_ERANGE);
    return;
  }
  constexpr double u = 1.0 / (double)(1ll << kSumBits);
  set_sums(m, u * (double)(long long)m->acc[0], u * (double)(long long)m->acc[1], u * (double)(long long)m->acc[2],
           a.pc.sigma2, nullptr, a.status);
}

// Persistent over the (template, column tile) items of a chunk: the grid is
// sized to the resident blocks, each builds the stage tables once.
template <typename R, int L1, int C, int NT, int SRC, int TAPS>
__global__ void __launch_bounds__(NT, (min_blocks<R>(NT, cols_smem<R, L1, C>()))) k_cols(ColsArgs<R> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[96];
  Pair<R>* buf = reinterpret_cast<Pair<R>*>(smem_raw);
  let_next_start();
  cols_tables<R, L1, C, NT>(a.tw, buf);
  wait_for_previous();
  const int total = a.tiles_max * a.c.nt;
#pragma unroll 1
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const int t = w / a.tiles_max;
    const int tile = w - t * a.tiles_max;
    const TmplMeta& m = a.c.meta[t];
    if constexpr (loads(SRC)) {
      // the rows below n_b of the next tile's resampled block, into L2
      const int wn = w + gridDim.x;
      if (threadIdx.x == 0 && wn < total) {
        const int tn = wn / a.tiles_max;
        const int tilen = wn - tn * a.tiles_max;
        const TmplMeta& mn = a.c.meta[tn];
        const int ln = mn.log2n;
        if (mn.status == FSTAT_OK && tilen < (1 << (ln - L1)) / C) {
          const int64_t first = (int64_t)tilen * C;                        // c0 of that tile
          const int64_t rows = mn.n_b > first ? (mn.n_b - first + (1 << (ln - L1)) - 1) >> (ln - L1) : 0;
          const unsigned bytes = (unsigned)((rows < (1 << L1) ? rows : (1 << L1)) * C * sizeof(Pair<R>));
          if (bytes >= 16)
            prefetch_l2(reinterpret_cast<const Pair<R>*>(a.c.wa) + (int64_t)tn * a.c.z_stride + first * (1 << L1),
                        bytes);
        }
      }
    }
    if (tile >= (1 << (m.log2n - L1)) / C || m.status != FSTAT_OK) continue;
    Pair<R>* za = reinterpret_cast<Pair<R>*>(a.c.za) + (int64_t)t * a.c.z_stride;
    cols_tile<R, L1, C, NT, SRC, TAPS>(a, t, tile, buf, red, za, a.rr, a.log2rr);
    if constexpr (loads(SRC)) {
      if (tile == 0 && threadIdx.x == 0) finish_sums<R>(a, t, m.log2n - L1);
    }
    __syncthreads();                      // the next tile reuses buf and its twiddle factors
  }
}

// --------------------------------------------------------------- pass B

// Stage twiddle tables of pass B (all threads of the block; read after a barrier).
template <typename R, int L2, int RR, int NT>
__device__ __forceinline__ void rows_tables(const Tw<R>& tw, Pair<R>* buf) {
  using PB = PlanB<L2>;
  cpx<R>* tws = reinterpret_cast<cpx<R>*>(buf + RR * FftGeom<L2, RR>::STRIDE);
  build_mid_tw<R, L2, PB::NSL_LAST - PB::RB0, NT>(tws, tw.tl[L2]);
  build_last_tw<R, L2, PB::NSL_LAST, PB::RBL, NT>(tws + PB::MID_TW, tw.tl[L2]);
}

// One row block of pass B for template t (stage tables from rows_tables);
// za: the template's intermediate.
// INPLACE: the intermediate lies in pass A's column order [k2 / C][p1][k2 % C]
// instead of row blocks.
// BAND: the plan writes a partial output band (bins band_lo <= q < band_hi
// only); without it every bin is stored, with no band test.
template <typename R, int L2, int RR, int G, int NT, bool BAND, bool INPLACE>
__device__ __forceinline__ void rows_tile(const RowsArgs<R>& a, int t, int blk, Pair<R>* __restrict__ buf,
                                          const Pair<R>* __restrict__ zbase) {
  using Cx = cpx<R>;
  constexpr int N2 = 1 << L2;
  constexpr int STRIDE = FftGeom<L2, RR>::STRIDE;
  const TmplMeta& m = a.c.meta[t];
  const int L = m.log2n;
  const int N1 = 1 << (L - L2);
  const int r0 = blk * RR;
  float* out = a.out + m.out_off;
  // with BAND, bin q (ascending frequency) goes to out[q - band_lo] when
  // band_lo <= q < band_hi (bins are below 2^24: 32-bit offsets)
  int lo = 0, hi = 0;
  if constexpr (BAND) {
    lo = (int)a.pc.band_lo;
    hi = (int)(a.pc.band_hi < ((int64_t)1 << L) ? a.pc.band_hi : ((int64_t)1 << L));
    out -= lo;
  }
  if (m.status_2f != FSTAT_OK) {
    for (int i = threadIdx.x; i < RR * N2; i += NT) {
      const int r = i & (RR - 1), p2 = i / RR;
      if constexpr (BAND) {
        const int qb = (r0 + r) + N1 * ((p2 + N2 / 2) & (N2 - 1));
        if (qb >= lo && qb < hi) out[qb] = __int_as_float(0x7fc00000);
      } else {
        out[(int64_t)(r0 + r) + (int64_t)N1 * ((p2 + N2 / 2) & (N2 - 1))] = __int_as_float(0x7fc00000);
      }
    }
    return;
  }
  // this block's rows lie in one contiguous run of N2 * G pairs, element
  // (k2, r) at k2 * G + r.  First radix-16 stage straight from there: lanes
  // run over r, then j.
  const Pair<R>* zr = zbase + (int64_t)(r0 / G) * (N2 * G) + (r0 & (G - 1));
  using PB = PlanB<L2>;
  using F = FftPlan<L2, PB::RBL, RR>;
  Cx* tws = reinterpret_cast<Cx*>(buf + RR * STRIDE);   // shared-memory stages (rows_tables)
  Cx* tlast = tws + PB::MID_TW;           // last stage, rows of powers
  constexpr int RB0 = PB::RB0;
  constexpr int RAD0 = 1 << RB0;
  constexpr int Q0 = N2 / RAD0;                   // butterflies per sequence
  each_unit<RR * Q0, NT>([&](int u) {
    const int r = u & (RR - 1);
    const int j = u / RR;
    const Pair<R>* src = zr + r + j * G;
    Cx xa[RAD0], xb[RAD0];
#pragma unroll
    for (int q = 0; q < RAD0; ++q) {
      Pair<R> v;
      if constexpr (INPLACE) {
        const int k2 = j + q * Q0;
        v = ldcs(zbase + ((int64_t)(k2 >> a.log2cols) << (L - L2 + a.log2cols)) + ((r0 + r) << a.log2cols) +
                 (k2 & (a.cols - 1)));
      } else {
        v = ldcs(src + q * (Q0 * G));
      }
      xa[q] = v.a;
      xb[q] = v.b;
    }
    Dft<Cx, RAD0>::run(xa);
    Dft<Cx, RAD0>::run(xb);
    Pair<R>* dst = buf + r * STRIDE;
#pragma unroll
    for (int q = 0; q < RAD0; ++q) dst[F::place(q, j)] = Pair<R>{xa[q], xb[q]};
  });
  __syncthreads();
  // middle stages in shared memory; in the last stage both series of a
  // butterfly are in one thread, so that 2F is formed in registers
  constexpr int NSL_LAST = PB::NSL_LAST;
  mid_stage<R, L2, PB::RBL, NT, RR, STRIDE>(buf, tws);
  R ca, cb, cc;
  if constexpr (std::is_same<R, float>::value) {
    ca = m.ca; cb = m.cb; cc = m.cc;
  } else {
    const double D = m.A * m.B - m.C * m.C;
    const double sc = 1.0 / (a.pc.sigma2 * D);
    ca = 2.0 * m.B * sc; cb = 2.0 * m.A * sc; cc = -4.0 * m.C * sc;
  }
  constexpr int RADL = PB::RADL;
  constexpr int NS = PB::NS;
#pragma unroll 1
  for (int u = threadIdx.x; u < RR * NS; u += NT) {
    const int r = u & (RR - 1);
    const int j = u / RR;
    Cx fa[RADL], fb[RADL];
    {
      Cx tq[RADL];
      last_twiddles<R, NSL_LAST, PB::RBL>(tlast + j, cmk<Cx, R>((R)1, (R)0), tq);
      const int p0 = j & 15, q1 = j >> 4;
      const Pair<R>* src = buf + r * STRIDE + p0 * F::SUB + q1 * RADL;
      const int key = F::key(p0);
#pragma unroll
      for (int q = 0; q < RADL; ++q) {
        const Pair<R> v = src[q ^ key];
        fa[q] = q == 0 ? v.a : cmul(v.a, tq[q]);
        fb[q] = q == 0 ? v.b : cmul(v.b, tq[q]);
      }
    }
    Dft<Cx, RADL>::run(fa);
    Dft<Cx, RADL>::run(fb);
    // p2 = j + q NS goes to row (p2 + N2/2) mod N2: + N2/2 for the first half
    // of q (p2 < N2/2), - N2/2 for the second
    float* oq = out + (int64_t)(r0 + r) + (int64_t)N1 * j;
    const int64_t s1 = (int64_t)N1 * NS, hh = (int64_t)N1 * (N2 / 2);
#pragma unroll
    for (int q = 0; q < RADL; ++q) {
      const R v = ca * (fa[q].x * fa[q].x + fa[q].y * fa[q].y) + cb * (fb[q].x * fb[q].x + fb[q].y * fb[q].y)
                + cc * (fa[q].x * fb[q].x + fa[q].y * fb[q].y);
      if constexpr (BAND) {
        const int qb = (r0 + r) + N1 * j + q * (N1 * NS) + (q < RADL / 2 ? 1 : -1) * (N1 * (N2 / 2));
        if (qb < lo || qb >= hi) continue;
      }
      __stcs(oq + q * s1 + (q < RADL / 2 ? hh : -hh), (float)v);
    }
  }
}

// Persistent over the (template, row block) items of a chunk.
template <typename R, int L2, int RR, int NT, bool BAND, bool INPLACE>
__global__ void __launch_bounds__(NT, (min_blocks<R>(NT, rows_smem<R, L2, RR>()))) k_rows(RowsArgs<R> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Pair<R>* buf = reinterpret_cast<Pair<R>*>(smem_raw);
  rows_tables<R, L2, RR, NT>(a.tw, buf);
  wait_for_previous();
  __syncthreads();
  const int total = a.blocks_max * a.c.nt;
#pragma unroll 1
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const int t = w / a.blocks_max;
    const int blk = w - t * a.blocks_max;
    const TmplMeta& m = a.c.meta[t];
    if constexpr (!INPLACE) {
      // the run of the intermediate that the next row block needs, into L2
      // (by the block that has the run's first rows)
      constexpr int G = rows_group<R>(L2);
      const int wn = w + gridDim.x;
      if (threadIdx.x == 0 && wn < total) {
        const int tn = wn / a.blocks_max;
        const int rn = (wn - tn * a.blocks_max) * RR;
        const int ln = a.c.meta[tn].log2n;
        if (rn < (1 << (ln - L2)) && (rn & (G - 1)) == 0)
          prefetch_l2(reinterpret_cast<const Pair<R>*>(a.c.za) + (int64_t)tn * a.c.z_stride + (int64_t)rn * (1 << L2),
                      (unsigned)((1u << L2) * G * sizeof(Pair<R>)));
      }
    }
    if (blk * RR >= (1 << (m.log2n - L2))) continue;
    const Pair<R>* za = reinterpret_cast<const Pair<R>*>(a.c.za) + (int64_t)t * a.c.z_stride;
    rows_tile<R, L2, RR, rows_group<R>(L2), NT, BAND, INPLACE>(a, t, blk, buf, za);
    __syncthreads();                      // the next block reuses buf
  }
}

}  // namespace fs
