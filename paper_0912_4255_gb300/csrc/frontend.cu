// SFT front end (Sec. III.B): SFTs -> normalised -> merged into the band of
// the long transform (Eq. e9) -> windowed -> inverse transformed -> stitched
// into the heterodyned series.
//
// Eq. e9 is evaluated in an exactly equivalent order.  With b = k* M + r
// (0 <= r < M), e^{-2 pi i b alpha / M} = e^{-2 pi i r alpha / M} and
// P_{b,k} depends on r and j = k - k* only, so
//   X_b = sum_j P(r, j) D_{k*+j}(r),   D_k(r) = sum_alpha X^_{alpha,k} e^{-2 pi i r alpha / M},
// a length-M DFT over the SFT index of every stored bin (k_dft_alpha) and a
// (2 dk + 1)-term sum per output bin (k_merge).  The inverse transform of
// length N_out = N1 M splits the same way (m = kappa M + r, n = n1 + N1 n2):
//   z[n1 + N1 n2] = sum_r e^{2 pi i r n2 / M} e^{2 pi i r n1 / N_out}
//                   sum_kappa Y[r][kappa] e^{2 pi i kappa n1 / N1},
// two passes (over kappa, as mixed-radix stages where N1 = 2^a 3^b 5^c, else
// split as N1 = P Q, and k_idft_n2 over r) with twiddle indices taken exactly in integers.  The lengths (N1 = band bins per SFT,
// M = SFTs per chunk) are arbitrary, not powers of two.
#include "fstat_internal.cuh"

#include <math.h>

#include <vector>

namespace fs {

namespace {

constexpr int kFeThreads = 256;
constexpr int kMaxBins = 32768;      // stored bins per SFT (running median in shared memory)
constexpr int kMaxN1 = 8192;         // band bins per SFT (inverse pass over kappa: 3 rows in shared memory)
constexpr int kMaxWindow = 1023;

// Step 2: X^ = X / sqrt(S), S = (lower) median of |X|^2 over the window / ln 2.
// One block per SFT, |X|^2 of the SFT in shared memory (so that the output
// may take the input's place); every warp slides the window along runs of 64
// bins.  The window's values lie in the lanes' registers, value i at place
// i mod w (S places a lane, an unused one holds kNone), so that the value that
// enters takes the place of the one that leaves; the median m is
// followed by the counts of values below m and up to m: a bin more and a bin
// less move it by at most a neighbour or two, found by one warp reduction
// each.  |X|^2 >= 0, so its bits order as unsigned integers (a NaN, its sign
// cleared, above all numbers).  432 SFTs of 3648 bins, window 101: 907 us
// when every thread kept a sorted window in shared memory and moved half of
// it per bin, 172 us now, bound by instruction issue.
constexpr int kMedThreads = 512;
constexpr int kMedRun = 64;
constexpr unsigned kNone = 0xffffffffu;

template <int S>
__global__ void __launch_bounds__(kMedThreads)
k_normalize(const float2* __restrict__ X, float2* __restrict__ Xh, int K, int w) {
  extern __shared__ unsigned P[];
  const float2* x = X + (int64_t)blockIdx.x * K;
  float2* y = Xh + (int64_t)blockIdx.x * K;
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    const float2 v = x[k];
    P[k] = __float_as_uint(v.x * v.x + v.y * v.y) & 0x7fffffffu;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int h = w / 2;
  for (int k0 = (threadIdx.x >> 5) * kMedRun; k0 < K; k0 += (kMedThreads / 32) * kMedRun) {
    unsigned v[S];
    auto below = [&](unsigned m) {                 // values below m
      unsigned c = 0;
#pragma unroll
      for (int i = 0; i < S; ++i) c += v[i] < m;
      return (int)__reduce_add_sync(0xffffffffu, c);
    };
    const int lo0 = max(0, k0 - h), hi0 = min(K, k0 + h + 1);
    const int first = lo0 % w;
#pragma unroll
    for (int i = 0; i < S; ++i) {
      const int place = lane + 32 * i;
      const int e = lo0 + (place >= first ? place - first : place - first + w);   // the value of this place
      v[i] = place < w && e < hi0 ? P[e] : kNone;
    }
    int t = (hi0 - lo0 - 1) / 2;                   // rank of the (lower) median
    int place = (k0 + h + 1) % w;                  // of the next value to enter
    unsigned m = 0;
#pragma unroll 1
    for (int bit = 30; bit >= 0; --bit)
      if (below(m | (1u << bit)) <= t) m |= 1u << bit;
    int lt = below(m), le = below(m + 1);
    unsigned med = 0;
    const int k1 = min(K, k0 + kMedRun);
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
      if (k > k0) {
        const int ro = k - h - 1, ni = k + h;      // the value that leaves, and the one that enters
        const unsigned vo = ro >= 0 ? P[ro] : kNone, vn = ni < K ? P[ni] : kNone;
        lt += (int)(vn < m) - (int)(vo < m);
        le += (int)(vn <= m) - (int)(vo <= m);
        const bool mine = lane == (place & 31);
        const int reg = place >> 5;
#pragma unroll
        for (int i = 0; i < S; ++i)
          if (mine && i == reg) v[i] = vn;
        if (++place == w) place = 0;
        t = (min(K, ni + 1) - max(0, ro + 1) - 1) / 2;
        while (t < lt) {                           // the largest value below m
          unsigned c = 0;
#pragma unroll
          for (int i = 0; i < S; ++i) c = v[i] < m && v[i] > c ? v[i] : c;
          m = __reduce_max_sync(0xffffffffu, c);
          le = lt;
          lt = below(m);
        }
        while (t >= le) {                          // the smallest value above m
          unsigned c = kNone;
#pragma unroll
          for (int i = 0; i < S; ++i) c = v[i] > m && v[i] < c ? v[i] : c;
          m = __reduce_min_sync(0xffffffffu, c);
          lt = le;
          le = below(m + 1);
        }
      }
      if (lane == (k & 31)) med = m;
      if ((k & 31) == 31 || k + 1 == k1) {
        const int kk = (k & ~31) + lane;
        if (kk <= k) {
          // 1 / sqrt(median / ln 2); a zero estimate (a window of zeros) gives zero
          const float mf = __uint_as_float(med);
          const float sc = mf > 0.f ? rsqrtf(mf * 1.4426950408889634f) : 0.f;
          const float2 q = x[kk];
          y[kk] = make_float2(q.x * sc, q.y * sc);
        }
      }
    }
  }
}

template <int S>
cudaError_t run_normalize(const float2* X, float2* Xh, int64_t n_sft, int K, int w, cudaStream_t s) {
  static DeviceOnce once;
  const cudaError_t e = kernel_setup(once, k_normalize<S>, kMedThreads, (size_t)kMaxBins * 4, nullptr);
  if (e != cudaSuccess) return e;
  k_normalize<S><<<(unsigned)n_sft, kMedThreads, (size_t)K * 4, s>>>(X, Xh, K, w);
  return cudaGetLastError();
}

// The same for short windows: a thread takes a run of consecutive bins and keeps
// its window sorted in a column of shared memory ([j][thread]), one removal and
// one insertion a bin.  The same element of the same multiset, in the same order.
__global__ void __launch_bounds__(kFeThreads)
k_normalize_sorted(const float2* __restrict__ X, float2* __restrict__ Xh, int K, int w) {
  extern __shared__ unsigned P[];
  const float2* x = X + (int64_t)blockIdx.x * K;
  float2* y = Xh + (int64_t)blockIdx.x * K;
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    const float2 v = x[k];
    P[k] = __float_as_uint(v.x * v.x + v.y * v.y) & 0x7fffffffu;
  }
  __syncthreads();
  const int h = w / 2;
  const int run = (K + kFeThreads - 1) / kFeThreads;
  const int k0 = threadIdx.x * run, k1 = min(K, k0 + run);
  if (k0 >= k1) return;
  unsigned* win = P + K + threadIdx.x;             // element j at win[j * kFeThreads]
  int cnt = 0;
  auto insert = [&](unsigned v) {
    int j = cnt;
    while (j > 0 && win[(j - 1) * kFeThreads] > v) { win[j * kFeThreads] = win[(j - 1) * kFeThreads]; --j; }
    win[j * kFeThreads] = v;
    ++cnt;
  };
  auto remove = [&](unsigned v) {
    int j = 0;
    while (j < cnt - 1 && win[j * kFeThreads] != v) ++j;
    for (; j < cnt - 1; ++j) win[j * kFeThreads] = win[(j + 1) * kFeThreads];
    --cnt;
  };
  for (int i = max(0, k0 - h); i < min(K, k0 + h + 1); ++i) insert(P[i]);
  for (int k = k0; k < k1; ++k) {
    if (k > k0) {
      if (k - h - 1 >= 0) remove(P[k - h - 1]);
      if (k + h < K) insert(P[k + h]);
    }
    const float med = __uint_as_float(win[((cnt - 1) / 2) * kFeThreads]);
    const float sc = med > 0.f ? rsqrtf(med * 1.4426950408889634f) : 0.f;
    const float2 v = x[k];
    y[k] = make_float2(v.x * sc, v.y * sc);
  }
}

size_t sorted_smem(int K, int w) { return ((size_t)K + (size_t)kFeThreads * (size_t)w) * sizeof(unsigned); }

// Whether the sorted windows are faster, by the time of each in microseconds
// (windows of 1 .. 61, bands of 200 .. 32000 bins, 1 .. 2000 SFTs, within 15 %
// of the fits).  Sorted: a thread's first window costs the square of its length,
// a bin its length, and shared memory limits the blocks that run at once.
// Counts: a warp's runs of 64 bins one after another, 16 warps a block; a
// second block on an SM already shares its issue slots.  (sorted | counts) 432
// SFTs of 3648 bins, window 5 22 | 150, 31 74 | 148, 51 136 | 148, 61 307 | 148; 20 of 932
// bins, window 5 9 | 19, 31 31 | 19.
bool sorted_is_faster(int64_t n_sft, int K, int w) {
  const size_t smem = sorted_smem(K, w);
  if (w > 63 || smem > 200 * 1024) return false;
  const int run = (K + kFeThreads - 1) / kFeThreads;
  const size_t room = 228 * 1024 / (smem + 1024);
  const int64_t at_once = 152 * (int64_t)(room < 8 ? room : 8);
  const double waves = (double)((n_sft + at_once - 1) / at_once);
  const double sorted = waves * (4.0 + 0.0185 * w * w + (run - 1) * (0.3 + 0.095 * w));
  const double shared = 3.0 + 12.2 * (double)n_sft / 152.0;
  const double counts = ((K + 1023) / 1024) * (shared > 16.0 ? shared : 16.0);
  return 1.06 * sorted < counts;
}

// Step 2 on n_sft SFTs: sorted windows or, by the window's places per lane, counts.
cudaError_t launch_normalize(const float2* X, float2* Xh, int64_t n_sft, int K, int w, cudaStream_t s) {
  if (sorted_is_faster(n_sft, K, w)) {
    static DeviceOnce once;
    const cudaError_t e = kernel_setup(once, k_normalize_sorted, kFeThreads, (size_t)200 * 1024, nullptr);
    if (e != cudaSuccess) return e;
    k_normalize_sorted<<<(unsigned)n_sft, kFeThreads, sorted_smem(K, w), s>>>(X, Xh, K, w);
    return cudaGetLastError();
  }
  if (w <= 32 * 2) return run_normalize<2>(X, Xh, n_sft, K, w, s);
  if (w <= 32 * 4) return run_normalize<4>(X, Xh, n_sft, K, w, s);
  if (w <= 32 * 8) return run_normalize<8>(X, Xh, n_sft, K, w, s);
  return run_normalize<32>(X, Xh, n_sft, K, w, s);
}

// The chunks of one launch (passed by value: no copy to the device, and a
// captured launch keeps its own table).  Chunks partition consecutive SFTs,
// so every per-SFT row (of D, Y, U and the M-tables) is addressed by its
// global SFT index g; chunk c holds rows a[c] .. a[c] + m[c] - 1.
constexpr int kChunksPerLaunch = 32;
constexpr int kN2PerBlock = 32;        // y-blocks of k_dft_alpha and k_idft_n2 cover 32 r or n2 each
struct ChunkTab {
  int n;                               // chunks in this launch
  int rows;                            // SFTs they hold: a[0] .. a[0] + rows - 1
  int a[kChunksPerLaunch], m[kChunksPerLaunch];
  int yb[kChunksPerLaunch + 1];        // prefix sums of ceil(m / 32)
  long long off[kChunksPerLaunch];     // output offset of the chunk
  float gc[kChunksPerLaunch], gs[kChunksPerLaunch];   // chunk factor e^{-2 pi i f_h (t_c - t_s)}
  float sc[kChunksPerLaunch];          // 1 / sqrt(M N_out)
};

__device__ __forceinline__ int chunk_of_row(const ChunkTab& t, int g) {
  int c = 0;
  while (c + 1 < t.n && g >= t.a[c] + t.m[c]) ++c;
  return c;
}
__device__ __forceinline__ int chunk_of_yblock(const ChunkTab& t, int y) {
  int c = 0;
  while (c + 1 < t.n && y >= t.yb[c + 1]) ++c;
  return c;
}

// Twiddle tables: tm[g] = (cos, sin, 1 - cos) of 2 pi j / M for row g = a + j
// of a chunk of M SFTs, tn[j] = (cos, sin) of 2 pi j / N1, from FP64.
__global__ void k_tables(ChunkTab tab, float4* __restrict__ tm, float2* __restrict__ tn, int N1) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < tab.rows) {
    const int g = tab.a[0] + i;
    const int c = chunk_of_row(tab, g);
    const int j = g - tab.a[c], M = tab.m[c];
    double s, co, sh, ch;
    sincospi(2.0 * j / M, &s, &co);
    sincospi((double)j / M, &sh, &ch);
    tm[g] = make_float4((float)co, (float)s, (float)(2.0 * sh * sh), 0.f);
  }
  if (i < N1) {
    double s, co;
    sincospi(2.0 * i / N1, &s, &co);
    tn[i] = make_float2((float)co, (float)s);
  }
}

// The length-M DFT over the SFTs of a chunk, in either direction:
//   out[r][c] = sum_a in[a][c] e^{-+2 pi i r a / M},
// rows of `ld` values.  A block takes 32 r and 128 columns, a warp 8 r and 64
// columns (two a lane), so that a row of input is read once per 8 outputs and
// a twiddle, staged in shared memory for 32 a at a time, serves 64 columns:
// with one column a lane and the index (r a) mod M stepped per product, the
// integer work was as large as the products'.  Both passes of 432 SFTs: 57 +
// 84 us then.  grid (ceil(columns / 128), yb[n]).
constexpr int kDftA = 32, kDftR = kN2PerBlock, kDftCols = 128, kDftPerWarp = 8;
template <bool INVERSE, typename F>
__device__ __forceinline__ void dft_tile(const float2* __restrict__ in, int M, int ncol, const float4* __restrict__ tm,
                                         int r_base, F&& out) {
  __shared__ __align__(16) float2 tw[kDftA][kDftR];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rw = (warp & 3) * kDftPerWarp;
  const int c0 = blockIdx.x * kDftCols + (warp >> 2) * 64 + lane, c1 = c0 + 32;
  float2 acc[2][kDftPerWarp];
#pragma unroll
  for (int q = 0; q < kDftPerWarp; ++q) acc[0][q] = acc[1][q] = make_float2(0.f, 0.f);
  for (int a0 = 0; a0 < M; a0 += kDftA) {
    const int an = min(kDftA, M - a0);
    __syncthreads();
    for (int e = threadIdx.x; e < an * kDftR; e += kFeThreads) {
      const unsigned r = r_base + (e & (kDftR - 1)), a = a0 + e / kDftR;
      const float4 t = __ldg(tm + (r * a) % (unsigned)M);       // r a < 2^32 for M <= 65535
      tw[e / kDftR][e & (kDftR - 1)] = make_float2(t.x, INVERSE ? t.y : -t.y);
    }
    __syncthreads();
    if (r_base + rw < M) {
#pragma unroll 4
      for (int a = 0; a < an; ++a) {
        const float2* row = in + (int64_t)(a0 + a) * ncol;
        const float2 v0 = c0 < ncol ? __ldg(row + c0) : make_float2(0.f, 0.f);
        const float2 v1 = c1 < ncol ? __ldg(row + c1) : make_float2(0.f, 0.f);
        const float4* tq = reinterpret_cast<const float4*>(&tw[a][rw]);
#pragma unroll
        for (int q = 0; q < kDftPerWarp; q += 2) {
          const float4 t = tq[q / 2];
          acc[0][q].x += v0.x * t.x - v0.y * t.y;     acc[0][q].y += v0.x * t.y + v0.y * t.x;
          acc[1][q].x += v1.x * t.x - v1.y * t.y;     acc[1][q].y += v1.x * t.y + v1.y * t.x;
          acc[0][q + 1].x += v0.x * t.z - v0.y * t.w; acc[0][q + 1].y += v0.x * t.w + v0.y * t.z;
          acc[1][q + 1].x += v1.x * t.z - v1.y * t.w; acc[1][q + 1].y += v1.x * t.w + v1.y * t.z;
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < kDftPerWarp; ++q) {
    const int r = r_base + rw + q;
    if (r >= M) break;
    if (c0 < ncol) out(r, c0, acc[0][q]);
    if (c1 < ncol) out(r, c1, acc[1][q]);
  }
}

// Step 4a: D[r][k] = sum_alpha Xh[alpha][k] e^{-2 pi i r alpha / M} per
// chunk (rows a + r of D).
__global__ void __launch_bounds__(kFeThreads)
k_dft_alpha(ChunkTab tab, const float2* __restrict__ Xh0, int K, const float4* __restrict__ tm0,
            float2* __restrict__ D0) {
  const int ch = chunk_of_yblock(tab, blockIdx.y);
  float2* D = D0 + (int64_t)tab.a[ch] * K;
  dft_tile<false>(Xh0 + (int64_t)tab.a[ch] * K, tab.m[ch], K, tm0 + tab.a[ch],
                  (blockIdx.y - tab.yb[ch]) * kDftR, [&](int r, int k, float2 v) { D[(int64_t)r * K + k] = v; });
}

// Step 4b + the Tukey window of step 5: for m = kappa M + r,
// Y[r][kappa + N1/2] = w_m sum_{j=-dk}^{dk} P(r, j) D[r][k_s + j],
// k_s = k_het - k_lo + kappa (rows a + r of D and Y).  grid (ceil(N1 / 256), rows).
constexpr int kMergeTerms = 128;       // reciprocals kept at a time
__global__ void __launch_bounds__(kFeThreads)
k_merge(ChunkTab tab, const float2* __restrict__ D, int K, int N1, int ks0, int dk, const float4* __restrict__ tm0,
        double tukey_e, float tukey_ef, float2* __restrict__ Y0) {
  const int g = tab.a[0] + blockIdx.y;
  const int ch = chunk_of_row(tab, g);
  const int M = tab.m[ch];
  const int r = g - tab.a[ch];
  const float4* tm = tm0 + tab.a[ch];
  float2* Y = Y0 + (int64_t)tab.a[ch] * N1;
  // 1 / y of every kernel term depends on r and j only: one division per term
  // and block
  __shared__ float iy[kMergeTerms];
  const float4 t = __ldg(tm + r);
  const float sn = t.y, omc = t.z;            // sin theta, 1 - cos theta
  const float th = 6.283185307179586f * ((float)r / (float)M);
  const int kp = blockIdx.x * blockDim.x + threadIdx.x;      // kappa + N1/2
  const int kappa = kp - N1 / 2;
  const int ks = ks0 + kappa;
  const float2* d = D + (int64_t)g * K;
  float2 acc = make_float2(0.f, 0.f);
  if (r == 0) {
    if (kp < N1) acc = __ldg(d + ks);         // y = 0 only at j = 0; P = 0 at the other SFT bins
  } else {
    float2 sum = make_float2(0.f, 0.f);
    for (int j0 = -dk; j0 <= dk; j0 += kMergeTerms) {
      const int n = min(kMergeTerms, dk + 1 - j0);
      __syncthreads();
      for (int i = threadIdx.x; i < n; i += blockDim.x) iy[i] = 1.0f / (th - 6.283185307179586f * (float)(j0 + i));
      __syncthreads();
      if (kp < N1) {
#pragma unroll 8
        for (int i = 0; i < n; ++i) {
          const float2 v = __ldg(d + ks + j0 + i);
          sum.x = fmaf(v.x, iy[i], sum.x);
          sum.y = fmaf(v.y, iy[i], sum.y);
        }
      }
    }
    // P = (sin theta - i (1 - cos theta)) / y
    acc = make_float2(sum.x * sn + sum.y * omc, sum.y * sn - sum.x * omc);
  }
  if (kp >= N1) return;
  // Tukey window over x = (i + 1/2) / N_out, i = m + N_out / 2; whole numbers
  // decide where it is flat (to one sample), FP64 only in the tapers
  const int64_t n_out = (int64_t)N1 * M;
  const int64_t i = (int64_t)kappa * M + r + n_out / 2;
  float w = 1.f;
  const int64_t edge = (int64_t)(tukey_ef * (float)n_out) + 1 + (n_out >> 20);
  if (tukey_e > 0.0 && (i <= edge || i >= n_out - 1 - edge)) {
    const double x = ((double)i + 0.5) / (double)n_out;
    if (x < tukey_e) w = (float)(0.5 * (1.0 - cospi(x / tukey_e)));
    else if (x > 1.0 - tukey_e) w = (float)(0.5 * (1.0 - cospi((1.0 - x) / tukey_e)));
  }
  Y[(int64_t)r * N1 + kp] = make_float2(acc.x * w, acc.y * w);
}

// Step 5, first pass: U[r][n1] = e^{2 pi i r n1 / N_out} (-1)^{n1}
// sum_{kp} Y[r][kp] e^{2 pi i kp n1 / N1}  (kp = kappa + N1/2).  One block per
// r, the row in shared memory.  The factor e^{2 pi i r n1 / N_out} is the
// product of one of 64 and one of N1/64 factors formed in FP64 once per block
// (its sine and cosine point by point were most of this pass's FP64 work).
constexpr int kRotLo = 64;
__device__ __forceinline__ void row_rotations(float2* __restrict__ rot, int r, int N1, int64_t n_out) {
  const int hi = (N1 + kRotLo - 1) / kRotLo;
  for (int i = threadIdx.x; i < kRotLo + hi; i += blockDim.x) {
    const int64_t n = i < kRotLo ? i : (int64_t)(i - kRotLo) * kRotLo;
    double s, c;
    sincospi(2.0 * (double)(((int64_t)r * n) % n_out) / (double)n_out, &s, &c);
    rot[i] = make_float2((float)c, (float)s);
  }
}
__device__ __forceinline__ float2 row_factor(const float2* __restrict__ rot, int n1) {
  const float2 f = cmul(rot[n1 % kRotLo], rot[kRotLo + n1 / kRotLo]);
  return (n1 & 1) ? make_float2(-f.x, -f.y) : f;   // e^{-pi i n1} from kappa = kp - N1/2
}

// In-register DFT of P points, e^{+2 pi i jk/P}, P = 2, 3, 4, 5.
template <int P>
__device__ __forceinline__ void dft_small(float2 (&v)[P]) {
  if constexpr (P == 2) {
    const float2 a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
  } else if constexpr (P == 4) {
    const float2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
    v[0] = cadd(a, c);
    v[2] = csub(a, c);
    v[1] = make_float2(b.x - d.y, b.y + d.x);      // b + i d
    v[3] = make_float2(b.x + d.y, b.y - d.x);
  } else {
    // pairs (j, P - j): sums s_j and differences d_j; output k is
    // v0 + sum_j cos(2 pi jk / P) s_j + i sum_j sin(2 pi jk / P) d_j
    constexpr int H = (P - 1) / 2;
    constexpr float cs3[2] = {-0.5f, 0.f}, sn3[2] = {0.866025403784438647f, 0.f};
    constexpr float cs5[3] = {0.f, 0.309016994374947424f, -0.809016994374947424f};
    constexpr float sn5[3] = {0.f, 0.951056516295153572f, 0.587785252292473129f};
    float2 s[H], d[H];
#pragma unroll
    for (int j = 0; j < H; ++j) { s[j] = cadd(v[j + 1], v[P - 1 - j]); d[j] = csub(v[j + 1], v[P - 1 - j]); }
    const float2 v0 = v[0];
#pragma unroll
    for (int j = 0; j < H; ++j) v[0] = cadd(v[0], s[j]);
#pragma unroll
    for (int k = 1; k <= H; ++k) {
      float2 e = v0, o = make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 1; j <= H; ++j) {
        const int m = (j * k) % P, mm = m <= H ? m : P - m;
        const float c = P == 3 ? cs3[0] : cs5[mm];
        const float sa = P == 3 ? sn3[0] : sn5[mm];
        const float sg = m <= H ? sa : -sa;
        e.x = fmaf(c, s[j - 1].x, e.x); e.y = fmaf(c, s[j - 1].y, e.y);
        o.x = fmaf(sg, d[j - 1].x, o.x); o.y = fmaf(sg, d[j - 1].y, o.y);
      }
      v[k] = make_float2(e.x - o.y, e.y + o.x);    // e + i o
      v[P - k] = make_float2(e.x + o.y, e.y - o.x);
    }
  }
}

// One Stockham stage of radix P after sub-transforms of length ns.
template <int P>
__device__ __forceinline__ void radix_stage(const float2* __restrict__ in, float2* __restrict__ out, int N1, int ns,
                                            const float2* __restrict__ ts) {
  const int q = N1 / P, tstep = q / ns;            // W_{ns P}^{r k} = table[r k N1 / (ns P)]
  for (int j = threadIdx.x; j < q; j += blockDim.x) {
    const int blk = j / ns, k = j - blk * ns;
    float2 v[P];
#pragma unroll
    for (int r = 0; r < P; ++r) v[r] = in[j + r * q];
#pragma unroll
    for (int r = 1; r < P; ++r) v[r] = cmul(v[r], ts[r * k * tstep]);
    dft_small<P>(v);
    float2* o = out + blk * ns * P + k;
#pragma unroll
    for (int r = 0; r < P; ++r) o[r * ns] = v[r];
  }
  __syncthreads();
}

// N1 = 2^a 3^b 5^c: Stockham stages of radix 4, 2, 3 and 5 between two rows of
// shared memory; four bits of `plan` a radix, the first stage lowest (N1 <=
// 8192 has at most eight of them).  N1 = 3600 takes 6 stages, about 60
// operations a point, where two short DFTs of 60 points took 960.
__global__ void __launch_bounds__(kFeThreads)
k_idft_n1_smooth(ChunkTab tab, const float2* __restrict__ Y, int N1, unsigned long long plan,
                 const float2* __restrict__ tn, float2* __restrict__ U) {
  extern __shared__ float2 sm[];
  float2* cur = sm;
  float2* nxt = sm + N1;
  float2* ts = sm + 2 * N1;
  float2* rot = sm + 3 * N1;
  const int g = tab.a[0] + blockIdx.x;          // global row; r within its chunk
  const int ch = chunk_of_row(tab, g);
  const int M = tab.m[ch];
  const int r = g - tab.a[ch];
  for (int i = threadIdx.x; i < N1; i += blockDim.x) {
    cur[i] = __ldg(Y + (int64_t)g * N1 + i);
    ts[i] = __ldg(tn + i);
  }
  row_rotations(rot, r, N1, (int64_t)N1 * M);
  __syncthreads();
  int ns = 1;
  for (unsigned long long pl = plan; pl; pl >>= 4) {
    const int p = (int)(pl & 15);
    if (p == 4) radix_stage<4>(cur, nxt, N1, ns, ts);
    else if (p == 2) radix_stage<2>(cur, nxt, N1, ns, ts);
    else if (p == 3) radix_stage<3>(cur, nxt, N1, ns, ts);
    else radix_stage<5>(cur, nxt, N1, ns, ts);
    ns *= p;
    float2* x = cur; cur = nxt; nxt = x;
  }
  for (int i = threadIdx.x; i < N1; i += blockDim.x) U[(int64_t)g * N1 + i] = cmul(cur[i], row_factor(rot, i));
}

// Radix plan of N1, or 0 if it has another prime factor.
unsigned long long radix_plan(int N1) {
  unsigned long long plan = 0;
  int shift = 0, n = N1;
  for (int p : {4, 2, 3, 5})
    while (n % p == 0) {
      plan |= (unsigned long long)p << shift;
      shift += 4;
      n /= p;
    }
  return n == 1 ? plan : 0;
}

// Other N1: two short DFTs with N1 = P Q (kp = Q k1 + k2, n1 = na + P nb):
//   V[k2][na] = e^{2 pi i k2 na / N1} sum_{k1 < P} Y[Q k1 + k2] e^{2 pi i k1 na / P},
//   sum = sum_{k2 < Q} V[k2][na] e^{2 pi i k2 nb / Q},
// N1 (P + Q) products per r instead of N1^2.  The P- and Q-point twiddles
// are every Q-th and P-th entry of the N1-table.
__global__ void __launch_bounds__(kFeThreads)
k_idft_n1(ChunkTab tab, const float2* __restrict__ Y, int N1, int P, const float2* __restrict__ tn,
          float2* __restrict__ U) {
  extern __shared__ float2 sm[];
  float2* ys = sm;
  float2* vs = sm + N1;
  float2* ts = sm + 2 * N1;
  float2* rot = sm + 3 * N1;
  const int Q = N1 / P;
  const int g = tab.a[0] + blockIdx.x;          // global row; r within its chunk
  const int ch = chunk_of_row(tab, g);
  const int M = tab.m[ch];
  const int r = g - tab.a[ch];
  for (int i = threadIdx.x; i < N1; i += blockDim.x) {
    ys[i] = __ldg(Y + (int64_t)g * N1 + i);
    ts[i] = __ldg(tn + i);
  }
  row_rotations(rot, r, N1, (int64_t)N1 * M);
  __syncthreads();
  for (int i = threadIdx.x; i < N1; i += blockDim.x) {
    const int k2 = i / P, na = i - k2 * P;
    float2 acc = make_float2(0.f, 0.f);
    int idx = 0;                                   // (k1 na) mod P
    for (int k1 = 0; k1 < P; ++k1) {
      const float2 y = ys[Q * k1 + k2], t = ts[idx * Q];
      acc.x += y.x * t.x - y.y * t.y;
      acc.y += y.x * t.y + y.y * t.x;
      idx += na;
      if (idx >= P) idx -= P;
    }
    const float2 t = ts[k2 * na];                  // k2 na < N1
    vs[i] = make_float2(acc.x * t.x - acc.y * t.y, acc.x * t.y + acc.y * t.x);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < N1; i += blockDim.x) {
    const int nb = i / P, na = i - nb * P;
    const int n1 = na + P * nb;
    float2 acc = make_float2(0.f, 0.f);
    int idx = 0;                                   // (k2 nb) mod Q
    for (int k2 = 0; k2 < Q; ++k2) {
      const float2 v = vs[k2 * P + na], t = ts[idx * P];
      acc.x += v.x * t.x - v.y * t.y;
      acc.y += v.x * t.y + v.y * t.x;
      idx += nb;
      if (idx >= Q) idx -= Q;
    }
    U[(int64_t)g * N1 + n1] = cmul(acc, row_factor(rot, n1));
  }
}

// Step 5, second pass, and step 6: x_h[off + n1 + N1 n2] =
// g taper(n) / sqrt(M N_out) sum_r U[r][n1] e^{2 pi i r n2 / M}.
__global__ void __launch_bounds__(kFeThreads)
k_idft_n2(ChunkTab tab, const float2* __restrict__ U0, int N1, const float4* __restrict__ tm0, int64_t taper,
          float2* __restrict__ x) {
  const int ch = chunk_of_yblock(tab, blockIdx.y);
  const int M = tab.m[ch];
  const float scale = tab.sc[ch], gc = tab.gc[ch], gs = tab.gs[ch];
  const int64_t off = tab.off[ch];
  const int64_t n_out = (int64_t)N1 * M;
  const int64_t e = taper < n_out / 2 ? taper : n_out / 2;
  dft_tile<true>(U0 + (int64_t)tab.a[ch] * N1, M, N1, tm0 + tab.a[ch], (blockIdx.y - tab.yb[ch]) * kDftR,
                 [&](int n2, int n1, float2 v) {
    const int64_t n = n1 + (int64_t)N1 * n2;
    float g = scale;
    if (e > 0) {
      if (n < e) g *= (float)(0.5 * (1.0 - cospi(((double)n + 0.5) / (double)e)));
      else if (n >= n_out - e) g *= (float)(0.5 * (1.0 - cospi(((double)(n_out - 1 - n) + 0.5) / (double)e)));
    }
    const float re = v.x * gc - v.y * gs, im = v.x * gs + v.y * gc;
    x[off + n] = make_float2(re * g, im * g);
  });
}

size_t a256(size_t v) { return (v + 255) & ~(size_t)255; }

struct FeLayout {
  size_t xh, d, y, u, tm, tn, total;
};

FeLayout layout(const fstat_sft_desc& d, int64_t n_sft) {
  FeLayout l;
  const size_t K = (size_t)d.n_bins, N1 = (size_t)d.band_bins, M = (size_t)n_sft;
  l.xh = 0;
  l.d = l.xh + a256(M * K * 8);
  l.y = l.d + a256(K * M * 8);
  l.u = l.y + a256(N1 * M * 8);
  l.tm = l.u + a256(N1 * M * 8);
  l.tn = l.tm + a256(M * 16);
  l.total = l.tn + a256(N1 * 8);
  return l;
}

int check(const fstat_sft_desc* d) {
  if (!d) return FSTAT_EINVAL;
  if (d->sft_len < 2 || !(d->dt_raw > 0.0) || d->n_bins < 1 || d->n_bins > kMaxBins || d->band_bins < 2 ||
      (d->band_bins & 1) || d->band_bins > kMaxN1 || d->dirichlet_terms < 0 || d->median_window < 0 ||
      (d->median_window > 0 && !(d->median_window & 1)) || d->median_window > kMaxWindow ||
      !(d->tukey_frac >= 0.0 && d->tukey_frac <= 1.0) || d->edge_taper < 0)
    return FSTAT_EINVAL;
  const int64_t need_lo = d->k_het - d->band_bins / 2 - d->dirichlet_terms;
  const int64_t need_hi = d->k_het + d->band_bins / 2 - 1 + d->dirichlet_terms;
  if (need_lo < d->k_lo || need_hi > d->k_lo + d->n_bins - 1) return FSTAT_ERANGE;
  return FSTAT_OK;
}

}  // namespace

}  // namespace fs

extern "C" int fstat_sft_normalize(const fstat_sft_desc* d, const float* sfts, int64_t n_sft, float* out,
                                   void* stream) {
  using namespace fs;
  if (!d || d->n_bins < 1 || d->n_bins > kMaxBins || d->median_window < 1 || !(d->median_window & 1) ||
      d->median_window > kMaxWindow || n_sft < 0)
    return FSTAT_EINVAL;
  if (n_sft == 0) return FSTAT_OK;
  if (!sfts || !out || ((uintptr_t)sfts & 7) || ((uintptr_t)out & 7)) return FSTAT_EINVAL;
  if (n_sft > 0x7fffffff) return FSTAT_ERANGE;
  return launch_normalize(reinterpret_cast<const float2*>(sfts), reinterpret_cast<float2*>(out), n_sft,
                          (int)d->n_bins, d->median_window, static_cast<cudaStream_t>(stream)) == cudaSuccess
             ? FSTAT_OK : FSTAT_ECUDA;
}

extern "C" size_t fstat_sft_workspace(const fstat_sft_desc* d, int64_t n_sft) {
  if (fs::check(d) != FSTAT_OK || n_sft < 0) return 0;
  return fs::layout(*d, n_sft > 0 ? n_sft : 1).total;
}

extern "C" int fstat_sft_series(const fstat_sft_desc* d, const float* sfts, const double* t_sft, int64_t n_sft,
                                double t_start, int64_t n_out, float* x_h, void* workspace, size_t ws_bytes,
                                void* stream) {
  using namespace fs;
  int rc = check(d);
  if (rc) return rc;
  if (n_sft < 0 || n_out < 0 || !x_h || ((uintptr_t)x_h & 7)) return FSTAT_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (n_out > 0 && cudaMemsetAsync(x_h, 0, (size_t)n_out * 8, s) != cudaSuccess) return FSTAT_ECUDA;
  if (n_sft == 0) return FSTAT_OK;
  if (!sfts || !t_sft || !workspace || ((uintptr_t)sfts & 7) || ((uintptr_t)workspace & 255)) return FSTAT_EINVAL;
  const FeLayout l = layout(*d, n_sft);
  if (ws_bytes < l.total) return FSTAT_ENOMEM;
  const double t_len = (double)d->sft_len * d->dt_raw;
  const double dt_out = t_len / (double)d->band_bins;
  const double f_h = (double)d->k_het / t_len;
  // chunks of consecutive SFTs, their output offsets
  struct Chunk1 { int64_t a, m, off; double tc; };
  std::vector<Chunk1> ch;
  int64_t a = 0;
  for (int64_t i = 1; i <= n_sft; ++i) {
    if (i < n_sft && !(t_sft[i] > t_sft[i - 1])) return FSTAT_EINVAL;
    if (i == n_sft || fabs(t_sft[i] - t_sft[i - 1] - t_len) > 1e-6 * t_len) {
      const double u = (t_sft[a] - t_start) / dt_out;
      const double ur = nearbyint(u);
      if (fabs(u - ur) > 1e-6 || ur < 0 || (int64_t)ur + (i - a) * d->band_bins > n_out) return FSTAT_ERANGE;
      if (i - a > 65535 || i - a > 0x7fffffff / d->band_bins) return FSTAT_ERANGE;   // grid y, int indices
      ch.push_back({a, i - a, (int64_t)ur, t_sft[a]});
      a = i;
    }
  }
  char* ws = static_cast<char*>(workspace);
  float2* xh = reinterpret_cast<float2*>(ws + l.xh);
  float2* D = reinterpret_cast<float2*>(ws + l.d);
  float2* Y = reinterpret_cast<float2*>(ws + l.y);
  float2* U = reinterpret_cast<float2*>(ws + l.u);
  float4* tm = reinterpret_cast<float4*>(ws + l.tm);
  float2* tn = reinterpret_cast<float2*>(ws + l.tn);
  const int K = (int)d->n_bins, N1 = (int)d->band_bins;
  const float2* X = reinterpret_cast<const float2*>(sfts);
  // step 2 over all SFTs
  if (d->median_window > 0) {
    if (n_sft > 0x7fffffff || launch_normalize(X, xh, n_sft, K, d->median_window, s) != cudaSuccess)
      return FSTAT_ECUDA;
    X = xh;
  }
  // three rows of N1 and the row factors
  const size_t n1_smem = ((size_t)3 * N1 + kRotLo + (N1 + kRotLo - 1) / kRotLo) * 8;
  constexpr size_t n1_smem_max = ((size_t)3 * kMaxN1 + kRotLo + kMaxN1 / kRotLo) * 8;
  const unsigned long long plan = radix_plan(N1);
  static DeviceOnce once_n1, once_n1s;
  if ((plan ? kernel_setup(once_n1s, k_idft_n1_smooth, kFeThreads, n1_smem_max, nullptr)
            : kernel_setup(once_n1, k_idft_n1, kFeThreads, n1_smem_max, nullptr)) != cudaSuccess)
    return FSTAT_ECUDA;
  // N1 = P Q with P the largest divisor of N1 not above sqrt(N1)
  int P = 1;
  for (int q = 1; (int64_t)q * q <= N1; ++q)
    if (N1 % q == 0) P = q;
  const int ks0 = (int)(d->k_het - d->k_lo);
  // the chunks in groups of at most kChunksPerLaunch chunks and 65535 SFTs
  // (grid y of k_merge): 5 launches per group
  for (size_t c0 = 0; c0 < ch.size();) {
    ChunkTab tab;
    int64_t rows = 0;
    tab.n = 0;
    while (c0 + tab.n < ch.size() && tab.n < kChunksPerLaunch && rows + ch[c0 + tab.n].m <= 65535)
      rows += ch[c0 + tab.n++].m;
    tab.yb[0] = 0;
    for (int i = 0; i < tab.n; ++i) {
      const Chunk1& c = ch[c0 + i];
      tab.a[i] = (int)c.a;
      tab.m[i] = (int)c.m;
      tab.yb[i + 1] = tab.yb[i] + (int)((c.m + kN2PerBlock - 1) / kN2PerBlock);
      tab.off[i] = c.off;
      double cyc = f_h * (c.tc - t_start);
      cyc -= floor(cyc);
      tab.gc[i] = (float)cos(2.0 * M_PI * cyc);
      tab.gs[i] = (float)(-sin(2.0 * M_PI * cyc));
      tab.sc[i] = (float)(1.0 / sqrt((double)c.m * ((double)N1 * (double)c.m)));
    }
    for (int i = tab.n; i < kChunksPerLaunch; ++i) { tab.a[i] = tab.m[i] = 0; tab.yb[i + 1] = tab.yb[tab.n]; }
    tab.rows = (int)(ch[c0 + tab.n - 1].a + ch[c0 + tab.n - 1].m - ch[c0].a);
    const int tmax = tab.rows > N1 ? tab.rows : N1;
    k_tables<<<(tmax + 255) / 256, 256, 0, s>>>(tab, tm, tn, N1);
    k_dft_alpha<<<dim3((K + kDftCols - 1) / kDftCols, tab.yb[tab.n]), kFeThreads, 0, s>>>(tab, X, K, tm, D);
    k_merge<<<dim3((N1 + 255) / 256, tab.rows), kFeThreads, 0, s>>>(tab, D, K, N1, ks0, d->dirichlet_terms, tm,
                                                                    d->tukey_frac / 2.0, (float)(d->tukey_frac / 2.0), Y);
    if (plan) k_idft_n1_smooth<<<(unsigned)tab.rows, kFeThreads, n1_smem, s>>>(tab, Y, N1, plan, tn, U);
    else k_idft_n1<<<(unsigned)tab.rows, kFeThreads, n1_smem, s>>>(tab, Y, N1, P, tn, U);
    k_idft_n2<<<dim3((N1 + kDftCols - 1) / kDftCols, tab.yb[tab.n]), kFeThreads, 0, s>>>(tab, U, N1, tm, d->edge_taper,
                                                                          reinterpret_cast<float2*>(x_h));
    c0 += tab.n;
  }
  return cudaGetLastError() == cudaSuccess ? FSTAT_OK : FSTAT_ECUDA;
}
