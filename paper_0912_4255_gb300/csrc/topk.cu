// Per-band top-k candidates of 2F spectra.  The paper computes 2F in every
// bin (Eq. 6, step 7 of Sec. III.A.2) for searches over many frequencies;
// it defines no candidate stage.  A search keeps the loudest bins: for each
// band of consecutive bins, the k largest values (descending; ties: lower bin
// first) with their bin indices.
//
// One block per (row, band).  It first samples the band and takes a lower bound
// of the k-th largest value from the sample; then it streams the band once and
// appends the few values at or above the bound to a buffer in shared memory.
// Between pieces of 16384 values a buffer that has filled up raises the bound
// to one from the buffer's own values and drops what is below.  At the end the
// same step leaves little more than k values, and each one's rank among them
// is its place in the result.  A value costs a maximum and a quarter of a
// comparison (lists of four in every thread's registers with an insertion
// where any of the 32 lanes had one ran at the issue limit), and 256 threads a
// block put all bands of a search's rows on the chip at once.  What bounds it is
// the read: 16 rows of 2^22 bins in bands of 65536, k = 16: 73 -> 43 us,
// 40 at the copy rate.
//
// A band whose values overflow the buffer all the same (a ramp: every value is
// above what came before) is done by a sweep that merges whenever it must: the
// threads' maxima of the first 1024 values give the bound, and the buffer is
// merged with the running list by a bitonic sort, which raises the bound to the
// list's k-th value.
//
// Few values of short bands are drawn by rounds instead (k_topk_short).
#include "fstat_internal.cuh"

#include <climits>

namespace fs {

namespace {

constexpr int kBandUnit = 2048;          // bands are multiples of this
template <int THREADS_, int UNROLL_, int MIN_BLOCKS_> struct TopForm {
  static constexpr int THREADS = THREADS_, UNROLL = UNROLL_, MIN_BLOCKS = MIN_BLOCKS_, WARPS = THREADS_ / 32;
  static constexpr int STEP = 4 * THREADS;          // values per step: one float4 per thread
  static constexpr int SORT_N = 8 * THREADS;        // sort buffer: the list (k <= 64) and the candidates
  static constexpr int PIECE = 16384 / STEP;        // steps between two looks at the buffer
};
using TopMany = TopForm<256, 4, 8>;
using TopFew = TopForm<512, 8, 2>;
constexpr int kMaxK = 64;

// key order: the larger value first, then the lower bin
__device__ __forceinline__ bool before(float va, int ia, float vb, int ib) {
  return va > vb || (va == vb && ia < ib);
}

// Bitonic sort of sv/si[0, n) into key order (n a power of two, 2..F::SORT_N);
// all threads; ends with a barrier.
template <class F>
__device__ void bitonic(float* sv, int* si, int n) {
  for (int size = 2; size <= n; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      __syncthreads();
      for (int t = threadIdx.x; t < n / 2; t += F::THREADS) {
        const int lo = 2 * t - (t & (stride - 1));     // the pair (lo, lo + stride)
        const int hi = lo + stride;
        const bool fwd = (lo & size) == 0;             // this run in key order, else reversed
        const float a = sv[lo], b = sv[hi];
        const int ia = si[lo], ib = si[hi];
        if (fwd ? before(b, ib, a, ia) : before(a, ia, b, ib)) {
          sv[lo] = b; sv[hi] = a; si[lo] = ib; si[hi] = ia;
        }
      }
    }
  }
  __syncthreads();
}

// the largest finite value of the four, or -inf
__device__ __forceinline__ float finite_max(float4 x) {
  const float a = x.x < INFINITY ? x.x : -INFINITY, b = x.y < INFINITY ? x.y : -INFINITY;
  const float c = x.z < INFINITY ? x.z : -INFINITY, d = x.w < INFINITY ? x.w : -INFINITY;
  return fmaxf(fmaxf(a, b), fmaxf(c, d));
}

template <class F>
__device__ __forceinline__ void clear(float* sv, int* si, int from, int to) {
  for (int i = from + (int)threadIdx.x; i < to; i += F::THREADS) { sv[i] = -INFINITY; si[i] = INT_MAX; }
}

__device__ __forceinline__ void append(float v, int b, float tau, float* sv, int* si, int* cnt, int k) {
  if (v >= tau && fabsf(v) < INFINITY) {     // false for NaN
    const int pos = atomicAdd(cnt, 1);
    sv[k + pos] = v;
    si[k + pos] = b;
  }
}

// list at [0, k), candidates at [k, k + cnt): sort them together, keep the
// first k, return the new bound (the k-th value)
template <class F>
__device__ float merge(float* sv, int* si, int* cnt, int k) {
  const int m = k + *cnt;
  int n = 2;
  while (n < m) n <<= 1;
  bitonic<F>(sv, si, n);
  const float tau = sv[k - 1];
  clear<F>(sv, si, k, n);
  __syncthreads();
  if (threadIdx.x == 0) *cnt = 0;
  __syncthreads();
  return tau;
}

// The sweep that keeps every candidate (all threads of the block).
template <class F>
__device__ void topk_sweep(const float* __restrict__ src, int base, int64_t o, int band_len, int k,
                           float* __restrict__ val, int* __restrict__ bin, float* sv, int* si, int& cnt) {
  // bound from the first step: the k-th largest of the threads' maxima
  float4 v4 = __ldcs(reinterpret_cast<const float4*>(src) + threadIdx.x);
  sv[threadIdx.x] = finite_max(v4);
  si[threadIdx.x] = (int)threadIdx.x;
  bitonic<F>(sv, si, F::THREADS);
  float tau = sv[k - 1];
  __syncthreads();
  clear<F>(sv, si, 0, F::SORT_N);
  if (threadIdx.x == 0) cnt = 0;
  __syncthreads();
#pragma unroll 1
  for (int s0 = 0; s0 < band_len; s0 += F::STEP) {
    if (s0 > 0) v4 = __ldcs(reinterpret_cast<const float4*>(src + s0) + threadIdx.x);
    const int b0 = base + s0 + 4 * (int)threadIdx.x;
    append(v4.x, b0, tau, sv, si, &cnt, k);
    append(v4.y, b0 + 1, tau, sv, si, &cnt, k);
    append(v4.z, b0 + 2, tau, sv, si, &cnt, k);
    append(v4.w, b0 + 3, tau, sv, si, &cnt, k);
    __syncthreads();
    // every warp has to see the same count: none goes on to append before all have read it
    const int n = cnt;
    __syncthreads();
    // the next step adds at most F::STEP candidates: merge while they still fit
    if (n > F::SORT_N - k - F::STEP || s0 + F::STEP >= band_len) tau = merge<F>(sv, si, &cnt, k);
  }
  for (int i = threadIdx.x; i < k; i += F::THREADS) {
    val[o + i] = sv[i];
    bin[o + i] = si[i] == INT_MAX ? -1 : si[i];
  }
}

// An integer whose signed order is the order of the (non-NaN) float (the
// two zeros, equal as floats, share a key).
__device__ __forceinline__ int order_key(float v) {
  const int i = __float_as_int(v == 0.0f ? 0.0f : v);
  return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float key_value(int key) { return __int_as_float(key ^ ((key >> 31) & 0x7fffffff)); }

// A candidate as one number, larger first in the result's order: the value's
// key, then the lower bin.
__device__ __forceinline__ unsigned long long pack(float v, int b) {
  return ((unsigned long long)((unsigned)order_key(v) ^ 0x80000000u) << 32) | (unsigned)~b;
}
__device__ __forceinline__ float packed_value(unsigned long long c) {
  return key_value((int)((unsigned)(c >> 32) ^ 0x80000000u));
}

// A lower bound of the k-th largest of the block's values from every thread's
// largest one (vmax; the values of different threads are different ones): the
// lowest over the warps of each one's ceil(k / warps)-th largest lane maximum.
// All threads; scratch: F::WARPS keys.
template <class F>
__device__ float lower_bound_of_kth(float vmax, int k, int* scratch) {
  int key = order_key(vmax), m = INT_MIN;
  for (int r = 0; r < (k + F::WARPS - 1) / F::WARPS; ++r) {
    m = __reduce_max_sync(0xffffffffu, key);
    const unsigned who = __ballot_sync(0xffffffffu, key == m);
    if ((threadIdx.x & 31) == __ffs(who) - 1) key = INT_MIN;       // one of them is out
  }
  if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = m;
  __syncthreads();
  m = scratch[0];
#pragma unroll
  for (int w = 1; w < F::WARPS; ++w) m = min(m, scratch[w]);
  __syncthreads();
  return key_value(m);                    // -inf where a warp has too few finite values
}

// The buffer's n candidates cut to those at or above a bound from themselves
// (at least k of them, if there were k); returns the bound.  All threads; ends
// with a barrier.
template <class F>
__device__ float refine(unsigned long long* buf, int n, int k, float tau, int* cnt, int* scratch) {
  float mx = -INFINITY;
  // candidate i to warp i % F::WARPS, so that every warp has its share
  for (int i = (threadIdx.x >> 5) + F::WARPS * (threadIdx.x & 31); i < n; i += F::THREADS)
    mx = fmaxf(mx, packed_value(buf[i]));
  tau = fmaxf(tau, lower_bound_of_kth<F>(mx, k, scratch));
  if (threadIdx.x == 0) *cnt = 0;
  for (int i0 = 0; i0 < n; i0 += F::THREADS) {
    // what is kept goes below i0 + F::THREADS, where all has been read
    const int i = i0 + threadIdx.x;
    const unsigned long long c = i < n ? buf[i] : 0;
    __syncthreads();
    if (i < n && packed_value(c) >= tau) buf[atomicAdd(cnt, 1)] = c;
  }
  __syncthreads();
  return tau;
}

// Values sampled per thread (float4): noise leaves about 2 k band / sample
// candidates.  A buffer above kRefineAt is refined before the next piece.
constexpr int kSample = 4;
constexpr int kRefineAt = 512;
constexpr int kRankAll = 128;      // so few are ranked as they are

// The largest of the warp's candidates, in every lane.
__device__ __forceinline__ unsigned long long warp_best(unsigned long long c) {
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(c >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(c >> 32) == hi ? (unsigned)c : 0u);
  return ((unsigned long long)hi << 32) | lo;
}

// Few values of a short band: k <= 2 of up to four values a step, or k <= 4 of one
// step, whose values the threads hold.  Every warp draws its k largest by rounds,
// then one warp the block's: one barrier, where a bound, a buffer and ranks take
// five.  In a graph (buffer | rounds): one band of 2048 at k = 1 2.7 | 1.7 us, k = 4
// 2.8 | 2.3, 128 bands at k = 1 3.7 | 2.0, one of 8192 at k = 2 3.3 | 2.9.
template <class F> bool few_of_short(int band_len, int k) {
  const int n_steps = band_len / F::STEP;
  return (k <= 2 && n_steps <= 4) || (k <= 4 && n_steps == 1);
}

template <class F>
__global__ void __launch_bounds__(F::THREADS, F::MIN_BLOCKS)
k_topk_short(const float* __restrict__ two_f, int64_t row_len, int band_len, int k, float* __restrict__ val,
             int* __restrict__ bin) {
  using Cand = unsigned long long;
  __shared__ Cand lists[4][F::WARPS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int base = blockIdx.x * band_len;
  const int64_t o = ((int64_t)blockIdx.y * (row_len / band_len) + blockIdx.x) * k;
  const float4* src = reinterpret_cast<const float4*>(two_f + blockIdx.y * row_len + base) + threadIdx.x;
  const int n_steps = band_len / F::STEP;
  Cand c[4], d[4];                             // descending; no candidate is 0
  const auto load = [&](Cand (&q)[4], float4 x, int u) {
    const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      q[e] = fabsf(v[e]) < INFINITY ? pack(v[e], base + u * F::STEP + 4 * (int)threadIdx.x + e) : 0;
  };
  const auto down = [](Cand& x, Cand& y) {     // the larger of the two to x
    const Cand hi = x > y ? x : y;
    y = x > y ? y : x;
    x = hi;
  };
  float4 xs[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) xs[u] = __ldg(src + (int64_t)(u < n_steps ? u : 0) * F::THREADS);
  load(c, xs[0], 0);
  down(c[0], c[1]); down(c[2], c[3]); down(c[0], c[2]); down(c[1], c[3]); down(c[1], c[2]);
#pragma unroll
  for (int u = 1; u < 4; ++u)
    if (u < n_steps) {                         // two are enough
      load(d, xs[u], u);
      down(d[0], d[1]); down(d[2], d[3]); down(d[0], d[2]); down(d[1], d[2]);
      down(c[0], d[0]); down(c[1], d[0]); down(c[1], d[1]);
    }
  for (int r = 0; r < k; ++r) {
    const Cand w = warp_best(c[0]);
    if (lane == 0) lists[r][warp] = w;
    if (c[0] == w) { c[0] = c[1]; c[1] = c[2]; c[2] = c[3]; c[3] = 0; }
  }
  __syncthreads();
  if (warp != 0) return;
  int p = 0;
  c[0] = lane < F::WARPS ? lists[0][lane] : 0;
  for (int r = 0; r < k; ++r) {
    const Cand w = warp_best(c[0]);
    if (lane == 0) {
      val[o + r] = w ? packed_value(w) : -INFINITY;
      bin[o + r] = w ? (int)~(unsigned)w : -1;
    }
    if (c[0] == w && w != 0) c[0] = ++p < k ? lists[p][lane] : 0;
  }
}

template <class F>
__global__ void __launch_bounds__(F::THREADS, F::MIN_BLOCKS)
k_topk(const float* __restrict__ two_f, int64_t row_len, int band_len, int k, float* __restrict__ val,
       int* __restrict__ bin) {
  __shared__ union {
    unsigned long long cand[F::SORT_N];
    struct { float v[F::SORT_N]; int b[F::SORT_N]; } sort;
  } sh;
  __shared__ int cnt;
  __shared__ int scratch[F::WARPS];
  const int band = blockIdx.x;
  const int64_t row = blockIdx.y;
  const float* src = two_f + row * row_len + (int64_t)band * band_len;
  const int base = band * band_len;
  const int64_t o = (row * (row_len / band_len) + band) * k;
  const float4* src4 = reinterpret_cast<const float4*>(src) + threadIdx.x;
  const int n_steps = band_len / F::STEP;
  if (threadIdx.x == 0) cnt = 0;
  float mx = -INFINITY;
  // steps spread over the band, so that a trend does not mislead the bound; a
  // short band is the sample
  const int ns = n_steps < kSample ? n_steps : kSample;
  float4 xs[kSample];
#pragma unroll
  for (int u = 0; u < kSample; ++u) xs[u] = __ldg(src4 + (int64_t)(u < ns ? u * n_steps / ns : 0) * F::THREADS);
#pragma unroll
  for (int u = 0; u < kSample; ++u) mx = fmaxf(mx, finite_max(xs[u]));
  float tau = lower_bound_of_kth<F>(mx, k, scratch);
  const auto look = [&](float4 x, int step) {
    if (fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)) >= tau) {
      const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (v[c] >= tau && fabsf(v[c]) < INFINITY) {
          const int at = atomicAdd(&cnt, 1);
          if (at < F::SORT_N) sh.cand[at] = pack(v[c], base + step * F::STEP + 4 * (int)threadIdx.x + c);
        }
    }
  };
  if (n_steps <= kSample) {
#pragma unroll
    for (int u = 0; u < kSample; ++u)
      if (u < n_steps) look(xs[u], u);
  } else
#pragma unroll 1
  for (int p0 = 0; p0 < n_steps; p0 += F::PIECE) {
    if (p0 > 0) {
      __syncthreads();
      const int n = cnt;
      if (n > F::SORT_N) break;
      __syncthreads();
      if (n > kRefineAt) tau = refine<F>(sh.cand, n, k, tau, &cnt, scratch);
    }
    const int p1 = p0 + F::PIECE < n_steps ? p0 + F::PIECE : n_steps;
    int s = p0;
#pragma unroll 1
    for (; s + F::UNROLL <= p1; s += F::UNROLL) {
      float4 x[F::UNROLL];
#pragma unroll
      for (int u = 0; u < F::UNROLL; ++u) x[u] = __ldcs(src4 + (int64_t)(s + u) * F::THREADS);
#pragma unroll
      for (int u = 0; u < F::UNROLL; ++u) look(x[u], s + u);
    }
    for (; s < p1; ++s) look(__ldcs(src4 + (int64_t)s * F::THREADS), s);
  }
  __syncthreads();
  int n = cnt;
  __syncthreads();
  if (n > F::SORT_N) {
    topk_sweep<F>(src, base, o, band_len, k, val, bin, sh.sort.v, sh.sort.b, cnt);
    return;
  }
  if (n > kRankAll) {
    refine<F>(sh.cand, n, k, tau, &cnt, scratch);
    n = cnt;
  }
  for (int i = threadIdx.x; i < n; i += F::THREADS) {
    const unsigned long long c = sh.cand[i];
    int rank = 0;
    for (int e = 0; e < n; ++e) rank += sh.cand[e] > c;
    if (rank < k) {
      val[o + rank] = packed_value(c);
      bin[o + rank] = (int)~(unsigned)c;
    }
  }
  for (int i = n + threadIdx.x; i < k; i += F::THREADS) {
    val[o + i] = -INFINITY;
    bin[o + i] = -1;
  }
}

}  // namespace

}  // namespace fs

extern "C" int fstat_topk(const float* twoF, int64_t n_rows, int64_t row_len, int64_t band_len, int k,
                          float* val, int32_t* bin, void* stream) {
  using namespace fs;
  if (!twoF || !val || !bin || ((uintptr_t)twoF & 15) || ((uintptr_t)val & 3) || ((uintptr_t)bin & 3))
    return FSTAT_EINVAL;
  if (k < 1 || k > kMaxK || n_rows < 0 || band_len < kBandUnit || band_len % kBandUnit || row_len % band_len ||
      row_len > ((int64_t)1 << 30))
    return FSTAT_EINVAL;
  if (n_rows > 65535 || row_len / band_len > 65535) return FSTAT_ERANGE;
  if (n_rows == 0) return FSTAT_OK;
  dim3 grid((unsigned)(row_len / band_len), (unsigned)n_rows);
  // With no more bands than two to an SM, more threads and more loads in flight
  // for each (many | few): 16 bands of 262144 65 | 35 us, 256 of them 71 | 46, 256 of
  // 8192 12.4 | 10.3; 512 bands of 65536 31 | 34, 1024 of them 43 | 60.
  if ((int64_t)grid.x * grid.y <= 2 * 152 && few_of_short<TopFew>((int)band_len, k))
    k_topk_short<TopFew><<<grid, TopFew::THREADS, 0, static_cast<cudaStream_t>(stream)>>>(twoF, row_len, (int)band_len, k, val, bin);
  else if ((int64_t)grid.x * grid.y <= 2 * 152)
    k_topk<TopFew><<<grid, TopFew::THREADS, 0, static_cast<cudaStream_t>(stream)>>>(twoF, row_len, (int)band_len, k, val, bin);
  else
    k_topk<TopMany><<<grid, TopMany::THREADS, 0, static_cast<cudaStream_t>(stream)>>>(twoF, row_len, (int)band_len, k, val, bin);
  return cudaGetLastError() == cudaSuccess ? FSTAT_OK : FSTAT_ECUDA;
}
