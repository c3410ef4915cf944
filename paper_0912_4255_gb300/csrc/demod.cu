// SFT-domain demodulation F-statistic: the earlier method that the paper's
// speed comparison (Sec. IV.A) measures resampling against, derived from
// Eq. 7 and the Dirichlet kernel of Eq. e9.  Within SFT alpha the template
// phase is taken as linear and a, b as constant at the SFT midpoint, so
//   F_a = sum_alpha a_alpha e^{-2 pi i (Phi_alpha / 2 pi - kappa_alpha / 2)}
//         sum_{k = k* - dk}^{k* + dk} X^_{alpha,k} P(kappa_alpha - k),
// kappa_alpha = fhat_alpha T_SFT the instantaneous frequency in SFT bins,
// P = sin y / y - i (1 - cos y) / y, y = 2 pi (kappa - k); F_b with b_alpha;
// for normalised SFTs A = sum a^2, B = sum b^2, C = sum ab.
//
// The per-(template, SFT) quantities are computed once in FP64
// (k_demod_setup); along the frequency grid f_q = f_0 + q df both kappa and
// the phase are linear in q.  They are laid down in 64-bit fixed point (kappa -
// k_lo with 44 fractional bits, the phase as a fraction of a cycle) and taken
// from there at every frequency where the terms are summed one by one, and at
// the centre of a segment of 32 or 64 frequencies where the far terms are
// expanded; inside a segment they are stepped in 32 bits (2^-30 bins, the step
// to 2^-36 bins or finer; 2^-32 cycles).  The sum over SFTs and terms is FP32.
#include "fstat_internal.cuh"

#include <math.h>

namespace fs {

namespace {

constexpr int kFracBits = 44;
constexpr int kSetupThreads = 32;
constexpr float kInv24 = 5.9604644775390625e-8f;      // 2^-24
constexpr long long kMask = (1ll << kFracBits) - 1;

struct DemodRec {
  long long rel0, drel;              // (kappa - k_lo) at q = 0 and per q step, 2^-44 bins
  unsigned long long ph0, dph;       // phase - kappa / 2 at q = 0 and per step, 2^-64 cycles
  float a, b;
  int pad_[2];
};

// x mod 1 in [0, 1): x - floor(x) rounds to 1.0 for tiny negative x
__device__ __forceinline__ double frac_d(double x) {
  const double v = x - floor(x);
  return v < 1.0 ? v : 0.0;
}

// grid (ceil(n_sft / kSetupThreads), n_t): the latency of FP64 binds; blocks of a
// warp spread over the SMs (432 SFTs x 4 templates 10.5 us, in blocks of 256 19 us).
__global__ void k_demod_setup(PlanConst pc, const fstat_template* __restrict__ tm, const double* __restrict__ t_sft,
                              int n_sft, double t_len, double k_lo, double f0, double df, DemodRec* __restrict__ rec,
                              int* status) {
  const int t = blockIdx.y;
  const int al = blockIdx.x * blockDim.x + threadIdx.x;
  if (al >= n_sft) return;
  const fstat_template tp = tm[t];
  DemodRec r;
  if (!(isfinite(tp.alpha) && isfinite(tp.delta) && isfinite(tp.fdot) && isfinite(tp.fddot)) ||
      fabs(tp.delta) > 1.5707963267948967) {
    if (al == 0) set_status(status, FSTAT_EINVAL);
    r.rel0 = r.drel = 0; r.ph0 = r.dph = 0; r.a = r.b = 0.f; r.pad_[0] = 1; r.pad_[1] = 0;
    rec[(int64_t)t * n_sft + al] = r;
    return;
  }
  const Sky<double> sky = make_sky<double>(pc, tp.alpha, tp.delta);
  const double tmid = t_sft[al] + 0.5 * t_len;
  double t_m, rate, sH, cH;
  roemer<double>(pc, sky, tmid, &t_m, &rate, &sH, &cH);
  double a, b, da, db;
  beams_h<double>(pc, sky, sH, cH, &a, &b, &da, &db);
  const double tau = tmid - pc.t_start + t_m;
  const double fdot_t = tp.fdot * tau + 0.5 * tp.fddot * tau * tau;
  const double kap0 = (f0 + fdot_t) * (1.0 + rate) * t_len;
  const double dkap = df * (1.0 + rate) * t_len;
  const double cyc0 = frac_d(f0 * tau) + frac_d(0.5 * tp.fdot * tau * tau) + frac_d(tp.fddot * tau * tau * tau / 6.0)
                      - 0.5 * kap0;
  const double dcyc = df * tau - 0.5 * dkap;
  const double s44 = 17592186044416.0;                  // 2^44
  const double s64 = 18446744073709551616.0;            // 2^64
  r.rel0 = llrint((kap0 - k_lo) * s44);
  r.drel = llrint(dkap * s44);
  r.ph0 = (unsigned long long)(frac_d(cyc0) * s64);
  r.dph = (unsigned long long)(frac_d(dcyc) * s64);
  r.a = (float)a;
  r.b = (float)b;
  r.pad_[0] = 0;
  r.pad_[1] = 0;
  rec[(int64_t)t * n_sft + al] = r;
}

// x / d added to T
__device__ __forceinline__ void add_term(float2& T, float2 x, float d) {
  const float iv = rcp_approx(d);
  T.x = fmaf(x.x, iv, T.x);
  T.y = fmaf(x.y, iv, T.y);
}

// sin(pi f) / pi, f in [0, 1) a multiple of 2^-24 (1 - f is exact, so the
// result is accurate relative to the distance from 0 and 1): polynomial in x^2
// on [0, 1/2] fitted for the least relative error, 1.2e-8 with the coefficients as
// written.
__device__ __forceinline__ float sinpi_over_pi(float f) {
  const float x = fminf(f, 1.0f - f);
  const float u = x * x;
  return x * fmaf(u, fmaf(u, fmaf(u, fmaf(u, 0.0246882383f, -0.190426379f), 0.811712424f), -1.644933129f), 1.0f);
}

// sin(pi v) and cos(pi v), |v| <= 1/2: the polynomial above times pi, and one
// in v^2 with its value at 0 held at 1 (absolute error 2.5e-8).
__device__ __forceinline__ void sincospi_half(float v, float* s, float* c) {
  const float u = v * v;
  *s = v * fmaf(u, fmaf(u, fmaf(u, fmaf(u, 0.0775603876f, -0.598242104f), 2.55006981f), -5.16770983f), 3.14159274f);
  *c = fmaf(u, fmaf(u, fmaf(u, fmaf(u, fmaf(u, -0.0244207f, 0.234953925f), -1.33521605f), 4.0587096f), -4.93480206f), 1.0f);
}

// How a block expands: PL frequencies a lane (a segment is 32 PL), the NEAR terms
// around kappa one by one, the others by ORDER coefficients.
// One SFT over one segment (centre q_c, kappa_c = k0 + fc): the terms outside
// k0 - NEAR/2 + 1 .. k0 + NEAR/2 are at least NEAR/2 bins away, so for a kappa d
// off the centre, |d| <= spread, their sum
//   sum_j X_j / (y_j + d), y_j = fc - j,
// is sum_n (-d)^n c_n with c_n = sum_j X_j / y_j^(n+1), and what is left out is
// below (2 spread / NEAR)^ORDER of a term: 2.4e-8 and 6e-8 in the forms below.
// WARPS a block, PARTS of them share a segment (SFTs p, p + PARTS, ..).
// ORDER 0: no expansions, every term one by one.
template <int PL_, int NEAR_, int ORDER_, int WARPS_, int PARTS_> struct DemodForm {
  static constexpr bool EXPANDS = ORDER_ > 0;
  static constexpr int PL = PL_, SEG = 32 * PL_;
  [[maybe_unused]] static constexpr int NEAR = NEAR_, ORDER = ORDER_;
  static constexpr int WARPS = WARPS_, PARTS = PARTS_, SEGS = WARPS_ / PARTS_, THREADS = 32 * WARPS_;
  static constexpr int TILE = THREADS / SEGS < 128 ? THREADS / SEGS : 128;   // SFTs at a time
  static constexpr int MIN_BLOCKS = (!EXPANDS && PARTS_ == 8 ? 32 : NEAR_ == 2 ? 28 : 20) / WARPS_;
  [[maybe_unused]] static constexpr float kSpread = NEAR_ == 2 ? 0.03f : 0.25f;
  [[maybe_unused]] static constexpr int BITS = NEAR_ == 2 ? 41 : 36;      // of the step: below 2^31 with the spread
};
template <int WARPS, int PARTS> struct DemodForms {
  using Fine = DemodForm<2, 2, 5, WARPS, PARTS>;
  using Mid = DemodForm<2, 4, 8, WARPS, PARTS>;
  using Wide = DemodForm<1, 4, 8, WARPS, PARTS>;
  using Terms = DemodForm<1, 0, 0, WARPS, PARTS>;
};

template <class F> struct __align__(16) DemodFar {
  float2 c[F::ORDER];
  float2 x[F::NEAR];                 // X at k0 - NEAR/2 + 1 ..
  int rel, drel;                     // kappa - k0 at q_c, 2^-30 bins; its step, 2^-BITS bins
  unsigned ph, dph;                  // phase at q_c and its step, 2^-32 cycles
  float a, b;
  float dkap;                        // the step in bins, FP32
  int k0, mode;                      // FAR_*
};
// kappa - k0 of the frequency dq steps from the centre, 2^-30 bins
template <class F> __device__ __forceinline__ int far_pos(int rel, int drel, int dq) {
  return rel + __mulhi(dq << (62 - F::BITS), drel);
}
enum { FAR_NONE, FAR_WHOLE, FAR_EDGES };   // FAR_EDGES: kappa passes a whole number in the segment, so the
                                           // windows differ: the c_n hold only the terms that all share

template <class F>
__device__ __forceinline__ DemodFar<F> expand_far(const DemodRec& r, const float2* __restrict__ X, long long qc, int K, int dk) {
  const long long relc = r.rel0 + qc * r.drel;
  const long long kc = relc >> kFracBits;
  DemodFar<F> f;
  f.rel = (int)((relc & kMask) >> (kFracBits - 30));
  f.drel = (int)(r.drel >> (kFracBits - F::BITS));      // 31 bits where the expansion holds
  f.ph = (unsigned)((r.ph0 + (unsigned long long)qc * r.dph + 0x80000000ull) >> 32);
  f.dph = (unsigned)((r.dph + 0x80000000ull) >> 32);
  f.dkap = (float)r.drel * 5.684341886080801e-14f;      // 2^-44
  f.k0 = (int)kc;
  f.a = r.a;
  f.b = r.b;
  const bool narrow = fabsf(f.dkap) * (F::SEG / 2) <= F::kSpread;
  const int e0 = far_pos<F>(f.rel, f.drel, -F::SEG / 2), e1 = far_pos<F>(f.rel, f.drel, F::SEG / 2 - 1);
  const bool edges = min(e0, e1) < 0 || max(e0, e1) >= 1 << 30;
  const bool ok = r.pad_[0] == 0 && dk > F::NEAR / 2 && narrow && kc - dk - (edges ? 1 : 0) >= 0 &&
                  kc + dk + (edges ? 1 : 0) < K;
  f.mode = ok ? (edges ? FAR_EDGES : FAR_WHOLE) : FAR_NONE;
#pragma unroll
  for (int n = 0; n < F::ORDER; ++n) f.c[n] = make_float2(0.f, 0.f);
#pragma unroll
  for (int n = 0; n < F::NEAR; ++n) f.x[n] = make_float2(0.f, 0.f);
  if (ok) {
    const float fc = (float)(f.rel >> 6) * kInv24;
    const float2* xr = X + f.k0;
#pragma unroll
    for (int n = 0; n < F::NEAR; ++n) f.x[n] = __ldg(xr + n - F::NEAR / 2 + 1);
    const int h = edges ? dk - 1 : dk;
    const auto add = [&](int j) {
      const float2 v = __ldg(xr + j);
      const float iv = rcp_approx(fc - (float)j);
      float p = iv;
#pragma unroll
      for (int n = 0; n < F::ORDER; ++n) {
        f.c[n].x = fmaf(v.x, p, f.c[n].x);
        f.c[n].y = fmaf(v.y, p, f.c[n].y);
        p *= iv;
      }
    };
#pragma unroll 4
    for (int j = -h; j <= -F::NEAR / 2; ++j) add(j);
#pragma unroll 4
    for (int j = F::NEAR / 2 + 1; j <= h; ++j) add(j);
  }
  return f;
}

// A warp has a segment of frequencies and every PARTS-th SFT.  Per tile of SFTs
// each thread first expands the far terms of one (SFT, segment); then a lane
// adds per SFT and frequency the near terms and the expansion instead of
// 2 dk + 1 terms with a reciprocal each.  With sin y - i (1 - cos y) =
// 2 sin(pi fr) e^{-i pi fr}, y = 2 pi (fr - j), the SFT's factor joins its phase:
// one rotation per SFT and frequency.  Positions and phases are stepped from
// the segment's centre in 32 bits (2^-30 bins, 2^-32 cycles).  Bound by issue
// (78 % of the slots).  432 SFTs x 4 templates x 32768 frequencies at dk = 16:
// 240 us, 915 with every term one by one in every thread.
// grid (ceil(n_q / (SEGS SEG)), n_t).
template <class F>
__global__ void __launch_bounds__(F::THREADS, F::MIN_BLOCKS)
k_demod(const DemodRec* __restrict__ rec, const float2* __restrict__ X, int n_sft, int K, int dk, int64_t n_q,
        float* __restrict__ out, int* status) {
  __shared__ DemodRec rs[F::TILE];
  using Far = std::conditional_t<F::EXPANDS, DemodFar<F>, int>;
  __shared__ Far far[F::EXPANDS ? F::TILE : 1][F::SEGS];
  __shared__ float4 sum[F::SEGS][F::PARTS - 1][F::PL][32];
  __shared__ int bads[F::SEGS][F::PARTS - 1][F::PL][32];
  __shared__ double abc_sh[3][F::WARPS];
  const int t = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int seg = warp / F::PARTS, part = warp % F::PARTS;
  const int64_t qs = ((int64_t)blockIdx.x * F::SEGS + seg) * F::SEG;   // the segment's first frequency
  float2 Fa[F::PL], Fb[F::PL];
#pragma unroll
  for (int i = 0; i < F::PL; ++i) Fa[i] = Fb[i] = make_float2(0.f, 0.f);
  int bad[F::PL] = {0};
  double A = 0, B = 0, C = 0;
  for (int a0 = 0; a0 < n_sft; a0 += F::TILE) {
    const int an = min(F::TILE, n_sft - a0);
    __syncthreads();
    for (int i = threadIdx.x; i < an; i += blockDim.x) {
      const DemodRec r = rec[(int64_t)t * n_sft + a0 + i];
      rs[i] = r;
      // A, B, C of the FP32 values the demodulation uses, in FP64
      A += (double)r.a * (double)r.a; B += (double)r.b * (double)r.b; C += (double)r.a * (double)r.b;
    }
    __syncthreads();
    if constexpr (F::EXPANDS) {
      const int i = threadIdx.x / F::SEGS, sg = threadIdx.x % F::SEGS;
      if (i < an)
        far[i][sg] = expand_far<F>(rs[i], X + (int64_t)(a0 + i) * K,
                                   ((long long)blockIdx.x * F::SEGS + sg) * F::SEG + F::SEG / 2, K, dk);
      __syncthreads();
    }
    if (qs >= n_q) continue;
#pragma unroll 1
    for (int i = part; i < an; i += F::PARTS) {
      const Far& fm = far[F::EXPANDS ? i : 0][seg];
      int mode = FAR_NONE;
      if constexpr (F::EXPANDS) mode = fm.mode;
      const float2* xs = X + (int64_t)(a0 + i) * K;
      float2 T[F::PL];
      float fr[F::PL];
      unsigned th[F::PL];                            // 2^-32 cycles
      float a, b;
      if constexpr (F::EXPANDS) if (mode != FAR_NONE) {
        const DemodFar<F> f = fm;
        a = f.a; b = f.b;
#pragma unroll
        for (int u = 0; u < F::PL; ++u) {
          const int dq = lane + 32 * u - F::SEG / 2;
          const int pos = far_pos<F>(f.rel, f.drel, dq);
          // the fraction's top 24 bits: exact in FP32 and below 1
          const int f24 = (pos >> 6) & 0xffffff;
          fr[u] = (float)f24 * kInv24;
          th[u] = f.ph + (unsigned)dq * f.dph + ((unsigned)f24 << 7);   // phase and fr / 2
          const float d = -(float)dq * f.dkap;
          T[u] = f.c[F::ORDER - 1];
#pragma unroll
          for (int n = F::ORDER - 2; n >= 0; --n) {
            T[u].x = fmaf(T[u].x, d, f.c[n].x);
            T[u].y = fmaf(T[u].y, d, f.c[n].y);
          }
          float y[F::NEAR];                               // kappa less the near terms' bins
#pragma unroll
          for (int n = 0; n < F::NEAR; ++n) y[n] = fr[u] - (float)(n - F::NEAR / 2 + 1);
          if (mode == FAR_EDGES) {
            const int sh = pos >> 30;                     // -1, 0 or 1
            // the terms that only some windows have: dk and dk - 1 bins away on the
            // sides that this kappa's window has
            const float2* xr = xs + f.k0 + sh;
            if (sh <= 0) add_term(T[u], __ldg(xr - dk), fr[u] + (float)dk);
            if (sh < 0) add_term(T[u], __ldg(xr - dk + 1), fr[u] + (float)(dk - 1));
            if (sh >= 0) add_term(T[u], __ldg(xr + dk), fr[u] - (float)dk);
            if (sh > 0) add_term(T[u], __ldg(xr + dk - 1), fr[u] - (float)(dk - 1));
            // (from fr and a whole number: as exact as in the terms one by one)
#pragma unroll
            for (int n = 0; n < F::NEAR; ++n) y[n] = fr[u] - (float)(n - F::NEAR / 2 + 1 - sh);
          }
#pragma unroll
          for (int n = 0; n < F::NEAR; ++n) add_term(T[u], f.x[n], y[n]);
        }
      }
      if (mode == FAR_NONE) {
        const DemodRec r = rs[i];
        a = r.a; b = r.b;
#pragma unroll
        for (int u = 0; u < F::PL; ++u) {
          T[u] = make_float2(0.f, 0.f);
          fr[u] = 0.f;
          th[u] = 0;
          const long long qq = qs + lane + 32 * u < n_q ? qs + lane + 32 * u : n_q - 1;
          const long long rel = r.rel0 + qq * r.drel;
          const int kst = (int)(rel >> kFracBits);
          if (r.pad_[0]) { bad[u] = 1; continue; }
          if (kst - dk < 0 || kst + dk >= K) { bad[u] = 2; continue; }
          // (converting all 44 bits could round up to 1.0 and put y = 0 on the next term)
          const int f24 = (int)((rel & kMask) >> (kFracBits - 24));
          fr[u] = (float)f24 * kInv24;
          th[u] = (unsigned)((r.ph0 + (unsigned long long)qq * r.dph + 0x80000000ull) >> 32) + ((unsigned)f24 << 7);
          for (int j = -dk; j <= dk; ++j) add_term(T[u], __ldg(xs + kst + j), fr[u] - (float)j);
          if (fr[u] == 0.f) T[u] = __ldg(xs + kst);
        }
      }
#pragma unroll
      for (int u = 0; u < F::PL; ++u) {
        // S = (sin y - i (1 - cos y)) / 2 pi * T = sin(pi fr) / pi e^{-i pi fr} T, and
        // the template's phase; at fr = 0 the window's own bin is all that is left
        float sc = sinpi_over_pi(fr[u]);
        if (fr[u] == 0.f) {
          sc = 1.f;
          if constexpr (F::EXPANDS) if (mode != FAR_NONE) {
            const int dq = lane + 32 * u - F::SEG / 2;
            T[u] = __ldg(xs + fm.k0 + (far_pos<F>(fm.rel, fm.drel, dq) >> 30));
          }
        }
        // e^{-2 pi i th}: whole half turns to the sign, the rest |v| <= 1/2 half turns
        const float v = (float)(int)(th[u] << 1) * 2.3283064365386963e-10f;      // 2^-32
        sc = __int_as_float(__float_as_int(sc) ^ (int)((th[u] + 0x40000000u) & 0x80000000u));
        float sn, cs;
        sincospi_half(v, &sn, &cs);
        const float2 w = cmul(make_float2(T[u].x * sc, T[u].y * sc), make_float2(cs, -sn));
        Fa[u].x = fmaf(a, w.x, Fa[u].x); Fa[u].y = fmaf(a, w.y, Fa[u].y);
        Fb[u].x = fmaf(b, w.x, Fb[u].x); Fb[u].y = fmaf(b, w.y, Fb[u].y);
      }
    }
  }
  // A, B, C over the block's threads
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    A += __shfl_xor_sync(0xffffffffu, A, o);
    B += __shfl_xor_sync(0xffffffffu, B, o);
    C += __shfl_xor_sync(0xffffffffu, C, o);
  }
  if (lane == 0) { abc_sh[0][warp] = A; abc_sh[1][warp] = B; abc_sh[2][warp] = C; }
  if (part > 0) {
#pragma unroll
    for (int u = 0; u < F::PL; ++u) {
      sum[seg][part - 1][u][lane] = make_float4(Fa[u].x, Fa[u].y, Fb[u].x, Fb[u].y);
      bads[seg][part - 1][u][lane] = bad[u];
    }
  }
  __syncthreads();
  A = B = C = 0.0;
#pragma unroll
  for (int w = 0; w < F::WARPS; ++w) { A += abc_sh[0][w]; B += abc_sh[1][w]; C += abc_sh[2][w]; }
  const double D = A * B - C * C;
  const float ca = (float)(2.0 * B / D), cb = (float)(2.0 * A / D), cc = (float)(-4.0 * C / D);
#pragma unroll
  for (int u = 0; u < F::PL; ++u) {
    const int64_t q = qs + lane + 32 * u;
    if (q >= n_q || part > 0) continue;
#pragma unroll
    for (int p = 0; p < F::PARTS - 1; ++p) {
      const float4 v = sum[seg][p][u][lane];
      Fa[u].x += v.x; Fa[u].y += v.y; Fb[u].x += v.z; Fb[u].y += v.w;
      if (bad[u] == 0) bad[u] = bads[seg][p][u][lane];
    }
    float v = __int_as_float(0x7fc00000);
    if (bad[u]) set_status(status, bad[u] == 1 ? FSTAT_EINVAL : FSTAT_ERANGE);
    else
      v = ca * (Fa[u].x * Fa[u].x + Fa[u].y * Fa[u].y) + cb * (Fb[u].x * Fb[u].x + Fb[u].y * Fb[u].y) +
          cc * (Fa[u].x * Fb[u].x + Fa[u].y * Fb[u].y);
    out[(int64_t)t * n_q + q] = v;
  }
}

}  // namespace

size_t demod_workspace(int64_t n_sft, int64_t n_t) {
  return ((size_t)n_t * (size_t)n_sft * sizeof(DemodRec) + 255) & ~(size_t)255;
}

cudaError_t launch_demod(const PlanConst& pc, const fstat_sft_desc& d, const float2* X, const double* t_sft,
                         int64_t n_sft, const fstat_template* tm, int64_t n_t, double f0, double df, int64_t n_q,
                         float* out, void* ws, int* status, cudaStream_t s) {
  const double t_len = (double)d.sft_len * d.dt_raw;
  DemodRec* rec = static_cast<DemodRec*>(ws);
  k_demod_setup<<<dim3((unsigned)((n_sft + kSetupThreads - 1) / kSetupThreads), (unsigned)n_t), kSetupThreads, 0, s>>>(
      pc, tm, t_sft, (int)n_sft, t_len, (double)d.k_lo, f0, df, rec, status);
  const auto launch = [&](auto form) {
    using F = decltype(form);
    constexpr int per_block = F::SEGS * F::SEG;
    k_demod<F><<<dim3((unsigned)((n_q + per_block - 1) / per_block), (unsigned)n_t), F::THREADS, 0, s>>>(
        rec, X, (int)n_sft, (int)d.n_bins, d.dirichlet_terms, n_q, out, status);
  };
  // The step of kappa decides how far a segment reaches.  (The Doppler factor is
  // within 2e-4 of 1; the kernel checks each SFT's own step all the same and
  // takes the terms one by one where it is wider.)  4 templates x 32768 frequencies,
  // expanded | one by one in every thread: 240 SFTs (Mid) 190 | 600 us, 48 (Wide)
  // 68 | 140.
  const double step = fabs(df * t_len) * 1.0003;
  // No SFT is expanded where the step is too wide for any form, or where the kernel
  // has near terms only: a form without the expansions' registers and shared
  // memory.  8 SFTs, 4 templates x 32768 frequencies, dk = 16: 55 us in the last form,
  // 45 in this one; 240 SFTs, 4 x 16384, dk = 1: 139 | 84.  (In 48 registers 47 and 90, and
  // 16 SFTs, 4 x 8192, 37 where both others take 33 to 35.)
  const bool any = fabs(df * t_len) * 0.9997 * (DemodForms<4, 2>::Wide::SEG / 2) <= DemodForms<4, 2>::Wide::kSpread &&
                   d.dirichlet_terms > 1;
  const auto demod = [&](auto forms) {
    using L = decltype(forms);
    if (!any) launch(typename L::Terms{});
    else if (step * (L::Fine::SEG / 2) <= L::Fine::kSpread) launch(typename L::Fine{});
    else if (step * (L::Mid::SEG / 2) <= L::Mid::kSpread) launch(typename L::Mid{});
    else launch(typename L::Wide{});
  };
  // Few frequencies leave the chip idle unless more warps share a segment: per
  // pass with eight sharing | with two, 480 SFTs: 1000 frequencies 53 | 105 us,
  // 16000 72 | 107, 32768 117 | 121, 65536 193 | 180; 48 SFTs: 1000 27 | 33, 16000
  // 33 | 35, 32768 48 | 37.
  if (n_q * n_t <= 16384) demod(DemodForms<8, 8>{});
  else demod(DemodForms<4, 2>{});
  return cudaGetLastError();
}

}  // namespace fs
