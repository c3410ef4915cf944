// Internal declarations of the F-statistic library: plan constants, the
// per-template metadata, knot records of the time map, device math helpers
// and the in-place shared-memory FFT stages used by both FFT passes.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <atomic>
#include <type_traits>

#include "../../include/fstat.h"

namespace fs {

// ---------------------------------------------------------------- constants

constexpr double kC = 299792458.0;        // speed of light, m/s
constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr int kTwLog = 12;                // twiddle tables split at 2^12
constexpr int kTwLo = 1 << kTwLog;
constexpr int kMaxLog = 24;               // largest FFT: 2^24
constexpr int kMinLog = 12;               // smallest FFT: 2^12

// Plan constants passed by value to every kernel.
struct PlanConst {
  double dt, t_start, f_het, sigma2;
  int64_t n_data;
  int32_t interp, taps, window, precision;
  double lat, lon, gamma, radius;                 // detector
  double au, year, sid, obliq, orb0, sid0;        // ephemeris
  int32_t log2h;                                  // knot spacing (samples)
  int32_t pad_;
  // derived on the host (FP64): trigonometric constants of the plan
  double ce, se;                                  // cos, sin of the obliquity
  double sl, cl, s2l, c2l;                        // latitude
  double s2g, c2g;                                // arm-bisector angle
  double auc, rc;                                 // AU/c, R/c (s)
  double wo, ws;                                  // orbital and sidereal rates (rad/s)
  double th0;                                     // sidereal angle of the meridian at t = 0
  double inv_dt;                                  // 1 / dt
  double beta;                                    // bound of |dt_m/dt|: orbital and diurnal speed over c
  // output band: 2F is written for bins band_lo <= q < band_hi only, at
  // out_off + q - band_lo
  int64_t band_lo, band_hi;
};

// Bits of a unit of the sums of A, B, C: 2^24 points of scaled beam patterns,
// |a|, |b| <= 1 (scale_beams), stay below 2^61.
constexpr int kSumBits = 36;

// Per-template state produced by the time-map kernel and completed by the
// first FFT pass (sums A, B, C and the 2F coefficients).  One cache line.
struct TmplMeta {
  double tb0;        // t_b of grid point 0
  double A, B, C;    // masked antenna sums (Eq. 9 as sums)
  // the same while the tiled resampler adds them up, in units of 2^-kSumBits:
  // whole numbers, so that the order of the warps' additions does not matter
  unsigned long long acc[3];
  int64_t n_b;       // resampled length N_b
  int64_t out_off;   // output offset in floats
  int64_t span_lo, span_hi, gap_off, n_gaps;
  int32_t log2n;     // FFT length of this template
  int32_t status;    // FSTAT_OK or the error of this template, as the time map found it
  // the same, or FSTAT_ERANGE where A, B, C give no 2F, for the second pass.  Not
  // in `status`: the first pass sets it while other blocks still choose by
  // `status` whether a tile of this template is theirs, and the warps of a
  // block have to choose alike.
  int32_t status_2f;
  float ca, cb, cc;  // 2F = ca |Fa|^2 + cb |Fb|^2 + cc Re(Fa Fb*)
};
static_assert(sizeof(TmplMeta) == 128, "the second pass reads one line of it before its tile");

// Knot interval record, single precision evaluation (80 bytes).  On the
// interval [k_j, k_j + h) with s = k - k_j:
//   u(s)     = I + s + F + ((u3 s + u2) s + u1) s      fractional data index
//   P(s)     = P + ((p3 s + p2) s + p1) s              phase to remove, cycles
//   a(s)     = a0 + ((a3 s + a2) s + a1) s             beam pattern a(T^k)
//   b(s)     = b0 + ((b3 s + b2) s + b1) s
// I is exact, F = frac(U_j) and P = frac(P_j) are reduced in FP64, so only
// small deviations are carried in FP32.
struct __align__(16) KnotF {
  int32_t I; float F, u1, u2;
  float u3, P, p1, p2;
  float p3, a0, a1, a2;
  float a3, b0, b1, b2;
  float b3, r0, r1, r2;
};
// Double precision record (128 bytes); U is the full fractional index.
struct __align__(16) KnotD {
  double U, u1, u2, u3;
  double P, p1, p2, p3;
  double a0, a1, a2, a3;
  double b0, b1, b2, b3;
};

template <typename R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };
template <typename R> using cpx = typename Cx<R>::T;

// One element of both series, w_a and w_b side by side: the two transforms
// take the same indices and twiddles, so every thread carries both, one
// 16-byte access (FP32) moves a value of each and a twiddle is fetched (or
// formed) once for the two.
template <typename R> struct alignas(16) Pair { cpx<R> a, b; };

template <typename R> struct KnotOf;
template <> struct KnotOf<float> { using T = KnotF; };
template <> struct KnotOf<double> { using T = KnotD; };

// Twiddle tables: tl[L][m] = exp(-2 pi i m / 2^L) for m < min(2^L, 4096);
// th[L][m] = exp(-2 pi i m 4096 / 2^L) for L > 12, m < 2^(L-12).
template <typename R> struct Tw {
  const cpx<R>* tl[kMaxLog + 1];
  const cpx<R>* th[kMaxLog + 1];
};

// ---------------------------------------------------------------- launch settings
// A launch whose blocks may start while the kernel before it in the stream still
// runs (let_next_start, wait_for_previous): its launch, its blocks' start and
// the tables that they build are hidden behind the other's last blocks.  Worth it
// where a launch is short: (after one another | early) 1 template of 2^17 points
// 32.5 | 26.6 us, 64 of them 144 | 140, 1 of 2^22 86 | 82, 2 147 | 142.  At 2^24 points
// there is nothing to hide (8 templates of 2^21 262 | 262, 1 of 2^24 352 | 360), and
// a chunk of 64 x 2^22 takes 3079 | 3142; FP64, 1 of 2^22, 2031 | 2188.
template <typename R> inline bool starts_early(int64_t points) { return sizeof(R) == 4 && points <= (1 << 23); }

template <typename... P, typename... A>
cudaError_t launch_after(bool early, void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                         A... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = early ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
  if (e != cudaSuccess) (void)cudaGetLastError();      // reported here, not by a later call
  return e;
}

// Kernel attributes and the persistent grid sizes derived from them belong
// to a device, and a process may drive several GPUs: they are applied and
// cached per device (the current one at the call; devices 0..63).
constexpr int kMaxDevices = 64;
struct DeviceOnce {
  std::atomic<unsigned long long> done{0};
  std::atomic<int> value[kMaxDevices] = {};
};

// Runs set(dev, &v) once for the current device and returns its v in *out.
template <typename F>
inline cudaError_t device_once(DeviceOnce& o, int* out, F&& set) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  const unsigned long long bit = 1ull << dev;
  if (!(o.done.load(std::memory_order_acquire) & bit)) {
    int v = 0;
    e = set(dev, &v);
    if (e != cudaSuccess) return e;
    o.value[dev].store(v, std::memory_order_relaxed);
    o.done.fetch_or(bit, std::memory_order_release);
  }
  if (out) *out = o.value[dev].load(std::memory_order_relaxed);
  return cudaSuccess;
}

// Dynamic shared memory of a kernel, and the blocks of it that fit on the
// current device at once, set and measured once per device.
template <typename K>
inline cudaError_t kernel_setup(DeviceOnce& o, K kern, int threads, size_t smem, int* resident) {
  return device_once(o, resident, [&](int dev, int* v) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int sms = 0, per_sm = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    *v = sms * per_sm;
    return e;
  });
}

// ---------------------------------------------------------------- complex

__host__ __device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__host__ __device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__host__ __device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
template <typename T> __host__ __device__ __forceinline__ T czero();
template <> __host__ __device__ __forceinline__ float2 czero<float2>() { return make_float2(0.f, 0.f); }
template <> __host__ __device__ __forceinline__ double2 czero<double2>() { return make_double2(0.0, 0.0); }
template <typename T, typename S> __host__ __device__ __forceinline__ T cmk(S re, S im);
template <> __host__ __device__ __forceinline__ float2 cmk<float2, float>(float re, float im) { return make_float2(re, im); }
template <> __host__ __device__ __forceinline__ double2 cmk<double2, double>(double re, double im) { return make_double2(re, im); }

// multiply by -i (used by the in-register butterflies)
__device__ __forceinline__ float2 cmul_mi(float2 a) { return make_float2(a.y, -a.x); }
__device__ __forceinline__ double2 cmul_mi(double2 a) { return make_double2(a.y, -a.x); }

// ---------------------------------------------------------------- status

__device__ __forceinline__ void set_status(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

// ---------------------------------------------------------------- geometry
// Roemer delay t_m = n.r_d/c (Eq. 4pt2) and its rate n.v_d/c (Eq. 11c) for
// the analytic ephemeris, plus the JKS beam patterns a, b (Eqs. 2-3) in
// coefficient form a = e0 + e1 cos x + e2 sin x + e3 cos 2x + e4 sin 2x,
// b = f1 cos x + f2 sin x + f3 cos 2x + f4 sin 2x, x = alpha - theta(t).

template <typename R>
struct Sky {
  R nx, ny, nz;                 // unit vector to the source
  R ox, oy;                     // n . (cos phi, sin phi cos eps + ...) orbital projections
  R rz;                         // R sin(lat) nz / c
  R rxy;                        // R cos(lat) cos(delta) / c
  R alpha;
  R e0, e1, e2, e3, e4, f1, f2, f3, f4;
};

// sa, ca, sd, cd: sines and cosines of alpha and delta
template <typename R>
__device__ __forceinline__ Sky<R> make_sky(const PlanConst& pc, R alpha, R sa, R ca, R sd, R cd) {
  Sky<R> s;
  s.nx = cd * ca; s.ny = cd * sa; s.nz = sd;
  const R auc = (R)pc.auc;
  s.ox = auc * s.nx;                         // coefficient of cos(phi)
  s.oy = auc * ((R)pc.ce * s.ny + (R)pc.se * s.nz);      // coefficient of sin(phi)
  const R sl = (R)pc.sl, cl = (R)pc.cl;
  s.rz = (R)pc.rc * sl * sd;
  s.rxy = (R)pc.rc * cl * cd;
  s.alpha = alpha;
  const R s2g = (R)pc.s2g, c2g = (R)pc.c2g;
  const R c2l = (R)pc.c2l, s2l = (R)pc.s2l;
  const R c2d = cd * cd - sd * sd, s2d = 2 * sd * cd;
  s.e3 = s2g * (3 - c2l) * (3 - c2d) / 16;
  s.e4 = -c2g * sl * (3 - c2d) / 4;
  s.e1 = s2g * s2l * s2d / 4;
  s.e2 = -c2g * cl * s2d / 2;
  s.e0 = (R)0.75 * s2g * cl * cl * cd * cd;
  s.f3 = c2g * sl * sd;
  s.f4 = s2g * (3 - c2l) * sd / 4;
  s.f1 = c2g * cl * cd;
  s.f2 = s2g * s2l * cd / 2;
  return s;
}

template <typename R>
__device__ __forceinline__ void rsincos(R x, R* s, R* c) {
  if constexpr (std::is_same<R, float>::value) sincosf(x, s, c); else sincos(x, s, c);
}

template <typename R>
__device__ __forceinline__ Sky<R> make_sky(const PlanConst& pc, R alpha, R delta) {
  R sa, ca, sd, cd;
  rsincos<R>(alpha, &sa, &ca);
  rsincos<R>(delta, &sd, &cd);
  return make_sky<R>(pc, alpha, sa, ca, sd, cd);
}

// 2^-e with 2^e above the sum of the amplitudes, the bound of a pattern at any
// hour angle (a pattern below what FP32 holds is left as it is)
__device__ __forceinline__ float beam_scale(float amplitudes) {
  return amplitudes > 1e-37f && amplitudes < 1e37f ? __int_as_float((253 << 23) - (__float_as_int(amplitudes) & 0x7f800000))
                                                   : 1.0f;
}

// a and b each times a power of two that brings its bound to 1/2 .. 1.  2F is
// the same to the last bit (a^2 |Fb|^2, b^2 |Fa|^2 and ab Fa Fb* all over a^2 b^2 in
// Eq. 6), and the sums of A, B, C in fixed units keep their accuracy for
// patterns of any size: for a detector at the pole b is sin(delta) of its size
// elsewhere.
template <typename R>
__device__ __forceinline__ void scale_beams(Sky<R>& s) {
  const float ka = beam_scale(fabsf((float)s.e0) + fabsf((float)s.e1) + fabsf((float)s.e2) + fabsf((float)s.e3) +
                              fabsf((float)s.e4));
  const float kb = beam_scale(fabsf((float)s.f1) + fabsf((float)s.f2) + fabsf((float)s.f3) + fabsf((float)s.f4));
  s.e0 *= ka; s.e1 *= ka; s.e2 *= ka; s.e3 *= ka; s.e4 *= ka;
  s.f1 *= kb; s.f2 *= kb; s.f3 *= kb; s.f4 *= kb;
}
// The same by a warp, a coefficient a lane, on constants in shared memory: three
// instructions of the FP64 pipe, which the time map's other warps wait for.
__device__ __forceinline__ void scale_beams_warp(Sky<double>& s) {
  static_assert(sizeof(Sky<double>) == 17 * sizeof(double), "e0 .. e4, f1 .. f4 are the last nine of 17");
  const int lane = threadIdx.x & 31;
  double* c = reinterpret_cast<double*>(&s) + 8 + (lane < 9 ? lane : 0);
  const double v = *c;
  float a = lane < 5 ? fabsf((float)v) : 0.f, b = lane >= 5 && lane < 9 ? fabsf((float)v) : 0.f;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (lane < 9) *c = v * (double)beam_scale(lane < 5 ? a : b);
}

// t_m(t) and dt_m/dt; sH, cH: sin and cos of the hour angle theta(t) - alpha.
template <typename R>
__device__ __forceinline__ void roemer(const PlanConst& pc, const Sky<R>& s, R t, R* tm, R* rate,
                                       R* sH_out = nullptr, R* cH_out = nullptr) {
  const R wo = (R)pc.wo, ws = (R)pc.ws;
  R sp, cp, st, ct;
  rsincos<R>((R)pc.orb0 + wo * t, &sp, &cp);
  // hour-angle form: n . r_rot = R cos(lat) cos(delta) cos(theta - alpha) + R sin(lat) sin(delta)
  rsincos<R>((R)pc.th0 + ws * t - s.alpha, &st, &ct);
  *tm = s.ox * cp + s.oy * sp + s.rxy * ct + s.rz;
  *rate = wo * (s.oy * cp - s.ox * sp) - ws * s.rxy * st;
  if (sH_out) { *sH_out = st; *cH_out = ct; }
}

// a, b and their time derivatives from the hour angle H = theta - alpha
// (x = alpha - theta = -H).
template <typename R>
__device__ __forceinline__ void beams_h(const PlanConst& pc, const Sky<R>& s, R sH, R cH,
                                        R* a, R* b, R* da, R* db) {
  const R ws = (R)pc.ws;
  const R sx = -sH, cx = cH;
  const R c2x = cx * cx - sx * sx, s2x = 2 * sx * cx;
  *a = s.e0 + s.e1 * cx + s.e2 * sx + s.e3 * c2x + s.e4 * s2x;
  *b = s.f1 * cx + s.f2 * sx + s.f3 * c2x + s.f4 * s2x;
  // dx/dt = -ws
  *da = -ws * (-s.e1 * sx + s.e2 * cx - 2 * s.e3 * s2x + 2 * s.e4 * c2x);
  *db = -ws * (-s.f1 * sx + s.f2 * cx - 2 * s.f3 * s2x + 2 * s.f4 * c2x);
}

// a, b and their time derivatives at detector time t.
template <typename R>
__device__ __forceinline__ void beams(const PlanConst& pc, const Sky<R>& s, R t,
                                      R* a, R* b, R* da, R* db) {
  R sH, cH;
  rsincos<R>((R)pc.th0 + (R)pc.ws * t - s.alpha, &sH, &cH);
  beams_h<R>(pc, s, sH, cH, a, b, da, db);
}

// sin and cos of a small angle x (|x| <= 0.1) by their Taylor series to x^13
// and x^12 (truncation below 1e-19 relative).
template <typename R>
__device__ __forceinline__ void sincos_small(R x, R* s, R* c) {
  const R x2 = x * x;
  // coefficients 1/((2k)(2k+1)) and 1/((2k-1)(2k)) as compile-time constants
  *s = x * (1 - x2 * (R)(1.0 / 6) * (1 - x2 * (R)(1.0 / 20) * (1 - x2 * (R)(1.0 / 42) * (1 - x2 * (R)(1.0 / 72) *
       (1 - x2 * (R)(1.0 / 110) * (1 - x2 * (R)(1.0 / 156)))))));
  *c = 1 - x2 * (R)0.5 * (1 - x2 * (R)(1.0 / 12) * (1 - x2 * (R)(1.0 / 30) * (1 - x2 * (R)(1.0 / 56) *
       (1 - x2 * (R)(1.0 / 90) * (1 - x2 * (R)(1.0 / 132))))));
}

// (sin, cos) of an angle advanced by d: rotate (s, c) by d, d small when
// possible, else a full evaluation of the advanced angle a + d.
template <typename R>
__device__ __forceinline__ void advance(R a, R d, R* s, R* c) {
  if (fabs(d) <= (R)0.1) {
    R sd, cd;
    if (fabs(d) <= (R)1e-3) {
      // the same series to x^5 and x^6: the terms left out are below 1e-24
      const R x2 = d * d;
      sd = d * (1 - x2 * (R)(1.0 / 6) * (1 - x2 * (R)(1.0 / 20)));
      cd = 1 - x2 * (R)0.5 * (1 - x2 * (R)(1.0 / 12) * (1 - x2 * (R)(1.0 / 30)));
    } else if (fabs(d) <= (R)2e-2) {
      // to x^9 and x^8: below 1e-20
      const R x2 = d * d;
      sd = d * (1 - x2 * (R)(1.0 / 6) * (1 - x2 * (R)(1.0 / 20) * (1 - x2 * (R)(1.0 / 42) * (1 - x2 * (R)(1.0 / 72)))));
      cd = 1 - x2 * (R)0.5 * (1 - x2 * (R)(1.0 / 12) * (1 - x2 * (R)(1.0 / 30) * (1 - x2 * (R)(1.0 / 56) *
           (1 - x2 * (R)(1.0 / 90)))));
    } else {
      sincos_small<R>(d, &sd, &cd);
    }
    const R s0 = *s, c0 = *c;
    *s = s0 * cd + c0 * sd;
    *c = c0 * cd - s0 * sd;
  } else {
    rsincos<R>(a + d, s, c);
  }
}

// Detector time T with T + t_m(T) = tb (Eq. 21), by one Newton step from
// T0 = tb - t_m(tb): |dt_m/dt| <~ 1e-4 puts T0 within ~5e-2 s of T and
// |d2t_m/dt2| <~ 1e-10 s^-1 leaves ~1e-13 s after the step, below the
// rounding of T.  The orbital phase and hour angle at T0 and T are those at
// tb rotated by small angles (|t_m| <= AU/c + R/c), so only tb needs full
// sines and cosines.  Returns t_m(T), its rate and the hour-angle
// sine/cosine at T, and 1 / (1 + dt_m/dt).  Used by the all-FP32 time map; the
// FP64 one steps twice from the detector grid (timemap.cu).
__device__ __forceinline__ float inverse_time(const PlanConst& pc, const Sky<float>& s, float tb, float* tm_out,
                                              float* rate_out, float* sH, float* cH, float* inv1r_out) {
  const float wo = (float)pc.wo, ws = (float)pc.ws;
  const float phi = (float)pc.orb0 + wo * tb, hh = (float)pc.th0 + ws * tb - s.alpha;
  float sp, cp, st, ct;
  rsincos<float>(phi, &sp, &cp);
  rsincos<float>(hh, &st, &ct);
  float tm = s.ox * cp + s.oy * sp + s.rxy * ct + s.rz;
  // T0 = tb - tm: phases move by -w tm
  const float d0 = -tm;
  advance<float>(phi, wo * d0, &sp, &cp);
  advance<float>(hh, ws * d0, &st, &ct);
  const float T0 = tb + d0;
  tm = s.ox * cp + s.oy * sp + s.rxy * ct + s.rz;
  const float rate = wo * (s.oy * cp - s.ox * sp) - ws * s.rxy * st;
  const float inv1r = 1 / (1 + rate);
  const float dT = -(T0 + tm - tb) * inv1r;
  *inv1r_out = inv1r;
  // the hour angle at T to first order in ws dT (|ws dT| <~ 4e-6)
  const float e = ws * dT;
  *sH = st + ct * e;
  *cH = ct - st * e;
  *tm_out = tm + rate * dT;
  *rate_out = rate;
  return T0 + dT;
}

// ---------------------------------------------------------------- samples

// Read a complex64 sample as R-precision complex.
template <typename R>
__device__ __forceinline__ cpx<R> ldx(const float2* __restrict__ x, int j) {
  const float2 v = __ldg(x + j);
  return cmk<cpx<R>, R>((R)v.x, (R)v.y);
}

// Validity of data sample j for a template: inside its span and outside its
// gaps.  The cursor g only moves forward: callers query ascending j (the
// taps of one sample ascend, and every thread visits its samples in
// ascending order), so a thread walks the sorted gap list once in total.
struct GapCursor {
  const int64_t* __restrict__ gaps;  // pairs [start, end)
  int n, g;
  int lo, hi;
  int cs, ce;                        // the current gap [cs, ce), INT_MAX past the last
  __device__ __forceinline__ void load() {
    if (g < n) { cs = (int)__ldg(gaps + 2 * g); ce = (int)__ldg(gaps + 2 * g + 1); }
    else { cs = 0x7fffffff; ce = 0x7fffffff; }
  }
  __device__ __forceinline__ bool valid(int j) {
    if (j < lo || j >= hi) return false;
    while (ce <= j) { ++g; load(); }
    return j < cs;
  }
  // the first gap that ends after j (binary search; the cursor then
  // advances from there)
  __device__ __forceinline__ void seek(int j) {
    int a = 0, b = n;
    while (a < b) {
      const int mid = (a + b) >> 1;
      if ((int)__ldg(gaps + 2 * mid + 1) <= j) a = mid + 1; else b = mid;
    }
    g = a;
    load();
  }
  // the first gap that ends after j (j ascending)
  __device__ __forceinline__ void advance(int j) {
    while (ce <= j) { ++g; load(); }
  }
  // true iff every sample of [j0, j1] is valid; advances the cursor to j0
  __device__ __forceinline__ bool window_valid(int j0, int j1) {
    if (j0 < lo || j1 >= hi) return false;
    while (ce <= j0) { ++g; load(); }
    return j1 < cs;
  }
};

__device__ __forceinline__ GapCursor make_cursor(const TmplMeta& m, const int64_t* gaps) {
  GapCursor gc;
  gc.gaps = gaps + 2 * m.gap_off;
  gc.n = (int)m.n_gaps;
  gc.g = 0;
  gc.lo = (int)m.span_lo;
  gc.hi = (int)m.span_hi;
  gc.load();
  return gc;
}

// cos and sin of 2 pi k / 16 for k = 0..15
__host__ __device__ constexpr double c16(int k) {
  return k == 0 ? 1.0 : k == 1 ? 0.92387953251128675613 : k == 2 ? 0.70710678118654752440
       : k == 3 ? 0.38268343236508977173 : k == 4 ? 0.0 : k == 5 ? -0.38268343236508977173
       : k == 6 ? -0.70710678118654752440 : k == 7 ? -0.92387953251128675613 : k == 8 ? -1.0
       : k == 9 ? -0.92387953251128675613 : k == 10 ? -0.70710678118654752440
       : k == 11 ? -0.38268343236508977173 : k == 12 ? 0.0 : k == 13 ? 0.38268343236508977173
       : k == 14 ? 0.70710678118654752440 : 0.92387953251128675613;
}
__host__ __device__ constexpr double s16(int k) { return c16((k + 12) & 15); }  // sin(2 pi k/16) = cos(2 pi (k-4)/16)

// Rounding without conversion instructions: adding and subtracting 1.5 * 2^23
// rounds a float to the nearest integer (ties to even) exactly for
// |x| < 2^22, and the integer is the low mantissa bits of the sum.
__device__ __forceinline__ float round_nearest(float x, int* i) {
  const float t = __fadd_rn(x, 12582912.0f);
  *i = __float_as_int(t) - 0x4B400000;
  return __fsub_rn(t, 12582912.0f);
}
// Between two kernels of one stream where the second is launched by
// launch_after: the first allows the second's blocks to start once all of its
// own have (they take what room is left), and the second waits, before it
// touches anything the first writes, until the first is complete and its writes
// are visible.  Every block waits, also one with nothing to do: a kernel that
// is complete then vouches for all before it.  Loads that the compiler may move
// (read-only and streaming ones) of what the first kernel wrote stand behind a
// branch on the template's metadata, which is loaded after the wait; before it
// a kernel reads the plan's tables only and writes its own shared memory only.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// exact float of a small non-negative integer (< 2^23)
__device__ __forceinline__ float small_int_to_float(int k) {
  return __fsub_rn(__int_as_float(0x4B000000 | k), 8388608.0f);
}

// sin and cos of pi x for |x| <= 1/4 by their Taylor series (terms to x^9
// and x^10; truncation below 2e-9), single precision.
__device__ __forceinline__ void sincospi_small(float x, float* s, float* c) {
  const float t = 3.14159265358979f * x;
  const float t2 = t * t;
  *s = t * fmaf(t2, fmaf(t2, fmaf(t2, fmaf(t2, 2.75573192e-6f, -1.98412698e-4f), 8.33333333e-3f),
                         -1.66666667e-1f), 1.0f);
  *c = fmaf(t2, fmaf(t2, fmaf(t2, fmaf(t2, fmaf(t2, -2.75573192e-7f, 2.48015873e-5f), -1.38888889e-3f),
                               4.16666667e-2f), -0.5f), 1.0f);
}

// exp(-2 pi i r) for |r| <= 1/2: quarter turns split off exactly, the rest
// (|f| <= 1/8) by sincospi_small.
__device__ __forceinline__ float2 expm2pi(float r) {
  int qi;
  const float q = round_nearest(4.0f * r, &qi);
  const float f = fmaf(-0.25f, q, r);
  float sn, cs;
  sincospi_small(2.0f * f, &sn, &cs);
  // exp(-2 pi i f) = (cs, -sn), times (-i)^q
  qi &= 3;
  float re = cs, im = -sn;
  if (qi & 1) { const float t = re; re = im; im = -t; }   // times -i
  if (qi & 2) { re = -re; im = -im; }                      // times -1
  return make_float2(re, im);
}

// Window constants cos/sin(pi m / H), m = -H..H: FP64 at wcs[0..63], the
// same values rounded to FP32 right after them (wcs + 64 doubles).
template <typename R> __device__ __forceinline__ const R* win_table(const double* wcs);
template <> __device__ __forceinline__ const double* win_table<double>(const double* wcs) { return wcs; }
template <> __device__ __forceinline__ const float* win_table<float>(const double* wcs) {
  return reinterpret_cast<const float*>(wcs + 64);
}

__device__ __forceinline__ float rcp_approx(float v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

// Step 4 of Sec. III.A.2 with the 8-tap windowed sinc in single precision.
// n0 = floor(u), f = u - n0 in [0, 1), qoff = (f >= 1/2), dn = f - qoff (so
// that jnn = n0 + qoff is the nearest sample and dn = u - jnn).  Tap i
// (i = 0..7, sample j = n0 - 3 + i) sits at x_i = f + 3 - i; the nearest tap
// gets x = dn exactly (f - 1 is exact for f >= 1/2), so its weight and
// sin(pi dn) come from the same number.  With s = sin(pi f):
//   sin(pi x_i) = (-1)^(3-i) s,
//   sin(pi x_i / 4) = sin(pi f/4) cos(pi (3-i)/4) + cos(pi f/4) sin(pi (3-i)/4),
// and x_{i+4} = x_i - 4 turns sin(pi x / 4) into its negative.  Lanczos:
// K(x) = 4 sin(pi x) sin(pi x/4) / (pi^2 x^2); plain truncation: sin(pi x)/(pi x).
// The common factor s leaves the sum over taps.  Returns the mask (the
// nearest sample is valid data); taps on invalid samples weigh zero.
// The taps of a window that touches a gap or the span's edge: each tap on
// an invalid sample weighs zero; the result is valid when the nearest sample
// is.  w0..w3: the window factors of taps 0..3 (sinc8_f32).
__device__ __forceinline__ bool sinc8_f32_edge(const float2* __restrict__ x, GapCursor& gc, bool lanczos,
                                            int jlo, int jnn, float f, float w0, float w1, float w2,
                                            float w3, float2& acc) {
  bool msk = false;
  acc = make_float2(0.f, 0.f);
  for (int i = 0; i < 8; ++i) {
    const int j = jlo + i;
    const bool ok = gc.valid(j);
    if (j == jnn) msk = ok;
    if (!ok) continue;
    const float2 t = __ldg(x + j);
    const float xi = f + (float)(3 - i);
    const float sg = ((3 - i) & 1) ? -1.0f : 1.0f;              // (-1)^(3-i)
    const int q = i & 3;
    const float wq = q == 0 ? w0 : (q == 1 ? w1 : (q == 2 ? w2 : w3));
    const float w = lanczos ? sg * (i < 4 ? wq : -wq) * rcp_approx(xi * xi) : sg * rcp_approx(xi);
    acc.x = fmaf(w, t.x, acc.x);
    acc.y = fmaf(w, t.y, acc.y);
  }
  return msk;
}

__device__ __forceinline__ bool sinc8_f32(const float2* __restrict__ x, GapCursor& gc, bool lanczos,
                                          int n0, int qoff, float f, float dn, float2& z) {
  const int jlo = n0 - 3;
  const int jnn = n0 + qoff;
  if (fabsf(dn) < 1e-7f) {
    // u on a sample (to the precision of u): the interpolant is that sample
    if (!gc.valid(jnn)) return false;
    z = __ldg(x + jnn);
    return true;
  }
  const bool full = gc.window_valid(jlo, jlo + 7);
  float2 v[8];
  if (full) {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __ldg(x + jlo + i);
  }
  // sin, cos of pi dn / 4 by the polynomial; sin(pi dn) by two doublings
  float sh, ch;
  sincospi_small(0.25f * dn, &sh, &ch);
  const float s2 = 2.0f * sh * ch, c2 = fmaf(ch, ch, -sh * sh);
  const float sdn = 2.0f * s2 * c2;
  const float sf = qoff ? -sdn : sdn;                     // sin(pi f)
  float2 acc = make_float2(0.f, 0.f);
  // sin(pi x_i / 4) for i = 0..3: with p = (sin + cos)(pi dn/4) / sqrt 2 and
  // m = (cos - sin)(pi dn/4) / sqrt 2 these are (m, cos, p, sin) for
  // qoff = 0 and (-sin, m, cos, p) for qoff = 1 (f/4 = dn/4 + 1/4)
  const float r2 = 0.70710678118654752f;
  const float p = (sh + ch) * r2, m = (ch - sh) * r2;
  const float w0 = qoff ? -sh : m, w1 = qoff ? m : ch, w2 = qoff ? ch : p, w3 = qoff ? p : sh;
  if (lanczos) {
    // sign (-1)^(3-i) times the window, i = 0..3; taps 4..7 take the negatives
    float g[8];
    g[0] = -w0; g[1] = w1; g[2] = -w2; g[3] = w3;
    g[4] = w0; g[5] = -w1; g[6] = w2; g[7] = -w3;
    if (full) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float xi = f + (float)(3 - i);
        const float w = g[i] * rcp_approx(xi * xi);
        acc.x = fmaf(w, v[i].x, acc.x);
        acc.y = fmaf(w, v[i].y, acc.y);
      }
    }
  } else {
    if (full) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float w = rcp_approx(f + (float)(3 - i));
        if ((3 - i) & 1) {
          acc.x = fmaf(-w, v[i].x, acc.x);
          acc.y = fmaf(-w, v[i].y, acc.y);
        } else {
          acc.x = fmaf(w, v[i].x, acc.x);
          acc.y = fmaf(w, v[i].y, acc.y);
        }
      }
    }
  }
  if (!full && !sinc8_f32_edge(x, gc, lanczos, jlo, jnn, f, w0, w1, w2, w3, acc)) return false;
  const float sc = lanczos ? sf * (float)(4.0 / (3.14159265358979323846 * 3.14159265358979323846))
                           : sf * (float)(1.0 / 3.14159265358979323846);
  z = make_float2(acc.x * sc, acc.y * sc);
  return true;
}

// sin and cos of pi x for |x| <= 1/4 by their Taylor series (terms to x^17 and
// x^16; truncation below 4e-20), double precision.  The FP64 pipe is what the
// double-precision resampler waits for, so its elementary functions are kept
// to what their arguments need.
__device__ __forceinline__ void sincospi_small(double x, double* s, double* c) {
  const double t = 3.14159265358979323846 * x;
  const double u = t * t;
  *s = t * fma(u, fma(u, fma(u, fma(u, fma(u, fma(u, fma(u, fma(u, 1.0 / 355687428096000.0, -1.0 / 1307674368000.0),
           1.0 / 6227020800.0), -1.0 / 39916800.0), 1.0 / 362880.0), -1.0 / 5040.0), 1.0 / 120.0), -1.0 / 6.0), 1.0);
  *c = fma(u, fma(u, fma(u, fma(u, fma(u, fma(u, fma(u, fma(u, 1.0 / 20922789888000.0, -1.0 / 87178291200.0),
           1.0 / 479001600.0), -1.0 / 3628800.0), 1.0 / 40320.0), -1.0 / 720.0), 1.0 / 24.0), -0.5), 1.0);
}

// exp(-2 pi i r) for |r| <= 1/2, as the single-precision form.
__device__ __forceinline__ double2 expm2pi(double r) {
  const double q = rint(4.0 * r);
  double sn, cs;
  sincospi_small(2.0 * fma(-0.25, q, r), &sn, &cs);
  const int qi = (int)q & 3;
  double re = cs, im = -sn;
  if (qi & 1) { const double t = re; re = im; im = -t; }   // times -i
  if (qi & 2) { re = -re; im = -im; }                      // times -1
  return make_double2(re, im);
}

// The weights of the 8-tap windowed sinc in double precision at the fraction
// f (x_i = f + 3 - i, dn = f or f - 1 the offset from the nearest sample, not
// 0).  The products x_i x_{7-i} = f (f - 1) - (0, 2, 6, 12) share one
// reciprocal, and 1 / x_i = x_{7-i} / (x_i x_{7-i}); sin(pi x_i) and
// sin(pi x_i / 4) come from sin, cos(pi dn / 4): about 75 FP64 operations
// where eight divisions and two sincospi took over 200.
__device__ __forceinline__ void sinc8_weights(double f, double dn, int qoff, bool lanczos, double (&w)[8]) {
  double sh, ch;
  sincospi_small(0.25 * dn, &sh, &ch);
  const double s2 = 2.0 * sh * ch, c2 = fma(ch, ch, -sh * sh);
  const double sdn = 2.0 * s2 * c2;
  const double sf = qoff ? -sdn : sdn;                     // sin(pi f)
  const double q = f * (qoff ? dn : f - 1.0);              // f (f - 1): both factors exact
  const double q1 = q - 2.0, q2 = q - 6.0, q3 = q - 12.0;
  const double p01 = q * q1, p23 = q2 * q3;
  const double r = __drcp_rn(p01 * p23);
  const double r01 = r * p23, r23 = r * p01;
  const double ip[4] = {r23 * q2, r23 * q3, r01 * q, r01 * q1};   // 1 / (x_i x_{7-i}), i = 0 .. 3
  double ix[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double xa = i == 3 && qoff == 0 ? dn : f + (double)(3 - i);
    const double xb = i == 3 && qoff ? dn : f + (double)(i - 4);
    ix[i] = xb * ip[i];
    ix[7 - i] = xa * ip[i];
  }
  if (lanczos) {
    const double r2 = 0.70710678118654752440;
    const double p = (sh + ch) * r2, m = (ch - sh) * r2;
    const double k = sf * (4.0 / (3.14159265358979323846 * 3.14159265358979323846));
    // (-1)^(3-i) sin(pi x_i / 4) for i = 0 .. 3; taps 4 .. 7 take the negatives
    const double g[4] = {-k * (qoff ? -sh : m), k * (qoff ? m : ch), -k * (qoff ? ch : p), k * (qoff ? p : sh)};
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = (i < 4 ? g[i & 3] : -g[i & 3]) * (ix[i] * ix[i]);
  } else {
    const double k = sf * (1.0 / 3.14159265358979323846);
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = (((3 - i) & 1) ? -k : k) * ix[i];
  }
}

// Phase P + ((p3 s + p2) s + p1) s of a knot interval, mod 1: the linear
// term reaches many cycles at the end of an interval, so its whole cycles come
// off exactly before the terms are added.
__device__ __forceinline__ float knot_phase(float P, float p1, float p2, float p3, float s) {
  int n;
  const float whole = round_nearest(p1 * s, &n);
  return P + fmaf((p3 * s + p2) * s, s, fmaf(p1, s, -whole));
}

// Per-sample time map and weights (steps 2-5) at grid point k < N_b of a
// template: returns the mask and writes wa = m a y, wb = m b y with
// y = z(T^k) exp(-2 pi i P(k)), and the beam values a, b.
template <typename R, int INTERP, int TAPS>
__device__ __forceinline__ bool sample_weights(
    const PlanConst& pc, const typename KnotOf<R>::T* __restrict__ kn,
    int k, const float2* __restrict__ x, GapCursor& gc,
    const double* __restrict__ wcs, cpx<R>& wa, cpx<R>& wb, R& a, R& b) {
  using C = cpx<R>;
  const int jint = k >> pc.log2h;
  const int sk = k & ((1 << pc.log2h) - 1);
  R s;
  if constexpr (std::is_same<R, float>::value) s = small_int_to_float(sk); else s = (R)sk;
  int ibase;       // integer part of u before the deviation
  R dev;           // u = ibase + dev
  R ph;            // phase cycles
  if constexpr (std::is_same<R, float>::value) {
    const float4* q = reinterpret_cast<const float4*>(kn + jint);
    const float4 r0 = __ldg(q), r1 = __ldg(q + 1), r2 = __ldg(q + 2), r3 = __ldg(q + 3), r4 = __ldg(q + 4);
    ibase = __float_as_int(r0.x) + sk;
    dev = r0.y + ((r1.x * s + r0.w) * s + r0.z) * s;
    ph = knot_phase(r1.y, r1.z, r1.w, r2.x, s);
    a = r2.y + ((r3.x * s + r2.w) * s + r2.z) * s;
    b = r3.y + ((r4.x * s + r3.w) * s + r3.z) * s;
  } else {
    const KnotD& q = kn[jint];
    const double u = q.U + s + ((q.u3 * s + q.u2) * s + q.u1) * s;
    const double fl = floor(u);
    ibase = (int)fl;
    dev = u - fl;
    ph = q.P + ((q.p3 * s + q.p2) * s + q.p1) * s;
    a = q.a0 + ((q.a3 * s + q.a2) * s + q.a1) * s;
    b = q.b0 + ((q.b3 * s + q.b2) * s + q.b1) * s;
  }
  C z;
  if constexpr (std::is_same<R, float>::value && INTERP == FSTAT_SINC && TAPS == 8) {
    // n0 = floor(u) = ibase + fl, f = dev - fl exactly
    int fl_i;
    float fl = round_nearest(dev, &fl_i);
    if (fl > dev) { fl -= 1.0f; --fl_i; }
    const float f = dev - fl;
    const int qoff = f >= 0.5f ? 1 : 0;
    const float dn = qoff ? f - 1.0f : f;
    float2 zz;
    if (!sinc8_f32(x, gc, pc.window == FSTAT_WIN_LANCZOS, ibase + fl_i, qoff, f, dn, zz)) {
      wa = czero<C>(); wb = czero<C>(); return false;
    }
    z = zz;
  } else if constexpr (std::is_same<R, double>::value && INTERP == FSTAT_SINC && TAPS == 8) {
    const int qoff = dev >= 0.5 ? 1 : 0;
    const double dn = qoff ? dev - 1.0 : dev;   // dev = u - floor(u)
    const int jlo = ibase - 3, jnn = ibase + qoff;
    if (dn == 0.0) {
      // u on a sample: the interpolant is that sample
      if (!gc.valid(jnn)) { wa = czero<C>(); wb = czero<C>(); return false; }
      z = ldx<R>(x, jnn);
    } else {
      const bool full = gc.window_valid(jlo, jlo + 7);
      float2 v[8];
      if (full) {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = __ldg(x + jlo + i);
      }
      double w[8];
      sinc8_weights(dev, dn, qoff, pc.window == FSTAT_WIN_LANCZOS, w);
      double2 acc = make_double2(0.0, 0.0);
      bool msk = full;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float2 t = v[i];
        if (!full) {
          const bool ok = gc.valid(jlo + i);
          if (jlo + i == jnn) msk = ok;
          t = ok ? __ldg(x + jlo + i) : make_float2(0.f, 0.f);
        }
        acc.x = fma(w[i], (double)t.x, acc.x);
        acc.y = fma(w[i], (double)t.y, acc.y);
      }
      if (!msk) { wa = czero<C>(); wb = czero<C>(); return false; }
      z = acc;
    }
  } else {
  int jnn_off;                        // jnn - ibase = floor(dev + 1/2)
  R jnn_f;
  if constexpr (std::is_same<R, float>::value) {
    // floor(dev + 1/2): round to nearest, step down where that rounded up
    // past dev + 1/2 (dev + 1/2 lies in (-1, 3), far inside the exact range)
    jnn_f = round_nearest(dev + 0.5f, &jnn_off);
    if (jnn_f > dev + 0.5f) { jnn_f -= 1.0f; --jnn_off; }
  } else {
    jnn_f = floor(dev + 0.5);
    jnn_off = (int)jnn_f;
  }
  const int jnn = ibase + jnn_off;
  if constexpr (INTERP == FSTAT_NEAREST) {
    if (!gc.valid(jnn)) { wa = czero<C>(); wb = czero<C>(); return false; }
    z = ldx<R>(x, jnn);
  } else {
    // (8 taps have a form of their own above)
    static_assert(TAPS == 0, "the number of taps is the plan's");
    const int taps = pc.taps;
    const int half = taps >> 1;
    // offset from the nearest sample, dn = u - jnn in [-1/2, 1/2]; every
    // weight is formed from sin/cos of pi dn and pi dn / H, so the tap next
    // to u gets its value without cancellation and the others have |x| >= 1/2
    const R dn = dev - jnn_f;
    const int qoff = dn >= (R)0 ? 0 : 1;       // jnn - floor(u)
    const int n0 = jnn - qoff;                 // floor(u)
    if (dn == (R)0) {
      bool ok = false;
      for (int j = n0 - half + 1; j <= jnn; ++j) ok = gc.valid(j);
      if (!ok) { wa = czero<C>(); wb = czero<C>(); return false; }
      z = ldx<R>(x, jnn);
    } else {
      // x = u - j = dn + mq with mq = jnn - j; sin(pi x) = (-1)^mq sin(pi dn);
      // sin(pi x / H) = sin(pi dn/H) cos(pi mq/H) + cos(pi dn/H) sin(pi mq/H)
      constexpr int NTAP = 16;
      // the common case: the whole window is valid data; the loads then go
      // out from one base pointer before any weight arithmetic
      const int jlo = n0 + 1 - half;
      const bool full = gc.window_valid(jlo, jlo + taps - 1);
      C v[NTAP];
      if (full) {
        const float2* xb = x + jlo;
#pragma unroll
        for (int i = 0; i < NTAP; ++i) {
          if (i >= taps) break;
          const float2 t2 = __ldg(xb + i);
          v[i] = cmk<C, R>((R)t2.x, (R)t2.y);
        }
      } else {
#pragma unroll
        for (int i = 0; i < NTAP; ++i) {
          if (i >= taps) break;
          int j = jlo + i;
          j = j < gc.lo ? gc.lo : (j >= gc.hi ? gc.hi - 1 : j);
          v[i] = ldx<R>(x, j);
        }
      }
      R S, Cd, sh, chh;
      if constexpr (std::is_same<R, float>::value) {
        sincospif(dn, &S, &Cd);
        sincospif(dn / (R)half, &sh, &chh);
      } else {
        sincospi(dn, &S, &Cd);
        sincospi(dn / (R)half, &sh, &chh);
      }
      const R inv_pi2 = (R)(1.0 / (3.14159265358979323846 * 3.14159265358979323846));
      const bool lanczos = pc.window == FSTAT_WIN_LANCZOS;
      const R* wt = win_table<R>(wcs);
      // tap i sits at x = dn + mq with mq = (half - 1 - i) + qoff: dn is added
      // to an exact small integer, so the tap at the nearest sample keeps x = dn
      // exactly;
      // (-1)^mq = (-1)^(half-1-i) (-1)^qoff: the qoff factor goes into Sp
      const R Sp = (qoff ? -S : S) * inv_pi2;
      C acc = czero<C>();
      bool msk = false;
      [[maybe_unused]] R inv = (R)0, inv_next = (R)0;
#pragma unroll
      for (int i = 0; i < NTAP; ++i) {
        if (i >= taps) break;
        const int mq = half - 1 - i + qoff;       // jnn - j
        const int j = n0 + 1 - half + i;
        const R xx = dn + (R)mq;
        R w;
        if constexpr (std::is_same<R, float>::value) {
          w = __fdividef(Sp, xx * xx);
        } else {
          // one division for two taps (one template of 2^22, 16 taps: 3019 -> 2588 us)
          if ((i & 1) == 0) {
            const R xn = dn + (R)(mq - 1);
            const R r = (R)1 / (xx * xn);
            inv = r * xn;
            inv_next = r * xx;
          } else {
            inv = inv_next;
          }
          w = Sp * (inv * inv);
        }
        if ((mq & 1) != qoff) w = -w;
        if (lanczos) {
          const R cm = __ldg(wt + 2 * (mq + half)), sm = __ldg(wt + 2 * (mq + half) + 1);
          w *= (R)half * (sh * cm + chh * sm);
        } else {
          w *= (R)3.14159265358979323846 * xx;   // plain truncated sinc: sin(pi x)/(pi x)
        }
        if (!full) {
          const bool ok = gc.valid(j);
          if (j == jnn) msk = ok;
          if (!ok) w = (R)0;
        }
        if constexpr (std::is_same<R, float>::value) {
          acc.x = fmaf(w, v[i].x, acc.x);
          acc.y = fmaf(w, v[i].y, acc.y);
        } else {
          acc.x = fma(w, v[i].x, acc.x);
          acc.y = fma(w, v[i].y, acc.y);
        }
      }
      if (full) msk = true;
      if (!msk) { wa = czero<C>(); wb = czero<C>(); return false; }
      z = acc;
    }
  }
  }
  // remove exp(2 pi i P): multiply by exp(-2 pi i r), r = P - rint(P)
  C e;
  if constexpr (std::is_same<R, float>::value) {
    int dummy;
    const float r = ph - round_nearest(ph, &dummy);
    e = expm2pi(r);
  } else {
    e = expm2pi(ph - rint(ph));
  }
  const C y = cmul(z, e);
  wa = cmk<C, R>(a * y.x, a * y.y);
  wb = cmk<C, R>(b * y.x, b * y.y);
  return true;
}

// ---------------------------------------------------------------- FFT
// In-register DFT of RAD points (forward, e^{-2 pi i jk/RAD}) by radix-2
// decimation in time; twiddles are compile-time constants.

template <typename T, int RAD, int STRIDE = 1>
struct Dft {
  // v[0], v[STRIDE], ... hold the RAD inputs; outputs in natural order at the same slots
  __device__ __forceinline__ static void run(T* v) {
    if constexpr (RAD == 1) {
      return;
    } else {
      // even/odd split: evens at stride 2*STRIDE from 0, odds from STRIDE
      Dft<T, RAD / 2, 2 * STRIDE>::run(v);
      Dft<T, RAD / 2, 2 * STRIDE>::run(v + STRIDE);
      T tmp[RAD];
#pragma unroll
      for (int k = 0; k < RAD / 2; ++k) {
        const T e = v[2 * k * STRIDE];
        T o = v[(2 * k + 1) * STRIDE];
        constexpr int step = 16 / RAD;
        const int kk = k * step;                // W_RAD^k = W_16^(k*16/RAD)
        if (kk == 4) {
          o = cmul_mi(o);
        } else if (kk != 0) {
          using R = decltype(o.x);
          const T w = cmk<T, R>((R)c16(kk), (R)(-s16(kk)));
          o = cmul(o, w);
        }
        tmp[k] = cadd(e, o);
        tmp[k + RAD / 2] = csub(e, o);
      }
#pragma unroll
      for (int k = 0; k < RAD; ++k) v[k * STRIDE] = tmp[k];
    }
  }
};

// A transform of N = 16 RM RL points in shared memory, in place.  With
//   k = lo + RL (mid + RM hi)   and   p = p0 + 16 (q1 + RM q2)
// its stages run over hi (radix 16), mid (radix RM, if any) and lo (radix RL),
// and a butterfly's outputs take the places of its inputs, [p0][q1][lo]: only
// one barrier lies between two stages, where writing a stage in transform
// order needs a second one between its reads and its writes.  The low bits of a place are
// xored with its first digit, so that the accesses of a quarter-warp (8
// lanes of 16 bytes), which run over lo in the first two stages and over p0
// in the last, fall on distinct banks without padding.
// With COUNT >= 8 interleaved sequences the lanes run over these, on distinct
// banks by their stride, and the key is left out.
template <int LOGN, int RBL, int COUNT> struct FftPlan {
  static constexpr int RBM = LOGN - 4 - RBL;
  static constexpr int RM = 1 << RBM, RL = 1 << RBL;
  static constexpr int SUB = RM * RL;               // points of one hi digit: N / 16
  static constexpr int KEYS = COUNT >= 8 ? 0 : (SUB < 8 ? SUB - 1 : 7);
  static __device__ __forceinline__ int key(int hi) { return hi & KEYS; }
  // place of (hi, j), j = mid RL + lo
  static __device__ __forceinline__ int place(int hi, int j) { return hi * SUB + (j ^ key(hi)); }
};
// Sequence stride in shared memory, in pairs.  Fills and epilogues interleave
// C sequences across the lanes of a quarter-warp; a stride congruent to 8/C
// mod 8 puts them on distinct banks.
template <int LOGN, int C> struct FftGeom {
  static constexpr int N = 1 << LOGN;
  static constexpr int WANT = C >= 8 ? 1 : 8 / C;
  static constexpr int STRIDE = N + (WANT & 7);
};

// Twiddles of the middle stage, held in shared memory: input mid = r of the
// butterfly (p0, lo) takes W_{16 RM}^{r p0}, table [r - 1][p0], r = 1 .. RM - 1.
constexpr int mid_tw_count(int rbm) { return ((1 << rbm) - 1) << 4; }
// Filled from the length-2^LOGN table tw (all threads).
template <typename R, int LOGN, int RBM, int NT>
__device__ __forceinline__ void build_mid_tw(cpx<R>* __restrict__ dst, const cpx<R>* __restrict__ tw) {
  for (int e = threadIdx.x; e < mid_tw_count(RBM); e += NT)
    dst[e] = __ldg(tw + ((((e >> 4) + 1) * (e & 15)) << (LOGN - 4 - RBM)));
}
// The last stage (radix 2^RB at NS = 2^NSL, LOGN = NSL + RB) keeps only the
// powers W^k, W^{2k}, W^{4k}, ...: row p holds W_{2^LOGN}^{2^p k}, k < NS.  A
// thread forms the others as products, once for both series: the rows in
// full would take 30 KB of shared memory and 15 loads at radix 16.
template <int NSL, int RB> constexpr int last_tw_count() { return RB << NSL; }
template <typename R, int LOGN, int NSL, int RB, int NT>
__device__ __forceinline__ void build_last_tw(cpx<R>* __restrict__ dst, const cpx<R>* __restrict__ tw) {
  static_assert(LOGN == NSL + RB, "the last stage completes the transform");
  for (int e = threadIdx.x; e < last_tw_count<NSL, RB>(); e += NT) {
    const int p = e >> NSL, k = e & ((1 << NSL) - 1);
    dst[e] = __ldg(tw + (k << p));
  }
}
// t[q] = first * W^{q k}, q < 2^RB, from the rows of build_last_tw (lt points
// at column k): one product each, at most RB deep.
template <typename R, int NSL, int RB>
__device__ __forceinline__ void last_twiddles(const cpx<R>* __restrict__ lt, cpx<R> first, cpx<R>* __restrict__ t) {
  t[0] = first;
#pragma unroll
  for (int p = 0; p < RB; ++p) {
    const cpx<R> w = lt[p << NSL];
#pragma unroll
    for (int q = 0; q < (1 << p); ++q) t[(1 << p) + q] = cmul(t[q], w);
  }
}

// The first stage in shared memory (persistent mode; elsewhere its inputs come
// from global memory) over COUNT interleaved sequences f at buf + f * STRIDE.
template <typename R, int LOGN, int RBL, int NT, int COUNT, int STRIDE>
__device__ __forceinline__ void first_stage(Pair<R>* __restrict__ buf) {
  using C = cpx<R>;
  using P = FftPlan<LOGN, RBL, COUNT>;
#pragma unroll 1
  for (int u = threadIdx.x; u < COUNT * P::SUB; u += NT) {
    Pair<R>* x = buf + (u % COUNT) * STRIDE;
    const int j = u / COUNT;
    C va[16], vb[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) { const Pair<R> v = x[P::place(r, j)]; va[r] = v.a; vb[r] = v.b; }
    Dft<C, 16>::run(va);
    Dft<C, 16>::run(vb);
#pragma unroll
    for (int r = 0; r < 16; ++r) x[P::place(r, j)] = Pair<R>{va[r], vb[r]};
  }
  __syncthreads();
}

// The middle stage: butterflies (p0, lo) over mid, twiddles tws
// (build_mid_tw); lanes run over the sequences, then lo, then p0.
template <typename R, int LOGN, int RBL, int NT, int COUNT, int STRIDE>
__device__ __forceinline__ void mid_stage(Pair<R>* __restrict__ buf, const cpx<R>* __restrict__ tws) {
  using C = cpx<R>;
  using P = FftPlan<LOGN, RBL, COUNT>;
  if constexpr (P::RBM > 0) {
    constexpr int UNITS = COUNT * 16 * P::RL;
#pragma unroll
    for (int u0 = 0; u0 < UNITS; u0 += NT) {
      const int u = u0 + threadIdx.x;
      if (UNITS % NT == 0 || u < UNITS) {
        const int b = u / COUNT;
        const int lo = b & (P::RL - 1), p0 = b >> RBL;
        Pair<R>* x = buf + (u % COUNT) * STRIDE + p0 * P::SUB;
        const int o = lo ^ P::key(p0);
        C va[P::RM], vb[P::RM];
#pragma unroll
        for (int r = 0; r < P::RM; ++r) {
          const Pair<R> v = x[o + r * P::RL];
          va[r] = v.a;
          vb[r] = v.b;
          if (r > 0) {
            const C w = tws[((r - 1) << 4) + p0];
            va[r] = cmul(va[r], w);
            vb[r] = cmul(vb[r], w);
          }
        }
        Dft<C, P::RM>::run(va);
        Dft<C, P::RM>::run(vb);
#pragma unroll
        for (int r = 0; r < P::RM; ++r) x[o + r * P::RL] = Pair<R>{va[r], vb[r]};
      }
    }
    __syncthreads();
  }
}

// streaming access to one pair (both planes of an FP32 pair in 16 bytes)
__device__ __forceinline__ Pair<float> ldcs(const Pair<float>* p) {
  const float4 v = __ldcs(reinterpret_cast<const float4*>(p));
  return Pair<float>{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ Pair<double> ldcs(const Pair<double>* p) {
  return Pair<double>{__ldcs(&p->a), __ldcs(&p->b)};
}
__device__ __forceinline__ void stcs(Pair<float>* p, const Pair<float>& v) {
  __stcs(reinterpret_cast<float4*>(p), make_float4(v.a.x, v.a.y, v.b.x, v.b.y));
}
__device__ __forceinline__ void stcs(Pair<double>* p, const Pair<double>& v) {
  __stcs(&p->a, v.a);
  __stcs(&p->b, v.b);
}

// exp(-2 pi i m / 2^L) from the two-level tables
template <typename R>
__device__ __forceinline__ cpx<R> twiddle(const Tw<R>& tw, int L, uint32_t m) {
  if (L <= kTwLog) return __ldg(tw.tl[L] + m);
  return cmul(__ldg(tw.th[L] + (m >> kTwLog)), __ldg(tw.tl[L] + (m & (kTwLo - 1))));
}

// Block-wide sum of three values (any block size multiple of 32, <= 1024):
// warp sums in FP32, the sum over warps in FP64 (the result is in thread 0).
__device__ __forceinline__ void block_sum3(float fx, float fy, float fz, double& x, double& y, double& z,
                                           double* sh /*[3*32]*/) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    fx += __shfl_down_sync(0xffffffffu, fx, o);
    fy += __shfl_down_sync(0xffffffffu, fy, o);
    fz += __shfl_down_sync(0xffffffffu, fz, o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) { sh[wid] = fx; sh[32 + wid] = fy; sh[64 + wid] = fz; }
  __syncthreads();
  x = y = z = 0.0;
  if (threadIdx.x == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    for (int w = 0; w < nw; ++w) { x += sh[w]; y += sh[32 + w]; z += sh[64 + w]; }
  }
}

// A, B, C (Eq. 8) of a template and the coefficients of 2F (Eq. 6 with
// D = AB - C^2); a template without valid samples, or with a and b
// proportional, gets FSTAT_ERANGE.
__device__ __forceinline__ void set_sums(TmplMeta* meta, double A, double B, double Cc, double sigma2,
                                         double* abcd, int* status) {
  const double D = A * B - Cc * Cc;
  meta->A = A; meta->B = B; meta->C = Cc;
  if (!(D > 0.0) || !isfinite(D)) {
    meta->status_2f = FSTAT_ERANGE;
    set_status(status, FSTAT_ERANGE);
  }
  const double s = 1.0 / (sigma2 * D);
  meta->ca = (float)(2.0 * B * s);
  meta->cb = (float)(2.0 * A * s);
  meta->cc = (float)(-4.0 * Cc * s);
  if (abcd) { abcd[0] = A; abcd[1] = B; abcd[2] = Cc; abcd[3] = D; }
}

// The last block of a template to finish its partial sums reduces them in
// index order (deterministic) and fills A, B, C and the 2F coefficients.
__device__ __forceinline__ void finalize_sums(TmplMeta* meta, const double* __restrict__ partials,
                                              int nparts, int* counter, double sigma2, double* abcd,
                                              int* status) {
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = (atomicAdd(counter, 1) == nparts - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x == 0) {
    double A = 0, B = 0, Cc = 0;
    for (int i = 0; i < nparts; ++i) {
      A += __ldcg(partials + 3 * i);
      B += __ldcg(partials + 3 * i + 1);
      Cc += __ldcg(partials + 3 * i + 2);
    }
    set_sums(meta, A, B, Cc, sigma2, abcd, status);
    *counter = 0;
  }
}

// ---------------------------------------------------------------- launchers
// (host side, defined in the .cu files)

struct Chunk {
  // one batch of templates: device pointers into the workspace
  const fstat_template* tmpl;
  TmplMeta* meta;
  void* knots;            // [nt][knot_stride] records
  int64_t knot_stride;    // records per template
  double* partials;       // [nt][part_stride][3]
  int64_t part_stride;
  int* counters;          // [nt]
  void* za;               // FFT intermediate [nt][n] pairs
  int64_t z_stride;       // pairs per template (n)
  void* wa;               // unfused path: resampled series [nt][n] pairs, column-tiled
  int nt;
};

struct Shape {
  int log2n, l1, l2, cols, rows;
};

// The resampler's tiles (8 rows x 32 columns) of the row tiles with a point
// below n_b.
__host__ __device__ __forceinline__ int live_tiles(int64_t n_b, int l2) {
  return n_b <= 0 ? 0 : (int)(((n_b - 1) >> (l2 + 3)) + 1) << (l2 - 5);
}

// Default factorisation N = N1 N2 of the four-step FFT: the longest first
// pass (N1 <= 2^12, N2 >= 2^6), so that a second-pass block holds as many
// rows as its shared memory allows and its 2F stores form longer runs.
// Knot spacing of the time map, 2^log2h grid points.  The cubic Hermite
// pieces between knots err by about (w h)^4 / 384 relative, w the fastest
// angular rate in the time delay and the beam patterns (twice the sidereal
// rate, for a and b): 1.3e-6 at h dt = 1024 s.  The phase within a piece
// is evaluated in FP32, so its span in cycles bounds h too: 2^11 points
// while |f_het dt| <= 50 cycles per sample and dt <= 0.5 s, 2^10 to 100,
// 2^9 beyond.
__host__ __device__ inline int default_knot_log2(double f_het, double dt) {
  const double c = fabs(f_het * dt);
  return (c <= 50.0 && dt <= 0.5) ? 11 : (c <= 100.0 ? 10 : 9);
}

__host__ __device__ inline int default_log2_n1(int L) {
  int l1 = L - 6;
  if (l1 > 12) l1 = 12;
  if (l1 < 6) l1 = 6;
  return l1;
}

size_t demod_workspace(int64_t n_sft, int64_t n_t);
cudaError_t launch_demod(const PlanConst& pc, const fstat_sft_desc& d, const float2* X, const double* t_sft,
                         int64_t n_sft, const fstat_template* tm, int64_t n_t, double f0, double df, int64_t n_q,
                         float* out, void* ws, int* status, cudaStream_t s);
cudaError_t launch_inject(const PlanConst& pc, const fstat_injection* inj, int64_t n_inj, int64_t max_span,
                          float2* x, int* status, cudaStream_t s);
cudaError_t launch_timemap(const PlanConst& pc, const Chunk& c, int log2n_plan, int mode, bool scaled,
                           const int64_t* gaps, int64_t n_gaps_total, int* status,
                           int64_t tmpl_base, cudaStream_t s);
cudaError_t launch_resample_w(const PlanConst& pc, const Chunk& c, int ti, int log2n, const float2* x,
                              const int64_t* gaps, const double* wcs, void* out_a, void* out_b,
                              int64_t out_stride, int out_double, double* abcd, int* status,
                              cudaStream_t s);
cudaError_t launch_resample_t(const PlanConst& pc, const Chunk& c, const Shape& sh, const float2* x,
                              const int64_t* gaps, int64_t n_gaps_total, const double* wcs, cudaStream_t s);
int resample_covered(const PlanConst& pc, const Shape& sh);
cudaError_t launch_cols_w(const PlanConst& pc, const Chunk& c, const Shape& sh, int inplace, const void* twf,
                          const void* twd, int* status, cudaStream_t s);
cudaError_t launch_rows_w(const PlanConst& pc, const Chunk& c, const Shape& sh, int inplace, const void* twf,
                          const void* twd, float* out, cudaStream_t s);
cudaError_t launch_grad_pass(const PlanConst& pc, const Chunk& c, const float2* x, const int64_t* gaps,
                             const double* wcs, const double* df, double* work, double* twoF,
                             double* grad, int* status, int pass, cudaStream_t s);
size_t grad_work_doubles(int nt);
int cols_per_block(int precision, int l1);
int persist_slots();
size_t persist_smem();
cudaError_t launch_persist(const PlanConst& pc, const Chunk& c, const float2* x, const int64_t* gaps,
                           const double* wcs, const void* twf, float* out, int* status, void* zslots,
                           int64_t z_stride, int* counters, int* sched, int* cnt, int spin_limit,
                           int stall_template, cudaStream_t s);
int rows_per_block(int precision, int l2);

// Fill the derived trigonometric constants of a PlanConst (host, FP64).
inline void derive_constants(PlanConst& pc) {
  pc.ce = cos(pc.obliq); pc.se = sin(pc.obliq);
  pc.sl = sin(pc.lat); pc.cl = cos(pc.lat);
  pc.s2l = sin(2 * pc.lat); pc.c2l = cos(2 * pc.lat);
  pc.s2g = sin(2 * pc.gamma); pc.c2g = cos(2 * pc.gamma);
  pc.auc = pc.au / kC; pc.rc = pc.radius / kC;
  pc.wo = kTwoPi / pc.year; pc.ws = kTwoPi / pc.sid;
  pc.th0 = pc.sid0 + pc.lon;
  pc.inv_dt = 1.0 / pc.dt;
  pc.beta = pc.wo * pc.auc + pc.ws * pc.rc;
}

// Host-side validation of a plan descriptor: FSTAT_OK or the error code
// fstat_plan returns for it (api.cu).
int check_plan_desc(const fstat_plan_desc* d);

// Host copy of the t_b-grid computation (same formulas, FP64) used to size
// work and by fstat_template_nb.
int64_t host_nb(const PlanConst& pc, const fstat_template& t, double* tb0);

}  // namespace fs
