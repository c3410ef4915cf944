// Time map (step 3 of Sec. III.A.2, Eqs. 11, 21): for every template the
// uniform barycentric grid t_b^k = t_b(t_s) + k dt and, at knots every
// h = 2^log2h grid points, the detector time T^k, the fractional data index
// u = (T^k - t_start)/dt, the phase to remove
// P = f_h t_m(T^k) + fdot tau_b^2 / 2 + fddot tau_b^3 / 6 (cycles, Eq. absorb with
// Eq. phi-s-explain, tau_b = t_b - t_start) and the beam patterns a, b at
// T^k (Eqs. 2-3), each with its derivative along the grid.  Consecutive
// knots are joined by cubic Hermite pieces; the per-interval coefficients
// are what the resampling kernels evaluate per sample.
//
// Everything here runs once per knot (h ~ 1024 samples), so FP64 costs
// little even at the FP64 rate of this GPU; the per-sample work only adds
// small FP32 deviations to FP64-reduced bases.
#include "fstat_internal.cuh"

#include <math.h>

namespace fs {

namespace {

// Values at one knot in FP32 (the precision study).
struct KnotVal {
  float U, dU, P, dP, a, da, b, db;
};

__device__ KnotVal knot_value(const PlanConst& pc, const Sky<float>& sky, double tb0, int64_t k, float fdot,
                              float fddot) {
  KnotVal v;
  const float tb = (float)(tb0 + (double)k * pc.dt);
  float tm, rate, sH, cH, inv1r;
  const float T = inverse_time(pc, sky, tb, &tm, &rate, &sH, &cH, &inv1r);
  const float dTdk = (float)pc.dt * inv1r;
  v.U = (T - (float)pc.t_start) * (float)pc.inv_dt;
  v.dU = inv1r;
  const float taub = tb - (float)pc.t_start;
  // spindown phase of Eq. 4 to s = 2 in barycentric time, and its rate
  v.P = (float)pc.f_het * tm + taub * taub * ((float)0.5 * fdot + fddot * taub * (float)(1.0 / 6));
  v.dP = (float)pc.f_het * rate * dTdk + taub * (fdot + (float)0.5 * fddot * taub) * (float)pc.dt;
  float a, b, da, db;
  beams_h<float>(pc, sky, sH, cH, &a, &b, &da, &db);
  v.a = a; v.b = b; v.da = da * dTdk; v.db = db * dTdk;
  return v;
}

// Cubic Hermite coefficients over an interval of H grid points; iH = 1/H
// (H a power of two: exact).
template <typename R>
__device__ __forceinline__ void hermite(R f0, R d0, R f1, R d1, R H, R iH, R* c1, R* c2, R* c3) {
  const R D = f1 - f0;
  *c1 = d0;
  *c2 = (3 * D - (2 * d0 + d1) * H) * (iH * iH);
  *c3 = (-2 * D + (d0 + d1) * H) * (iH * iH * iH);
}

// FP32 time map (precision study): the same record built from FP32 values.
__device__ __forceinline__ void write_record(KnotF* out, const KnotVal& k0, const KnotVal& k1, float H) {
  KnotF r;
  const float iH = (float)1 / H;
  float c1, c2, c3;
  const float fl = floorf(k0.U);
  r.I = (int32_t)fl;
  r.F = k0.U - fl;
  hermite(k0.U, k0.dU, k1.U, k1.dU, H, iH, &c1, &c2, &c3);
  r.u1 = c1 - 1.f; r.u2 = c2; r.u3 = c3;
  r.P = k0.P - floorf(k0.P);
  hermite(k0.P, k0.dP, k1.P, k1.dP, H, iH, &c1, &c2, &c3);
  r.p1 = c1; r.p2 = c2; r.p3 = c3;
  hermite(k0.a, k0.da, k1.a, k1.da, H, iH, &c1, &c2, &c3);
  r.a0 = k0.a; r.a1 = c1; r.a2 = c2; r.a3 = c3;
  hermite(k0.b, k0.db, k1.b, k1.db, H, iH, &c1, &c2, &c3);
  r.b0 = k0.b; r.b1 = c1; r.b2 = c2; r.b3 = c3;
  r.r0 = r.r1 = r.r2 = 0.f;
  *out = r;
}

// Whether the block's first interval lies beyond any grid of the template: the
// launch covers n_fft points, and a span of span_len samples maps to at most
// span_len (1 + beta) of them.
__device__ __forceinline__ bool beyond_span(const PlanConst& pc, const fstat_template& tp, int64_t first) {
  // (FP32 with a margin of 2e-6: FP64 is this kernel's bottleneck)
  const float beta = 1.02f * (float)pc.beta + 2e-6f;
  return first > 0 && (float)(first << pc.log2h) > (float)tp.span_len * (1.0f + beta) + 3.0f;
}

// t_b(t) = t + t_m(t) at the span's first and last sample into tb[0], tb[1],
// and the sky constants, by one warp: the sines and cosines of the sky
// position and of the four angles take one FP64 latency in six lanes.
__device__ __forceinline__ Sky<double> span_ends(const PlanConst& pc, const fstat_template& tp, double* tb) {
  const int lane = threadIdx.x & 31;
  const double t_s = pc.t_start + (double)tp.span_start * pc.dt;
  const double t_e = pc.t_start + (double)(tp.span_start + tp.span_len - 1) * pc.dt;
  const double tt = lane < 4 ? t_s : t_e;
  const double ang = lane == 0 ? tp.alpha : lane == 1 ? tp.delta
                     : (lane & 1) == 0 ? pc.orb0 + pc.wo * tt : pc.th0 + pc.ws * tt - tp.alpha;
  double sn, cs;
  sincos(ang, &sn, &cs);
  const double sa = __shfl_sync(0xffffffffu, sn, 0), ca = __shfl_sync(0xffffffffu, cs, 0);
  const double sd = __shfl_sync(0xffffffffu, sn, 1), cd = __shfl_sync(0xffffffffu, cs, 1);
  const int o = lane == 1 ? 4 : 2;
  const double sp = __shfl_sync(0xffffffffu, sn, o), cp = __shfl_sync(0xffffffffu, cs, o);
  const double ct = __shfl_sync(0xffffffffu, cs, o + 1);
  const Sky<double> s = make_sky<double>(pc, tp.alpha, sa, ca, sd, cd);
  if (lane < 2) tb[lane] = (lane == 0 ? t_s : t_e) + (s.ox * cp + s.oy * sp + s.rxy * ct + s.rz);
  return s;
}

// Grid length, FFT length and validity of a template whose span maps to
// [tb0, tbe] (every block of the template computes the same).
struct TmplGrid { int64_t n_b; int n_int, log2n, status; };
__device__ __forceinline__ TmplGrid tmpl_grid(const PlanConst& pc, const fstat_template& tp, double tb0, double tbe,
                                              int log2n_plan, int allow_ragged, int64_t n_gaps_total) {
  int st = FSTAT_OK;
  if (!(isfinite(tp.alpha) && isfinite(tp.delta) && isfinite(tp.fdot) && isfinite(tp.fddot)) ||
      fabs(tp.delta) > 1.5707963267948967)
    st = FSTAT_EINVAL;
  if (tp.span_start < 0 || tp.span_len < 2 || tp.span_start + tp.span_len > pc.n_data) st = FSTAT_ERANGE;
  if (tp.n_gaps < 0 || tp.gap_off < 0 || tp.gap_off + tp.n_gaps > n_gaps_total) st = FSTAT_EINVAL;
  int log2n = log2n_plan;
  if (tp.n_fft != 0) {
    const int64_t nf = tp.n_fft;
    const int l = 63 - __clzll((unsigned long long)max(nf, (int64_t)1));
    if ((nf & (nf - 1)) != 0 || l < kMinLog || l > log2n_plan) st = st ? st : FSTAT_ERANGE;
    else if (!allow_ragged && l != log2n_plan) st = st ? st : FSTAT_ENOTSUP;
    else log2n = l;
  }
  // a partial output band is defined on the plan's n_fft only
  if (log2n != log2n_plan && (pc.band_lo != 0 || pc.band_hi != ((int64_t)1 << log2n_plan)))
    st = st ? st : FSTAT_ENOTSUP;
  TmplGrid g;
  g.n_b = (int64_t)floor((tbe - tb0) / pc.dt) + 1;
  if (st == FSTAT_OK && g.n_b > ((int64_t)1 << log2n)) st = FSTAT_ERANGE;
  if (st != FSTAT_OK) g.n_b = 0;
  g.n_int = (int)((g.n_b + (1 << pc.log2h) - 1) >> pc.log2h);
  g.log2n = log2n;
  g.status = st;
  return g;
}

// The template's metadata, and the check of its gap list: sorted, disjoint,
// non-empty intervals (all threads of its first block).
__device__ __forceinline__ void write_meta(const PlanConst& pc, const fstat_template& tp, const TmplGrid& g, double tb0,
                                           int64_t index, TmplMeta* __restrict__ meta,
                                           const int64_t* __restrict__ gaps, int* status) {
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  if (g.status == FSTAT_OK) {
    for (int64_t i = threadIdx.x; i < tp.n_gaps; i += blockDim.x) {
      const int64_t s0 = gaps[2 * (tp.gap_off + i)], e0 = gaps[2 * (tp.gap_off + i) + 1];
      bool ok = s0 < e0 && s0 >= 0 && e0 <= pc.n_data;
      if (i + 1 < tp.n_gaps) ok = ok && e0 <= gaps[2 * (tp.gap_off + i + 1)];
      if (!ok) bad = 1;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int st = bad && g.status == FSTAT_OK ? FSTAT_EINVAL : g.status;
    TmplMeta m;
    m.tb0 = tb0;
    m.A = m.B = m.C = 0.0;
    m.acc[0] = m.acc[1] = m.acc[2] = 0;
    m.n_b = st == FSTAT_OK ? g.n_b : 0;
    m.out_off = tp.out_off >= 0 ? tp.out_off : index * (pc.band_hi - pc.band_lo);
    m.span_lo = tp.span_start;
    m.span_hi = tp.span_start + tp.span_len;
    m.gap_off = tp.gap_off;
    m.n_gaps = tp.n_gaps;
    m.log2n = g.log2n;
    m.status = st;
    m.ca = m.cb = m.cc = 0.f;
    m.status_2f = st;
    *meta = m;
    if (st != FSTAT_OK) set_status(status, st);
  }
}

// 1 / (1 + r)
__device__ __forceinline__ double inv_one_plus(double r) {
  if (fabs(r) < 5e-4) return 1.0 - r * (1.0 - r * (1.0 - r * (1.0 - r * (1.0 - r))));   // r^6 < 2e-20
  return 1.0 / (1.0 + r);
}

// FP64 time map.  A group of 31 intervals (32 knots, one per lane) goes
// through four warps in stages, because one thread per knot is a chain of
// 1400 instructions, most of them waiting for the FP64 result before:
//   the angles at t_s + k dt (warps 1, 2) beside the span's ends (warp 0);
//   Newton's steps for T^k (warp 0);
//   the phase P (warp 1) and the beams a, b (warp 2) with their slopes;
//   the Hermite pieces of u, P, a, b, one quantity a warp.
// An FP64 instruction of a warp holds an SM's pipe for 16 cycles, so nothing
// is computed twice, and 1 / (1 + dt_m/dt) is a series in the 1e-4 of dt_m/dt.
// T = s_k + delta with s_k = t_s + k dt and delta = t_m(t_s) - t_m(T)
// (Eq. 21): the first step from s_k leaves delta^2 t_m'' / 2 (5e-7 s for the
// 86 s of 10 days), the second, at s_k + delta, below 1e-12 of that.  The
// angles there are those at s_k rotated by w delta.  A block takes `groups`
// groups after one evaluation of the ends.  With one knot per thread in blocks
// of 256 one template took 42 us, 64 took 95.
constexpr int kTmThreads = 128;
constexpr int kTmKnots = 32;

template <typename REC>
__global__ void __launch_bounds__(kTmThreads)
k_timemap(PlanConst pc, const fstat_template* __restrict__ tmpl, TmplMeta* __restrict__ meta,
          REC* __restrict__ knots, int64_t knot_stride, int log2n_plan, int allow_ragged, bool scaled,
          const int64_t* __restrict__ gaps, int64_t n_gaps_total, int* status, int64_t tmpl_base, int groups) {
  __shared__ double tb_sh[2];
  __shared__ Sky<double> sky;
  __shared__ double ang[4][kTmKnots];              // sin, cos of the orbital phase and of the hour angle
  __shared__ double val[4][kTmKnots], slope[4][kTmKnots];   // u, P, a, b at the knots
  __shared__ double geo[5][kTmKnots];              // t_m, rate, sin H, cos H, dT/dk
  __shared__ TmplGrid grid_sh;
  let_next_start();
  const int t = blockIdx.y;
  const fstat_template tp = tmpl[t];
  const int64_t g0 = (int64_t)blockIdx.x * groups;
  if (beyond_span(pc, tp, g0 * (kTmKnots - 1))) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double t_s = pc.t_start + (double)tp.span_start * pc.dt;
  const double H = (double)(1 << pc.log2h), iH = 1.0 / H;     // a power of two: exact
  TmplGrid g;
  double tb0 = 0.0;
  for (int64_t gi = g0; gi < g0 + groups; ++gi) {
    const int64_t j0 = gi * (kTmKnots - 1);
    const double kdt = (double)((j0 + lane) << pc.log2h) * pc.dt;
    const double sk = t_s + kdt;
    // --- angles; the span's ends with the first group
    if (warp == 0 && gi == g0) {
      const Sky<double> s = span_ends(pc, tp, tb_sh);
      __syncwarp();
      if (lane == 0) {
        sky = s;
        grid_sh = tmpl_grid(pc, tp, tb_sh[0], tb_sh[1], log2n_plan, allow_ragged, n_gaps_total);
      }
    } else if (warp == 1) {
      sincos(pc.orb0 + pc.wo * sk, &ang[0][lane], &ang[1][lane]);
    } else if (warp == 2) {
      sincos(pc.th0 + pc.ws * sk - tp.alpha, &ang[2][lane], &ang[3][lane]);
    }
    __syncthreads();
    if (gi == g0) {
      tb0 = tb_sh[0];
      g = grid_sh;
      if (blockIdx.x == 0) write_meta(pc, tp, g, tb0, tmpl_base + t, meta + t, gaps, status);
      if (g.status != FSTAT_OK) return;
    }
    if (j0 >= g.n_int) return;
    const double tb = tb0 + kdt;
    // --- T^k
    if (warp == 0) {
      double sp = ang[0][lane], cp = ang[1][lane], st = ang[2][lane], ct = ang[3][lane];
      const double tm0 = tb0 - t_s;
      double tm = sky.ox * cp + sky.oy * sp + sky.rxy * ct + sky.rz;
      double rate = pc.wo * (sky.oy * cp - sky.ox * sp) - pc.ws * sky.rxy * st;
      const double delta = (tm0 - tm) * inv_one_plus(rate);
      advance<double>(pc.orb0 + pc.wo * sk, pc.wo * delta, &sp, &cp);
      advance<double>(pc.th0 + pc.ws * sk - tp.alpha, pc.ws * delta, &st, &ct);
      const double T1 = sk + delta;
      tm = sky.ox * cp + sky.oy * sp + sky.rxy * ct + sky.rz;
      rate = pc.wo * (sky.oy * cp - sky.ox * sp) - pc.ws * sky.rxy * st;
      const double inv1r = inv_one_plus(rate);
      const double dT = -(T1 + tm - tb) * inv1r;
      // the hour angle at T to first order in ws dT
      const double e = pc.ws * dT;
      geo[0][lane] = tm + rate * dT;
      geo[1][lane] = rate;
      geo[2][lane] = st + ct * e;
      geo[3][lane] = ct - st * e;
      geo[4][lane] = pc.dt * inv1r;
      val[0][lane] = (T1 + dT - pc.t_start) * pc.inv_dt;
      slope[0][lane] = inv1r;
    } else if (warp == 3 && gi == g0 && scaled) {
      scale_beams_warp(sky);                       // (warp 0 reads the orbit only)
    }
    __syncthreads();
    // --- P (cycles to remove), a, b and their slopes along the grid
    if (warp == 1) {
      const double taub = tb - pc.t_start;
      val[1][lane] = pc.f_het * geo[0][lane] + taub * taub * (0.5 * tp.fdot + tp.fddot * taub * (1.0 / 6));
      slope[1][lane] = pc.f_het * geo[1][lane] * geo[4][lane] + taub * (tp.fdot + 0.5 * tp.fddot * taub) * pc.dt;
    } else if (warp == 2) {
      double a, b, da, db;
      beams_h<double>(pc, sky, geo[2][lane], geo[3][lane], &a, &b, &da, &db);
      val[2][lane] = a;
      val[3][lane] = b;
      slope[2][lane] = da * geo[4][lane];
      slope[3][lane] = db * geo[4][lane];
    }
    __syncthreads();
    // --- the pieces between neighbouring knots
    if (lane < kTmKnots - 1 && j0 + lane < g.n_int) {
      const double f0 = val[warp][lane];
      double c1, c2, c3;
      hermite(f0, slope[warp][lane], val[warp][lane + 1], slope[warp][lane + 1], H, iH, &c1, &c2, &c3);
      REC* r = knots + (int64_t)t * knot_stride + j0 + lane;
      if constexpr (std::is_same<REC, KnotF>::value) {
        const double fl = floor(f0);
        if (warp == 0) {
          r->I = (int32_t)fl; r->F = (float)(f0 - fl);
          r->u1 = (float)(c1 - 1.0); r->u2 = (float)c2; r->u3 = (float)c3;
          r->r0 = r->r1 = r->r2 = 0.f;
        } else {
          float* o = warp == 1 ? &r->P : (warp == 2 ? &r->a0 : &r->b0);
          o[0] = (float)(warp == 1 ? f0 - fl : f0);
          o[1] = (float)c1; o[2] = (float)c2; o[3] = (float)c3;
        }
      } else {
        double* o = warp == 0 ? &r->U : (warp == 1 ? &r->P : (warp == 2 ? &r->a0 : &r->b0));
        o[0] = warp == 1 ? f0 - floor(f0) : f0;
        o[1] = warp == 0 ? c1 - 1.0 : c1; o[2] = c2; o[3] = c3;
      }
    }
    __syncthreads();                               // before the next group rewrites the arrays
  }
}

// All-FP32 knots (precision study): one knot per thread, neighbouring blocks
// evaluating their common knot twice.
constexpr int kKnotThreads = 128;

__global__ void __launch_bounds__(kKnotThreads)
k_timemap_f32(PlanConst pc, const fstat_template* __restrict__ tmpl, TmplMeta* __restrict__ meta,
              KnotF* __restrict__ knots, int64_t knot_stride, int log2n_plan, int allow_ragged, bool scaled,
              const int64_t* __restrict__ gaps, int64_t n_gaps_total, int* status, int64_t tmpl_base) {
  __shared__ KnotVal kv[kKnotThreads];
  __shared__ double tb_sh[2];
  let_next_start();
  const int t = blockIdx.y;
  const fstat_template tp = tmpl[t];
  const int64_t j0 = (int64_t)blockIdx.x * (kKnotThreads - 1);
  if (beyond_span(pc, tp, j0)) return;
  if (threadIdx.x < 32) span_ends(pc, tp, tb_sh);
  __syncthreads();
  const double tb0 = tb_sh[0];
  const TmplGrid g = tmpl_grid(pc, tp, tb0, tb_sh[1], log2n_plan, allow_ragged, n_gaps_total);
  if (blockIdx.x == 0) write_meta(pc, tp, g, tb0, tmpl_base + t, meta + t, gaps, status);
  if (g.status != FSTAT_OK || j0 >= g.n_int) return;
  Sky<float> sky = make_sky<float>(pc, (float)tp.alpha, (float)tp.delta);
  if (scaled) scale_beams(sky);
  const int64_t j = j0 + threadIdx.x;
  if (j <= g.n_int) kv[threadIdx.x] = knot_value(pc, sky, tb0, j << pc.log2h, (float)tp.fdot, (float)tp.fddot);
  __syncthreads();
  if (threadIdx.x < kKnotThreads - 1 && j < g.n_int)
    write_record(knots + (int64_t)t * knot_stride + j, kv[threadIdx.x], kv[threadIdx.x + 1], (float)(1 << pc.log2h));
}

}  // namespace

// scaled: a, b times the powers of two of scale_beams, for the passes that only
// form 2F from them
cudaError_t launch_timemap(const PlanConst& pc, const Chunk& c, int log2n_plan, int mode, bool scaled,
                           const int64_t* gaps, int64_t n_gaps_total, int* status,
                           int64_t tmpl_base, cudaStream_t s) {
  const int64_t max_int = (((int64_t)1 << log2n_plan) >> pc.log2h) + 1;
  const int ragged = mode == FSTAT_MODE_PERSISTENT;
  if (pc.precision == FSTAT_PREC_FP32) {
    const dim3 grid((unsigned)((max_int + kKnotThreads - 2) / (kKnotThreads - 1)), (unsigned)c.nt);
    k_timemap_f32<<<grid, kKnotThreads, 0, s>>>(pc, c.tmpl, c.meta, (KnotF*)c.knots, c.knot_stride, log2n_plan,
                                                ragged, scaled, gaps, n_gaps_total, status, tmpl_base);
    return cudaGetLastError();
  }
  // one group of knots per block while the blocks are few enough to be on the
  // chip at once (8 on each of 152 SMs), two after that: 64 templates of 846
  // knots 60 us with one, 53 with two, 83 with four; one template 15, 21, -
  const int64_t all = (max_int + kTmKnots - 2) / (kTmKnots - 1);
  const int groups = all * c.nt <= 8 * 152 ? 1 : 2;
  const dim3 grid((unsigned)((all + groups - 1) / groups), (unsigned)c.nt);
  if (pc.precision == FSTAT_PREC_FP64)
    k_timemap<<<grid, kTmThreads, 0, s>>>(pc, c.tmpl, c.meta, (KnotD*)c.knots, c.knot_stride, log2n_plan, ragged, scaled, gaps,
                                          n_gaps_total, status, tmpl_base, groups);
  else
    k_timemap<<<grid, kTmThreads, 0, s>>>(pc, c.tmpl, c.meta, (KnotF*)c.knots, c.knot_stride, log2n_plan, ragged, scaled, gaps,
                                          n_gaps_total, status, tmpl_base, groups);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ host copy
// The grid length N_b on the host, same FP64 formulas as span_ends above.
int64_t host_nb(const PlanConst& pc, const fstat_template& t, double* tb0_out) {
  if (t.span_start < 0 || t.span_len < 2 || t.span_start + t.span_len > pc.n_data) return -1;
  const double ca = cos(t.alpha), sa = sin(t.alpha), cd = cos(t.delta), sd = sin(t.delta);
  const double nx = cd * ca, ny = cd * sa, nz = sd;
  const double auc = pc.au / kC;
  const double ox = auc * nx, oy = auc * (cos(pc.obliq) * ny + sin(pc.obliq) * nz);
  const double rz = pc.radius / kC * sin(pc.lat) * sd, rxy = pc.radius / kC * cos(pc.lat) * cd;
  auto tb = [&](double tt) {
    const double phi = pc.orb0 + kTwoPi / pc.year * tt;
    const double hh = pc.sid0 + pc.lon + kTwoPi / pc.sid * tt - t.alpha;
    return tt + ox * cos(phi) + oy * sin(phi) + rxy * cos(hh) + rz;
  };
  const double t_s = pc.t_start + (double)t.span_start * pc.dt;
  const double t_e = pc.t_start + (double)(t.span_start + t.span_len - 1) * pc.dt;
  const double b0 = tb(t_s), b1 = tb(t_e);
  if (tb0_out) *tb0_out = b0;
  return (int64_t)floor((b1 - b0) / pc.dt) + 1;
}

}  // namespace fs
