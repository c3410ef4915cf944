// Gradient of 2F at one continuous frequency offset per template.
//
// Forward pass: F_a(df) = sum_k w_a[k] E_k, F_b alike, with
// E_k = exp(-2 pi i df tau_b,k) (Eqs. 19-20 evaluated off the FFT grid) and
// the sums A, B, C; the last block forms 2F (Eq. 6) and the cotangents
//   G_a = d2F/dF_a* = 2 (2 B F_a - 2 C F_b) / (sigma2 D),  G_b alike,
//   g_A, g_B, g_C = d2F/dA, dB, dC.
// Adjoint pass: every sample contributes
//   Re(conj(G_a) dW_a/dtheta + conj(G_b) dW_b/dtheta) + g_A dA_k/dtheta + ...
// with W = w E, i.e. the conjugate transform of the cotangent restricted to
// the one bin.  The derivatives follow the time map: with
// g0 = dt_m/dtheta at the span start (the grid start t_b0 moves with the sky),
//   dT^k/dtheta = (g0 - dt_m/dtheta(T^k)) / (1 + dt_m/dt(T^k))      (Eq. 21),
//   du_k = dT^k / dt,  dtau_k = g0 - dT^k,  dtau_b,k = g0,
// the interpolation kernel derivative K'(u - j), the heterodyne and
// spindown phases, and a(T^k), b(T^k) (explicit and through T^k).
#include "passes.cuh"
#include "sinc_run.cuh"

namespace fs {

namespace {

constexpr int kGradThreads = 256;
constexpr int kGradBlocks = 128;       // blocks per template
constexpr int kPartW = 8;              // doubles per block partial
constexpr int kCotW = 16;              // doubles of per-template state
constexpr int kConW = 48;              // doubles of per-template adjoint constants (AdjConst)

template <typename R>
struct GradArgs {
  PlanConst pc;
  Chunk c;
  const float2* x;
  const int64_t* gaps;
  const double* wcs;
  const double* df;       // [nt]
  double* part;           // [nt][kGradBlocks][kPartW]
  double* cot;            // [nt][kCotW]
  double* con;            // [nt][kConW]: AdjConst<R>
  int nblk;               // blocks per template (<= kGradBlocks)
  int* counters;          // [nt] (forward) ; [nt] (adjoint) at counters + nt
  double* twoF;           // [nt]
  double* grad;           // [nt][4]
  int* status;
};

template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double* sh /* [NV*32] */) {
#pragma unroll
  for (int i = 0; i < NV; ++i)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_down_sync(0xffffffffu, v[i], o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0)
#pragma unroll
    for (int i = 0; i < NV; ++i) sh[i * 32 + wid] = v[i];
  __syncthreads();
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      v[i] = lane < nw ? sh[i * 32 + lane] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_down_sync(0xffffffffu, v[i], o);
    }
  }
}

// last-block election; returns true in every thread of the last block
__device__ __forceinline__ bool last_block(int* counter, int nblocks) {
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(counter, 1) == nblocks - 1;
    if (last) *counter = 0;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// sinc(y) and its derivative; series near y = 0 avoids the cancellation of
// (cos(pi y) - sinc(y)) / y
// ry = 1 / y (used only when |y| >= 0.05): one reciprocal per tap serves
// the sinc and, scaled, the window, instead of a division for each term.
template <typename R>
__device__ __forceinline__ void sinc_d(R y, R ry, R sy, R cy, R& s, R& ds) {
  const R pi = (R)3.14159265358979323846;
  if (fabs(y) < (R)0.05) {
    const R p2 = pi * pi * y * y;
    s = (R)1 - p2 * (R)(1.0 / 6) + p2 * p2 * (R)(1.0 / 120);
    ds = pi * pi * y * ((R)(-1.0 / 3.0) + p2 * (R)(1.0 / 30));
  } else {
    s = sy * ry * (R)(1.0 / 3.14159265358979323846);
    ds = (cy - s) * ry;
  }
}

// Resampled value z(u_k) and dz/du with the windowed-sinc kernel, the
// mask, the phase P (cycles) and a, b at grid point k.
template <typename R, int TAPS>
__device__ __forceinline__ bool sample_with_derivative(
    const PlanConst& pc, const typename KnotOf<R>::T* __restrict__ kn, int k,
    const float2* __restrict__ x, GapCursor& gc, const double* __restrict__ wcs,
    cpx<R>& z, cpx<R>& dz, R& u_rel, R& ph, R& a, R& b) {
  using C = cpx<R>;
  const int jint = k >> pc.log2h;
  const int sk = k & ((1 << pc.log2h) - 1);
  const R s = (R)sk;
  int ibase;
  R dev;
  if constexpr (std::is_same<R, float>::value) {
    const KnotF q = kn[jint];
    ibase = q.I + sk;
    dev = q.F + ((q.u3 * s + q.u2) * s + q.u1) * s;
    ph = q.P + ((q.p3 * s + q.p2) * s + q.p1) * s;
    a = q.a0 + ((q.a3 * s + q.a2) * s + q.a1) * s;
    b = q.b0 + ((q.b3 * s + q.b2) * s + q.b1) * s;
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
  const int taps = TAPS > 0 ? TAPS : pc.taps;
  const int half = taps >> 1;
  const R ihalf = (R)1 / (R)half;
  const int jnn_off = (int)floor(dev + (R)0.5);
  const int jnn = ibase + jnn_off;
  const R dn = dev - (R)jnn_off;                // u - jnn in [-1/2, 1/2]
  const int qoff = dn >= (R)0 ? 0 : 1;
  const int n0 = jnn - qoff;
  u_rel = (R)jnn + dn;                          // u in samples from t_start
  R S, Cd, sh, chh;
  if constexpr (std::is_same<R, float>::value) {
    sincospif(dn, &S, &Cd);
    sincospif(dn * ihalf, &sh, &chh);
  } else {
    sincospi(dn, &S, &Cd);
    sincospi(dn * ihalf, &sh, &chh);
  }
  const bool lanczos = pc.window == FSTAT_WIN_LANCZOS;
  C acc = czero<C>(), dacc = czero<C>();
  bool msk = false;
#pragma unroll
  for (int i = 0; i < (TAPS > 0 ? TAPS : 16); ++i) {
    if (TAPS == 0 && i >= taps) break;
    const int mq = half - 1 - i + qoff;
    const int j = n0 + 1 - half + i;
    const R xx = dn + (R)mq;
    const R sg = (mq & 1) ? (R)-1 : (R)1;
    R k0, k1;
    const R rx = (R)1 / xx;
    sinc_d<R>(xx, rx, sg * S, sg * Cd, k0, k1);
    if (lanczos) {
      const R* wt = win_table<R>(wcs);
      const R cm = __ldg(wt + 2 * (mq + half)), sm = __ldg(wt + 2 * (mq + half) + 1);
      const R shm = sh * cm + chh * sm, chm = chh * cm - sh * sm;
      R w0, w1;
      sinc_d<R>(xx * ihalf, rx * (R)half, shm, chm, w0, w1);
      const R kk = k0 * w0;
      k1 = k1 * w0 + k0 * w1 * ihalf;
      k0 = kk;
    }
    const bool ok = gc.valid(j);
    if (j == jnn) msk = ok;
    if (ok) {
      const C v = ldx<R>(x, j);
      acc.x = fma(k0, v.x, acc.x);
      acc.y = fma(k0, v.y, acc.y);
      dacc.x = fma(k1, v.x, dacc.x);
      dacc.y = fma(k1, v.y, dacc.y);
    }
  }
  z = acc;
  dz = dacc;
  return msk;
}

// frac(s k) for the sample index k >= 0 without FP64 work per sample: with
// F = frac(s) as a 64-bit binary fraction, F k mod 2^64 is exact in integer
// arithmetic, and its top 24 bits are frac(s k) to FP32 precision (F itself
// carries the 2^-53 rounding of the FP64 s, as the FP64 product s k would).
// A warp's FP64 instruction costs 64 issue cycles at this GPU's FP64 rate,
// so the four FP64 operations of frac(s k) per sample were the kernels'
// largest cost.
__device__ __forceinline__ unsigned long long frac_fix64(double s) {
  const double f = s - floor(s);                  // [0, 1)
  return __double2ull_rz(f * 18446744073709551616.0);   // f 2^64 < 2^64
}
__device__ __forceinline__ float frac_mul(unsigned long long F, int k) {
  return (float)((F * (unsigned long long)k) >> 40) * (1.0f / 16777216.0f);
}

template <typename R>
__device__ __forceinline__ cpx<R> expm(R cyc) {   // exp(-2 pi i cyc)
  R sp, cp;
  const R r = cyc - rint(cyc);
  if constexpr (std::is_same<R, float>::value) sincospif(2.f * r, &sp, &cp); else sincospi(2.0 * r, &sp, &cp);
  return cmk<cpx<R>, R>(cp, -sp);
}

// Per-template constants of the adjoint, from FP64: projections of the orbit
// and of the site on the derivatives of the sky vector, beam coefficients and
// their delta derivatives, angles at t_start reduced for single precision,
// dt_m/dtheta at the span start.
template <typename R>
struct AdjConst {
  R ox, oy, oxa, oya, oxd, oyd;        // orbital projections and their alpha, delta derivatives
  R rxy, rxyd, rzd;                    // R/c cos(lat) cos(delta); R/c cos(lat) sin(delta); R/c sin(lat) cos(delta)
  R g0a, g0d;                          // dt_m/dalpha, dt_m/ddelta at t_s
  R phi0, hh0, wo, ws;
  R e1, e2, e3, e4, f1, f2, f3, f4;
  R de0, de1, de2, de3, de4, df1, df2, df3, df4;
  R tb0, fdot, fddot, fh, dt, idt;
};
static_assert(sizeof(AdjConst<double>) <= kConW * sizeof(double), "fits its slot");

// One warp; lanes 0..3 take one sine and cosine each (the FP64 latency of one
// instead of four).
template <typename R>
__device__ void adj_constants(const PlanConst& pc, const fstat_template& tp, double tb0, AdjConst<R>* out) {
  const int lane = threadIdx.x & 31;
  const double t_s = pc.t_start + (double)tp.span_start * pc.dt;
  const double ang = lane == 0 ? tp.alpha : lane == 1 ? tp.delta : lane == 2 ? pc.orb0 + pc.wo * t_s
                                                                  : pc.th0 + pc.ws * t_s - tp.alpha;
  double sn, cs;
  sincos(ang, &sn, &cs);
  const double sa = __shfl_sync(0xffffffffu, sn, 0), ca = __shfl_sync(0xffffffffu, cs, 0);
  const double sd = __shfl_sync(0xffffffffu, sn, 1), cd = __shfl_sync(0xffffffffu, cs, 1);
  const double sp = __shfl_sync(0xffffffffu, sn, 2), cp = __shfl_sync(0xffffffffu, cs, 2);
  const double sH = __shfl_sync(0xffffffffu, sn, 3), cH = __shfl_sync(0xffffffffu, cs, 3);
  if (lane != 0) return;
  // dn/dalpha = (-cd sa, cd ca, 0), dn/ddelta = (-sd ca, -sd sa, cd)
  const double oxa = pc.auc * (-cd * sa), oya = pc.auc * (pc.ce * cd * ca);
  const double oxd = pc.auc * (-sd * ca), oyd = pc.auc * (pc.ce * (-sd * sa) + pc.se * cd);
  const double rcl = pc.rc * pc.cl, rsl = pc.rc * pc.sl;
  AdjConst<R> k;
  k.ox = (R)(pc.auc * cd * ca);
  k.oy = (R)(pc.auc * (pc.ce * cd * sa + pc.se * sd));
  k.oxa = (R)oxa; k.oya = (R)oya; k.oxd = (R)oxd; k.oyd = (R)oyd;
  k.rxy = (R)(rcl * cd); k.rxyd = (R)(rcl * sd); k.rzd = (R)(rsl * cd);
  k.g0a = (R)(oxa * cp + oya * sp + rcl * cd * sH);
  k.g0d = (R)(oxd * cp + oyd * sp - rcl * sd * cH + rsl * cd);
  k.phi0 = (R)fmod(pc.orb0 + pc.wo * pc.t_start, kTwoPi);
  k.hh0 = (R)fmod(pc.th0 + pc.ws * pc.t_start - tp.alpha, kTwoPi);
  k.wo = (R)pc.wo; k.ws = (R)pc.ws;
  const double c2d = cd * cd - sd * sd, s2d = 2 * sd * cd;
  k.e1 = (R)(pc.s2g * pc.s2l * s2d / 4); k.e2 = (R)(-pc.c2g * pc.cl * s2d / 2);
  k.e3 = (R)(pc.s2g * (3 - pc.c2l) * (3 - c2d) / 16); k.e4 = (R)(-pc.c2g * pc.sl * (3 - c2d) / 4);
  k.f1 = (R)(pc.c2g * pc.cl * cd); k.f2 = (R)(pc.s2g * pc.s2l * cd / 2);
  k.f3 = (R)(pc.c2g * pc.sl * sd); k.f4 = (R)(pc.s2g * (3 - pc.c2l) * sd / 4);
  k.de0 = (R)(-0.75 * pc.s2g * pc.cl * pc.cl * s2d); k.de1 = (R)(pc.s2g * pc.s2l * c2d / 2);
  k.de2 = (R)(-pc.c2g * pc.cl * c2d); k.de3 = (R)(pc.s2g * (3 - pc.c2l) * s2d / 8);
  k.de4 = (R)(-pc.c2g * pc.sl * s2d / 2);
  k.df1 = (R)(-pc.c2g * pc.cl * sd); k.df2 = (R)(-pc.s2g * pc.s2l * sd / 2);
  k.df3 = (R)(pc.c2g * pc.sl * cd); k.df4 = (R)(pc.s2g * (3 - pc.c2l) * cd / 4);
  k.tb0 = (R)(tb0 - pc.t_start);
  k.fdot = (R)tp.fdot; k.fddot = (R)tp.fddot; k.fh = (R)pc.f_het; k.dt = (R)pc.dt; k.idt = (R)(1.0 / pc.dt);
  *out = k;
}

// Geometry of the adjoint at u samples after t_start: dT/dalpha, dT/ddelta,
// the total derivatives of a and b, and (SLOPE) how these change per sample.
template <typename R>
struct AdjGeo {
  R dTa, dTd, da_a, db_a, da_d, db_d;
  R dTa1, dTd1, da_a1, db_a1, da_d1, db_d1;
};
template <typename R, bool SLOPE>
__device__ __forceinline__ AdjGeo<R> adj_geometry(const AdjConst<R>& q, R u) {
  AdjGeo<R> g;
  const R tt = u * q.dt;                        // T^k - t_start
  R sp, cp, sH, cH;
  rsincos<R>(q.phi0 + q.wo * tt, &sp, &cp);
  rsincos<R>(q.hh0 + q.ws * tt, &sH, &cH);
  const R rate = q.wo * (q.oy * cp - q.ox * sp) - q.ws * q.rxy * sH;
  const R dtma = q.oxa * cp + q.oya * sp + q.rxy * sH;
  const R dtmd = q.oxd * cp + q.oyd * sp - q.rxyd * cH + q.rzd;
  const R inv = (R)1 / ((R)1 + rate);
  g.dTa = (q.g0a - dtma) * inv;
  g.dTd = (q.g0d - dtmd) * inv;
  // beam patterns: x = -H
  const R c2x = cH * cH - sH * sH, s2x = -2 * sH * cH;   // cos 2x, sin 2x
  const R cx = cH, sx = -sH;
  const R dadx = -q.e1 * sx + q.e2 * cx - 2 * q.e3 * s2x + 2 * q.e4 * c2x;
  const R dbdx = -q.f1 * sx + q.f2 * cx - 2 * q.f3 * s2x + 2 * q.f4 * c2x;
  const R dad_T = q.de0 + q.de1 * cx + q.de2 * sx + q.de3 * c2x + q.de4 * s2x;
  const R dbd_T = q.df1 * cx + q.df2 * sx + q.df3 * c2x + q.df4 * s2x;
  // total derivatives (dx/dalpha = 1 explicit, dx/dt = -ws through T)
  const R ea = (R)1 - q.ws * g.dTa, ed = q.ws * g.dTd;
  g.da_a = dadx * ea; g.db_a = dbdx * ea;
  g.da_d = dad_T - dadx * ed; g.db_d = dbd_T - dbdx * ed;
  if constexpr (SLOPE) {
    // per sample: T moves by dt / (1 + rate), x by -ws of it; the rates of
    // inv and of dT inside ea, ed are below 1e-8 of the terms kept
    const R st = q.dt * inv, xs = -q.ws * st;
    g.dTa1 = -(q.wo * (q.oya * cp - q.oxa * sp) + q.ws * q.rxy * cH) * inv * st;
    g.dTd1 = -(q.wo * (q.oyd * cp - q.oxd * sp) + q.ws * q.rxyd * sH) * inv * st;
    const R d2a = xs * (-q.e1 * cx - q.e2 * sx - 4 * q.e3 * c2x - 4 * q.e4 * s2x);
    const R d2b = xs * (-q.f1 * cx - q.f2 * sx - 4 * q.f3 * c2x - 4 * q.f4 * s2x);
    g.da_a1 = d2a * ea; g.db_a1 = d2b * ea;
    g.da_d1 = xs * (-q.de1 * sx + q.de2 * cx - 2 * q.de3 * s2x + 2 * q.de4 * c2x) - d2a * ed;
    g.db_d1 = xs * (-q.df1 * sx + q.df2 * cx - 2 * q.df3 * s2x + 2 * q.df4 * c2x) - d2b * ed;
  }
  return g;
}

// Cotangents of one template in R.
template <typename R>
struct Cot { R Gar, Gai, Gbr, Gbi, gA, gB, gC; };
template <typename R>
__device__ __forceinline__ Cot<R> load_cot(const double* cot) {
  return Cot<R>{(R)cot[0], (R)cot[1], (R)cot[2], (R)cot[3], (R)cot[4], (R)cot[5], (R)cot[6]};
}

// frac(df dt k) of grid point k
template <typename R>
__device__ __forceinline__ R bin_phase(unsigned long long fdt64, double fdt, int k) {
  if constexpr (std::is_same<R, float>::value) {
    return frac_mul(fdt64, k);
  } else {
    const double ck = fdt * (double)k;
    return (R)(ck - floor(ck));
  }
}

// The contribution of grid point k to dF2/d(alpha, delta, f, fdot).
template <typename R, int TAPS>
__device__ __forceinline__ void adj_point(const PlanConst& pc, const typename KnotOf<R>::T* __restrict__ kn, int k,
                                          const float2* __restrict__ x, GapCursor& gc, const double* __restrict__ wcs,
                                          const AdjConst<R>& q, const Cot<R>& ct, unsigned long long fdt64, double fdt,
                                          R c0f, R df, R& ga, R& gd, R& gf, R& gfd) {
  using C = cpx<R>;
  const R twopi = (R)kTwoPi;
  C z, dz;
  R u, ph, a, b;
  if (!sample_with_derivative<R, TAPS>(pc, kn, k, x, gc, wcs, z, dz, u, ph, a, b)) return;
  const AdjGeo<R> g = adj_geometry<R, false>(q, u);   // smooth quantities, single precision is ample
  // phase Phi (cycles) and its derivatives
  const R taub = q.tb0 + (R)k * q.dt;
  const C e = expm<R>(ph + bin_phase<R>(fdt64, fdt, k) + c0f);
  const R fb = taub * (q.fdot + (R)0.5 * q.fddot * taub) + df;   // d(Phi_s + df tau_b)/dt_b, cycles/s
  const R dPa = q.fh * (q.g0a - g.dTa) + fb * q.g0a;
  const R dPd = q.fh * (q.g0d - g.dTd) + fb * q.g0d;
  // y = z e, W_a = a y, W_b = b y
  const C y = cmul(z, e);
  const C dy = cmul(dz, e);
  // dW_a/dtheta = da y + a (dy du/dtheta - 2 pi i y dPhi)
  auto contrib = [&](R dA, R dB, R du, R dP) {
    // V_a = dA y + a (du dy - 2 pi i dP y) ; -2 pi i dP y = 2 pi dP (y.y, -y.x)
    const R vx = du * dy.x + twopi * dP * y.y;
    const R vy = du * dy.y - twopi * dP * y.x;
    const R Var = dA * y.x + a * vx, Vai = dA * y.y + a * vy;
    const R Vbr = dB * y.x + b * vx, Vbi = dB * y.y + b * vy;
    return ct.Gar * Var + ct.Gai * Vai + ct.Gbr * Vbr + ct.Gbi * Vbi
         + ct.gA * 2 * a * dA + ct.gB * 2 * b * dB + ct.gC * (dA * b + a * dB);
  };
  ga += contrib(g.da_a, g.db_a, g.dTa * q.idt, dPa);
  gd += contrib(g.da_d, g.db_d, g.dTd * q.idt, dPd);
  // f and fdot: dW/dtheta = -2 pi i c W, Re(conj(G)(-2 pi i c W)) = 2 pi c Im(conj(G) W)
  const R im = a * (ct.Gar * y.y - ct.Gai * y.x) + b * (ct.Gbr * y.y - ct.Gbi * y.x);
  gf += twopi * taub * im;
  gfd += twopi * (R)0.5 * taub * taub * im;
}

// Sum of NV values over a template's block partials (warp 0 of its last
// block; the result in every lane, in a fixed order).
template <int NV>
__device__ __forceinline__ void sum_partials(const double* __restrict__ p0, int nblk, double (&s)[NV]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < NV; ++i) s[i] = 0.0;
  for (int b = lane; b < nblk; b += 32)
#pragma unroll
    for (int i = 0; i < NV; ++i) s[i] += __ldcg(p0 + b * kPartW + i);
#pragma unroll
  for (int i = 0; i < NV; ++i)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s[i] += __shfl_xor_sync(0xffffffffu, s[i], o);
}

// An invalid template (all threads of block 0).
template <typename R>
__device__ __forceinline__ void fwd_invalid(const GradArgs<R>& g, int t) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    g.twoF[t] = __longlong_as_double(0x7ff8000000000000ll);
    for (int i = 0; i < 4; ++i) g.grad[4 * t + i] = __longlong_as_double(0x7ff8000000000000ll);
  }
}

// The end of the forward pass (all threads): block sums, and in the
// template's last block 2F and the cotangents.  v: F_a, F_b (re, im), A, B, C.
template <typename R>
__device__ __forceinline__ void fwd_finish(const GradArgs<R>& g, int t, double (&v)[7], double* red) {
  block_sum<7>(v, red);
  double* part = g.part + ((int64_t)t * kGradBlocks + blockIdx.x) * kPartW;
  if (threadIdx.x == 0)
    for (int i = 0; i < 7; ++i) part[i] = v[i];
  if (!last_block(g.counters + t, g.nblk)) return;
  if (threadIdx.x >= 32) return;
  double s[7];
  sum_partials<7>(g.part + (int64_t)t * kGradBlocks * kPartW, g.nblk, s);
  if (threadIdx.x != 0) return;
  const double Far = s[0], Fai = s[1], Fbr = s[2], Fbi = s[3], A = s[4], B = s[5], Cc = s[6];
  const double D = A * B - Cc * Cc;
  const double s2 = g.pc.sigma2;
  const double fa2 = Far * Far + Fai * Fai, fb2 = Fbr * Fbr + Fbi * Fbi, re = Far * Fbr + Fai * Fbi;
  const double N = B * fa2 + A * fb2 - 2.0 * Cc * re;
  double* cot = g.cot + (int64_t)t * kCotW;
  if (!(D > 0.0)) {
    set_status(g.status, FSTAT_ERANGE);
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    g.twoF[t] = nan;
    for (int i = 0; i < kCotW; ++i) cot[i] = 0.0;
    cot[15] = 1.0;   // flag: skip the adjoint
    return;
  }
  const double k2 = 2.0 / (s2 * D);
  g.twoF[t] = k2 * N;
  cot[0] = k2 * (2.0 * B * Far - 2.0 * Cc * Fbr);   // G_a
  cot[1] = k2 * (2.0 * B * Fai - 2.0 * Cc * Fbi);
  cot[2] = k2 * (2.0 * A * Fbr - 2.0 * Cc * Far);   // G_b
  cot[3] = k2 * (2.0 * A * Fbi - 2.0 * Cc * Fai);
  cot[4] = (2.0 / s2) * (fb2 / D - N * B / (D * D));          // d2F/dA
  cot[5] = (2.0 / s2) * (fa2 / D - N * A / (D * D));          // d2F/dB
  cot[6] = (2.0 / s2) * (-2.0 * re / D + 2.0 * N * Cc / (D * D));  // d2F/dC
  cot[15] = 0.0;
}

// The end of the adjoint pass (all threads).
template <typename R>
__device__ __forceinline__ void adj_finish(const GradArgs<R>& g, int t, double (&v)[4], double* red) {
  block_sum<4>(v, red);
  double* part = g.part + ((int64_t)t * kGradBlocks + blockIdx.x) * kPartW;
  if (threadIdx.x == 0)
    for (int i = 0; i < 4; ++i) part[i] = v[i];
  if (!last_block(g.counters + g.c.nt + t, g.nblk)) return;
  if (threadIdx.x >= 32) return;
  double s[4];
  sum_partials<4>(g.part + (int64_t)t * kGradBlocks * kPartW, g.nblk, s);
  if (threadIdx.x == 0)
    for (int i = 0; i < 4; ++i) g.grad[4 * t + i] = s[i];
}

// True in all threads when the adjoint of template t has nothing to do.
template <typename R>
__device__ __forceinline__ bool adj_skip(const GradArgs<R>& g, int t) {
  if (g.c.meta[t].status != FSTAT_OK) return true;
  if (g.cot[(int64_t)t * kCotW + 15] == 0.0) return false;
  if (blockIdx.x == 0 && threadIdx.x == 0)
    for (int i = 0; i < 4; ++i) g.grad[4 * t + i] = __longlong_as_double(0x7ff8000000000000ll);
  return true;
}

template <typename R>
__device__ __forceinline__ AdjConst<R>* con_of(const GradArgs<R>& g, int t) {
  return reinterpret_cast<AdjConst<R>*>(g.con + (int64_t)t * kConW);
}

// Point by point: FP64, and tap counts other than 8.
template <typename R, int TAPS>
__global__ void __launch_bounds__(kGradThreads) k_grad_fwd(GradArgs<R> g) {
  using C = cpx<R>;
  using Knot = typename KnotOf<R>::T;
  __shared__ double red[7 * 32];
  const int t = blockIdx.y;
  const TmplMeta m = g.c.meta[t];
  if (m.status != FSTAT_OK) { fwd_invalid(g, t); return; }
  if (blockIdx.x == 0 && threadIdx.x >= kGradThreads - 32) adj_constants<R>(g.pc, g.c.tmpl[t], m.tb0, con_of(g, t));
  const Knot* kn = reinterpret_cast<const Knot*>(g.c.knots) + (int64_t)t * g.c.knot_stride;
  const double df = g.df[t];
  const double c0 = df * (m.tb0 - g.pc.t_start);
  const R c0f = (R)(c0 - floor(c0));
  const double fdt = df * g.pc.dt;
  const unsigned long long fdt64 = frac_fix64(fdt);
  R far = 0, fai = 0, fbr = 0, fbi = 0, sa = 0, sb = 0, sc = 0;
  GapCursor gc = make_cursor(m, g.gaps);
  for (int k = blockIdx.x * kGradThreads + threadIdx.x; k < (int)m.n_b; k += gridDim.x * kGradThreads) {
    C wa, wb;
    R aa, bb;
    if (!sample_weights<R, FSTAT_SINC, TAPS>(g.pc, kn, k, g.x, gc, g.wcs, wa, wb, aa, bb))
      continue;
    const C e = expm<R>(bin_phase<R>(fdt64, fdt, k) + c0f);
    const C xa = cmul(wa, e), xb = cmul(wb, e);
    far += xa.x; fai += xa.y; fbr += xb.x; fbi += xb.y;
    sa += aa * aa; sb += bb * bb; sc += aa * bb;
  }
  double v[7] = {far, fai, fbr, fbi, sa, sb, sc};
  fwd_finish(g, t, v, red);
}

template <typename R, int TAPS>
__global__ void __launch_bounds__(kGradThreads) k_grad_adj(GradArgs<R> g) {
  using Knot = typename KnotOf<R>::T;
  __shared__ double red[4 * 32];
  const int t = blockIdx.y;
  if (adj_skip(g, t)) return;
  const TmplMeta m = g.c.meta[t];
  const PlanConst& pc = g.pc;
  const Knot* kn = reinterpret_cast<const Knot*>(g.c.knots) + (int64_t)t * g.c.knot_stride;
  const AdjConst<R> q = *con_of(g, t);
  const Cot<R> ct = load_cot<R>(g.cot + (int64_t)t * kCotW);
  const double df = g.df[t];
  const double c0 = df * (m.tb0 - pc.t_start);
  const R c0f = (R)(c0 - floor(c0));
  const double fdt = df * pc.dt;
  const unsigned long long fdt64 = frac_fix64(fdt);
  R ga = 0, gd = 0, gf = 0, gfd = 0;
  GapCursor gc = make_cursor(m, g.gaps);
  for (int k = blockIdx.x * kGradThreads + threadIdx.x; k < (int)m.n_b; k += gridDim.x * kGradThreads)
    adj_point<R, TAPS>(pc, kn, k, g.x, gc, g.wcs, q, ct, fdt64, fdt, c0f, (R)df, ga, gd, gf, gfd);
  double v[4] = {ga, gd, gf, gfd};
  adj_finish(g, t, v, red);
}

// FP32, 8 taps: runs of eight consecutive grid points per lane, 256 per warp
// and step, with the expansions of the resampler (sinc_run.cuh): one weight
// expansion, one set of knot cubics and (adjoint) one evaluation of the
// geometry per run, the phase with the bin's included.  The adjoint of a run
// needs only the sums over its points of Re(conj(G) y), Re(conj(G) dy) and
// Im(conj(G) W) with weights 1 and tau, because everything they multiply is
// linear over a run (a few samples of a sidereal day) to single precision.
// Point by point the adjoint took two sincosf, three sincospif and 17
// divisions a point, and every thread of every block its own FP64 constants:
// 64 candidates of 864,000 samples 573 us forward and 3523 us adjoint, now 245
// and 358 (bound by instruction issue).  The samples of a step (272 from the one before its
// first tap) are copied a step ahead into the warp's shared memory.
constexpr int kGrSamples = 272;
constexpr int kGrUnits = kGrSamples / 2;           // 16-byte pieces
constexpr int kGrPad = kGrUnits + kGrUnits / 4;    // one piece of padding every four: lanes 8 samples apart on distinct banks
constexpr int kGrWarps = kGradThreads / 32;
__device__ __forceinline__ int gr_unit(int u) { return u + (u >> 2); }

// What a run of a lane needs, computed from its knot record.
struct RunState {
  int k0, n0, base;           // first point, floor(u) there, first staged sample
  float f, d1, d2;            // fraction at the centre, and how u moves
  float pc0, p1, p2;          // phase to remove (cycles), the bin's included
  float a0, a1, a2, b0, b1, b2;
  float spread;
};

template <typename F>
__device__ __forceinline__ void for_slow_runs(bool slow_run, int k0, int g, F&& point) {
  const int lane = threadIdx.x & 31;
  unsigned slow = __ballot_sync(0xffffffffu, slow_run);
  while (slow) {
    // four runs at a time, eight lanes a run
    int src = -1;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (lane >> 3 == r) src = __ffs(slow) - 1;
      slow &= slow - 1;
    }
    const int sl = src < 0 ? 0 : src;
    const int ks = __shfl_sync(0xffffffffu, k0, sl), gs = __shfl_sync(0xffffffffu, g, sl);
    if (src >= 0) point(ks + (lane & 7), gs);
    __syncwarp();
  }
}

__device__ __noinline__ void fwd_slow(const GradArgs<float>& g, const KnotF* kn, int k, int n_b, GapCursor gc, int gi,
                                      unsigned long long fdt64, float c0f, float (&acc)[7]) {
  if (k >= n_b) return;
  gc.g = gi;
  gc.load();
  float2 wa, wb;
  float aa, bb;
  if (!sample_weights<float, FSTAT_SINC, 8>(g.pc, kn, k, g.x, gc, g.wcs, wa, wb, aa, bb)) return;
  const float2 e = expm<float>(frac_mul(fdt64, k) + c0f);
  const float2 xa = cmul(wa, e), xb = cmul(wb, e);
  acc[0] += xa.x; acc[1] += xa.y; acc[2] += xb.x; acc[3] += xb.y;
  acc[4] += aa * aa; acc[5] += bb * bb; acc[6] += aa * bb;
}

__device__ __noinline__ void adj_slow(const GradArgs<float>& g, const KnotF* kn, int k, int n_b, GapCursor gc, int gi,
                                      const AdjConst<float>& q, const Cot<float>& ct, unsigned long long fdt64,
                                      float c0f, float df, float (&acc)[4]) {
  if (k >= n_b) return;
  gc.g = gi;
  gc.load();
  adj_point<float, 8>(g.pc, kn, k, g.x, gc, g.wcs, q, ct, fdt64, 0.0, c0f, df, acc[0], acc[1], acc[2], acc[3]);
}

// Both passes.  QUAD: the weights' square in d is kept (u moves faster than
// kRunNarrow allows for the linear form).
template <bool LANCZOS, bool QUAD, bool ADJ>
__global__ void __launch_bounds__(kGradThreads, 2) k_grad_run(GradArgs<float> g) {
  constexpr int NV = ADJ ? 4 : 7;
  __shared__ double red[NV * 32];
  __shared__ float4 buf[kGrWarps][2][kGrPad];
  __shared__ AdjConst<float> q;
  const int t = blockIdx.y;
  const TmplMeta m = g.c.meta[t];
  if constexpr (ADJ) {
    if (adj_skip(g, t)) return;
    if (threadIdx.x < sizeof(AdjConst<float>) / 4)
      reinterpret_cast<float*>(&q)[threadIdx.x] = reinterpret_cast<const float*>(con_of(g, t))[threadIdx.x];
    __syncthreads();
  } else {
    if (m.status != FSTAT_OK) { fwd_invalid(g, t); return; }
    if (blockIdx.x == 0 && threadIdx.x >= kGradThreads - 32)
      adj_constants<float>(g.pc, g.c.tmpl[t], m.tb0, con_of(g, t));
  }
  const PlanConst& pc = g.pc;
  const KnotF* kn = reinterpret_cast<const KnotF*>(g.c.knots) + (int64_t)t * g.c.knot_stride;
  const int n_b = (int)m.n_b;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double dfd = g.df[t];
  const double c0 = dfd * (m.tb0 - pc.t_start);
  const float c0f = (float)(c0 - floor(c0));
  const double fdt = dfd * pc.dt;
  const unsigned long long fdt64 = frac_fix64(fdt), half64 = frac_fix64(0.5 * fdt);
  // the bin's phase step (cycles a point) less an even number: tau, an odd
  // number of halves, turns it into whole cycles
  const float fdt1 = (float)(fdt - 2.0 * rint(0.5 * fdt));
  const int odd = (int)(((uintptr_t)g.x >> 3) & 1);
  const int x_end = (((int)pc.n_data + odd) & ~1) - odd;
  const int hmask = (1 << pc.log2h) - 1;
  [[maybe_unused]] Cot<float> ct;
  if constexpr (ADJ) ct = load_cot<float>(g.cot + (int64_t)t * kCotW);

  auto prepare = [&](int step, int u) {
    RunState r;
    r.k0 = step * 256 + 8 * lane;
    const int kc = r.k0 < n_b ? r.k0 : n_b - 1;
    const int sk = kc & hmask;
    const float4* kp = reinterpret_cast<const float4*>(kn + (kc >> pc.log2h));
    const float4 q0 = __ldg(kp), q1 = __ldg(kp + 1), q2 = __ldg(kp + 2), q3 = __ldg(kp + 3), q4 = __ldg(kp + 4);
    const float s = small_int_to_float(sk) + 3.5f;       // the run's centre
    const float dev = fmaf(fmaf(fmaf(q1.x, s, q0.w), s, q0.z), s, q0.y);
    int fl;
    float flf = round_nearest(dev, &fl);
    if (flf > dev) { flf -= 1.0f; --fl; }
    r.f = dev - flf;
    r.n0 = __float_as_int(q0.x) + sk + fl;
    r.d1 = q0.z + s * (2.0f * q0.w + 3.0f * q1.x * s); r.d2 = q0.w + 3.0f * q1.x * s;
    r.spread = 3.5f * fabsf(r.d1) + 12.25f * fabsf(r.d2);
    // the phase with the bin's, frac(df dt (k0 + 7/2)) = frac(df dt / 2 (2 k0 + 7)) exactly
    const float bin = (float)((half64 * (unsigned long long)(2ll * r.k0 + 7)) >> 40) * (1.0f / 16777216.0f);
    r.pc0 = knot_phase(q1.y, q1.z, q1.w, q2.x, s) + bin + c0f;
    r.p1 = q1.z + s * (2.0f * q1.w + 3.0f * q2.x * s) + fdt1; r.p2 = q1.w + 3.0f * q2.x * s;
    r.a0 = q2.y + ((q3.x * s + q2.w) * s + q2.z) * s;
    r.a1 = q2.z + s * (2.0f * q2.w + 3.0f * q3.x * s); r.a2 = q2.w + 3.0f * q3.x * s;
    r.b0 = q3.y + ((q4.x * s + q3.w) * s + q3.z) * s;
    r.b1 = q3.z + s * (2.0f * q3.w + 3.0f * q4.x * s); r.b2 = q3.w + 3.0f * q4.x * s;
    const int first = __shfl_sync(0xffffffffu, r.n0, 0) - 4;
    r.base = ((first + odd) & ~1) - odd;
    float4* dst = buf[warp][u];
    if (r.base >= odd && r.base + kGrSamples <= x_end) {
      // 32 pieces on, the padded place is 40 on
      const float2* src = g.x + r.base + 2 * lane;
#pragma unroll
      for (int i = 0; i < (kGrUnits + 31) / 32; ++i)
        if (32 * i + 32 <= kGrUnits || lane < kGrUnits % 32) copy_async16(dst + gr_unit(lane) + 40 * i, src + 64 * i, true);
    } else {
#pragma unroll 1
      for (int un = lane; un < kGrUnits; un += 32) {
        const int jx = r.base + 2 * un;
        const bool inside = jx >= odd && jx < x_end;
        copy_async16(dst + gr_unit(un), inside ? g.x + jx : g.x + odd, inside);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    return r;
  };

  GapCursor gc = make_cursor(m, g.gaps);
  float acc[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) acc[i] = 0.f;
  const int steps = (n_b + 255) >> 8;
  const int stride = gridDim.x * kGrWarps;
  const int first_step = blockIdx.x * kGrWarps + warp;
  if (first_step < steps) {
    RunState r = prepare(first_step, 0);
    if (gc.n > 0) gc.seek(r.n0 - 64);                    // the lane's points only move forward
    int u = 0;
#pragma unroll 1
    for (int step = first_step; step < steps; step += stride) {
      const RunState nx = prepare(step + stride < steps ? step + stride : step, u ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncwarp();
      gc.advance(r.n0 - 5);
      const bool live = r.k0 < n_b;
      const bool smooth = r.spread <= (QUAD ? kRunSpread : kRunNarrow);
      const bool masked = smooth && gc.cs < r.n0 && r.n0 + 9 < gc.ce;
      const int off = r.n0 - 3 - r.base, j0 = r.n0 - 3, j1 = r.n0 + 11;
      const bool fast = live && smooth && r.k0 + 7 < n_b && off >= 0 && off + 16 <= kGrSamples && j0 >= odd &&
                        j1 < x_end && j0 >= gc.lo && j1 < gc.hi && j1 < gc.cs &&
                        ((LANCZOS && !QUAD && !ADJ) || (r.f >= r.spread + 1e-6f && r.f + r.spread < 1.0f - 1e-6f)) &&
                        12.25f * fabsf(r.p2) <= 1e-5f;
      if (fast) {
        float w0[8], w1[8], w2[8];
        if constexpr (ADJ) run_weights_d<LANCZOS>(r.f - 0.5f, w0, w1, w2);
        else run_weights<LANCZOS>(r.f - 0.5f, w0, w1, w2);
        if constexpr (!QUAD) {
          const float hs = 0.5f * r.spread * r.spread;
#pragma unroll
          for (int tp = 0; tp < 8; ++tp) w0[tp] = fmaf(hs, w2[tp], w0[tp]);
        }
        float2 v[16];
        const float4* xr = buf[warp][u];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float4 p = xr[gr_unit((off >> 1) + j)];
          v[2 * j] = make_float2(p.x, p.y);
          v[2 * j + 1] = make_float2(p.z, p.w);
        }
        if (off & 1) {
#pragma unroll
          for (int j = 0; j < 15; ++j) v[j] = v[j + 1];
        }
        int di;
        const float2 ec = expm2pi(r.pc0 - round_nearest(r.pc0, &di));
        // sums over the run of p = Re(conj(G_a) y), Re(conj(G_b) y), of
        // Re(conj(a G_a + b G_b) dy) and of Im(conj(a G_a + b G_b) y), with
        // weights 1 and tau
        [[maybe_unused]] float P0 = 0.f, P1 = 0.f, Q0 = 0.f, Q1 = 0.f, D0 = 0.f, D1 = 0.f, I0 = 0.f, I1 = 0.f;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const float th = (float)h + 0.5f, t2 = th * th;
          const float lin = th * r.p1;
          const float2 e = expm2pi(lin - round_nearest(lin, &di));     // (cos, -sin)
          const float eps = (6.28318531f * t2) * r.p2;
          const float ex = fmaf(eps, ec.y, ec.x), ey = fmaf(-eps, ec.x, ec.y);
          const float xc = ex * e.x, yc = ey * e.x;
          const float2 rot[2] = {make_float2(fmaf(ey, e.y, xc), fmaf(-ex, e.y, yc)),     // tau = -th
                                 make_float2(fmaf(-ey, e.y, xc), fmaf(ex, e.y, yc))};    // tau = +th
#pragma unroll
          for (int sd = 0; sd < 2; ++sd) {
            const int i = sd ? 4 + h : 3 - h;
            const float tau = sd ? th : -th;
            const float d = fmaf(tau, r.d1, t2 * r.d2);
            float2 z = make_float2(0.f, 0.f);
            [[maybe_unused]] float2 dz = make_float2(0.f, 0.f);
#pragma unroll
            for (int tp = 0; tp < 8; ++tp) {
              float w;
              if constexpr (QUAD) w = fmaf(d, fmaf(d, w2[tp], w1[tp]), w0[tp]);
              else w = fmaf(d, w1[tp], w0[tp]);
              z.x = fmaf(w, v[i + tp].x, z.x);
              z.y = fmaf(w, v[i + tp].y, z.y);
              if constexpr (ADJ) {
                const float dw = fmaf(2.0f * d, w2[tp], w1[tp]);
                dz.x = fmaf(dw, v[i + tp].x, dz.x);
                dz.y = fmaf(dw, v[i + tp].y, dz.y);
              }
            }
            const float a = fmaf(tau, r.a1, fmaf(t2, r.a2, r.a0));
            const float bb = fmaf(tau, r.b1, fmaf(t2, r.b2, r.b0));
            const float2 y = cmul(z, rot[sd]);
            if constexpr (ADJ) {
              const float2 dy = cmul(dz, rot[sd]);
              const float hr = fmaf(a, ct.Gar, bb * ct.Gbr), hi = fmaf(a, ct.Gai, bb * ct.Gbi);
              const float p = fmaf(ct.Gar, y.x, ct.Gai * y.y), pq = fmaf(ct.Gbr, y.x, ct.Gbi * y.y);
              const float qd = fmaf(hr, dy.x, hi * dy.y), im = fmaf(hr, y.y, -hi * y.x);
              P0 += p; P1 = fmaf(tau, p, P1);
              Q0 += pq; Q1 = fmaf(tau, pq, Q1);
              D0 += qd; D1 = fmaf(tau, qd, D1);
              I0 += im; I1 = fmaf(tau, im, I1);
            } else {
              acc[0] = fmaf(a, y.x, acc[0]); acc[1] = fmaf(a, y.y, acc[1]);
              acc[2] = fmaf(bb, y.x, acc[2]); acc[3] = fmaf(bb, y.y, acc[3]);
            }
          }
        }
        if constexpr (ADJ) {
          const float twopi = 6.28318531f;
          const AdjGeo<float> ge = adj_geometry<float, true>(q, (float)r.n0 + (r.f + 3.5f));
          const float taub = fmaf((float)r.k0 + 3.5f, q.dt, q.tb0);
          const float df = (float)dfd;
          const float fb = taub * (q.fdot + 0.5f * q.fddot * taub) + df;
          const float fb1 = q.dt * (q.fdot + q.fddot * taub);
          auto contrib = [&](float dA, float dB, float dA1, float dB1, float dT, float dT1, float g0) {
            const float dP = q.fh * (g0 - dT) + fb * g0, dP1 = fb1 * g0 - q.fh * dT1;
            return dA * P0 + dA1 * P1 + dB * Q0 + dB1 * Q1 + q.idt * (dT * D0 + dT1 * D1) +
                   twopi * (dP * I0 + dP1 * I1) +
                   ct.gA * 2.0f * (8.0f * r.a0 * dA + 42.0f * r.a1 * dA1) +
                   ct.gB * 2.0f * (8.0f * r.b0 * dB + 42.0f * r.b1 * dB1) +
                   ct.gC * (8.0f * (dA * r.b0 + r.a0 * dB) + 42.0f * (dA1 * r.b1 + r.a1 * dB1));
          };
          acc[0] += contrib(ge.da_a, ge.db_a, ge.da_a1, ge.db_a1, ge.dTa, ge.dTa1, q.g0a);
          acc[1] += contrib(ge.da_d, ge.db_d, ge.da_d1, ge.db_d1, ge.dTd, ge.dTd1, q.g0d);
          acc[2] += twopi * (taub * I0 + q.dt * I1);
          acc[3] += 0.5f * twopi * taub * (taub * I0 + 2.0f * q.dt * I1);
        } else {
          acc[4] += fmaf(8.0f * r.a0, r.a0, fmaf(42.0f, fmaf(r.a1, r.a1, 2.0f * r.a0 * r.a2), 388.5f * r.a2 * r.a2));
          acc[5] += fmaf(8.0f * r.b0, r.b0, fmaf(42.0f, fmaf(r.b1, r.b1, 2.0f * r.b0 * r.b2), 388.5f * r.b2 * r.b2));
          acc[6] += fmaf(8.0f * r.a0, r.b0, fmaf(42.0f, fmaf(r.a1, r.b1, fmaf(r.a0, r.b2, r.a2 * r.b0)), 388.5f * r.a2 * r.b2));
        }
      }
      for_slow_runs(live && !fast && !masked, r.k0, gc.g, [&](int k, int gi) {
        if constexpr (ADJ) adj_slow(g, kn, k, n_b, gc, gi, q, ct, fdt64, c0f, (float)dfd, acc);
        else fwd_slow(g, kn, k, n_b, gc, gi, fdt64, c0f, acc);
      });
      __syncwarp();
      r = nx;
      u ^= 1;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }
  double v[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = (double)acc[i];
  if constexpr (ADJ) adj_finish(g, t, v, red);
  else fwd_finish(g, t, v, red);
}

template <typename R>
cudaError_t run_grad(const PlanConst& pc, const Chunk& c, const float2* x, const int64_t* gaps,
                     const double* wcs, const double* df, double* work, double* twoF, double* grad,
                     int* status, int pass, cudaStream_t s) {
  GradArgs<R> g;
  g.pc = pc; g.c = c; g.x = x; g.gaps = gaps; g.wcs = wcs; g.df = df;
  g.part = work;
  g.cot = work + (int64_t)c.nt * kGradBlocks * kPartW;
  g.con = g.cot + (int64_t)c.nt * kCotW;
  g.counters = c.counters;
  g.twoF = twoF; g.grad = grad; g.status = status;
  g.nblk = kGradBlocks;
  if constexpr (std::is_same<R, float>::value) {
    // knot intervals of whole runs; h >= 16 always holds
    if (pc.taps == 8) {
      // four rounds of the 16 warps x 152 SMs that hold the kernel at once
      const int want = 4 * 2 * 152 / c.nt;
      g.nblk = want < 16 ? 16 : (want > kGradBlocks ? kGradBlocks : want);
      const dim3 grid((unsigned)g.nblk, (unsigned)c.nt);
      const bool lz = pc.window == FSTAT_WIN_LANCZOS, quad = runs_need_square(pc);
      auto go = [&](auto fwd, auto adj) {
        if (pass == 0) fwd<<<grid, kGradThreads, 0, s>>>(g);
        else adj<<<grid, kGradThreads, 0, s>>>(g);
      };
      if (lz && !quad) go(k_grad_run<true, false, false>, k_grad_run<true, false, true>);
      else if (lz) go(k_grad_run<true, true, false>, k_grad_run<true, true, true>);
      else if (!quad) go(k_grad_run<false, false, false>, k_grad_run<false, false, true>);
      else go(k_grad_run<false, true, false>, k_grad_run<false, true, true>);
      return cudaGetLastError();
    }
  }
  dim3 grid(kGradBlocks, (unsigned)c.nt);
  if constexpr (std::is_same<R, double>::value) {
    if (pc.taps == 8) {
      if (pass == 0) k_grad_fwd<R, 8><<<grid, kGradThreads, 0, s>>>(g);
      else k_grad_adj<R, 8><<<grid, kGradThreads, 0, s>>>(g);
      return cudaGetLastError();
    }
  }
  if (pass == 0) k_grad_fwd<R, 0><<<grid, kGradThreads, 0, s>>>(g);
  else k_grad_adj<R, 0><<<grid, kGradThreads, 0, s>>>(g);
  return cudaGetLastError();
}

}  // namespace

size_t grad_work_doubles(int nt) { return (size_t)nt * (kGradBlocks * kPartW + kCotW + kConW); }

// pass 0: forward (2F, cotangents); pass 1: adjoint (gradient)
cudaError_t launch_grad_pass(const PlanConst& pc, const Chunk& c, const float2* x, const int64_t* gaps,
                             const double* wcs, const double* df, double* work, double* twoF,
                             double* grad, int* status, int pass, cudaStream_t s) {
  if (pc.precision == FSTAT_PREC_FP64)
    return run_grad<double>(pc, c, x, gaps, wcs, df, work, twoF, grad, status, pass, s);
  return run_grad<float>(pc, c, x, gaps, wcs, df, work, twoF, grad, status, pass, s);
}

}  // namespace fs
