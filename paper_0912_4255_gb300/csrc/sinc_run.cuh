// Windowed-sinc weights for a run of consecutive grid points (step 4 of
// Sec. III.A.2, 8 taps, single precision).
//
// Along a run of eight grid points the fractional index u - k moves by a few
// 1e-4 only (dt_m/dt ~ 1e-4, Eq. 4pt2), so the eight tap weights are
// expanded once per run: at the run's centre u = n + f, f = g + 1/2, tap i
// has x_i = f + 3 - i and
//   w_i(f + d) = K(x_i) + d K'(x_i) + d^2 K''(x_i) / 2,
// with |d| <= kRunSpread = 1.5e-3 the neglected d^3 K''' / 6 is below 2e-8
// (2e-10 at the Earth's 3.7e-4).  K is the Lanczos window times the sinc or
// the plain sinc.  K is even, so taps i and 7 - i take the even and odd parts
// of one polynomial in g:  K(x_i) = E(g^2) + g O(g^2), K(x_{7-i}) = E - g O.
// The polynomials interpolate K, K' and K'' / 2 at the Chebyshev nodes of
// |g| <= 1/2; they have no singularity at the sample nearest to u, so no
// reciprocal, sine or special case is left.  Per point: 8 FMAs for the
// weights (16 with the square in d) and 16 for the sum, against 62
// instructions and 8 reciprocals for weights formed point by point.
#pragma once

#include "fstat_internal.cuh"

namespace fs {

constexpr float kRunSpread = 1.5e-3f;
constexpr float kRunNarrow = 4.5e-4f;   // |d| up to which a linear form of the weights is used

// Coefficients of g^k for tap p (0..3), ascending.
// K_p(g): degree 10.  The coefficients are rounded to single precision one after
// the other, the constant first, each time with a new fit of those that follow, so
// that the mean error over g stays near zero: a coherent sum of samples sees the
// mean.  Error as written below 7e-10 (tap 0) to 3e-8 (tap 3), mean below 4e-9; rounded
// from one fit they erred by up to 5.5e-8, with a mean of 2.7e-8.  (The errors stated
// for K' and K''/2 are those of the fits; rounding adds half a unit in the last
// place of each coefficient.)
template <bool LANCZOS>
__host__ __device__ constexpr float sinc_c0(int p, int k) {
  constexpr float lz[4][11] = {
      {-0.0126608778f, 0.0312413145f, 0.0495652221f, -0.15180859f, 0.0118439076f, 0.115309335f, -0.0331076756f, -0.0328786187f, 0.0124566918f, 0.00453863107f, -0.00207216316f},
      {0.0599094816f, -0.0674174875f, -0.269770414f, 0.324785233f, 0.118619673f, -0.235903755f, 0.0100880126f, 0.0640243962f, -0.0103230393f, -0.00901622791f, 0.0021423921f},
      {-0.166415229f, 0.167748332f, 0.722850561f, -0.765625536f, -0.231783688f, 0.401936233f, 0.0106301596f, -0.0969409868f, 0.00629437901f, 0.0132465046f, -0.00165375881f},
      {0.620383024f, -1.30521214f, -0.513493776f, 1.34897912f, 0.130107567f, -0.541389048f, -0.00873297732f, 0.119500615f, -0.00101422041f, -0.0161359441f, -0.000913758879f}};
  constexpr float rc[4][11] = {
      {-0.0909456834f, 0.0259844773f, 0.441374958f, -0.126106843f, -0.333095193f, 0.0951634347f, 0.094278127f, -0.0268735122f, -0.013841561f, 0.00369112426f, 0.00139993429f},
      {0.127323955f, -0.0509295799f, -0.607946754f, 0.243178457f, 0.419500947f, -0.167793885f, -0.102900557f, 0.041093424f, 0.0135331191f, -0.00512069976f, -0.00114567636f},
      {-0.212206587f, 0.141471058f, 0.952883184f, -0.635255396f, -0.437773645f, 0.291846991f, 0.0887024775f, -0.0591107421f, -0.0101380497f, 0.00664602965f, 0.000274523074f},
      {0.636619747f, -1.27323949f, -0.59511131f, 1.19022477f, 0.203347757f, -0.406769395f, -0.0359162949f, 0.0726720765f, 0.00178920047f, -0.0074517983f, 0.00313225482f}};
  return LANCZOS ? lz[p][k] : rc[p][k];
}

// K_p'(g): degree 6 (error below 2e-5)
template <bool LANCZOS>
__host__ __device__ constexpr float sinc_c1(int p, int k) {
  constexpr float lz[4][7] = {
      {0.031241317f, 0.0992852604f, -0.455355985f, 0.042386143f, 0.574313236f, -0.15788033f, -0.212283071f},
      {-0.0674174939f, -0.539665916f, 0.974217125f, 0.478519001f, -1.17508254f, 0.0273248969f, 0.412678687f},
      {0.167748344f, 1.44577476f, -2.2966732f, -0.929521004f, 2.00316529f, 0.0835524577f, -0.626447058f},
      {-1.3052121f, -1.02700845f, 4.0466865f, 0.521077616f, -2.6989857f, -0.05718888f, 0.772958918f}};
  constexpr float rc[4][7] = {
      {0.0259844805f, 0.882571174f, -0.378263846f, -1.32663619f, 0.474001432f, 0.519135787f, -0.173585281f},
      {-0.0509295818f, -1.21571705f, 0.729456602f, 1.67233756f, -0.836449449f, -0.571603333f, 0.267495691f},
      {0.141471061f, 1.90562973f, -1.90566396f, -1.74671991f, 1.45596423f, 0.497110084f, -0.387611461f},
      {-1.27323954f, -1.19017423f, 3.57056225f, 0.81191073f, -2.03019802f, -0.204973338f, 0.479392981f}};
  return LANCZOS ? lz[p][k] : rc[p][k];
}

// K_p''(g) / 2: degree 3 (error below 2e-2)
template <bool LANCZOS>
__host__ __device__ constexpr float sinc_c2(int p, int k) {
  constexpr float lz[4][4] = {
      {0.052803632f, -0.450350369f, -0.0351086202f, 0.989411992f},
      {-0.270429034f, 0.964484836f, 0.734868266f, -2.04065128f},
      {0.721292117f, -2.28190245f, -1.34206937f, 3.53648812f},
      {-0.512398638f, 4.02846435f, 0.745876279f, -4.81824363f}};
  constexpr float rc[4][4] = {
      {0.431056993f, -0.374170831f, -1.66548724f, 0.817812094f},
      {-0.596606229f, 0.723153128f, 2.15124766f, -1.4722748f},
      {0.943037043f, -1.89653514f, -2.30938126f, 2.62121704f},
      {-0.59105728f, 3.55927542f, 1.08975598f, -3.70084816f}};
  return LANCZOS ? lz[p][k] : rc[p][k];
}

// K_p'(g): degree 9 (error below 4e-8)
template <bool LANCZOS>
__host__ __device__ constexpr float sinc_d1(int p, int k) {
  constexpr float lz[4][10] = {
      {0.0312413086f, 0.0991304465f, -0.455424834f, 0.0473753765f, 0.576523968f, -0.198639391f, -0.229977672f, 0.0995995716f, 0.0404449701f, -0.0205903271f},
      {-0.0674174752f, -0.539541132f, 0.974353708f, 0.474493299f, -1.17946992f, 0.0603136499f, 0.44779701f, -0.0813661277f, -0.0802709001f, 0.0190777152f},
      {0.167748317f, 1.44570152f, -2.2968739f, -0.927154448f, 2.00961249f, 0.0640745622f, -0.678053448f, 0.0486742003f, 0.117958162f, -0.0132871303f},
      {-1.30521206f, -1.02698568f, 4.04692699f, 0.52034084f, -2.70671128f, -0.0511003817f, 0.834798099f, -0.0153959277f, -0.141347547f, 0.00473270745f}};
  constexpr float rc[4][10] = {
      {0.0259844735f, 0.882749625f, -0.378319861f, -1.33236664f, 0.475800224f, 0.565460635f, -0.187982888f, -0.109550496f, 0.0329089655f, 0.0117268684f},
      {-0.0509295727f, -1.21589339f, 0.729534227f, 1.67799893f, -0.838941572f, -0.617336481f, 0.287442022f, 0.10790067f, -0.0455917963f, -0.0107754865f},
      {0.14147105f, 1.90576702f, -1.90576482f, -1.75112652f, 1.45920181f, 0.532685048f, -0.413523395f, -0.0837676551f, 0.0592274895f, 0.00785010607f},
      {-1.27323953f, -1.19022713f, 3.57067894f, 0.813608461f, -2.03394302f, -0.218674528f, 0.50936557f, 0.0322260373f, -0.0685090036f, -0.0029085598f}};
  return LANCZOS ? lz[p][k] : rc[p][k];
}

// K_p''(g) / 2: degree 5 (error below 3e-4)
template <bool LANCZOS>
__host__ __device__ constexpr float sinc_d2(int p, int k) {
  constexpr float lz[4][6] = {
      {0.0497184741f, -0.455346178f, 0.0599841419f, 1.14736038f, -0.375646415f, -0.629265561f},
      {-0.269893902f, 0.974197673f, 0.720661722f, -2.3476518f, 0.0530455575f, 1.22298468f},
      {0.722922997f, -2.29664462f, -1.39596167f, 4.00263719f, 0.217765087f, -1.85722311f},
      {-0.513515251f, 4.04665225f, 0.782135258f, -5.39354566f, -0.145711919f, 2.29237298f}};
  constexpr float rc[4][6] = {
      {0.441197254f, -0.378255867f, -1.98574012f, 0.946972642f, 1.27543225f, -0.514585218f},
      {-0.607771175f, 0.729445542f, 2.50433721f, -1.67147182f, -1.40683572f, 0.793938371f},
      {0.952746821f, -1.90564958f, -2.61683094f, 2.91007477f, 1.22549331f, -1.15172895f},
      {-0.595060887f, 3.57054562f, 1.21661355f, -4.05825198f, -0.505770076f, 1.4253332f}};
  return LANCZOS ? lz[p][k] : rc[p][k];
}


// E(t) + g O(t) of the coefficients C(p, 0 .. DEG): *plus = E + g O (tap p),
// *minus = E - g O (tap 7 - p).
#define FS_EVEN_ODD(C, DEG, p, g, t, plus, minus)                                    \
  {                                                                                  \
    constexpr int e1 = (DEG) & ~1, o1 = ((DEG) - 1) | 1;                             \
    float E = C(p, e1), O = C(p, o1);                                                \
    _Pragma("unroll") for (int k = e1 - 2; k >= 0; k -= 2) E = fmaf(E, t, C(p, k));  \
    _Pragma("unroll") for (int k = o1 - 2; k >= 1; k -= 2) O = fmaf(O, t, C(p, k));  \
    plus = fmaf(g, O, E);                                                            \
    minus = fmaf(-g, O, E);                                                          \
  }

// Weights of the eight taps at the run's centre and their expansion in the
// offset from it: w(d) = w0 + d (w1 + d w2).
template <bool LANCZOS>
__device__ __forceinline__ void run_weights(float g, float (&w0)[8], float (&w1)[8], float (&w2)[8]) {
  const float t = g * g;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    FS_EVEN_ODD(sinc_c0<LANCZOS>, 10, p, g, t, w0[p], w0[7 - p]);
    FS_EVEN_ODD(sinc_c1<LANCZOS>, 6, p, g, t, w1[p], w1[7 - p]);
    w1[7 - p] = -w1[7 - p];          // d/du of K(x_{7-p}) = K_p(-g)
    FS_EVEN_ODD(sinc_c2<LANCZOS>, 3, p, g, t, w2[p], w2[7 - p]);
  }
}

// The same with K' to single precision, for the derivative of the
// interpolant: dw(d) = w1 + 2 d w2.
template <bool LANCZOS>
__device__ __forceinline__ void run_weights_d(float g, float (&w0)[8], float (&w1)[8], float (&w2)[8]) {
  const float t = g * g;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    FS_EVEN_ODD(sinc_c0<LANCZOS>, 10, p, g, t, w0[p], w0[7 - p]);
    FS_EVEN_ODD(sinc_d1<LANCZOS>, 9, p, g, t, w1[p], w1[7 - p]);
    w1[7 - p] = -w1[7 - p];
    FS_EVEN_ODD(sinc_d2<LANCZOS>, 5, p, g, t, w2[p], w2[7 - p]);
  }
}

// u - k moves by at most beta (1 + beta) samples a grid point: whether that
// leaves the linear form of the weights (kRunNarrow over 3.5 points; the
// Earth's motion gives 3.7e-4).
inline bool runs_need_square(const PlanConst& pc) {
  const double beta = pc.beta;
  return 3.5 * beta * (1.0 + 2.0 * beta) > 0.98 * kRunNarrow;
}

// 16 bytes into shared memory, behind the thread's back; zeros if !inside.
__device__ __forceinline__ void copy_async16(void* dst, const void* src, bool inside) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(inside ? 16 : 0) : "memory");
}

}  // namespace fs
