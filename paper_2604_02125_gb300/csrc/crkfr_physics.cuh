// crkfr_physics.cuh -- device physics of the cRKFR hot path (sm_103a).
//
// System u_t + f(u)_x + B(u) g(u)_x = 0 (paper: eq. flux.and.non.cons).
// Point-wise physical flux, spectral radius of f' + B g' (eqs.
// rusanov.wave.speed / combined.wave.speed), two-point volume fluxes f_S of
// the flux-differencing form (Sec. 3, eq. entropy.cons.flux.dev) and the
// non-conservative product of eq. entropy.cons.noncons.dev.
//
// Every routine works on "pair data" q[P]: primitive values of one node that
// the two-point fluxes need, computed once per node and stage.  Templated on
// the arithmetic type R (double for the FP64 path, float for the FP32
// pair-flux form).
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace crk {

constexpr int VOL_EC = 0, VOL_KEP = 1, VOL_CENTRAL = 2;

__host__ __device__ constexpr int ipow(int b, int e) { return e == 0 ? 1 : b * ipow(b, e - 1); }

template <typename R>
struct PhysParams {
  R gamma, inv_gm1, c_h;
  R inv4;   // 4 / (gamma - 1): the energy row of the scaled two-point fluxes
  R ch2;    // 2 c_h
};
template <typename R>
__host__ __device__ __forceinline__ PhysParams<R> make_phys(double gamma, double c_h) {
  return PhysParams<R>{R(gamma), R(1.0 / (gamma - 1.0)), R(c_h), R(4.0 / (gamma - 1.0)), R(2.0 * c_h)};
}

// a b + c with one rounding, where a sum of two products would leave the choice
// of the fused one to the compiler: every kernel that evaluates a flux then
// rounds it the same way
__device__ __forceinline__ double mad(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
// a product that is rounded by itself, never fused into a sum
__device__ __forceinline__ double mulr(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mulr(float a, float b) { return __fmul_rn(a, b); }

// ---------------------------------------------------------------------------
// Logarithmic mean L(a,b) = (a-b)/(ln a - ln b) and its inverse.
// For a ~ b both use polynomials in u = ((a-b)/(a+b))^2:
//   L = (a+b) / (2 F(u)),  F(u) = artanh(sqrt u) / sqrt u = 1 + u/3 + u^2/5 + ...
//   and 1/F(u) = 1 - u/3 - 4u^2/45 - ...
// FP64: degree 8 below u = 1/16 (least-maximum fits on [0, 1/16]; with the
// coefficients as written F is within 1.8e-17 and 1/F within 3.1e-18 in exact arithmetic, below a sixth
// of half an ulp), inside it the series in two FP32 parts below u = 2^-11 (unit_plus); above 1/16 the ratio a/b exceeds 1.66 and log(a/b) is
// well conditioned (at u = 1e-4 the quotient's rounding costs log(a/b) 1e-16 / 0.02).
// FP32: degree 3 below u = 0.05 (least-maximum fits on [0, 0.05]; F within 1.2e-8, 1/F
// within 3.7e-9, a fifth and an eighth of half an ulp); above it the ratio a/b exceeds 1.57.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double series_F(double u) {
  return 1.0 + u * (0.33333333333331369 + u * (0.20000000000836662 + u * (0.14285714148744664 + u * (0.11111122319976208
      + u * (0.090903954153249859 + u * (0.077060649643451390 + u * (0.064540716251361030 + u * 0.076102246025017837)))))));
}
__device__ __forceinline__ double series_invF(double u) {
  return 1.0 + u * (-0.33333333333332982 + u * (-0.088888888890384454 + u * (-0.046560846315972715 + u * (-0.030194023571221005
      + u * (-0.021795885119032539 + u * (-0.016812176252078610 + u * (-0.013121851935549912 + u * -0.014306111787604733)))))));
}
__device__ __forceinline__ float series_F(float u) {
  return 1.0f + u * (0.33333710f + u * (0.19962572f + u * 0.15462606f));
}
__device__ __forceinline__ float series_invF(float u) {
  return 1.0f + u * (-0.33333435f + u * (-0.088788078f + u * -0.049737233f));
}
__device__ __forceinline__ float series_invF4(float u) {   // 1/(4 F(u))
  return 0.25f + u * (-0.25f * 0.33333435f + u * (-0.25f * 0.088788078f + u * (-0.25f * 0.049737233f)));
}
template <typename R> struct LogMeanEps;
template <> struct LogMeanEps<double> { static constexpr double v = 0.0625; };
template <> struct LogMeanEps<float> { static constexpr float v = 0.05f; };

// FP64: the reciprocal unit's approximation r of 1/x (relative error about
// 2^-20) and one third-order Householder iteration, r (1 + e + e^2) with
// e = 1 - x r: three FP64 fused multiply-adds, error e^3 plus one rounding.  The
// unit takes subnormal operands and results for zero, so this holds for 2^-1022 <=
// |x| < 2^1022 (rcp_normal); fast_rcp scales the others into that range and back, and
// leaves zero and the infinities (e is NaN) to the unit.
// FP32: the MUFU reciprocal (rcp.approx, about 1 ulp), no slow-path branch.
__device__ __forceinline__ double rcp_unit(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ double rcp_normal(double x) {
  const double r = rcp_unit(x), e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ bool rcp_holds(double x) {
  return (((unsigned)__double2hiint(x) >> 20) & 0x7FFu) - 1u < 2044u;
}
__device__ __forceinline__ double rcp_scaled(double x) {
  const double sc = fabs(x) < 1.0 ? 1.2676506002282294e30 : 7.8886090522101181e-31;   // 2^100, 2^-100
  const double y = x * sc, r = rcp_unit(y), e = fma(-y, r, 1.0);
  return e == e ? fma(r, fma(e, e, e), r) * sc : r;
}
__device__ __forceinline__ double fast_rcp(double x) { return rcp_holds(x) ? rcp_normal(x) : rcp_scaled(x); }
__device__ __forceinline__ float fast_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double plain_log(double x) { return log(x); }
__device__ __forceinline__ float plain_log(float x) { return logf(x); }

template <typename R>
__device__ __forceinline__ R logmean(R a, R b) {
  R s = a + b, d = a - b;
  R rs = fast_rcp(s);
  R f = d * rs;
  R u = f * f;
  if (u < LogMeanEps<R>::v) return R(0.5) * s * series_invF(u);
  return d * fast_rcp(plain_log(a * fast_rcp(b)));
}

template <typename R>
__device__ __forceinline__ R inv_logmean(R a, R b) {
  R s = a + b, d = a - b;
  R rs = fast_rcp(s);
  R f = d * rs;
  R u = f * f;
  if (u < LogMeanEps<R>::v) return R(2) * series_F(u) * rs;
  return plain_log(a * fast_rcp(b)) * fast_rcp(d);
}

// Out of line so that the compiler cannot if-convert it into the common path
// (a predicated copy would be executed by every pair).
template <typename R>
__device__ __noinline__ void logmean_pair_general(R a1, R b1, R a2, R b2, R& H1, R& T2) {
  H1 = R(0.5) * logmean(a1, b1);
  T2 = R(0.5) * inv_logmean(a2, b2);
}

// Both logarithmic means of a pair in the scale the two-point fluxes take them
// (powers of two folded into the polynomials or the callers' coefficients):
// H1 = L(a1,b1) / 2 and T2 = 1 / (2 L(a2,b2)), and rs2 = 1/(a2 + b2).  One
// reciprocal, 1/(s1 s2), gives both 1/s1 and 1/s2, and one branch decides for
// both which form applies (the polynomials on resolved data; otherwise each
// takes its own branch above).
__device__ __forceinline__ void logmean_pair(float a1, float b1, float a2, float b2, float& H1, float& T2,
                                             float& rs2) {
  const float s1 = a1 + b1, d1 = a1 - b1, s2 = a2 + b2, d2 = a2 - b2;
  const float r = fast_rcp(s1 * s2);
  const float rs1 = s2 * r;
  rs2 = s1 * r;
  const float f1 = d1 * rs1, f2 = d2 * rs2;
  const float u1 = f1 * f1, u2 = f2 * f2;
  if (fmaxf(u1, u2) < LogMeanEps<float>::v) {
    H1 = s1 * series_invF4(u1);
    T2 = series_F(u2) * rs2;
  } else {
    logmean_pair_general(a1, b1, a2, b2, H1, T2);
  }
}

// u = (d/s)^2 as the sum of two FP32 values (relative error about 2^-45), from the
// bits of d and s: both are scaled by the power of two that takes s to [1, 2).
// False where that fails: |d| >= 2 |s| (or not finite), |s| below 2^-895, where the
// exponent of d = 0 would not be small beside that of s, or |s| beyond rcp_normal's range.
__device__ __forceinline__ bool ratio_squared(double d, double s, float& uh, float& ul) {
  const unsigned sH = (unsigned)__double2hiint(s), sL = (unsigned)__double2loint(s);
  const unsigned dH = (unsigned)__double2hiint(d), dL = (unsigned)__double2loint(d);
  const int es = (int)((sH >> 20) & 0x7FFu), k = (int)((dH >> 20) & 0x7FFu) - es;
  const float two46 = 1.4210854715202004e-14f;   // 2^-46
  // leading 24 bits, and the next 23 as a number (2^23 + bits, minus 2^23)
  const float sh = __uint_as_float(0x3F800000u | (__funnelshift_l(sL, sH, 3) & 0x7FFFFFu));
  const float sl = (__uint_as_float(0x4B000000u | ((sL >> 6) & 0x7FFFFFu)) - 8388608.0f) * two46;
  const float sc = __uint_as_float(k > -126 ? (unsigned)(127 + k) << 23 : 0u);
  const float dh = __uint_as_float(0x3F800000u | (__funnelshift_l(dL, dH, 3) & 0x7FFFFFu)) * sc;
  const float dl = (__uint_as_float(0x4B000000u | ((dL >> 6) & 0x7FFFFFu)) - 8388608.0f) * (two46 * sc);
  // quotient by the approximate reciprocal, its remainder divided twice
  const float r = fast_rcp(sh), q0 = dh * r;
  const float rem = __fmaf_rn(-q0, sh, dh) + __fmaf_rn(-q0, sl, dl);
  float q1 = rem * r;
  q1 = __fmaf_rn(__fmaf_rn(-q1, sh, rem), r, q1);
  uh = __fmul_rn(q0, q0);
  ul = __fmaf_rn(q0 + q0, q1, __fmaf_rn(q0, q0, -uh));
  return (unsigned)(es - 128) < 1917u && k <= 0;
}

// 1 + u (c1 + u (c2 + u (c3 + u (c4 + u c5)))) for 0 <= u < 2^-11 as a double,
// times the power of two whose high word is `unit`: the series beyond 1 in two
// FP32 parts (c1 and c2 too), whose sum is at most 2^-12.6 and right to 2^-57, then
// added to the bits of the unit as a fixed-point number -- in steps of 2^-52 above
// 1, of 2^-53 below (NEG: c1 < 0).  Rounding to integers by adding 1.5 2^23.
template <bool NEG>
__device__ __forceinline__ double unit_plus(float uh, float ul, float c1h, float c1l, float c2h, float c2l, float c3,
                                            float c4, float c5, unsigned unit) {
  const float t = uh * __fmaf_rn(uh, __fmaf_rn(uh, c5, c4), c3);
  const float mh = __fadd_rn(c2h, t), ml = __fadd_rn(t, -__fadd_rn(mh, -c2h)) + c2l;
  const float nh = __fmul_rn(uh, mh), nl = __fmaf_rn(uh, mh, -nh) + __fmaf_rn(uh, ml, ul * mh);
  const float oh = __fadd_rn(c1h, nh), ol = __fadd_rn(nh, -__fadd_rn(oh, -c1h)) + c1l + nl;
  const float ch = __fmul_rn(uh, oh), cl = __fmaf_rn(uh, oh, -ch) + __fmaf_rn(uh, ol, ul * oh);
  const float magic = 12582912.0f;   // 1.5 2^23
  // ch in steps of 2^-34 (at most 2^21.4 of them): the rest, below 2^-35, keeps its bits to 2^-59 when
  // cl joins it.  In steps of 2^-31 that sum was rounded at 2^-57, close to the final 2^-54.
  const float x = __fmaf_rn(ch, 17179869184.0f, magic);
  const float rem = __fmaf_rn(-__fadd_rn(x, -magic), 5.820766091346741e-11f, ch) + cl;
  const float y = __fmaf_rn(rem, NEG ? 9007199254740992.0f : 4503599627370496.0f, magic);
  const int ih = __float_as_int(x) - 0x4B400000, il = __float_as_int(y) - 0x4B400000;
  const long long i = (long long)ih * (1ll << (NEG ? 19 : 18)) + il + ((long long)unit << 32);
  return __longlong_as_double(i);
}

// the pairs beyond the two-part series: out of line, since most pairs of a
// resolved flow do not come here
static __device__ __noinline__ void logmean_pair_far(double a1, double b1, double a2, double b2, double rs2, double& H1,
                                                     double& T2) {
  const double s1 = a1 + b1;
  const double f1 = (a1 - b1) * fast_rcp(s1), f2 = (a2 - b2) * rs2;
  const double u1 = f1 * f1, u2 = f2 * f2;
  if (fmax(u1, u2) < LogMeanEps<double>::v) {
    H1 = s1 * (0.25 * series_invF(u1));
    T2 = series_F(u2) * rs2;
  } else {
    logmean_pair_general(a1, b1, a2, b2, H1, T2);
  }
}

// FP64.  The FP64 pipe bounds these kernels (a warp instruction occupies it for
// about 18 cycles, in which the SM can issue 70 others), so everything that is
// needed to less than 53 bits is done beside it: the two polynomials' part beyond
// 1 is a correction below 2^-12.6, two FP32 parts give it to 2^-57, and integer
// arithmetic adds it to 1.  Nine FP64 instructions a pair (four sums, a
// three-FMA reciprocal, two products) against 22 with the polynomials in FP64;
// the result's error is that of its one rounding, as there (against 113 bits, for
// u < 1e-4: root mean square 3.2e-17 for 1/F and 6.4e-17 for F, FP64 Horner 3.2e-17 and 6.4e-17;
// L 7.4e-17 either way, 1/L 1.04e-16 against 1.23e-16 with the reciprocal of a product).  Volume launch: 256^2, N = 3 1558 -> 1227
// us, 97x61 N = 5 1266 -> 951, 64-element 1D wave 64 -> 53, GLM-MHD 128^2 N = 4 3267 ->
// 2933.  Above 2^-11 (a/b > 1.045) the degree-8
// polynomials in FP64, above 1/16 the logarithms (a single FP64 series bound at
// 1e-4 with logarithms beyond cost 124 against 71 us per volume launch on the
// 64-element 1D wave and 2138 against 1846 us on the 256^2, N = 3 shear layer).
__device__ __forceinline__ void logmean_pair(double a1, double b1, double a2, double b2, double& H1, double& T2,
                                             double& rs2) {
  const double s1 = a1 + b1, d1 = a1 - b1, s2 = a2 + b2, d2 = a2 - b2;
  rs2 = rcp_normal(s2);
  float h1, l1, h2, l2;
  const bool ok1 = ratio_squared(d1, s1, h1, l1), ok2 = ratio_squared(d2, s2, h2, l2);
  if (ok1 && ok2 && fmaxf(h1, h2) < 4.8828125e-4f) {   // 2^-11
    // 1/F = 1 - u/3 - 4u^2/45 - 44u^3/945 - 428u^4/14175 - 10196u^5/467775, F = 1 + u/3 + u^2/5 + ...
    H1 = s1 * unit_plus<true>(h1, l1, -0.33333334f, 9.9341078e-9f, -0.088888891f, 2.1523899e-9f, -44.0f / 945.0f,
                              -428.0f / 14175.0f, -10196.0f / 467775.0f, 0x3FD00000u);
    T2 = rs2 * unit_plus<false>(h2, l2, 0.33333334f, -9.9341078e-9f, 0.2f, -2.9802323e-9f, 1.0f / 7.0f, 1.0f / 9.0f,
                                1.0f / 11.0f, 0x3FF00000u);
  } else {
    if (!rcp_holds(s2)) rs2 = rcp_scaled(s2);
    logmean_pair_far(a1, b1, a2, b2, rs2, H1, T2);
  }
}

// Exact float <-> double conversions with integer instructions only (the FP64
// pipe of this GPU is narrow and also executes the hardware conversions, and a
// predicated hardware fallback would still occupy it).  Values below the
// normal FP32 range become signed zero; overflow gives a signed infinity,
// NaN stays NaN.
__device__ __forceinline__ float d2f_int(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned e = (hi >> 20) & 0x7FFu;
  const unsigned sign = hi & 0x80000000u;
  const unsigned mant = ((hi & 0xFFFFFu) << 3) | (lo >> 29);
  const unsigned rest = lo & 0x1FFFFFFFu;
  unsigned bits = sign | ((e - 896u) << 23) | mant;
  bits += (rest > 0x10000000u) | ((rest == 0x10000000u) & (mant & 1u));   // round to nearest even
  const bool nan = e == 0x7FFu && ((hi & 0xFFFFFu) | lo) != 0u;
  bits = e < 897u ? sign : bits;
  bits = e > 1150u ? (sign | 0x7F800000u | (nan ? 0x400000u : 0u)) : bits;
  return __uint_as_float(bits);
}
__device__ __forceinline__ double f2d_int(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned e = (b >> 23) & 0xFFu;
  const unsigned ed = e == 255u ? 0x7FFu : e + 896u;
  unsigned hi = (b & 0x80000000u) | (ed << 20) | ((b & 0x7FFFFFu) >> 3);
  unsigned lo = b << 29;
  hi = e == 0u ? (b & 0x80000000u) : hi;
  lo = e == 0u ? 0u : lo;
  return __hiloint2double((int)hi, (int)lo);
}

// Double -> float rounded toward zero, for the FP32 physicality and wave-speed
// check of an updated state (a sign test and a maximum: the rounding
// direction does not matter there).  Values below the normal FP32 range give
// signed zero; values beyond it, infinities and NaNs give NaN, which fails the
// check.  About ten integer instructions against twenty-five for d2f_int.
__device__ __forceinline__ float d2f_rz(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned e = (hi >> 20) & 0x7FFu;
  const unsigned mant = __funnelshift_r(lo, hi, 29) & 0x7FFFFFu;
  const unsigned sign = hi & 0x80000000u;
  unsigned bits = sign | ((e - 896u) << 23) | mant;
  bits = e - 897u < 254u ? bits : (e < 897u ? sign : 0x7FC00000u);
  return __uint_as_float(bits);
}

// Reciprocal and square root of the CFL wave speeds: IEEE in FP64, the MUFU
// approximations (about 1 ulp) in FP32, where the result only enters the
// maximum that sets dt.
__device__ __forceinline__ double speed_rcp(double x) { return 1.0 / x; }
__device__ __forceinline__ float speed_rcp(float x) { return fast_rcp(x); }
__device__ __forceinline__ double speed_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float speed_sqrt(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// what the FP32 bound of the wave speeds needs of the mesh
struct MeshSpeeds {
  float gamma, gm1, c_h;   // gm1 = gamma - 1
  const float* inv_dx;
};

// Whether speed_bound's FP32 arithmetic held: density and its reciprocal, and every
// 1/dx, normal numbers; the energy so large that the squares lost below the
// normal range (1e-37) are within its error; the pressure above zero by more than
// its error; the square of the speed (a2) of a size whose own square, which GLM-MHD
// forms, is normal.  Too large a value makes up infinite or NaN.
template <int DIM>
__device__ __forceinline__ bool speed_range(float rho, float E, float p_low, float a2, float up, const MeshSpeeds& ms) {
  bool ok = rho > 1e-30f && rho < 1e30f && E > 1e-28f && p_low > 1e-25f && a2 > 1e-17f && up < 1e38f;
#pragma unroll
  for (int k = 0; k < DIM; ++k) ok = ok && ms.inv_dx[k] >= 1.17549435e-38f;
  return ok;
}

// ---------------------------------------------------------------------------
// Compressible Euler in DIM dimensions: u = (rho, rho v_1..rho v_DIM, E).
// Pair data q = (rho, v_1..v_DIM, p, aux); aux = rho/p for the EC flux,
// e = E/rho for the KEP and central fluxes.
// ---------------------------------------------------------------------------
template <int DIM_, int VOL_ = VOL_EC>
struct Euler {
  static constexpr int DIM = DIM_;
  static constexpr int VOL = VOL_;
  static constexpr int M = DIM_ + 2;
  static constexpr int P = DIM_ + 3;
  static constexpr bool NC = false;
  static constexpr bool NCS = false;   // stage-wise non-conservative flux (GLM-MHD only)
  static constexpr int IRHO = 0, IP = DIM_ + 1, IAUX = DIM_ + 2;

  // A product that becomes pair data.  1D: rounded by itself, since a thread that
  // holds a whole line would otherwise fuse it into the pairs' sums (v_a + v_b as
  // u_a (1/rho_a) + v_b), which the form with a lane per pair cannot: both
  // forms of the volume kernel take the same values.
  template <typename R>
  __device__ __forceinline__ static R value(R a, R b) {
    if constexpr (DIM == 1) return mulr(a, b);
    else return a * b;
  }

  template <typename R>
  __device__ __forceinline__ static void pair_data(const R* u, R* q, const PhysParams<R>& pp) {
    R rho = u[0];
    R E = u[DIM + 1];
    if constexpr (sizeof(R) == 8 && VOL == VOL_EC) {
      // one FP64 division for 1/rho and rho/p: p needs |m|^2 / rho, so
      // p rho = (gamma-1)(E rho - |m|^2/2) and 1/(rho p rho) gives both
      R mm = R(0);
#pragma unroll
      for (int k = 0; k < DIM; ++k) mm += u[1 + k] * u[1 + k];
      const R prho = (pp.gamma - R(1)) * (E * rho - R(0.5) * mm);   // p rho
      const R r = fast_rcp(prho * rho);
      const R ir = prho * r;                                         // 1 / rho
#pragma unroll
      for (int k = 0; k < DIM; ++k) q[1 + k] = value(u[1 + k], ir);
      q[0] = rho;
      q[IP] = value(prho, ir);
      q[IAUX] = value(rho * rho * rho, r);                                 // rho / p
      return;
    }
    R ir = fast_rcp(rho);
    R ke = R(0);
    q[0] = rho;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
      R v = value(u[1 + k], ir);
      q[1 + k] = v;
      ke += v * u[1 + k];
    }
    R p = value(pp.gamma - R(1), E - R(0.5) * ke);
    q[IP] = p;
    if constexpr (VOL == VOL_EC) q[IAUX] = value(rho, fast_rcp(p));
    else q[IAUX] = value(E, ir);
  }

  template <typename R>
  __device__ __forceinline__ static R total_energy(const R* q, const PhysParams<R>& pp) {
    if constexpr (VOL == VOL_EC) {
      R ke = R(0);
#pragma unroll
      for (int k = 0; k < DIM; ++k) ke += q[1 + k] * q[1 + k];
      return mad(q[IP], pp.inv_gm1, R(0.5) * q[0] * ke);
    }
    return value(q[0], q[IAUX]);
  }

  // conserved variables from pair data
  template <typename R>
  __device__ __forceinline__ static void cons_from_pair(const R* q, R* u, const PhysParams<R>& pp) {
    u[0] = q[0];
#pragma unroll
    for (int k = 0; k < DIM; ++k) u[1 + k] = q[0] * q[1 + k];
    u[DIM + 1] = total_energy(q, pp);
  }

  // physical flux in direction d from pair data
  template <typename R>
  __device__ __forceinline__ static void flux(int d, const R* q, R* f, const PhysParams<R>& pp) {
    R mflux = q[0] * q[1 + d];
    f[0] = mflux;
#pragma unroll
    for (int k = 0; k < DIM; ++k) f[1 + k] = mflux * q[1 + k] + (k == d ? q[IP] : R(0));
    f[DIM + 1] = q[1 + d] * (total_energy(q, pp) + q[IP]);
  }

  // Symmetric two-point flux f_S(q_a, q_b) in direction d, scaled so that sums
  // stand in for means: f_S,v = f[v] / 2 where half(v), else f[v]; the
  // differentiation coefficients, D_pq and 2 D_pq, carry the factor, so no
  // instruction multiplies by one half.  Kennedy-Gruber: every row halved,
  // with one addition more -- with two coefficients per pair the branch-free FP32
  // pair loops of degree 4 and 5 gave wrong results at optimisation levels above
  // 1 (CUDA 13.0; a constant state lost a fifth of its mass in a step, which the
  // per-variant tests caught).  The cause is not known: the EC flux takes two
  // coefficients in the same loops and its tests pass.
  __host__ __device__ static constexpr bool half(int v) { return VOL == VOL_KEP || v > 0; }
  template <typename R>
  __device__ __forceinline__ static void two_point(int d, const R* a, const R* b, R* f, const PhysParams<R>& pp) {
    static_assert(VOL != VOL_CENTRAL, "the central flux is differenced as sum_q D_pq f(q_q)");
    R vs[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) vs[k] = a[1 + k] + b[1 + k];
    const R ps = a[IP] + b[IP];
    if constexpr (VOL == VOL_EC) {
      // Ranocha: rho^ln {{v}}, momentum f_rho {{v}} + {{p}} n, energy with
      // 1/ln-mean(rho/p) and the product p_a v_b + p_b v_a
      R h, t, rs;
      logmean_pair(a[0], b[0], a[IAUX], b[IAUX], h, t, rs);
      const R f0 = h * vs[d];
      R w = pp.inv4 * t;
#pragma unroll
      for (int k = 0; k < DIM; ++k) w = mad(a[1 + k], b[1 + k], w);
      f[0] = f0;
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        if (k == d) f[1 + k] = mad(f0, vs[k], ps);
        else f[1 + k] = f0 * vs[k];
      }
      const R pv = a[IP] * b[1 + d];
      f[DIM + 1] = mad(f0, w, mad(b[IP], a[1 + d], pv));
    } else {
      // Kennedy-Gruber: arithmetic means of rho, v, p and e = E/rho
      const R rq = R(0.25) * (a[0] + b[0]);
      const R f0 = rq * vs[d];
      f[0] = f0 + f0;
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        if (k == d) f[1 + k] = mad(f0, vs[k], ps);
        else f[1 + k] = f0 * vs[k];
      }
      // 2 (rho e + p) v = (rq (e_a + e_b) + ps / 2) vs
      f[DIM + 1] = mad(rq, a[IAUX] + b[IAUX], R(0.5) * ps) * vs[d];
    }
  }

  template <typename R>
  __device__ __forceinline__ static R wave_speed(int d, const R* q, const PhysParams<R>& pp) {
    return fabs(q[1 + d]) + sqrt(pp.gamma * q[IP] / q[0]);
  }

  // g^d(u) for the non-conservative product: none for Euler
  template <typename R>
  __device__ __forceinline__ static void ncg(int, const R*, R*) {}
  template <typename R>
  __device__ __forceinline__ static void nc_apply(int, const R*, const R*, R*) {}

  // An upper bound of sum_d lambda_d / dx_d from the FP32 truncation of a state;
  // returns whether the state is certainly physical (else the bound says
  // nothing).  With e = 2^-23: the inputs, the reciprocal and the roundings leave
  // |p - p_32| < 16 e (gamma - 1)(E + |m|^2/(2 rho)) and every other factor
  // within a few e; the bound takes p at its upper end and 32 e on the sum.
  // That holds while no part leaves the normal FP32 range by an amount that
  // matters (speed_range): the kinetic energy is formed as m (m / rho), whose lost
  // parts stay below 1e-37 against E > 1e-28, never from bare squares.
  __device__ __forceinline__ static bool speed_bound(const float* u, const MeshSpeeds& ms, float& up) {
    const float e16 = 16.0f / 8388608.0f;
    const float rho = u[0], Et = u[DIM + 1], ir = fast_rcp(rho);
    float ke = 0.0f;
#pragma unroll
    for (int k = 0; k < DIM; ++k) ke += u[1 + k] * (u[1 + k] * ir);
    const float kr = 0.5f * ke, gm1 = ms.gm1;
    const float p = gm1 * (Et - kr), dp = e16 * gm1 * (Et + kr);
    const float c2 = ms.gamma * (p + dp) * ir, c = speed_sqrt(c2);
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < DIM; ++k) s += (fabsf(u[1 + k]) * ir + c) * ms.inv_dx[k];
    up = s * (1.0f + 2.0f * e16);
    return speed_range<DIM>(rho, Et, p - dp, c2, up, ms);
  }

  // physicality of a conserved state (rho > 0, p > 0, finite) and sum_d lambda_d / dx_d
  template <typename T>
  __device__ __forceinline__ static bool physical(const T* u, T gamma, T& lam_sum, const T* inv_dx) {
    T rho = u[0];
    T ke = T(0);
#pragma unroll
    for (int k = 0; k < DIM; ++k) ke += u[1 + k] * u[1 + k];
    T ir = speed_rcp(rho);
    T p = (gamma - T(1)) * (u[DIM + 1] - T(0.5) * ke * ir);
    T c = speed_sqrt(gamma * p * ir);
    T s = T(0);
#pragma unroll
    for (int k = 0; k < DIM; ++k) s += (fabs(u[1 + k] * ir) + c) * inv_dx[k];
    lam_sum = s;
    return rho > T(0) && p > T(0) && isfinite(s);
  }
};

// ---------------------------------------------------------------------------
// Ideal GLM-MHD (2D): u = (rho, rho v1..3, E, B1..3, psi),
// E = p/(gamma-1) + rho|v|^2/2 + |B|^2/2 + psi^2/2.
// Non-conservative term along d: phi_Powell(u) dB_d/dx_d + phi_GLM^d(u) dpsi/dx_d,
// phi_Powell = (0, B, v.B, v, 0), phi_GLM^d = (0, 0,0,0, v_d psi, 0,0,0, v_d),
// so g^d(u) = (B_d, psi).
// Pair data q = (rho, v1, v2, v3, p, B1, B2, B3, psi, beta = rho/(2p), |v|^2, |B|^2, v.B).
// ---------------------------------------------------------------------------
template <int VOL_ = VOL_EC>
struct GlmMhd {
  static constexpr int DIM = 2;
  static constexpr int VOL = VOL_;
  static constexpr int M = 9;
  static constexpr int P = 13;
  static constexpr bool NC = true;
  static constexpr bool NCS = false;
  static constexpr int IRHO = 0, IP = 4, IB = 5, IPSI = 8, IBETA = 9, IV2 = 10, IB2 = 11, IVB = 12;

  template <typename R>
  __device__ __forceinline__ static void pair_data(const R* u, R* q, const PhysParams<R>& pp) {
    R rho = u[0];
    R B1 = u[5], B2 = u[6], B3 = u[7], psi = u[8];
    R BB = B1 * B1 + B2 * B2 + B3 * B3;
    R ir, p, irp;   // 1/rho, p, rho/p
    if constexpr (sizeof(R) == 8) {
      // one FP64 division: p rho = (gamma-1)(rho (E - |B|^2/2 - psi^2/2) - |m|^2/2)
      const R mm = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
      const R prho = (pp.gamma - R(1)) * (rho * (u[4] - R(0.5) * BB - R(0.5) * psi * psi) - R(0.5) * mm);
      const R r = fast_rcp(prho * rho);
      ir = prho * r;
      p = prho * ir;
      irp = rho * rho * rho * r;
    } else {
      ir = fast_rcp(rho);
      const R w1 = u[1] * ir, w2 = u[2] * ir, w3 = u[3] * ir;
      const R vv0 = w1 * w1 + w2 * w2 + w3 * w3;
      p = (pp.gamma - R(1)) * (u[4] - R(0.5) * rho * vv0 - R(0.5) * BB - R(0.5) * psi * psi);
      irp = rho * fast_rcp(p);
    }
    R v1 = u[1] * ir, v2 = u[2] * ir, v3 = u[3] * ir;
    R vv = v1 * v1 + v2 * v2 + v3 * v3;
    q[0] = rho; q[1] = v1; q[2] = v2; q[3] = v3; q[4] = p;
    q[5] = B1; q[6] = B2; q[7] = B3; q[8] = psi;
    q[IBETA] = R(0.5) * irp;
    q[IV2] = vv; q[IB2] = BB; q[IVB] = v1 * B1 + v2 * B2 + v3 * B3;
  }

  // conserved variables from pair data
  template <typename R>
  __device__ __forceinline__ static void cons_from_pair(const R* q, R* u, const PhysParams<R>& pp) {
    const R rho = q[0];
    u[0] = rho;
    u[1] = rho * q[1]; u[2] = rho * q[2]; u[3] = rho * q[3];
    u[4] = q[IP] * pp.inv_gm1 + R(0.5) * (rho * q[IV2] + q[IB2] + q[IPSI] * q[IPSI]);
    u[5] = q[5]; u[6] = q[6]; u[7] = q[7]; u[8] = q[8];
  }

  template <typename R>
  __device__ __forceinline__ static void flux(int d, const R* q, R* f, const PhysParams<R>& pp) {
    R rho = q[0], p = q[IP], psi = q[IPSI];
    R vd = q[1 + d], Bd = q[IB + d];
    R mflux = rho * vd;
    f[0] = mflux;
#pragma unroll
    for (int k = 0; k < 3; ++k) f[1 + k] = mflux * q[1 + k] - Bd * q[IB + k] + (k == d ? p + R(0.5) * q[IB2] : R(0));
    f[4] = vd * (R(0.5) * rho * q[IV2] + pp.gamma * pp.inv_gm1 * p + q[IB2]) - Bd * q[IVB] + pp.c_h * psi * Bd;
#pragma unroll
    for (int k = 0; k < 3; ++k) f[5 + k] = (k == d) ? pp.c_h * psi : vd * q[IB + k] - q[1 + k] * Bd;
    f[8] = pp.c_h * Bd;
  }

  // entropy-conservative flux: satisfies [[w]].f = [[psi_d]] + {{theta}} [[B_d]]
  // with theta = w.phi_Powell = rho (v.B)/p (derived from the entropy
  // variables of S = -rho s/(gamma-1)).  Scaled so that sums stand in for
  // means: f_S = f / 4 in every row, so the coefficient of the pair is D_pq / 2.
  __host__ __device__ static constexpr bool half(int) { return false; }
  template <typename R>
  __device__ __forceinline__ static void two_point(int d, const R* a, const R* b, R* f, const PhysParams<R>& pp) {
    static_assert(VOL == VOL_EC, "the central flux is differenced as sum_q D_pq f(q_q)");
    R v[3], B[3];   // sums of both nodes
#pragma unroll
    for (int k = 0; k < 3; ++k) { v[k] = a[1 + k] + b[1 + k]; B[k] = a[IB + k] + b[IB + k]; }
    const R psi = a[IPSI] + b[IPSI];
    R h, t, rs2;
    logmean_pair(a[0], b[0], a[IBETA], b[IBETA], h, t, rs2);
    const R Bd = B[d];
    const R f0 = h * v[d];              // rho^ln {{v_d}}
    const R g0 = f0 + f0;
    f[0] = g0 + g0;
    // 4 (p~ + {{|B|^2}}/2), p~ = {{rho}} / (2 {{beta}})
    const R rs = a[0] + b[0];
    const R pt = mad(rs + rs, rs2, a[IB2] + b[IB2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const R m = k == d ? mad(g0, v[k], pt) : R(g0 * v[k]);
      f[1 + k] = mad(-Bd, B[k], m);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (k == d) f[5 + k] = pp.ch2 * psi;
      else f[5 + k] = mad(v[d], B[k], R(-(v[k] * Bd)));
    }
    f[8] = pp.ch2 * Bd;
    // 8 f_E = e + 2 z
    R z = Bd * (a[IVB] + b[IVB]);
    z = mad(-a[1 + d], a[IB2], z);
    z = mad(-b[1 + d], b[IB2], z);
    const R pb = a[IPSI] * a[IB + d];
    z = mad(-pp.ch2, mad(b[IPSI], b[IB + d], pb), z);
    R e = g0 * mad(pp.inv4, t, -(a[IV2] + b[IV2]));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      e = mad(f[1 + k], v[k], e);
      e = mad(f[5 + k], B[k], e);
    }
    f[4] = mad(R(0.5), mad(f[8], psi, e), z);
  }

  // |v_d| + max(c_f, c_h): the GLM pair travels at v_d -+ c_h
  template <typename R>
  __device__ __forceinline__ static R wave_speed(int d, const R* q, const PhysParams<R>& pp) {
    R ir = R(1) / q[0];
    R a2 = pp.gamma * q[IP] * ir;
    R b2 = q[IB2] * ir;
    R bd2 = q[IB + d] * q[IB + d] * ir;
    R s = a2 + b2;
    R cf = sqrt(R(0.5) * (s + sqrt(fmax(s * s - R(4) * a2 * bd2, R(0)))));
    return fabs(q[1 + d]) + fmax(cf, pp.c_h);
  }

  // g^d(u) = (B_d, psi)
  template <typename R>
  __device__ __forceinline__ static void ncg(int d, const R* q, R* g) { g[0] = q[IB + d]; g[1] = q[IPSI]; }

  // out += phi_Powell(q) g0 + phi_GLM^d(q) g1
  template <typename R>
  __device__ __forceinline__ static void nc_apply(int d, const R* q, const R* g, R* out) {
    R g0 = g[0], g1 = g[1];
    out[1] += q[IB + 0] * g0;
    out[2] += q[IB + 1] * g0;
    out[3] += q[IB + 2] * g0;
    out[4] += q[IVB] * g0 + q[1 + d] * q[IPSI] * g1;
    out[5] += q[1] * g0;
    out[6] += q[2] * g0;
    out[7] += q[3] * g0;
    out[8] += q[1 + d] * g1;
  }

  // as Euler's speed_bound; the root's argument takes 32 e of s^2 on top
  __device__ __forceinline__ static bool speed_bound(const float* u, const MeshSpeeds& ms, float& up) {
    const float e16 = 16.0f / 8388608.0f;
    const float rho = u[0], ir = fast_rcp(rho), gm1 = ms.gm1;
    const float BB = u[5] * u[5] + u[6] * u[6] + u[7] * u[7];
    const float q = 0.5f * (u[1] * (u[1] * ir) + u[2] * (u[2] * ir) + u[3] * (u[3] * ir) + BB + u[8] * u[8]);
    const float p = gm1 * (u[4] - q), dp = e16 * gm1 * (u[4] + q);
    const float a2 = ms.gamma * (p + dp) * ir, s = (a2 + BB * ir) * (1.0f + e16);
    float tot = 0.0f;
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      const float bd2 = u[5 + d] * u[5 + d] * ir * (1.0f - e16);
      const float arg = fmaxf(s * s * (1.0f + 2.0f * e16) - 4.0f * ms.gamma * fmaxf(p - dp, 0.0f) * ir * bd2, 0.0f);
      const float cf = speed_sqrt(0.5f * (s + speed_sqrt(arg) * (1.0f + e16)));
      tot += (fabsf(u[1 + d]) * ir + fmaxf(cf, ms.c_h)) * ms.inv_dx[d];
    }
    up = tot * (1.0f + 2.0f * e16);
    return speed_range<2>(rho, u[4], p - dp, a2, up, ms);
  }

  template <typename T>
  __device__ __forceinline__ static bool physical(const T* u, T gamma, T c_h, T& lam_sum, const T* inv_dx) {
    T rho = u[0];
    T ir = speed_rcp(rho);
    T v1 = u[1] * ir, v2 = u[2] * ir, v3 = u[3] * ir;
    T BB = u[5] * u[5] + u[6] * u[6] + u[7] * u[7];
    T p = (gamma - T(1)) * (u[4] - T(0.5) * rho * (v1 * v1 + v2 * v2 + v3 * v3) - T(0.5) * BB - T(0.5) * u[8] * u[8]);
    T a2 = gamma * p * ir, b2 = BB * ir, s = a2 + b2;
    T vv[2] = {v1, v2};
    T tot = T(0);
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      T bd2 = u[5 + d] * u[5 + d] * ir;
      T cf = speed_sqrt(T(0.5) * (s + speed_sqrt(fmax(s * s - T(4) * a2 * bd2, T(0)))));
      tot += (fabs(vv[d]) + fmax(cf, c_h)) * inv_dx[d];
    }
    lam_sum = tot;
    return rho > T(0) && p > T(0) && isfinite(tot);
  }
};

// GLM-MHD with the stage-wise non-conservative numerical flux of eq.
// bad.numflux.non.cons: sum_j b_j B(u^{(j),+-}) g^avg(u^(j)).  B(u) and g(u)
// depend on u through v, B and psi only, so each stage leaves these seven
// values of both face traces for the face kernel (stage_prims), which applies
// B(own) to the averaged g of both sides (nc_apply_prims).
template <int VOL_ = VOL_EC>
struct GlmMhdStages : GlmMhd<VOL_> {
  using Base = GlmMhd<VOL_>;
  static constexpr bool NCS = true;
  static constexpr int NPRIM = 7;   // v1, v2, v3, B1, B2, B3, psi
  template <typename R>
  __device__ __forceinline__ static void stage_prims(const R* q, R* o) {
    o[0] = q[1]; o[1] = q[2]; o[2] = q[3];
    o[3] = q[Base::IB]; o[4] = q[Base::IB + 1]; o[5] = q[Base::IB + 2]; o[6] = q[Base::IPSI];
  }
  // g^d of a primitive record: (B_d, psi)
  template <typename R>
  __device__ __forceinline__ static void ncg_prims(int d, const R* w, R* g) { g[0] = w[3 + d]; g[1] = w[6]; }
  // out += phi_Powell(w) g0 + phi_GLM^d(w) g1 (as nc_apply, from the primitives)
  template <typename R>
  __device__ __forceinline__ static void nc_apply_prims(int d, const R* w, const R* g, R* out) {
    const R g0 = g[0], g1 = g[1];
    out[1] += w[3] * g0;
    out[2] += w[4] * g0;
    out[3] += w[5] * g0;
    out[4] += (w[0] * w[3] + w[1] * w[4] + w[2] * w[5]) * g0 + w[d] * w[6] * g1;
    out[5] += w[0] * g0;
    out[6] += w[1] * g0;
    out[7] += w[2] * g0;
    out[8] += w[d] * g1;
  }
};

// ---------------------------------------------------------------------------
// Butcher tableaux per degree N (explicit RK of order N+1), as constexpr
// functions so that fully unrolled stage loops fold zero coefficients.
//  N=1 Heun RK2, N=2 Heun RK3, N=3 classical RK4, N=4 Butcher's 6-stage
//  order 5, N=5 Butcher's 7-stage order 6.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int rk_stages(int N) { return N == 1 ? 2 : N == 2 ? 3 : N == 3 ? 4 : N == 4 ? 6 : 7; }

__host__ __device__ constexpr double rk_a(int N, int i, int j) {
  // i, j zero-based stage indices, a_ij for j < i
  return N == 1 ? (i == 1 && j == 0 ? 1.0 : 0.0)
       : N == 2 ? ((i == 1 && j == 0) ? 1.0 / 3.0 : (i == 2 && j == 1) ? 2.0 / 3.0 : 0.0)
       : N == 3 ? ((i == 1 && j == 0) ? 0.5 : (i == 2 && j == 1) ? 0.5 : (i == 3 && j == 2) ? 1.0 : 0.0)
       : N == 4 ? (i == 1 ? (j == 0 ? 0.25 : 0.0)
                 : i == 2 ? (j == 0 ? 0.125 : j == 1 ? 0.125 : 0.0)
                 : i == 3 ? (j == 1 ? -0.5 : j == 2 ? 1.0 : 0.0)
                 : i == 4 ? (j == 0 ? 3.0 / 16.0 : j == 3 ? 9.0 / 16.0 : 0.0)
                 : i == 5 ? (j == 0 ? -3.0 / 7.0 : j == 1 ? 2.0 / 7.0 : j == 2 ? 12.0 / 7.0 : j == 3 ? -12.0 / 7.0 : j == 4 ? 8.0 / 7.0 : 0.0)
                 : 0.0)
       : (i == 1 ? (j == 0 ? 1.0 / 3.0 : 0.0)
        : i == 2 ? (j == 1 ? 2.0 / 3.0 : 0.0)
        : i == 3 ? (j == 0 ? 1.0 / 12.0 : j == 1 ? 1.0 / 3.0 : j == 2 ? -1.0 / 12.0 : 0.0)
        : i == 4 ? (j == 0 ? -1.0 / 16.0 : j == 1 ? 9.0 / 8.0 : j == 2 ? -3.0 / 16.0 : j == 3 ? -3.0 / 8.0 : 0.0)
        : i == 5 ? (j == 1 ? 9.0 / 8.0 : j == 2 ? -3.0 / 8.0 : j == 3 ? -3.0 / 4.0 : j == 4 ? 0.5 : 0.0)
        : i == 6 ? (j == 0 ? 9.0 / 44.0 : j == 1 ? -9.0 / 11.0 : j == 2 ? 63.0 / 44.0 : j == 3 ? 18.0 / 11.0 : j == 5 ? -16.0 / 11.0 : 0.0)
        : 0.0);
}

__host__ __device__ constexpr double rk_b(int N, int i) {
  return N == 1 ? 0.5
       : N == 2 ? (i == 0 ? 0.25 : i == 1 ? 0.0 : 0.75)
       : N == 3 ? (i == 0 || i == 3 ? 1.0 / 6.0 : 1.0 / 3.0)
       : N == 4 ? (i == 0 || i == 5 ? 7.0 / 90.0 : i == 1 ? 0.0 : i == 2 || i == 4 ? 32.0 / 90.0 : 12.0 / 90.0)
       : (i == 0 || i == 6 ? 11.0 / 120.0 : i == 1 ? 0.0 : i == 2 || i == 3 ? 27.0 / 40.0 : -4.0 / 15.0);
}

// true if R_j is needed by a later stage's combination
__host__ __device__ constexpr bool rk_needed_later(int N, int j) {
  bool need = false;
  for (int i = j + 1; i < rk_stages(N); ++i) need = need || (rk_a(N, i, j) != 0.0);
  return need;
}

}  // namespace crk
