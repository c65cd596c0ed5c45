// twofloat.cuh -- arithmetic on unevaluated sums of two floats (F2: about 48
// significant bits) and three floats (F3: about 72).
//
// Why: on GB300 the FP64 pipe issues one warp instruction in 16 cycles per SM
// and the FP32 pipes 64 in the same time.  An F2 sum or product is 7 to 12
// FP32 operations, so a right-hand side in F2 runs about an order of magnitude
// faster than in FP64, at a rounding error of a few 2^-47 per operation.  The
// ray tracer's steps carry a truncation error of rtol >= 1e-10 where this
// arithmetic is used (split_allowed), four orders of magnitude above that.
//
// The error-free transformations are the classical ones: the sums of Knuth
// and Dekker (Dekker, Numer. Math. 18, 1971), products by the fused
// multiply-add, double-word sums and products as analysed by Joldes, Muller &
// Popescu (ACM TOMS 44, 2017).  Every operation is an explicit
// round-to-nearest intrinsic, so nothing is contracted or reordered.  The
// functions also compile for the host, where the tests run them.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

namespace bhrt {

#define BH_HD __host__ __device__ __forceinline__
// out of line on the device: long and called from several places
#define BH_NI static __host__ __device__ __noinline__

#ifdef __CUDA_ARCH__
BH_HD float f_add(float a, float b) { return __fadd_rn(a, b); }
BH_HD float f_sub(float a, float b) { return __fsub_rn(a, b); }
BH_HD float f_mul(float a, float b) { return __fmul_rn(a, b); }
BH_HD float f_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
BH_HD float f_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
BH_HD int f_bits(float x) { return __float_as_int(x); }
BH_HD float bits_f(int x) { return __int_as_float(x); }
#else
BH_HD float f_add(float a, float b) { return a + b; }
BH_HD float f_sub(float a, float b) { return a - b; }
BH_HD float f_mul(float a, float b) { return a * b; }
BH_HD float f_fma(float a, float b, float c) { return std::fmaf(a, b, c); }
BH_HD float f_rcp(float x) { return 1.0f / x; }
BH_HD int f_bits(float x) {
  int i;
  std::memcpy(&i, &x, 4);
  return i;
}
BH_HD float bits_f(int i) {
  float x;
  std::memcpy(&x, &i, 4);
  return x;
}
#endif

struct F2 {
  float h, l;
};
struct F3 {
  float a, b, c;
};

BH_HD F2 mk2(float h, float l) {
  F2 r;
  r.h = h;
  r.l = l;
  return r;
}
BH_HD F2 neg(F2 x) { return mk2(-x.h, -x.l); }
// exact powers of two
BH_HD F2 twice(F2 x) { return mk2(f_add(x.h, x.h), f_add(x.l, x.l)); }
BH_HD F2 scale(F2 x, float p) { return mk2(f_mul(x.h, p), f_mul(x.l, p)); }

// a + b exactly as s + e: any order (6 operations), |a| >= |b| (3).
BH_HD F2 two_sum(float a, float b) {
  const float s = f_add(a, b), bb = f_sub(s, a);
  return mk2(s, f_add(f_sub(a, f_sub(s, bb)), f_sub(b, bb)));
}
BH_HD F2 quick_sum(float a, float b) {
  const float s = f_add(a, b);
  return mk2(s, f_sub(b, f_sub(s, a)));
}
BH_HD F2 two_prod(float a, float b) {
  const float p = f_mul(a, b);
  return mk2(p, f_fma(a, b, -p));
}

// Sums and products: absolute error of a sum within 2^-46 (|x| + |y|),
// relative error of a product within 2^-45.
BH_HD F2 add(F2 x, F2 y) {
  const F2 s = two_sum(x.h, y.h);
  return quick_sum(s.h, f_add(s.l, f_add(x.l, y.l)));
}
BH_HD F2 sub(F2 x, F2 y) {
  const F2 s = two_sum(x.h, -y.h);
  return quick_sum(s.h, f_add(s.l, f_sub(x.l, y.l)));
}
BH_HD F2 addf(F2 x, float y) {
  const F2 s = two_sum(x.h, y);
  return quick_sum(s.h, f_add(s.l, x.l));
}
// the product without the last renormalisation (|l| a few ulps of h): for
// operands of further sums
BH_HD F2 mul_raw(F2 x, F2 y) {
  const float p = f_mul(x.h, y.h);
  float e = f_fma(x.h, y.h, -p);
  e = f_fma(x.h, y.l, e);
  return mk2(p, f_fma(x.l, y.h, e));
}
BH_HD F2 mul(F2 x, F2 y) {
  const F2 p = mul_raw(x, y);
  return quick_sum(p.h, p.l);
}
BH_HD F2 sqr_raw(F2 x) {
  const float p = f_mul(x.h, x.h);
  return mk2(p, f_fma(f_add(x.h, x.h), x.l, f_fma(x.h, x.h, -p)));
}
BH_HD F2 sqr(F2 x) {
  const F2 p = sqr_raw(x);
  return quick_sum(p.h, p.l);
}
// float times F2, raw
BH_HD F2 mulf_raw(float x, F2 y) {
  const float p = f_mul(x, y.h);
  return mk2(p, f_fma(x, y.l, f_fma(x, y.h, -p)));
}
// c + x y
BH_HD F2 fma2(F2 x, F2 y, F2 c) { return add(c, mul_raw(x, y)); }
// a Horner step c + z t where |c| >= |z t|, left unnormalised
BH_HD F2 horner2(F2 z, F2 t, F2 c) {
  const F2 p = mul_raw(z, t);
  const F2 s = quick_sum(c.h, p.h);
  return mk2(s.h, f_add(s.l, f_add(c.l, p.l)));
}
// 1 / x: the approximate reciprocal r, its residual e = 1 - x r exact to
// 2^-47, and r (1 + e + e^2).
BH_HD F2 rcp2(F2 x) {
  const float r = f_rcp(x.h);
  float e = f_fma(-x.h, r, 1.0f);
  e = f_fma(-x.l, r, e);
  return quick_sum(r, f_mul(r, f_fma(e, e, e)));
}

// sqrt(x) for x > 0: the approximate reciprocal square root r, s = x r, and
// one correction by the residual x - s^2.
BH_HD F2 sqrt2(F2 x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x.h));
#else
  const float r = 1.0f / std::sqrt(x.h);
#endif
  const float s = f_mul(x.h, r);
  // one Newton step in float brings s to its last bit, the residual the rest
  const float s1 = f_fma(f_mul(0.5f, r), f_fma(-s, s, x.h), s);
  const float e = f_add(f_fma(-s1, s1, x.h), x.l);
  return quick_sum(s1, f_mul(f_mul(0.5f, r), e));
}

__host__ __device__ inline F2 f2_of(double x) {
  const float h = (float)x;
  return mk2(h, (float)(x - (double)h));
}
__host__ __device__ inline double f64_of(F2 x) { return (double)x.h + (double)x.l; }
__host__ __device__ inline F3 f3_of(double x) {
  F3 r;
  r.a = (float)x;
  const double y = x - (double)r.a;
  r.b = (float)y;
  r.c = (float)(y - (double)r.b);
  return r;
}
__host__ __device__ inline double f64_of(F3 x) { return (double)x.a + ((double)x.b + (double)x.c); }
BH_HD F2 f2_of(F3 x) { return mk2(x.a, x.b); }

// y + d for a state component: the state keeps about 72 bits, so that the
// sum over a ray's steps rounds less than a double's would.
BH_HD F3 add3(F3 y, F2 d) {
  const F2 s = two_sum(y.a, d.h), t = two_sum(y.b, d.l), u = two_sum(t.h, s.l);
  const float w = f_add(y.c, f_add(t.l, u.l));
  const F2 p = quick_sum(s.h, u.h), q = quick_sum(p.l, w);
  F3 r;
  r.a = p.h;
  r.b = q.h;
  r.c = q.l;
  return r;
}

// Tables of the exponential and the logarithm (gen_split_tables.py): 2^(j/64)
// as F2, and per bin of the leading six fraction bits of m in [1, 2) a factor
// r_j near 1/m with -log r_j as F2.
#define BH_EXP64 \
  1.0f, 0.0f, 1.01088929f, -5.71160541e-09f, 1.0218972f, -4.81155986e-08f, \
  1.03302491f, -2.80908932e-08f, 1.04427373f, 4.83347016e-08f, 1.05564523f, -4.90716943e-08f, \
  1.06714046f, -5.93375198e-08f, 1.07876074f, 5.46159455e-08f, 1.09050775f, -1.30775399e-08f, \
  1.10238254f, 4.260502e-08f, 1.1143868f, -5.43554002e-08f, 1.12652159f, 3.12364143e-08f, \
  1.13878858f, 5.38622231e-08f, 1.15118921f, 2.19222827e-08f, 1.1637249f, -4.05144149e-08f, \
  1.17639697f, 2.56697508e-08f, 1.18920708f, 3.79763527e-08f, 1.20215678f, -5.06975653e-08f, \
  1.21524739f, -3.26739489e-08f, 1.22848058f, -4.13620036e-08f, 1.24185777f, 4.4968381e-08f, \
  1.25538075f, 7.32223748e-09f, 1.26905096f, 1.41933332e-09f, 1.28287005f, -3.81662169e-08f, \
  1.29683959f, -4.01899953e-08f, 1.31096125f, -3.49657157e-08f, 1.32523668f, -3.49637332e-08f, \
  1.33966756f, -3.46167397e-08f, 1.35425556f, -1.01233493e-08f, 1.36900246f, -3.84588184e-08f, \
  1.38390994f, -5.87557736e-08f, 1.39897966f, 8.68943406e-09f, 1.41421354f, 2.4203235e-08f, \
  1.42961335f, -1.34299292e-08f, 1.44518077f, 3.32419994e-08f, 1.46091783f, -3.62865755e-08f, \
  1.47682619f, -4.50089885e-08f, 1.49290776f, -3.42362014e-08f, 1.50916445f, -2.49593732e-08f, \
  1.52559817f, -1.76285688e-08f, 1.54221082f, 8.07090483e-09f, 1.55900443f, -2.57646651e-08f, \
  1.5759809f, -5.66102543e-08f, 1.59314215f, -4.90313679e-10f, 1.61049032f, 9.83621717e-09f, \
  1.62802744f, -1.72600831e-08f, 1.64575553f, -5.12497209e-08f, 1.66367662f, -3.92029875e-08f, \
  1.68179286f, -2.47553267e-08f, 1.70010638f, -2.86514723e-08f, 1.71861935f, -4.8496176e-08f, \
  1.73733389f, -5.85022342e-08f, 1.75625217f, -9.23577037e-09f, 1.77537644f, 5.34319788e-08f, \
  1.79470909f, -1.14150449e-08f, 1.81425214f, 3.73625824e-08f, 1.8340081f, -1.1239278e-08f, \
  1.85397911f, 1.43656118e-08f, 1.87416768f, -4.66300563e-08f, 1.89457595f, 2.81033845e-08f, \
  1.91520655f, 9.84532811e-09f, 1.93606174f, 5.3570723e-08f, 1.95714414f, -1.70218044e-08f, \
  1.97845602f, 6.03272632e-09f
#define BH_LOG64 \
  1.0f, 0.0f, 0.0f, 0.977050781f, 0.0232166518f, -1.7692614e-10f, \
  0.962402344f, 0.0383226797f, -6.9178907e-10f, 0.948242188f, 0.0531453378f, -5.41727219e-10f, \
  0.934326172f, 0.0679296777f, 3.6284078e-09f, 0.920898438f, 0.0824055225f, 5.00289754e-10f, \
  0.907714844f, 0.0968249962f, 2.26457253e-09f, 0.895019531f, 0.110909738f, 6.7311362e-10f, \
  0.8828125f, 0.124642447f, -1.42987699e-09f, 0.870849609f, 0.13828598f, 1.7318893e-09f, \
  0.859130859f, 0.151834026f, 3.41871642e-09f, 0.84765625f, 0.165280089f, 2.15679252e-09f, \
  0.836669922f, 0.178325638f, 6.66972433e-09f, 0.825927734f, 0.191248f, -1.72948611e-09f, \
  0.815185547f, 0.204339534f, -7.26857641e-09f, 0.804931641f, 0.216997921f, 2.18078533e-09f, \
  0.794921875f, 0.22951144f, -2.03349657e-10f, 0.78515625f, 0.241872534f, 2.26464114e-09f, \
  0.775878906f, 0.253758818f, 1.71153436e-09f, 0.766357422f, 0.266106606f, 4.34760494e-09f, \
  0.757324219f, 0.277963817f, 5.86326099e-09f, 0.748535156f, 0.289637119f, -1.12903731e-08f, \
  0.739990234f, 0.301118284f, 5.1976583e-09f, 0.731445312f, 0.312732816f, 6.33974073e-09f, \
  0.723144531f, 0.324146181f, -9.45338652e-09f, 0.715087891f, 0.335349828f, -8.11322654e-09f, \
  0.707275391f, 0.346335173f, -3.70320485e-09f, 0.699462891f, 0.357442528f, 9.56108881e-09f, \
  0.691894531f, 0.368321747f, -1.19035323e-10f, 0.684570312f, 0.378963917f, 1.07104281e-09f, \
  0.677246094f, 0.389720559f, 6.7243886e-09f, 0.670166016f, 0.400229812f, 1.10731668e-09f, \
  0.663330078f, 0.410482556f, 1.66517311e-09f, 0.656494141f, 0.420841515f, -4.61376048e-09f, \
  0.649658203f, 0.431308895f, 3.92151978e-10f, 0.643310547f, 0.441127717f, -1.17510837e-08f, \
  0.63671875f, 0.451427251f, -7.4277402e-09f, 0.630615234f, 0.461059362f, 1.19272601e-08f, \
  0.624511719f, 0.470785171f, 1.37870222e-08f, 0.618408203f, 0.480606526f, -9.4187298e-09f, \
  0.612548828f, 0.49012661f, 1.0550675e-08f, 0.606689453f, 0.499738216f, 1.1788468e-08f, \
  0.600830078f, 0.509443104f, 1.20611672e-08f, 0.595458984f, 0.518422782f, -1.39176883e-08f, \
  0.58984375f, 0.527897596f, 1.13053851e-08f, 0.584472656f, 0.5370453f, -1.94054408e-08f, \
  0.579101562f, 0.546277404f, 2.77024581e-09f, 0.573974609f, 0.555170119f, -6.29472141e-10f, \
  0.568847656f, 0.564142644f, -2.42457681e-08f, 0.563964844f, 0.572763383f, -2.01850145e-08f, \
  0.558837891f, 0.581895828f, 1.85197067e-08f, 0.554199219f, 0.590231061f, -4.737855e-09f, \
  0.549316406f, 0.599080682f, -1.02799644e-08f, 0.544677734f, 0.607560992f, -1.99540953e-08f, \
  0.540039062f, 0.616113782f, 2.2148102e-08f, 0.535644531f, 0.624284506f, 2.00400514e-08f, \
  0.531005859f, 0.632982194f, 2.87728845e-08f, 0.526855469f, 0.640829027f, -5.79780224e-09f, \
  0.522460938f, 0.649205029f, 2.96926732e-08f, 0.518310547f, 0.657180727f, -2.15120792e-08f, \
  0.514160156f, 0.665220499f, -2.50132732e-08f, 0.510009766f, 0.673325419f, -1.42631862e-08f, \
  0.505859375f, 0.681496561f, 2.76639223e-09f, 0.501953125f, 0.689248562f, -2.17148433e-08f
static __device__ const float kExp64[128] = {BH_EXP64};
static __device__ const float kLog64[192] = {BH_LOG64};
#ifdef __CUDA_ARCH__
#define BH_TAB(t, i) __ldg(&t[i])
#else
static const float kExp64Host[128] = {BH_EXP64};
static const float kLog64Host[192] = {BH_LOG64};
#define BH_TAB(t, i) t##Host[i]
#endif
#undef BH_EXP64
#undef BH_LOG64

// e^x for an F2 argument: x = k ln2 / 64 + r, |r| <= ln2 / 128, e^r - 1 = r +
// r^2 / 2 + (r^3 / 6 + r^4 / 24 + r^5 / 120) with the square in F2, 2^(k/64) from the
// table.  0 below -87, +inf above 88.
BH_NI F2 exp2f2(F2 x) {
  if (!(x.h > -87.0f)) return mk2(x.h != x.h ? x.h : 0.0f, 0.0f);
  if (x.h > 88.0f) return mk2(bits_f(0x7f800000), 0.0f);
  const float km = f_fma(x.h, 92.3324826f, 12582912.0f);  // 64 / ln2, 1.5 * 2^23
  const float k = f_sub(km, 12582912.0f);
  const int ik = f_bits(km) - 0x4b400000;
  const F2 p = two_prod(k, 1.08304247e-2f);                // ln2 / 64, leading part
  const F2 d = two_sum(x.h, -p.h);
  const float lo = f_add(f_sub(x.l, p.l), f_fma(k, 2.97602221e-11f, d.l));
  const F2 r = quick_sum(d.h, lo);
  const float r2 = f_mul(r.h, r.h);
  const float hr = f_mul(0.5f, r.h);
  // r^2 / 2 = q exactly to 2^-48, r^3 / 6 + r^4 / 24 + r^5 / 120 in one float
  const float g = f_fma(r.h, f_fma(r.h, 8.33333377e-3f, 4.16666679e-2f), 1.66666672e-1f);
  F2 q = two_prod(hr, r.h);
  q.l = f_add(f_fma(r.h, r.l, q.l), f_mul(f_mul(r2, r.h), g));
  F2 s = quick_sum(r.h, q.h);
  s = mk2(s.h, f_add(s.l, f_add(r.l, q.l)));               // e^r - 1
  const int j = ik & 63;
  const F2 T = mk2(BH_TAB(kExp64, 2 * j), BH_TAB(kExp64, 2 * j + 1));
  const F2 w = mul_raw(T, s);
  const F2 u = quick_sum(T.h, w.h);
  const F2 y = quick_sum(u.h, f_add(u.l, f_add(T.l, w.l)));
  return scale(y, bits_f(((ik >> 6) + 127) << 23));
}

// log(1 + x) for x > -1 (F2): u = 1 + x = 2^e m, z = m r_j - 1 with |z| <=
// 1/64 (z = x itself for 0 <= x < 1/64, which keeps the relative precision
// there),
// log u = e ln2 + T_j + log(1 + z), the series in F2 to z^3 and in floats
// beyond.
BH_NI F2 log1p2(F2 x) {
  const F2 u = addf(x, 1.0f);
  const int ub = f_bits(u.h);
  int e = ((ub >> 23) & 0xff) - 127, j = (ub >> 17) & 63;
  const float sc = bits_f((127 - e) << 23);                // 2^-e
  const F2 m = scale(u, sc);
  const float r = BH_TAB(kLog64, 3 * j);
  const F2 p = two_prod(m.h, r);
  F2 z = two_sum(p.h, -1.0f);
  z = quick_sum(z.h, f_add(z.l, f_fma(m.l, r, p.l)));
  if (e == 0 && j == 0) z = x;
  float t = f_fma(z.h, -1.25e-1f, 1.42857149e-1f);         // -1/8, 1/7
  t = f_fma(z.h, t, -1.66666672e-1f);                      // -1/6
  t = f_fma(z.h, t, 2.00000003e-1f);                       // 1/5
  F2 P = horner2(z, mk2(t, 0.f), mk2(-0.25f, 0.f));
  P = horner2(z, P, mk2(3.33333343e-1f, -9.93410776e-9f));  // 1/3
  P = horner2(z, P, mk2(-0.5f, 0.f));
  const F2 w = mul_raw(sqr_raw(z), P);
  const F2 v = quick_sum(z.h, w.h);
  const F2 lz = quick_sum(v.h, f_add(v.l, f_add(z.l, w.l)));
  const F2 T = mk2(BH_TAB(kLog64, 3 * j + 1), BH_TAB(kLog64, 3 * j + 2));
  const F2 base = add(mulf_raw((float)e, mk2(6.93147182e-1f, -1.90465421e-9f)), T);
  return add(base, lz);
}

// ------------------------------------------------ pairs of two-float numbers
// The same operations on two numbers at a time in the packed FP32
// instructions (add, mul and fma .f32x2).  The FP32 pipes do the same work
// per clock either way (measured on GB300: 3.97 scalar or 2.00 packed fused
// multiply-adds per clock and SM); what packing saves is issue slots and
// instruction cache.
typedef unsigned long long fx2;
#ifdef __CUDA_ARCH__
BH_HD fx2 pk(float a, float b) {
  fx2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
BH_HD float lo_of(fx2 v) { return __uint_as_float((unsigned)v); }
BH_HD float hi_of(fx2 v) { return __uint_as_float((unsigned)(v >> 32)); }
BH_HD fx2 v_add(fx2 a, fx2 b) {
  fx2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
BH_HD fx2 v_sub(fx2 a, fx2 b) {
  fx2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
BH_HD fx2 v_mul(fx2 a, fx2 b) {
  fx2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
BH_HD fx2 v_fma(fx2 a, fx2 b, fx2 c) {
  fx2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
#else
BH_HD fx2 pk(float a, float b) {
  return (fx2)(unsigned)f_bits(a) | ((fx2)(unsigned)f_bits(b) << 32);
}
BH_HD float lo_of(fx2 v) { return bits_f((int)(unsigned)v); }
BH_HD float hi_of(fx2 v) { return bits_f((int)(unsigned)(v >> 32)); }
BH_HD fx2 v_add(fx2 a, fx2 b) { return pk(lo_of(a) + lo_of(b), hi_of(a) + hi_of(b)); }
BH_HD fx2 v_sub(fx2 a, fx2 b) { return pk(lo_of(a) - lo_of(b), hi_of(a) - hi_of(b)); }
BH_HD fx2 v_mul(fx2 a, fx2 b) { return pk(lo_of(a) * lo_of(b), hi_of(a) * hi_of(b)); }
BH_HD fx2 v_fma(fx2 a, fx2 b, fx2 c) {
  return pk(std::fmaf(lo_of(a), lo_of(b), lo_of(c)), std::fmaf(hi_of(a), hi_of(b), hi_of(c)));
}
#endif
BH_HD fx2 v_neg(fx2 a) { return pk(-lo_of(a), -hi_of(a)); }

struct F2x2 {
  fx2 h, l;
};
struct F3x2 {
  fx2 a, b, c;
};
BH_HD F2x2 mkv(fx2 h, fx2 l) {
  F2x2 r;
  r.h = h;
  r.l = l;
  return r;
}
BH_HD F2x2 pair(F2 x, F2 y) { return mkv(pk(x.h, y.h), pk(x.l, y.l)); }
BH_HD F2 first(F2x2 x) { return mk2(lo_of(x.h), lo_of(x.l)); }
BH_HD F2 second(F2x2 x) { return mk2(hi_of(x.h), hi_of(x.l)); }
BH_HD F2x2 v_two_sum(fx2 a, fx2 b) {
  const fx2 s = v_add(a, b), bb = v_sub(s, a);
  return mkv(s, v_add(v_sub(a, v_sub(s, bb)), v_sub(b, bb)));
}
BH_HD F2x2 v_quick_sum(fx2 a, fx2 b) {
  const fx2 s = v_add(a, b);
  return mkv(s, v_sub(b, v_sub(s, a)));
}
// raw: |l| up to a few ulps of h, as mul_raw
BH_HD F2x2 v_mul_raw(F2x2 x, F2x2 y) {
  const fx2 p = v_mul(x.h, y.h);
  return mkv(p, v_fma(x.l, y.h, v_fma(x.h, y.l, v_fma(x.h, y.h, v_neg(p)))));
}
BH_HD F2x2 v_norm(F2x2 x) { return v_quick_sum(x.h, x.l); }
BH_HD F2x2 v_sqr_raw(F2x2 x) {
  const fx2 p = v_mul(x.h, x.h);
  return mkv(p, v_fma(v_add(x.h, x.h), x.l, v_fma(x.h, x.h, v_neg(p))));
}
BH_HD F2x2 v_add_raw(F2x2 x, F2x2 y) {
  const F2x2 s = v_two_sum(x.h, y.h);
  return mkv(s.h, v_add(s.l, v_add(x.l, y.l)));
}
BH_HD F2x2 v_sub_raw(F2x2 x, F2x2 y) {
  const F2x2 s = v_two_sum(x.h, v_neg(y.h));
  return mkv(s.h, v_add(s.l, v_sub(x.l, y.l)));
}
BH_HD F2x2 v_horner(F2x2 z, F2x2 t, F2x2 c) {
  const F2x2 p = v_mul_raw(z, t), s = v_quick_sum(c.h, p.h);
  return mkv(s.h, v_add(s.l, v_add(c.l, p.l)));
}
BH_HD F2x2 v_rcp(F2x2 x) {
  const fx2 r = pk(f_rcp(lo_of(x.h)), f_rcp(hi_of(x.h)));
  const fx2 nr = v_neg(r);
  fx2 e = v_fma(x.h, nr, pk(1.0f, 1.0f));
  e = v_fma(x.l, nr, e);
  return v_quick_sum(r, v_mul(r, v_fma(e, e, e)));
}
// the same without the last renormalisation, scalar
BH_HD F2 add_raw(F2 x, F2 y) {
  const F2 s = two_sum(x.h, y.h);
  return mk2(s.h, f_add(s.l, f_add(x.l, y.l)));
}

// Sine and cosine of an F2 angle of a few radians: reduction by the nearest
// multiple q of pi/2 (three floats), Taylor polynomials on |r| <= pi/4, the
// two side by side, whose terms above 2^-24 of the result are F2 and the rest
// floats, rotation by q quarter turns.  Absolute error within 2^-44 (tests).
BH_HD void sincos2(F2 x, F2& sn, F2& cs) {
  const float qm = f_fma(x.h, 0.636619772f, 12582912.0f);  // 2/pi, 1.5 * 2^23
  const float q = f_sub(qm, 12582912.0f);
  const int iq = f_bits(qm);
  const F2 p1 = two_prod(q, 1.57079637f);                  // pi/2, leading part
  const F2 d = two_sum(x.h, -p1.h);
  // q times the second part against the low float exactly: r keeps its
  // relative precision near theta = pi, where 1 / sin(theta) enters
  const F2 p2 = two_prod(q, -4.37113883e-8f);
  const F2 e = two_sum(f_sub(x.l, p1.l), -p2.h);
  const F2 rr = quick_sum(d.h, e.h);
  const float lo = f_sub(f_add(e.l, d.l), f_fma(q, -1.71512451e-15f, p2.l));
  const F2 r = quick_sum(rr.h, f_add(rr.l, lo));
  const F2 zs = sqr_raw(r);
  const F2x2 z = pair(zs, zs);
  // sin r = r + r z S(z), cos r = 1 + z C(z): coefficients (S, C)
  fx2 t = v_fma(z.h, pk(-7.64716373e-13f, -1.14707454e-11f),   // -1/15!, -1/14!
                pk(1.60590444e-10f, 2.08767559e-9f));          // 1/13!, 1/12!
  t = v_fma(z.h, t, pk(-2.50521079e-8f, -2.755732e-7f));       // -1/11!, -1/10!
  F2x2 P = v_horner(z, mkv(t, 0ull), mkv(pk(2.75573188e-6f, 2.48015876e-5f),  // 1/9!, 1/8!
                                         pk(3.79357122e-14f, -3.40699609e-13f)));
  P = v_horner(z, P, mkv(pk(-1.98412701e-4f, -1.38888892e-3f),  // -1/7!, -1/6!
                         pk(2.72559687e-12f, 3.36310944e-11f)));
  P = v_horner(z, P, mkv(pk(8.33333377e-3f, 4.16666679e-2f),    // 1/5!, 1/4!
                         pk(-4.34617203e-10f, -1.24176347e-9f)));
  P = v_horner(z, P, mkv(pk(-1.66666672e-1f, -0.5f),            // -1/3!, -1/2
                         pk(4.96705388e-9f, 0.0f)));
  const F2x2 w = v_mul_raw(pair(mul_raw(r, zs), zs), P);
  const F2x2 u = v_quick_sum(pk(r.h, 1.0f), w.h);
  const F2x2 y = v_quick_sum(u.h, v_add(u.l, v_add(pk(r.l, 0.0f), w.l)));
  const F2 sr = first(y), cr = second(y);
  const bool odd = (iq & 1) != 0;
  const int ss = (iq & 2) << 30, cc = ((iq + 1) & 2) << 30;
  sn = mk2(bits_f(f_bits(odd ? cr.h : sr.h) ^ ss), bits_f(f_bits(odd ? cr.l : sr.l) ^ ss));
  cs = mk2(bits_f(f_bits(odd ? sr.h : cr.h) ^ cc), bits_f(f_bits(odd ? sr.l : cr.l) ^ cc));
}

}  // namespace bhrt
