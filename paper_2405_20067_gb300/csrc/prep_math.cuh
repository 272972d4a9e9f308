// prep_math.cuh -- the FP64 functions of the preparation (csrc/cull.cu): its
// exponentials, sigmoids and quotients.  The preparation is bound by FP64
// arithmetic (two lanes per clock and SM), so they take few FP64 operations,
// with errors no larger than those of exp() and `/`; ndg_selftest_math
// evaluates both side by side.  Measured: prep_kernel on 500,000 N = 10
// Gaussians 1.87 ms (2.46 with exp() and `/`), conditioned 3.12 ms (3.91).
#pragma once
#include <cuda_runtime.h>

namespace ndg {

// exp(v) after P. T. P. Tang, "Table-driven implementation of the exponential
// function in IEEE floating-point arithmetic" (ACM TOMS 15, 1989):
// k = round(64 v / ln 2) (from FP32: any nearby integer does),
// r = v - k ln2 / 64 with ln2 / 64 split so that k * high part is exact,
// exp(v) = 2^(k / 64) (1 + p(r)), the power as a pair high + low.  p is the
// Taylor polynomial of degree 6 with its last term economised on
// |r| <= a = ln2 / 128 (r^6 = 3/2 a^2 r^4 - 9/16 a^4 r^2 + ..., the rest below
// 3e-18).  Largest error 0.53 ulp: the last addition's half and the roundings
// of p (one table entry per power and degree 5 made 1.26).
__device__ const double2 kExp2Table[64] = {  // 2^(j / 64), high and low
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.02c9a3e778061p+0, -0x1.19083535b085dp-56},
    {0x1.059b0d3158574p+0, 0x1.d73e2a475b465p-55}, {0x1.0874518759bc8p+0, 0x1.186be4bb284ffp-57},
    {0x1.0b5586cf9890fp+0, 0x1.8a62e4adc610bp-54}, {0x1.0e3ec32d3d1a2p+0, 0x1.03a1727c57b52p-59},
    {0x1.11301d0125b51p+0, -0x1.6c51039449b3ap-54}, {0x1.1429aaea92de0p+0, -0x1.32fbf9af1369ep-54},
    {0x1.172b83c7d517bp+0, -0x1.19041b9d78a76p-55}, {0x1.1a35beb6fcb75p+0, 0x1.e5b4c7b4968e4p-55},
    {0x1.1d4873168b9aap+0, 0x1.e016e00a2643cp-54}, {0x1.2063b88628cd6p+0, 0x1.dc775814a8495p-55},
    {0x1.2387a6e756238p+0, 0x1.9b07eb6c70573p-54}, {0x1.26b4565e27cddp+0, 0x1.2bd339940e9d9p-55},
    {0x1.29e9df51fdee1p+0, 0x1.612e8afad1255p-55}, {0x1.2d285a6e4030bp+0, 0x1.0024754db41d5p-54},
    {0x1.306fe0a31b715p+0, 0x1.6f46ad23182e4p-55}, {0x1.33c08b26416ffp+0, 0x1.32721843659a6p-54},
    {0x1.371a7373aa9cbp+0, -0x1.63aeabf42eae2p-54}, {0x1.3a7db34e59ff7p+0, -0x1.5e436d661f5e3p-56},
    {0x1.3dea64c123422p+0, 0x1.ada0911f09ebcp-55}, {0x1.4160a21f72e2ap+0, -0x1.ef3691c309278p-58},
    {0x1.44e086061892dp+0, 0x1.89b7a04ef80d0p-59}, {0x1.486a2b5c13cd0p+0, 0x1.3c1a3b69062f0p-56},
    {0x1.4bfdad5362a27p+0, 0x1.d4397afec42e2p-56}, {0x1.4f9b2769d2ca7p+0, -0x1.4b309d25957e3p-54},
    {0x1.5342b569d4f82p+0, -0x1.07abe1db13cadp-55}, {0x1.56f4736b527dap+0, 0x1.9bb2c011d93adp-54},
    {0x1.5ab07dd485429p+0, 0x1.6324c054647adp-54}, {0x1.5e76f15ad2148p+0, 0x1.ba6f93080e65ep-54},
    {0x1.6247eb03a5585p+0, -0x1.383c17e40b497p-54}, {0x1.6623882552225p+0, -0x1.bb60987591c34p-54},
    {0x1.6a09e667f3bcdp+0, -0x1.bdd3413b26456p-54}, {0x1.6dfb23c651a2fp+0, -0x1.bbe3a683c88abp-57},
    {0x1.71f75e8ec5f74p+0, -0x1.16e4786887a99p-55}, {0x1.75feb564267c9p+0, -0x1.0245957316dd3p-54},
    {0x1.7a11473eb0187p+0, -0x1.41577ee04992fp-55}, {0x1.7e2f336cf4e62p+0, 0x1.05d02ba15797ep-56},
    {0x1.82589994cce13p+0, -0x1.d4c1dd41532d8p-54}, {0x1.868d99b4492edp+0, -0x1.fc6f89bd4f6bap-54},
    {0x1.8ace5422aa0dbp+0, 0x1.6e9f156864b27p-54}, {0x1.8f1ae99157736p+0, 0x1.5cc13a2e3976cp-55},
    {0x1.93737b0cdc5e5p+0, -0x1.75fc781b57ebcp-57}, {0x1.97d829fde4e50p+0, -0x1.d185b7c1b85d1p-54},
    {0x1.9c49182a3f090p+0, 0x1.c7c46b071f2bep-56}, {0x1.a0c667b5de565p+0, -0x1.359495d1cd533p-54},
    {0x1.a5503b23e255dp+0, -0x1.d2f6edb8d41e1p-54}, {0x1.a9e6b5579fdbfp+0, 0x1.0fac90ef7fd31p-54},
    {0x1.ae89f995ad3adp+0, 0x1.7a1cd345dcc81p-54}, {0x1.b33a2b84f15fbp+0, -0x1.2805e3084d708p-57},
    {0x1.b7f76f2fb5e47p+0, -0x1.5584f7e54ac3bp-56}, {0x1.bcc1e904bc1d2p+0, 0x1.23dd07a2d9e84p-55},
    {0x1.c199bdd85529cp+0, 0x1.11065895048ddp-55}, {0x1.c67f12e57d14bp+0, 0x1.2884dff483cadp-54},
    {0x1.cb720dcef9069p+0, 0x1.503cbd1e949dbp-56}, {0x1.d072d4a07897cp+0, -0x1.cbc3743797a9cp-54},
    {0x1.d5818dcfba487p+0, 0x1.2ed02d75b3707p-55}, {0x1.da9e603db3285p+0, 0x1.c2300696db532p-54},
    {0x1.dfc97337b9b5fp+0, -0x1.1a5cd4f184b5cp-54}, {0x1.e502ee78b3ff6p+0, 0x1.39e8980a9cc8fp-55},
    {0x1.ea4afa2a490dap+0, -0x1.e9c23179c2893p-54}, {0x1.efa1bee615a27p+0, 0x1.dc7f486a4b6b0p-54},
    {0x1.f50765b6e4540p+0, 0x1.9d3e12dd8a18bp-54}, {0x1.fa7c1819e90d8p+0, 0x1.74853f3a5931ep-55}};
constexpr float kExpRange = 690.0f;  // |v| below: every step in the normal range

// v as FP64 by moving its bits: a conversion would be another operation on the
// FP64 pipe.  FP32 zeros and subnormals become +-2^-127 (1 + ...), which the
// exponential cannot tell from them.
__device__ __forceinline__ double widen(float v) {
  const unsigned b = __float_as_uint(v);
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)),
                          (int)(b << 29));
}
__device__ __forceinline__ double exp_in_range(float v) {
  constexpr double A2 = 2.932499e-5;  // (ln2 / 128)^2
  const float kf = rintf(v * 92.33248261689366f);
  const int k = (int)kf;
  const double kd = widen(kf);
  double r = fma(kd, -0x1.62e42fee00000p-7, widen(v));
  r = fma(kd, -0x1.a39ef35793c76p-39, r);
  double q = fma(r, 1.0 / 120.0, 1.0 / 24.0 + 1.5 * A2 / 720.0);
  q = fma(q, r, 1.0 / 6.0);
  q = fma(q, r, 0.5 - 0.5625 * A2 * A2 / 720.0);
  q = fma(q * r, r, r);
  const double2 t = __ldg(kExp2Table + (k & 63));
  const double e = t.x + fma(t.x, q, t.y);
  return __hiloint2double(__double2hiint(e) + ((k >> 6) << 20), __double2loint(e));
}
__device__ __forceinline__ double exp_f32(float v) {
  return fabsf(v) < kExpRange ? exp_in_range(v) : exp((double)v);
}

// 1 / (1 + exp(-v)).  The reciprocal: the approximate one (2^-20 or better),
// one third-order correction x (1 + e + e^2), e = 1 - d x, and Markstein's
// final step (P. W. Markstein, IBM J. Res. Dev. 34, 1990), whose residual
// decides the last bit.
__device__ __forceinline__ double sigmoid(float v) {
  if (!(fabsf(v) < kExpRange)) return 1.0 / (1.0 + exp(-(double)v));
  const double d = 1.0 + exp_in_range(-v);
  double x;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(d));
  double e = fma(-d, x, 1.0);
  e = fma(e, e, e);
  x = fma(e, x, x);
  return fma(fma(-d, x, 1.0), x, x);
}
// Eq. 2's off-diagonal, 2 sigmoid - 1 (the doubling and the difference of the
// correctly rounded quotient round once, as 2 / (1 + exp(-v)) - 1 does).
__device__ __forceinline__ double off_diagonal(float v) { return fma(2.0, sigmoid(v), -1.0); }

// a / b from y = 1 / b: Markstein's step on the product a y.  The residual is
// exact for 2^-400 <= |a|, |b| < 2^400, and the quotient then that of the
// division; products out of the FP64 range stay as they are.
__device__ __forceinline__ double quotient(double a, double b, double y) {
  const double q = a * y;
  const double p = fma(fma(-b, q, a), y, q);
  return (__double2hiint(p) & 0x7ff00000) == 0x7ff00000 ? q : p;
}

}  // namespace ndg
