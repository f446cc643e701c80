// lean_fp64.cuh -- e^x and 1/sqrt(x) in FP64 with few FP64 instructions.
//
// On GB300 an FP64 instruction costs the issue slots of about 64 FP32 ones, and
// the passes that hold a field in FP64 are bound by their count.  Both
// functions work out in FP32 and integers what FP64 does not need to carry,
// and keep an error below 1 ulp (e^x) and 1.5 ulp (1/sqrt x) of FP64; arguments
// outside the ranges stated go to the CUDA functions.  The same code compiles
// as host C++ for testing.
#pragma once
#include "dfloat.cuh"

#ifdef __CUDACC__
#define LEAN_HD __host__ __device__ __forceinline__
#else
#define LEAN_HD static inline
#endif

// 2^(j/64), j = 0..63, rounded to FP64
#define LEAN_EXP2_TABLE \
  {                                                                            \
    0x1.0000000000000p+0, 0x1.02c9a3e778061p+0, 0x1.059b0d3158574p+0, 0x1.0874518759bc8p+0, \
    0x1.0b5586cf9890fp+0, 0x1.0e3ec32d3d1a2p+0, 0x1.11301d0125b51p+0, 0x1.1429aaea92de0p+0, \
    0x1.172b83c7d517bp+0, 0x1.1a35beb6fcb75p+0, 0x1.1d4873168b9aap+0, 0x1.2063b88628cd6p+0, \
    0x1.2387a6e756238p+0, 0x1.26b4565e27cddp+0, 0x1.29e9df51fdee1p+0, 0x1.2d285a6e4030bp+0, \
    0x1.306fe0a31b715p+0, 0x1.33c08b26416ffp+0, 0x1.371a7373aa9cbp+0, 0x1.3a7db34e59ff7p+0, \
    0x1.3dea64c123422p+0, 0x1.4160a21f72e2ap+0, 0x1.44e086061892dp+0, 0x1.486a2b5c13cd0p+0, \
    0x1.4bfdad5362a27p+0, 0x1.4f9b2769d2ca7p+0, 0x1.5342b569d4f82p+0, 0x1.56f4736b527dap+0, \
    0x1.5ab07dd485429p+0, 0x1.5e76f15ad2148p+0, 0x1.6247eb03a5585p+0, 0x1.6623882552225p+0, \
    0x1.6a09e667f3bcdp+0, 0x1.6dfb23c651a2fp+0, 0x1.71f75e8ec5f74p+0, 0x1.75feb564267c9p+0, \
    0x1.7a11473eb0187p+0, 0x1.7e2f336cf4e62p+0, 0x1.82589994cce13p+0, 0x1.868d99b4492edp+0, \
    0x1.8ace5422aa0dbp+0, 0x1.8f1ae99157736p+0, 0x1.93737b0cdc5e5p+0, 0x1.97d829fde4e50p+0, \
    0x1.9c49182a3f090p+0, 0x1.a0c667b5de565p+0, 0x1.a5503b23e255dp+0, 0x1.a9e6b5579fdbfp+0, \
    0x1.ae89f995ad3adp+0, 0x1.b33a2b84f15fbp+0, 0x1.b7f76f2fb5e47p+0, 0x1.bcc1e904bc1d2p+0, \
    0x1.c199bdd85529cp+0, 0x1.c67f12e57d14bp+0, 0x1.cb720dcef9069p+0, 0x1.d072d4a07897cp+0, \
    0x1.d5818dcfba487p+0, 0x1.da9e603db3285p+0, 0x1.dfc97337b9b5fp+0, 0x1.e502ee78b3ff6p+0, \
    0x1.ea4afa2a490dap+0, 0x1.efa1bee615a27p+0, 0x1.f50765b6e4540p+0, 0x1.fa7c1819e90d8p+0 \
  }
// what the rounding left out of each entry
#define LEAN_EXP2_LOW                                                          \
  {                                                                            \
    0.f, -1.52347793e-17f, 5.10922498e-17f, 7.60083857e-18f, \
    8.55188948e-17f, 1.75932569e-18f, -7.89985411e-17f, -6.65666054e-17f, \
    -3.04678214e-17f, 5.26603692e-17f, 1.04102784e-16f, 5.16585675e-17f, \
    8.91281287e-17f, 3.25071029e-17f, 3.82920467e-17f, 5.55420348e-17f, \
    3.98201537e-17f, 6.64498141e-17f, -7.71263071e-17f, -1.89878168e-17f, \
    4.65802774e-17f, -6.71138987e-18f, 2.6679321e-18f, 1.71359497e-17f, \
    2.5382502e-17f, -7.18153642e-17f, -2.85873123e-17f, 8.92728257e-17f, \
    7.70094827e-17f, 9.59379824e-17f, -6.77051169e-17f, -9.61421306e-17f, \
    -9.66729357e-17f, -1.20316423e-17f, -3.02375807e-17f, -5.60037737e-17f, \
    -3.48399441e-17f, 1.41929205e-17f, -1.01645535e-16f, -1.10249418e-16f, \
    7.94983501e-17f, 3.78120702e-17f, -1.01369164e-17f, -1.00944066e-16f, \
    2.47071934e-17f, -6.71295514e-17f, -1.012568e-16f, 5.89099239e-17f, \
    8.19901026e-17f, -8.02371977e-18f, -1.85138043e-17f, 3.16438936e-17f, \
    2.9601406e-17f, 6.42973181e-17f, 1.82274592e-17f, -9.96953147e-17f, \
    3.28310731e-17f, 9.7618873e-17f, -6.1227631e-17f, 3.40340353e-17f, \
    -1.06199462e-16f, 1.03323858e-16f, 8.9607675e-17f, 4.03887544e-17f \
  }
#ifdef __CUDACC__
static __device__ const double kLeanExp2[64] = LEAN_EXP2_TABLE;
static __device__ const float kLeanExp2Low[64] = LEAN_EXP2_LOW;
#endif
static const double kLeanExp2Host[64] = LEAN_EXP2_TABLE;
static const float kLeanExp2LowHost[64] = LEAN_EXP2_LOW;

// e^x by Tang's table-driven method (P. T. P. Tang, ACM TOMS 15 (1989) 144):
// x = k ln2/64 + r, |r| <= ln2/128, k rounded in FP32; the reduction by two
// fused multiply-adds with ln2/64 as a sum of two doubles; e^r - 1 from its
// Taylor series, whose terms from r^4 on (below 4e-11) are summed in FP32;
// the first omitted term is r^7/5040 < 3e-20.  Nine FP64 instructions.
LEAN_HD double lean_exp(double x) {
  const float xf = f_from_double_bits(x);
  if (!(xf > -690.f && xf < 690.f)) return exp(x);  // and NaN
  const float kf = rintf(DF_MUL(xf, 92.332482616893656877f));  // 64 / ln 2
  const int k = (int)kf;
  const double kd = d_from_float_bits(kf);
  double r = fma(kd, -0x1.62e42fefa39efp-7, x);
  r = fma(kd, -0x1.abc9e3b39803fp-62, r);
  const float rf = f_from_double_bits(r);
  const float q = DF_FMA(rf, DF_FMA(rf, 1.f / 720.f, 1.f / 120.f), 1.f / 24.f);
  double p = fma(r, d_from_float_bits(q), 1.0 / 6.0);
  p = fma(r, p, 0.5);
  p = fma(r * r, p, r);
#ifdef __CUDA_ARCH__
  const double t = __ldg(kLeanExp2 + (k & 63));
  const double lo = d_from_float_bits(__ldg(kLeanExp2Low + (k & 63)));
#else
  const double t = kLeanExp2Host[k & 63];
  const double lo = d_from_float_bits(kLeanExp2LowHost[k & 63]);
#endif
  // 2^(k div 64) enters the exponent: the result is normal for |x| < 690
  return dfrombits(dbits(t + fma(t, p, lo)) + ((unsigned long long)(long long)(k >> 6) << 52));
}

// 1/sqrt(x): an FP32 estimate y (relative error e/2 < 2e-7 in 1 - x y^2 = e),
// then y (1 + e/2 + 3 e^2/8), the omitted term 5 e^3/16 < 1e-20.  Five FP64
// instructions for 1e-30 < x < 1e30.
LEAN_HD double lean_rsqrt(double x) {
  const float xf = f_from_double_bits(x);
#ifdef __CUDA_ARCH__
  if (!(xf > 1e-30f && xf < 1e30f)) return rsqrt(x);
  const double y = d_from_float_bits(rsqrtf(xf));
#else
  if (!(xf > 1e-30f && xf < 1e30f)) return 1.0 / sqrt(x);
  const double y = d_from_float_bits(1.f / sqrtf(xf));
#endif
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}
