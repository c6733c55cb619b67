// FP64 exponential, logarithm and power of a positive base for the nodal closures of the FP64
// path (local-field mobility mu0 (|E| / E_ref)^p and Townsend alpha = A exp(-B/|E|)), with a
// few tens of FP64 operations each.  GB300 issues about one warp-wide FP64 instruction per 17
// cycles per SM, so general-purpose library routines, which handle every special case with full
// correct rounding, made these two closures most of the nodal kernel's time.  The arguments here
// are finite, the bases positive and normal.  exp and log are accurate to a few units in the
// last place; pow carries log's rounding times |p log x| (about 4e-16 (1 + |p log x|) relative),
// a few ulp for the mobility closure, whose |p log x| stays below 2 (tested against the CUDA
// math library on the device).
//
// Both are table-driven (P. T. P. Tang, ACM TOMS 15 (1989) and 16 (1990)), which halves the FP64
// operations of the plain series: nodal fields of 500,000 nodes 161 -> 131 us with them.
//
//   exp: x = (32 k + j) ln2 / 32 + r, |r| <= ln2 / 64, with ln2 split in a head of 32 significant
//        bits (the product with 32 k + j exact) and a tail; 2^(j/32) from a table of 32 rounded
//        values, e^r - 1 by its Taylor polynomial of degree 6 (truncation below 4e-18), 2^k added
//        to the exponent field (results below the smallest normal flush to zero).
//   log: x = m 2^e with m in [sqrt(1/2), sqrt(2)), split into 64 intervals with a rounded reciprocal
//        c of the interval's middle (1 in the interval around 1, so that log x keeps its relative
//        accuracy there); r = m c - 1, |r| < 2^-6.9; log m = -log c + log(1 + r) with a table of
//        -log c and the series of degree 8 (truncation below 3e-20).
//   pow: x^p = exp(p log x), x > 0.
#pragma once

namespace avip {

// 2^(j/32), j = 0 .. 31
static __device__ const double kExp2Table[32] = {
    0x1.0000000000000p+0, 0x1.059b0d3158574p+0, 0x1.0b5586cf9890fp+0, 0x1.11301d0125b51p+0,
    0x1.172b83c7d517bp+0, 0x1.1d4873168b9aap+0, 0x1.2387a6e756238p+0, 0x1.29e9df51fdee1p+0,
    0x1.306fe0a31b715p+0, 0x1.371a7373aa9cbp+0, 0x1.3dea64c123422p+0, 0x1.44e086061892dp+0,
    0x1.4bfdad5362a27p+0, 0x1.5342b569d4f82p+0, 0x1.5ab07dd485429p+0, 0x1.6247eb03a5585p+0,
    0x1.6a09e667f3bcdp+0, 0x1.71f75e8ec5f74p+0, 0x1.7a11473eb0187p+0, 0x1.82589994cce13p+0,
    0x1.8ace5422aa0dbp+0, 0x1.93737b0cdc5e5p+0, 0x1.9c49182a3f090p+0, 0x1.a5503b23e255dp+0,
    0x1.ae89f995ad3adp+0, 0x1.b7f76f2fb5e47p+0, 0x1.c199bdd85529cp+0, 0x1.cb720dcef9069p+0,
    0x1.d5818dcfba487p+0, 0x1.dfc97337b9b5fp+0, 0x1.ea4afa2a490dap+0, 0x1.f50765b6e4540p+0};
// per interval of the mantissa: c (a rounded reciprocal of its middle) and -log c
static __device__ const double kLogC[64] = {
    0x1.680cbcd75c447p+0, 0x1.6422f70fce190p+0, 0x1.604ebbd86ed05p+0, 0x1.5c8f5b36b5f7ap+0,
    0x1.58e42c98c7254p+0, 0x1.554c8e72ab8d1p+0, 0x1.51c7e5e1a7890p+0, 0x1.4e559e553c622p+0,
    0x1.4af5293d6fae2p+0, 0x1.47a5fdbdf9ca4p+0, 0x1.44679866047a0p+0, 0x1.41397aec297ffp+0,
    0x1.3e1b2bee6741cp+0, 0x1.3b0c36b5c7393p+0, 0x1.380c2afd77253p+0, 0x1.351a9cbd1ab0bp+0,
    0x1.323723f61fa13p+0, 0x1.2f615c83e29d7p+0, 0x1.2c98e5ee7644dp+0, 0x1.29dd633fe1b19p+0,
    0x1.272e7adbae92dp+0, 0x1.248bd658a1e75p+0, 0x1.21f5225c7cfd0p+0, 0x1.1f6a0e79a6c4ep+0,
    0x1.1cea4d0e9fc17p+0, 0x1.1a75932724e42p+0, 0x1.180b985ee791fp+0, 0x1.15ac16c5c2c72p+0,
    0x1.1356cac556ee6p+0, 0x1.110b7307f780bp+0, 0x1.0ec9d060d6e24p+0, 0x1.0c91a5b55e3b4p+0,
    0x1.0a62b7e7a03aap+0, 0x1.083ccdc1d6c93p+0, 0x1.061fafe2dcbc4p+0, 0x1.040b28ab9586fp+0,
    0x1.01ff042d35cc6p+0, 0x1.0000000000000p+0, 0x1.f80c5d11a2684p-1, 0x1.f0698d819db27p-1,
    0x1.e901160cae199p-1, 0x1.e1d063d89c40fp-1, 0x1.dad50a3b936f0p-1, 0x1.d40cc001e9fd6p-1,
    0x1.cd755ceee8d1dp-1, 0x1.c70cd772d5babp-1, 0x1.c0d1429125649p-1, 0x1.bac0cbf246f1cp-1,
    0x1.b4d9ba1cf7947p-1, 0x1.af1a6ad37a2eep-1, 0x1.a98151916fce0p-1, 0x1.a40cf6276378ap-1,
    0x1.9ebbf37167b25p-1, 0x1.998cf626676a3p-1, 0x1.947ebbbe07efcp-1, 0x1.8f90116b2ed26p-1,
    0x1.8abfd3296e17dp-1, 0x1.860ceadbc3a2fp-1, 0x1.81764f7b3e95dp-1, 0x1.7cfb04543f712p-1,
    0x1.789a185126283p-1, 0x1.7452a5515cb7bp-1, 0x1.7023cf8bc561ap-1, 0x1.6c0cc4fba9cedp-1};
static __device__ const double kLogL[64] = {
    -0x1.5d401699901fbp-2, -0x1.520f66629c64ap-2, -0x1.46fdadb7c4a33p-2, -0x1.3c0a43098441cp-2,
    -0x1.3134822a443dfp-2, -0x1.267bcc14a5204p-2, -0x1.1bdf86b4c6653p-2, -0x1.115f1cb45c41bp-2,
    -0x1.06f9fd496801ep-2, -0x1.f95f380ed4a55p-3, -0x1.e4fee165d342bp-3, -0x1.d0d1ee2e52a3ep-3,
    -0x1.bcd75dbbe1f04p-3, -0x1.a90e36d289f47p-3, -0x1.9575875de8192p-3, -0x1.820c642bbdb66p-3,
    -0x1.6ed1e8a9c1f43p-3, -0x1.5bc536a687a6cp-3, -0x1.48e576154b88ep-3, -0x1.3631d4d4821b2p-3,
    -0x1.23a98676fee40p-3, -0x1.114bc40f914ebp-3, -0x1.fe2f97fdeb17dp-4, -0x1.da19c387f3f66p-4,
    -0x1.b6549b9b77017p-4, -0x1.92deba9fba046p-4, -0x1.6fb6c4313fd6bp-4, -0x1.4cdb64d18a57ep-4,
    -0x1.2a4b519a3f19bp-4, -0x1.080547f38348dp-4, -0x1.cc101a9acb805p-5, -0x1.88a4ddb8616c5p-5,
    -0x1.45c682aefd356p-5, -0x1.0372c177df6e4p-5, -0x1.834ec03d80f5dp-6, -0x1.00c4649e005fbp-6,
    -0x1.fd08c72af8ec1p-8, 0x0.0p+0, 0x1.0073809b61d99p-6, 0x1.fa8e7ea7db662p-6,
    0x1.7873639e2b330p-5, 0x1.f1cc700489fe1p-5, 0x1.34b003beee67bp-4, 0x1.6f9d9b2997907p-4,
    0x1.a9b53d561f1bbp-4, 0x1.e2fce6417493fp-4, 0x1.0dbd2942908b4p-3, 0x1.299981652da3dp-3,
    0x1.45161f80ebbedp-3, 0x1.60358cb284e6ep-3, 0x1.7afa38a290ab0p-3, 0x1.95667ad5d0993p-3,
    0x1.af7c93e811547p-3, 0x1.c93eaeb33e210p-3, 0x1.e2aee16420b79p-3, 0x1.fbcf2e7e26c9fp-3,
    0x1.0a50c2e7b4a5bp-2, 0x1.1693e2ab0b8b5p-2, 0x1.22b1dd0c26444p-2, 0x1.2eab9077a5f5bp-2,
    0x1.3a81d3a37b68fp-2, 0x1.463575e92b4a2p-2, 0x1.51c73f9af8e78p-2, 0x1.5d37f2544ef66p-2};

__device__ __forceinline__ double exp_fp64(double x) {
  constexpr double k32Log2e = 32.0 * 1.4426950408889634;
  constexpr double kHi = 0.6931471806019545 / 32.0;       // ln 2 rounded to 32 significant bits, / 32
  constexpr double kLo = -4.2009150726810846e-11 / 32.0;  // (ln 2 - its head) / 32
  constexpr double kMagic = 6755399441055744.0;           // 1.5 * 2^52: the sum's low word is the integer
  const int hx = __double2hiint(x);
  if ((hx & 0x7fffffff) >= 0x40862000) {                  // |x| >= 708
    if (x > 709.0) return __longlong_as_double(0x7ff0000000000000LL);  // overflow: +inf
    if (x < -708.0) return 0.0;                                          // below the normal range
    if (x != x) return x;
  }
  const double nm = fma(x, k32Log2e, kMagic);
  const int n = __double2loint(nm);
  const double nd = nm - kMagic;
  double r = fma(-nd, kHi, x);
  r = fma(-nd, kLo, r);
  // e^r - 1 = r + r^2 (1/2 + r/6 + r^2/24 + r^3/120 + r^4/720)
  double p = 1.0 / 720.0;
  p = fma(p, r, 1.0 / 120.0);
  p = fma(p, r, 1.0 / 24.0);
  p = fma(p, r, 1.0 / 6.0);
  p = fma(p, r, 0.5);
  p = fma(p, r * r, r);
  const double t = __ldg(kExp2Table + (n & 31));
  const double v = fma(t, p, t);
  return __hiloint2double(__double2hiint(v) + ((n >> 5) << 20), __double2loint(v));
}

__device__ __forceinline__ double log_fp64(double x) {
  constexpr double kLn2Hi = 0.6931471806019545;
  constexpr double kLn2Lo = -4.2009150726810846e-11;
  const long long bits = __double_as_longlong(x);
  const long long ix = bits - 0x3fe6a09e00000000LL;  // (the high word of sqrt(1/2))
  const int e = (int)(ix >> 52), j = (int)(ix >> 46) & 63;
  const double m = __longlong_as_double(bits - (ix & (long long)0xfff0000000000000ULL));
  const double r = fma(m, __ldg(kLogC + j), -1.0);
  // log(1 + r) = r - r^2 (1/2 - r/3 + r^2/4 - r^3/5 + r^4/6 - r^5/7 + r^6/8)
  double t = -1.0 / 8.0;
  t = fma(t, r, 1.0 / 7.0);
  t = fma(t, r, -1.0 / 6.0);
  t = fma(t, r, 1.0 / 5.0);
  t = fma(t, r, -1.0 / 4.0);
  t = fma(t, r, 1.0 / 3.0);
  t = fma(t, r, -0.5);
  const double ed = (double)e;
  const double small = fma(t, r * r, fma(ed, kLn2Lo, r));
  return fma(ed, kLn2Hi, __ldg(kLogL + j) + small);
}

__device__ __forceinline__ double pow_pos_fp64(double x, double p) { return exp_fp64(p * log_fp64(x)); }

// 1 / d for a nonzero d: the hardware's approximate reciprocal refined by two Newton-Raphson
// steps y <- y + y (1 - d y) (each squares the relative error: about 2^-20 -> 2^-40 -> the FP64
// rounding), within a few ulp of the rounded quotient, for 5 FP64 instructions against about
// twice that for an IEEE division.  A subnormal d (exponent field zero; the approximation
// flushes it) takes the division.
__device__ __forceinline__ double recip_nr(double d) {
  if ((__double2hiint(d) & 0x7ff00000) == 0) return 1.0 / d;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  double e = fma(-d, y, 1.0);
  y = fma(y, e, y);
  e = fma(-d, y, 1.0);
  return fma(y, e, y);
}

// n / d for normal n, d and quotient: the Newton reciprocal's quotient corrected by its residual
// (Markstein, IBM J. Res. Dev. 34 (1990)), for two more FP64 instructions than n * recip_nr(d).
__device__ __forceinline__ double quotient_nr(double n, double d) {
  const double y = recip_nr(d), q = n * y;
  return fma(fma(-d, q, n), y, q);
}

}  // namespace avip
