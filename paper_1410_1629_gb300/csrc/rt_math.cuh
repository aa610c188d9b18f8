// Double-precision exponential and logarithm of the forced-scattering
// inversion (Sect. 1) and of the dust's emission, written for a device whose
// FP64 pipe issues one warp instruction per 16 cycles of an SM, whatever its
// active lanes: 1 - exp(-x) and exp(x) - 1 in 11 FP64 instructions, -ln(1 - v)
// in 14, table-driven (P. T. P. Tang, "Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic", ACM TOMS 15, 1989,
// and "... of the logarithm function ...", ACM TOMS 16, 1990).  The tables hold
// the leading bits of their values apart, so that the largest part of a result is
// exact and the rest, which is small against it, carries the roundings.  Where
// the result is as small as the reduced argument, the argument is not reduced.
// The range reduction, the remainders of constants and the high-order terms of
// the series use integer and FP32 instructions; where an FP32 value enters an
// FP64 sum its weight there is below 2^-32, so its rounding stays below 2^-56 of
// the result.
//
// Against 113-bit arithmetic (2e5 arguments in each of 17 ranges, on the
// device): 1 - exp(-x) within 0.55 ulp, exp(x) - 1 within 0.56, -ln(1 - v) within
// 0.58, their rms errors within 0.2 % of those of the correctly rounded values
// (0.289 ulp); the CUDA library's expm1 and log1p: 1.15 and 1.49 ulp, rms up to
// 0.325 and 0.387, in no range more than 0.1 % below these.  Measured with the
// library's functions in their place (time over that with these): 256 batched
// models (110 ms) 1.056, a 48^3 fit with an absorption target (20.3 ms) 1.070,
// dust temperatures and emission (7.0 ms) 1.37, 1e4 packets of a 32^3 cube (0.38
// ms) 1.04, a taped forward launch with its adjoint (32.7 ms) 0.99.  (A form that
// kept the rounding errors of the leading sums by two-sums, 15, 16 and 18
// instructions: 0.53 ulp, a replayed adjoint of 1e7 packets 414 against 392 ms.)
//
// The file compiles as CUDA (device functions) and as plain C++ (for tests).
#pragma once

#ifdef __CUDACC__
#define RT_FN __device__ __forceinline__
#define RT_TABLE static __device__ const
#else
#include <cmath>
#include <cstdint>
#include <cstring>
#define RT_FN static inline
#define RT_TABLE static const
#endif

namespace rtk {

#ifdef __CUDACC__
RT_FN long long bits_of(double v) { return __double_as_longlong(v); }
RT_FN double double_of(long long b) { return __longlong_as_double(b); }
RT_FN unsigned bits_of(float v) { return __float_as_uint(v); }
RT_FN float float_of(unsigned b) { return __uint_as_float(b); }
#else
RT_FN long long bits_of(double v) { long long b; std::memcpy(&b, &v, 8); return b; }
RT_FN double double_of(long long b) { double v; std::memcpy(&v, &b, 8); return v; }
RT_FN unsigned bits_of(float v) { unsigned b; std::memcpy(&b, &v, 4); return b; }
RT_FN float float_of(unsigned b) { float v; std::memcpy(&v, &b, 4); return v; }
#endif

// Exact widening of an FP32 value to FP64 with integer operations (rebias the
// exponent by 1023 - 127 and shift the significand), off the FP64 pipe.
// Subnormal and non-finite inputs take the ordinary conversion.
RT_FN double widen(float f) {
  const unsigned u = bits_of(f);
  const unsigned e = u & 0x7f800000u;
  if (e == 0u || e == 0x7f800000u) {
    if ((u & 0x7fffffffu) != 0u) return (double)f;
    return double_of((long long)((unsigned long long)u << 32));  // a zero keeps its sign
  }
  const unsigned hi = (((u & 0x7fffffffu) >> 3) + 0x38000000u) | (u & 0x80000000u);
  return double_of((long long)(((unsigned long long)hi << 32) | (unsigned long long)(u << 29)));
}

// FP64 to FP32 by cutting the significand to 24 bits, with integer
// operations; values outside the normal FP32 range take the ordinary
// conversion (a zero stays one).
RT_FN float cut(double v) {
  const long long b = bits_of(v);
  const int be = (int)((b >> 52) & 0x7ff);
  const unsigned top = (unsigned)((unsigned long long)b >> 32);
  if (be < 1023 - 126 || be > 1023 + 127) return (b << 1) == 0 ? float_of(top & 0x80000000u) : (float)v;
  return float_of((top & 0x80000000u) | ((unsigned)(be - 896) << 23) | ((unsigned)(b >> 29) & 0x7fffffu));
}

// 2^(-j/128), to 13 bits, and the remainder: hi - 2^(-j/128); in kExpUpTable
// 2^(j/128), to 13 bits, and the remainder 2^(j/128) - hi
struct ExpEntry {
  double t, hi, lo;
};
// a reciprocal of the middle of [1/2 + j/256, 1/2 + (j + 1)/256] to 13 bits
// (1 for the last three intervals, and for the one before them a value that
// keeps its |r| below 2^-9 wherever the result is below 2^-6), the same less one,
// and its logarithm to a multiple of 2^-40 and its remainder
struct alignas(16) LogEntry {
  double rc, c, ln;
  float ln_lo;
};

// ln 2 / 128 as a double and its remainder, ln 2 to a multiple of 2^-40 (sums of
// its multiples and of table entries are exact) and its remainder
constexpr double kLn2Over128 = 0x1.62e42fefa39efp-8;
constexpr float kLn2Over128Lo = 0x1.abc9e3b39803fp-63;
constexpr double kLn2 = 0x1.62e42fefa4p-1;
constexpr float kLn2Lo = -0x1.8432a1b0e2634p-43;
RT_TABLE ExpEntry kExpTable[128] = {
    {0x1.0000000000000p+0, 0x1.0p+0, 0x0.0p+0},
    {0x1.fd3c22b8f71f1p-1, 0x1.fd4p-1, 0x1.eea3847077b45p-16},
    {0x1.fa7c1819e90d8p-1, 0x1.fa8p-1, 0x1.f3f30b793e8b8p-16},
    {0x1.f7bfdad9cbe14p-1, 0x1.f7cp-1, 0x1.2931a0f63b762p-20},
    {0x1.f50765b6e4540p-1, 0x1.f5p-1, -0x1.d96db915019d4p-15},
    {0x1.f252b376bba97p-1, 0x1.f25p-1, -0x1.59bb5dd4ba743p-16},
    {0x1.efa1bee615a27p-1, 0x1.efap-1, -0x1.bee615a277720p-17},
    {0x1.ecf482d8e67f1p-1, 0x1.ecfp-1, -0x1.20b6399fc236cp-15},
    {0x1.ea4afa2a490dap-1, 0x1.ea5p-1, 0x1.41756dbc99e9cp-15},
    {0x1.e7a51fbc74c83p-1, 0x1.e7ap-1, -0x1.47ef1d320d2d5p-15},
    {0x1.e502ee78b3ff6p-1, 0x1.e5p-1, -0x1.773c59ffb139fp-16},
    {0x1.e264614f5a129p-1, 0x1.e26p-1, -0x1.1853d684a284ap-15},
    {0x1.dfc97337b9b5fp-1, 0x1.dfdp-1, 0x1.a3321192851a6p-15},
    {0x1.dd321f301b460p-1, 0x1.dd3p-1, -0x1.0f980da3025b5p-16},
    {0x1.da9e603db3285p-1, 0x1.daap-1, 0x1.9fc24cd7a8f74p-17},
    {0x1.d80e316c98398p-1, 0x1.d81p-1, 0x1.ce9367c68447bp-17},
    {0x1.d5818dcfba487p-1, 0x1.d58p-1, -0x1.8dcfba48725dap-17},
    {0x1.d2f87080d89f2p-1, 0x1.d3p-1, 0x1.e3dfc9d839d48p-15},
    {0x1.d072d4a07897cp-1, 0x1.d07p-1, -0x1.6a503c4bdc688p-16},
    {0x1.cdf0b555dc3fap-1, 0x1.cdfp-1, -0x1.6aabb87f3889fp-18},
    {0x1.cb720dcef9069p-1, 0x1.cb7p-1, -0x1.06e77c8348a82p-16},
    {0x1.c8f6d9406e7b5p-1, 0x1.c8fp-1, -0x1.b6501b9ed446bp-15},
    {0x1.c67f12e57d14bp-1, 0x1.c68p-1, 0x1.da3505d696bbep-18},
    {0x1.c40ab5fffd07ap-1, 0x1.c41p-1, 0x1.528000be164bbp-15},
    {0x1.c199bdd85529cp-1, 0x1.c1ap-1, 0x1.9089eab58f778p-15},
    {0x1.bf2c25bd71e09p-1, 0x1.bf3p-1, 0x1.ed21470fbbdfcp-16},
    {0x1.bcc1e904bc1d2p-1, 0x1.bccp-1, -0x1.e904bc1d2247cp-17},
    {0x1.ba5b030a1064ap-1, 0x1.ba6p-1, 0x1.3f3d7be6d9efdp-15},
    {0x1.b7f76f2fb5e47p-1, 0x1.b7fp-1, -0x1.dbcbed791baaap-15},
    {0x1.b59728de5593ap-1, 0x1.b59p-1, -0x1.ca379564e638ep-15},
    {0x1.b33a2b84f15fbp-1, 0x1.b34p-1, 0x1.751ec3a814250p-15},
    {0x1.b0e07298db666p-1, 0x1.b0ep-1, -0x1.ca636d9964211p-19},
    {0x1.ae89f995ad3adp-1, 0x1.ae9p-1, 0x1.819a94b14a85ep-15},
    {0x1.ac36bbfd3f37ap-1, 0x1.ac3p-1, -0x1.aeff4fcde7037p-15},
    {0x1.a9e6b5579fdbfp-1, 0x1.a9ep-1, -0x1.ad55e7f6fd0fbp-15},
    {0x1.a799e1330b358p-1, 0x1.a7ap-1, 0x1.87b33d329e435p-15},
    {0x1.a5503b23e255dp-1, 0x1.a55p-1, -0x1.d91f12ae45a12p-20},
    {0x1.a309bec4a2d33p-1, 0x1.a31p-1, 0x1.904ed74b329d0p-15},
    {0x1.a0c667b5de565p-1, 0x1.a0cp-1, -0x1.99ed779592ca7p-15},
    {0x1.9e86319e32323p-1, 0x1.9e8p-1, -0x1.8c678c8c8c609p-15},
    {0x1.9c49182a3f090p-1, 0x1.9c5p-1, 0x1.b9f5703dbf8e1p-15},
    {0x1.9a0f170ca07bap-1, 0x1.9a1p-1, 0x1.d1e6bf08c8b9ep-18},
    {0x1.97d829fde4e50p-1, 0x1.97ep-1, 0x1.f58086c6c1d18p-15},
    {0x1.95a44cbc8520fp-1, 0x1.95ap-1, -0x1.132f21483ba6dp-15},
    {0x1.93737b0cdc5e5p-1, 0x1.937p-1, -0x1.bd866e2f27a28p-16},
    {0x1.9145b0b91ffc6p-1, 0x1.914p-1, -0x1.6c2e47ff1622ap-15},
    {0x1.8f1ae99157736p-1, 0x1.8f2p-1, 0x1.459baa232751ap-15},
    {0x1.8cf3216b5448cp-1, 0x1.8cfp-1, -0x1.90b5aa245f795p-16},
    {0x1.8ace5422aa0dbp-1, 0x1.8adp-1, 0x1.abdd55f24a458p-17},
    {0x1.88ac7d98a6699p-1, 0x1.88bp-1, 0x1.c133accb34cd6p-16},
    {0x1.868d99b4492edp-1, 0x1.869p-1, 0x1.3325db689bf8ep-16},
    {0x1.8471a4623c7adp-1, 0x1.847p-1, -0x1.a4623c7acce53p-17},
    {0x1.82589994cce13p-1, 0x1.826p-1, 0x1.d99accc7b5d4cp-15},
    {0x1.80427543e1a12p-1, 0x1.804p-1, -0x1.3aa1f0d08db07p-16},
    {0x1.7e2f336cf4e62p-1, 0x1.7e3p-1, 0x1.99261633bdf46p-18},
    {0x1.7c1ed0130c132p-1, 0x1.7c2p-1, 0x1.2fecf3ecd83b7p-17},
    {0x1.7a11473eb0187p-1, 0x1.7a1p-1, -0x1.473eb0186d7d5p-17},
    {0x1.780694fde5d3fp-1, 0x1.78p-1, -0x1.a53f7974fd867p-15},
    {0x1.75feb564267c9p-1, 0x1.76p-1, 0x1.4a9bd98374091p-17},
    {0x1.73f9a48a58174p-1, 0x1.74p-1, 0x1.96dd69fa310a9p-15},
    {0x1.71f75e8ec5f74p-1, 0x1.71fp-1, -0x1.d7a3b17dcf749p-15},
    {0x1.6ff7df9519484p-1, 0x1.6ffp-1, -0x1.f7e546520f3e2p-15},
    {0x1.6dfb23c651a2fp-1, 0x1.6ep-1, 0x1.370e6b9744378p-15},
    {0x1.6c012750bdabfp-1, 0x1.6cp-1, -0x1.2750bdabeed77p-17},
    {0x1.6a09e667f3bcdp-1, 0x1.6a1p-1, 0x1.86660310cdbddp-15},
    {0x1.68155d44ca973p-1, 0x1.681p-1, -0x1.575132a5cc207p-15},
    {0x1.6623882552225p-1, 0x1.662p-1, -0x1.c412a91124894p-16},
    {0x1.6434634ccc320p-1, 0x1.643p-1, -0x1.18d3330c7f1dcp-15},
    {0x1.6247eb03a5585p-1, 0x1.624p-1, -0x1.fac0e95612c7cp-15},
    {0x1.605e1b976dc09p-1, 0x1.606p-1, 0x1.e468923f74f89p-17},
    {0x1.5e76f15ad2148p-1, 0x1.5e7p-1, -0x1.bc56b48521ba7p-15},
    {0x1.5c9268a5946b7p-1, 0x1.5c9p-1, -0x1.3452ca35b80e2p-16},
    {0x1.5ab07dd485429p-1, 0x1.5abp-1, -0x1.f752150a56325p-19},
    {0x1.58d12d497c7fdp-1, 0x1.58dp-1, -0x1.2d497c7fd252cp-17},
    {0x1.56f4736b527dap-1, 0x1.56fp-1, -0x1.1cdad49f699bbp-15},
    {0x1.551a4ca5d920fp-1, 0x1.552p-1, 0x1.6cd689b7c4eb4p-15},
    {0x1.5342b569d4f82p-1, 0x1.534p-1, -0x1.5ab4ea7c0ef85p-16},
    {0x1.516daa2cf6642p-1, 0x1.517p-1, 0x1.2ae984cdf1f77p-16},
    {0x1.4f9b2769d2ca7p-1, 0x1.4fap-1, 0x1.36258b4d654b3p-15},
    {0x1.4dcb299fddd0dp-1, 0x1.4ddp-1, 0x1.3598088bca713p-15},
    {0x1.4bfdad5362a27p-1, 0x1.4cp-1, 0x1.29564eaec715ep-16},
    {0x1.4a32af0d7d3dep-1, 0x1.4a3p-1, -0x1.5786be9ef3397p-16},
    {0x1.486a2b5c13cd0p-1, 0x1.487p-1, 0x1.7528fb0cbfb10p-15},
    {0x1.46a41ed1d0057p-1, 0x1.46ap-1, -0x1.07b474015dc94p-15},
    {0x1.44e086061892dp-1, 0x1.44ep-1, -0x1.0c0c3125a0627p-18},
    {0x1.431f5d950a897p-1, 0x1.432p-1, 0x1.44d5eaed2471fp-18},
    {0x1.4160a21f72e2ap-1, 0x1.416p-1, -0x1.443ee5c53f086p-18},
    {0x1.3fa4504ac801cp-1, 0x1.3fap-1, -0x1.1412b2006e830p-15},
    {0x1.3dea64c123422p-1, 0x1.3dfp-1, 0x1.66cfb72f77293p-15},
    {0x1.3c32dc313a8e5p-1, 0x1.3c3p-1, -0x1.6e189d4724200p-16},
    {0x1.3a7db34e59ff7p-1, 0x1.3a8p-1, 0x1.2658d30048af2p-16},
    {0x1.38cae6d05d866p-1, 0x1.38dp-1, 0x1.464be89e69e96p-15},
    {0x1.371a7373aa9cbp-1, 0x1.372p-1, 0x1.63231558d563bp-15},
    {0x1.356c55f929ff1p-1, 0x1.357p-1, 0x1.d5036b0079b5dp-16},
    {0x1.33c08b26416ffp-1, 0x1.33cp-1, -0x1.164c82dfe9939p-18},
    {0x1.32170fc4cd831p-1, 0x1.321p-1, -0x1.c3f13360c4d4ep-15},
    {0x1.306fe0a31b715p-1, 0x1.307p-1, 0x1.f5ce48ead2173p-21},
    {0x1.2ecafa93e2f56p-1, 0x1.2edp-1, 0x1.415b0742a7b8dp-15},
    {0x1.2d285a6e4030bp-1, 0x1.2d3p-1, 0x1.e9646ff3d2ffep-15},
    {0x1.2b87fd0dad990p-1, 0x1.2b8p-1, -0x1.ff436b663ff78p-15},
    {0x1.29e9df51fdee1p-1, 0x1.29fp-1, 0x1.882b80847b4f7p-15},
    {0x1.284dfe1f56381p-1, 0x1.285p-1, 0x1.00f054e3fb498p-16},
    {0x1.26b4565e27cddp-1, 0x1.26bp-1, -0x1.159789f37495fp-15},
    {0x1.251ce4fb2a63fp-1, 0x1.252p-1, 0x1.8d826ace0653fp-16},
    {0x1.2387a6e756238p-1, 0x1.238p-1, -0x1.e9b9d588e19b0p-15},
    {0x1.21f49917ddc96p-1, 0x1.21fp-1, -0x1.2645f77258955p-15},
    {0x1.2063b88628cd6p-1, 0x1.206p-1, -0x1.dc431466b1dc7p-16},
    {0x1.1ed5022fcd91dp-1, 0x1.1edp-1, -0x1.408bf36472e20p-15},
    {0x1.1d4873168b9aap-1, 0x1.1d5p-1, 0x1.e33a5d19561ffp-15},
    {0x1.1bbe084045cd4p-1, 0x1.1bcp-1, 0x1.f7bfba32c654ep-17},
    {0x1.1a35beb6fcb75p-1, 0x1.1a3p-1, -0x1.6fadbf2dd4f2ep-15},
    {0x1.18af9388c8deap-1, 0x1.18bp-1, 0x1.b1dcdc8591102p-19},
    {0x1.172b83c7d517bp-1, 0x1.173p-1, 0x1.1f0e0aba148c8p-15},
    {0x1.15a98c8a58e51p-1, 0x1.15bp-1, 0x1.9cdd69c6bb6e0p-15},
    {0x1.1429aaea92de0p-1, 0x1.143p-1, 0x1.95455b4881330p-15},
    {0x1.12abdc06c31ccp-1, 0x1.12bp-1, 0x1.08fe4f38d011bp-15},
    {0x1.11301d0125b51p-1, 0x1.113p-1, -0x1.d0125b50a4ebcp-21},
    {0x1.0fb66affed31bp-1, 0x1.0fbp-1, -0x1.9abffb4c6bc8dp-15},
    {0x1.0e3ec32d3d1a2p-1, 0x1.0e4p-1, 0x1.3cd2c2e5dfdf9p-17},
    {0x1.0cc922b7247f7p-1, 0x1.0cdp-1, 0x1.b75236e022fe1p-15},
    {0x1.0b5586cf9890fp-1, 0x1.0b5p-1, -0x1.61b3e6243d8a6p-15},
    {0x1.09e3ecac6f383p-1, 0x1.09ep-1, -0x1.f656379c1a291p-16},
    {0x1.0874518759bc8p-1, 0x1.087p-1, -0x1.1461d66f20231p-15},
    {0x1.0706b29ddf6dep-1, 0x1.07p-1, -0x1.aca777db771b7p-15},
    {0x1.059b0d3158574p-1, 0x1.05ap-1, 0x1.3cb3a9ea2f146p-15},
    {0x1.04315e86e7f85p-1, 0x1.043p-1, -0x1.5e86e7f84bd74p-17},
    {0x1.02c9a3e778061p-1, 0x1.02dp-1, 0x1.970621fe7c464p-15},
    {0x1.0163da9fb3335p-1, 0x1.016p-1, -0x1.ed4fd999ab6c2p-16},
};
RT_TABLE ExpEntry kExpUpTable[128] = {
    {0x1.0000000000000p+0, 0x1.0p+0, 0x0.0p+0},
    {0x1.0163da9fb3335p+0, 0x1.016p+0, 0x1.ed4fd999ab6c2p-15},
    {0x1.02c9a3e778061p+0, 0x1.02c8p+0, 0x1.a3e778060ee6fp-16},
    {0x1.04315e86e7f85p+0, 0x1.043p+0, 0x1.5e86e7f84bd74p-16},
    {0x1.059b0d3158574p+0, 0x1.0598p+0, 0x1.8698ac2ba1d74p-15},
    {0x1.0706b29ddf6dep+0, 0x1.0708p+0, -0x1.4d62209223924p-16},
    {0x1.0874518759bc8p+0, 0x1.0878p+0, -0x1.d73c5321bfb9ep-15},
    {0x1.09e3ecac6f383p+0, 0x1.09ep+0, 0x1.f656379c1a291p-15},
    {0x1.0b5586cf9890fp+0, 0x1.0b58p+0, -0x1.3c9833b784eb4p-15},
    {0x1.0cc922b7247f7p+0, 0x1.0cc8p+0, 0x1.22b7247f7407bp-16},
    {0x1.0e3ec32d3d1a2p+0, 0x1.0e4p+0, -0x1.3cd2c2e5dfdf9p-16},
    {0x1.0fb66affed31bp+0, 0x1.0fb8p+0, -0x1.950012ce50dcep-16},
    {0x1.11301d0125b51p+0, 0x1.113p+0, 0x1.d0125b50a4ebcp-20},
    {0x1.12abdc06c31ccp+0, 0x1.12a8p+0, 0x1.ee03618e5fdc9p-15},
    {0x1.1429aaea92de0p+0, 0x1.1428p+0, 0x1.aaea92ddfb341p-16},
    {0x1.15a98c8a58e51p+0, 0x1.15a8p+0, 0x1.8c8a58e512481p-16},
    {0x1.172b83c7d517bp+0, 0x1.1728p+0, 0x1.c1e3ea8bd6e70p-15},
    {0x1.18af9388c8deap+0, 0x1.18bp+0, -0x1.b1dcdc8591102p-18},
    {0x1.1a35beb6fcb75p+0, 0x1.1a38p+0, -0x1.20a481a4561a5p-15},
    {0x1.1bbe084045cd4p+0, 0x1.1bcp+0, -0x1.f7bfba32c654ep-16},
    {0x1.1d4873168b9aap+0, 0x1.1d48p+0, 0x1.cc5a2e6a9e017p-18},
    {0x1.1ed5022fcd91dp+0, 0x1.1ed8p+0, -0x1.7ee819371a3bfp-15},
    {0x1.2063b88628cd6p+0, 0x1.206p+0, 0x1.dc431466b1dc7p-15},
    {0x1.21f49917ddc96p+0, 0x1.21f8p+0, -0x1.b374111b4ed57p-15},
    {0x1.2387a6e756238p+0, 0x1.2388p+0, -0x1.6462a771e64f8p-18},
    {0x1.251ce4fb2a63fp+0, 0x1.252p+0, -0x1.8d826ace0653fp-15},
    {0x1.26b4565e27cddp+0, 0x1.26b8p+0, -0x1.d4d0ec1916d43p-15},
    {0x1.284dfe1f56381p+0, 0x1.285p+0, -0x1.00f054e3fb498p-15},
    {0x1.29e9df51fdee1p+0, 0x1.29e8p+0, 0x1.df51fdee12c26p-16},
    {0x1.2b87fd0dad990p+0, 0x1.2b88p+0, -0x1.79293380110aep-23},
    {0x1.2d285a6e4030bp+0, 0x1.2d28p+0, 0x1.69b900c2d0024p-18},
    {0x1.2ecafa93e2f56p+0, 0x1.2ec8p+0, 0x1.7d49f17ab08e5p-15},
    {0x1.306fe0a31b715p+0, 0x1.307p+0, -0x1.f5ce48ead2173p-20},
    {0x1.32170fc4cd831p+0, 0x1.3218p+0, -0x1.e07664f9d958cp-17},
    {0x1.33c08b26416ffp+0, 0x1.33cp+0, 0x1.164c82dfe9939p-17},
    {0x1.356c55f929ff1p+0, 0x1.357p+0, -0x1.d5036b0079b5dp-15},
    {0x1.371a7373aa9cbp+0, 0x1.3718p+0, 0x1.39b9d54e5538ap-15},
    {0x1.38cae6d05d866p+0, 0x1.38c8p+0, 0x1.73682ec32c2d5p-15},
    {0x1.3a7db34e59ff7p+0, 0x1.3a8p+0, -0x1.2658d30048af2p-15},
    {0x1.3c32dc313a8e5p+0, 0x1.3c3p+0, 0x1.6e189d4724200p-15},
    {0x1.3dea64c123422p+0, 0x1.3de8p+0, 0x1.326091a111adap-15},
    {0x1.3fa4504ac801cp+0, 0x1.3fa8p+0, -0x1.d7da9bff22fa0p-15},
    {0x1.4160a21f72e2ap+0, 0x1.416p+0, 0x1.443ee5c53f086p-17},
    {0x1.431f5d950a897p+0, 0x1.432p+0, -0x1.44d5eaed2471fp-17},
    {0x1.44e086061892dp+0, 0x1.44ep+0, 0x1.0c0c3125a0627p-17},
    {0x1.46a41ed1d0057p+0, 0x1.46a8p+0, -0x1.f09717fd446d7p-15},
    {0x1.486a2b5c13cd0p+0, 0x1.4868p+0, 0x1.15ae09e6809e1p-15},
    {0x1.4a32af0d7d3dep+0, 0x1.4a3p+0, 0x1.5786be9ef3397p-15},
    {0x1.4bfdad5362a27p+0, 0x1.4cp+0, -0x1.29564eaec715ep-15},
    {0x1.4dcb299fddd0dp+0, 0x1.4dc8p+0, 0x1.94cfeee86b1dap-15},
    {0x1.4f9b2769d2ca7p+0, 0x1.4f98p+0, 0x1.93b4e9653569ap-15},
    {0x1.516daa2cf6642p+0, 0x1.517p+0, -0x1.2ae984cdf1f77p-15},
    {0x1.5342b569d4f82p+0, 0x1.534p+0, 0x1.5ab4ea7c0ef85p-15},
    {0x1.551a4ca5d920fp+0, 0x1.5518p+0, 0x1.2652ec9076297p-15},
    {0x1.56f4736b527dap+0, 0x1.56f8p+0, -0x1.c64a56c12cc8ap-15},
    {0x1.58d12d497c7fdp+0, 0x1.58dp+0, 0x1.2d497c7fd252cp-16},
    {0x1.5ab07dd485429p+0, 0x1.5abp+0, 0x1.f752150a56325p-18},
    {0x1.5c9268a5946b7p+0, 0x1.5c9p+0, 0x1.3452ca35b80e2p-15},
    {0x1.5e76f15ad2148p+0, 0x1.5e78p+0, -0x1.0ea52deb79164p-16},
    {0x1.605e1b976dc09p+0, 0x1.606p+0, -0x1.e468923f74f89p-16},
    {0x1.6247eb03a5585p+0, 0x1.6248p+0, -0x1.4fc5aa7b4e0f0p-20},
    {0x1.6434634ccc320p+0, 0x1.6438p+0, -0x1.ce5999e701c48p-15},
    {0x1.6623882552225p+0, 0x1.662p+0, 0x1.c412a91124894p-15},
    {0x1.68155d44ca973p+0, 0x1.6818p+0, -0x1.515d9ab467bf2p-15},
    {0x1.6a09e667f3bcdp+0, 0x1.6a08p+0, 0x1.e667f3bcc908bp-16},
    {0x1.6c012750bdabfp+0, 0x1.6cp+0, 0x1.2750bdabeed77p-16},
    {0x1.6dfb23c651a2fp+0, 0x1.6df8p+0, 0x1.91e328d177910p-15},
    {0x1.6ff7df9519484p+0, 0x1.6ff8p+0, -0x1.035735be183c1p-19},
    {0x1.71f75e8ec5f74p+0, 0x1.71f8p+0, -0x1.42e27411845b9p-17},
    {0x1.73f9a48a58174p+0, 0x1.73f8p+0, 0x1.a48a58173bd5dp-16},
    {0x1.75feb564267c9p+0, 0x1.76p+0, -0x1.4a9bd98374091p-16},
    {0x1.780694fde5d3fp+0, 0x1.7808p+0, -0x1.6b021a2c09e65p-16},
    {0x1.7a11473eb0187p+0, 0x1.7a1p+0, 0x1.473eb0186d7d5p-16},
    {0x1.7c1ed0130c132p+0, 0x1.7c2p+0, -0x1.2fecf3ecd83b7p-16},
    {0x1.7e2f336cf4e62p+0, 0x1.7e3p+0, -0x1.99261633bdf46p-17},
    {0x1.80427543e1a12p+0, 0x1.804p+0, 0x1.3aa1f0d08db07p-15},
    {0x1.82589994cce13p+0, 0x1.8258p+0, 0x1.332999c25159fp-17},
    {0x1.8471a4623c7adp+0, 0x1.847p+0, 0x1.a4623c7acce53p-16},
    {0x1.868d99b4492edp+0, 0x1.869p+0, -0x1.3325db689bf8ep-15},
    {0x1.88ac7d98a6699p+0, 0x1.88bp+0, -0x1.c133accb34cd6p-15},
    {0x1.8ace5422aa0dbp+0, 0x1.8adp+0, -0x1.abdd55f24a458p-16},
    {0x1.8cf3216b5448cp+0, 0x1.8cfp+0, 0x1.90b5aa245f795p-15},
    {0x1.8f1ae99157736p+0, 0x1.8f18p+0, 0x1.74c8abb9b15ccp-15},
    {0x1.9145b0b91ffc6p+0, 0x1.9148p+0, -0x1.27a37001d3badp-15},
    {0x1.93737b0cdc5e5p+0, 0x1.937p+0, 0x1.bd866e2f27a28p-15},
    {0x1.95a44cbc8520fp+0, 0x1.95a8p+0, -0x1.d9a1bd6f88b26p-15},
    {0x1.97d829fde4e50p+0, 0x1.97d8p+0, 0x1.4fef2727c5cf5p-19},
    {0x1.9a0f170ca07bap+0, 0x1.9a1p+0, -0x1.d1e6bf08c8b9ep-17},
    {0x1.9c49182a3f090p+0, 0x1.9c48p+0, 0x1.182a3f0901c7cp-16},
    {0x1.9e86319e32323p+0, 0x1.9e88p+0, -0x1.ce61cdcdce7dbp-16},
    {0x1.a0c667b5de565p+0, 0x1.a0c8p+0, -0x1.984a21a9b4d65p-16},
    {0x1.a309bec4a2d33p+0, 0x1.a308p+0, 0x1.bec4a2d3358c1p-16},
    {0x1.a5503b23e255dp+0, 0x1.a55p+0, 0x1.d91f12ae45a12p-19},
    {0x1.a799e1330b358p+0, 0x1.a798p+0, 0x1.e1330b3586f2ep-16},
    {0x1.a9e6b5579fdbfp+0, 0x1.a9e8p+0, -0x1.4aa860240bc15p-16},
    {0x1.ac36bbfd3f37ap+0, 0x1.ac38p+0, -0x1.4402c0c863f24p-16},
    {0x1.ae89f995ad3adp+0, 0x1.ae88p+0, 0x1.f995ad3ad5e87p-16},
    {0x1.b0e07298db666p+0, 0x1.b0ep+0, 0x1.ca636d9964211p-18},
    {0x1.b33a2b84f15fbp+0, 0x1.b338p+0, 0x1.15c278afd7b60p-15},
    {0x1.b59728de5593ap+0, 0x1.b598p+0, -0x1.ae4354d8ce38fp-17},
    {0x1.b7f76f2fb5e47p+0, 0x1.b7f8p+0, -0x1.21a0943722ab1p-17},
    {0x1.ba5b030a1064ap+0, 0x1.ba58p+0, 0x1.818508324c206p-15},
    {0x1.bcc1e904bc1d2p+0, 0x1.bccp+0, 0x1.e904bc1d2247cp-16},
    {0x1.bf2c25bd71e09p+0, 0x1.bf3p+0, -0x1.ed21470fbbdfcp-15},
    {0x1.c199bdd85529cp+0, 0x1.c198p+0, 0x1.bdd85529c2221p-16},
    {0x1.c40ab5fffd07ap+0, 0x1.c408p+0, 0x1.5afffe83d368ap-15},
    {0x1.c67f12e57d14bp+0, 0x1.c68p+0, -0x1.da3505d696bbep-17},
    {0x1.c8f6d9406e7b5p+0, 0x1.c8f8p+0, -0x1.26bf9184aee53p-16},
    {0x1.cb720dcef9069p+0, 0x1.cb7p+0, 0x1.06e77c8348a82p-15},
    {0x1.cdf0b555dc3fap+0, 0x1.cdfp+0, 0x1.6aabb87f3889fp-17},
    {0x1.d072d4a07897cp+0, 0x1.d07p+0, 0x1.6a503c4bdc688p-15},
    {0x1.d2f87080d89f2p+0, 0x1.d2f8p+0, 0x1.c203627c62b78p-18},
    {0x1.d5818dcfba487p+0, 0x1.d58p+0, 0x1.8dcfba48725dap-16},
    {0x1.d80e316c98398p+0, 0x1.d81p+0, -0x1.ce9367c68447bp-16},
    {0x1.da9e603db3285p+0, 0x1.daap+0, -0x1.9fc24cd7a8f74p-16},
    {0x1.dd321f301b460p+0, 0x1.dd3p+0, 0x1.0f980da3025b5p-15},
    {0x1.dfc97337b9b5fp+0, 0x1.dfc8p+0, 0x1.7337b9b5eb969p-16},
    {0x1.e264614f5a129p+0, 0x1.e268p+0, -0x1.cf5852f6baf6cp-15},
    {0x1.e502ee78b3ff6p+0, 0x1.e5p+0, 0x1.773c59ffb139fp-15},
    {0x1.e7a51fbc74c83p+0, 0x1.e7a8p+0, -0x1.7021c59be5a56p-15},
    {0x1.ea4afa2a490dap+0, 0x1.ea48p+0, 0x1.7d152486cc2c8p-15},
    {0x1.ecf482d8e67f1p+0, 0x1.ecf8p+0, -0x1.be938cc07b928p-15},
    {0x1.efa1bee615a27p+0, 0x1.efap+0, 0x1.bee615a277720p-16},
    {0x1.f252b376bba97p+0, 0x1.f25p+0, 0x1.59bb5dd4ba743p-15},
    {0x1.f50765b6e4540p+0, 0x1.f508p+0, -0x1.34923757f3161p-17},
    {0x1.f7bfdad9cbe14p+0, 0x1.f7cp+0, -0x1.2931a0f63b762p-19},
    {0x1.fa7c1819e90d8p+0, 0x1.fa8p+0, -0x1.f3f30b793e8b8p-15},
    {0x1.fd3c22b8f71f1p+0, 0x1.fd4p+0, -0x1.eea3847077b45p-15},
};
RT_TABLE LogEntry kLogTable[128] = {
    {0x1.fep+0, 0x1.fcp-1, 0x1.60e32f4478p-1, 0x1.1b195p-42f},
    {0x1.fa1p+0, 0x1.f42p-1, 0x1.5ceb4e16f2p-1, -0x1.c852cep-42f},
    {0x1.f63p+0, 0x1.ec6p-1, 0x1.58fbcdcdb8p-1, 0x1.83e928p-46f},
    {0x1.f26p+0, 0x1.e4cp-1, 0x1.5514efdbb2p-1, 0x1.ac591ep-42f},
    {0x1.eeap+0, 0x1.dd4p-1, 0x1.5136f66336p-1, 0x1.92d78ap-42f},
    {0x1.eafp+0, 0x1.d5ep-1, 0x1.4d62242e94p-1, 0x1.53f70ep-42f},
    {0x1.e74p+0, 0x1.ce8p-1, 0x1.4985ece016p-1, 0x1.752b0ap-42f},
    {0x1.e3bp+0, 0x1.c76p-1, 0x1.45c414576ap-1, 0x1.d0daa2p-43f},
    {0x1.e02p+0, 0x1.c04p-1, 0x1.41fb1f835p-1, 0x1.adbb58p-42f},
    {0x1.dcap+0, 0x1.b94p-1, 0x1.3e3c23918ep-1, 0x1.db156cp-43f},
    {0x1.d93p+0, 0x1.b26p-1, 0x1.3a8766721ep-1, 0x1.a248e8p-42f},
    {0x1.d5dp+0, 0x1.abap-1, 0x1.36dd2e951ep-1, 0x1.998158p-42f},
    {0x1.d27p+0, 0x1.a4ep-1, 0x1.332c331256p-1, -0x1.9214eap-42f},
    {0x1.cf2p+0, 0x1.9e4p-1, 0x1.2f860b54dap-1, 0x1.2a7ab6p-45f},
    {0x1.cbep+0, 0x1.97cp-1, 0x1.2beaff89b8p-1, 0x1.3d7ea6p-42f},
    {0x1.c8bp+0, 0x1.916p-1, 0x1.285b5840fcp-1, -0x1.2caffep-46f},
    {0x1.c59p+0, 0x1.8b2p-1, 0x1.24d75e6134p-1, 0x1.7b622p-42f},
    {0x1.c27p+0, 0x1.84ep-1, 0x1.214d2b9d6cp-1, 0x1.6e49e8p-47f},
    {0x1.bf6p+0, 0x1.7ecp-1, 0x1.1dcef9ca56p-1, -0x1.8bf0bcp-44f},
    {0x1.bc5p+0, 0x1.78ap-1, 0x1.1a4aa38b78p-1, -0x1.874f36p-46f},
    {0x1.b95p+0, 0x1.72ap-1, 0x1.16d2a38aep-1, -0x1.426fe4p-42f},
    {0x1.b66p+0, 0x1.6ccp-1, 0x1.1367452adp-1, -0x1.e39c78p-43f},
    {0x1.b37p+0, 0x1.66ep-1, 0x1.0ff6041a2cp-1, -0x1.482edp-47f},
    {0x1.b09p+0, 0x1.612p-1, 0x1.0c91bc8186p-1, 0x1.9d086cp-42f},
    {0x1.adcp+0, 0x1.5b8p-1, 0x1.093abae514p-1, 0x1.d44462p-42f},
    {0x1.aafp+0, 0x1.55ep-1, 0x1.05de1c197p-1, 0x1.fe0386p-43f},
    {0x1.a83p+0, 0x1.506p-1, 0x1.028f1d69a6p-1, -0x1.cd9956p-53f},
    {0x1.a57p+0, 0x1.4aep-1, 0x1.fe7538ded4p-2, -0x1.805d36p-43f},
    {0x1.a2cp+0, 0x1.458p-1, 0x1.f7e82e661p-2, -0x1.47d962p-43f},
    {0x1.a02p+0, 0x1.404p-1, 0x1.f177b7dfd4p-2, 0x1.feb26cp-48f},
    {0x1.9d8p+0, 0x1.3bp-1, 0x1.eafcd2cea8p-2, 0x1.d71276p-42f},
    {0x1.9aep+0, 0x1.35cp-1, 0x1.e4775d2ec4p-2, 0x1.cfaeap-44f},
    {0x1.985p+0, 0x1.30ap-1, 0x1.de0f55682cp-2, 0x1.0d51fep-43f},
    {0x1.95dp+0, 0x1.2bap-1, 0x1.d7c55acb2p-2, -0x1.16724cp-43f},
    {0x1.935p+0, 0x1.26ap-1, 0x1.d1716d3f8cp-2, -0x1.511c9p-48f},
    {0x1.90dp+0, 0x1.21ap-1, 0x1.cb136d19p-2, -0x1.45be3ap-42f},
    {0x1.8e6p+0, 0x1.1ccp-1, 0x1.c4d45b6e8p-2, 0x1.746c68p-47f},
    {0x1.8cp+0, 0x1.18p-1, 0x1.beb4d9da7p-2, 0x1.b7bf78p-42f},
    {0x1.89ap+0, 0x1.134p-1, 0x1.b88bea5878p-2, 0x1.dfa3e6p-42f},
    {0x1.874p+0, 0x1.0e8p-1, 0x1.b2596fb0c4p-2, 0x1.5a502p-43f},
    {0x1.84fp+0, 0x1.09ep-1, 0x1.ac476d0204p-2, 0x1.0de07p-43f},
    {0x1.82ap+0, 0x1.054p-1, 0x1.a62c25e7fcp-2, -0x1.178e96p-42f},
    {0x1.806p+0, 0x1.00cp-1, 0x1.a0321ed14cp-2, 0x1.da47aap-42f},
    {0x1.7e2p+0, 0x1.f88p-2, 0x1.9a2f1c2edcp-2, -0x1.32f28cp-43f},
    {0x1.7bfp+0, 0x1.efcp-2, 0x1.944e23354cp-2, -0x1.2df2d6p-42f},
    {0x1.79cp+0, 0x1.e7p-2, 0x1.8e647999p-2, 0x1.f7ba32p-42f},
    {0x1.779p+0, 0x1.de4p-2, 0x1.88720582ecp-2, -0x1.663f44p-43f},
    {0x1.757p+0, 0x1.d5cp-2, 0x1.82a28d349p-2, 0x1.31fdf4p-44f},
    {0x1.735p+0, 0x1.cd4p-2, 0x1.7cca97da6cp-2, -0x1.dec59ap-42f},
    {0x1.713p+0, 0x1.c4cp-2, 0x1.76ea0c82ccp-2, 0x1.d9c596p-42f},
    {0x1.6f2p+0, 0x1.bc8p-2, 0x1.712d738158p-2, -0x1.28bc5ap-44f},
    {0x1.6d2p+0, 0x1.b48p-2, 0x1.6b9574b0f8p-2, 0x1.226274p-43f},
    {0x1.6b1p+0, 0x1.ac4p-2, 0x1.65c878c014p-2, 0x1.54332ap-42f},
    {0x1.691p+0, 0x1.a44p-2, 0x1.6020689b1cp-2, 0x1.d34784p-44f},
    {0x1.672p+0, 0x1.9c8p-2, 0x1.5a9ded96bcp-2, 0x1.93f1fep-44f},
    {0x1.652p+0, 0x1.948p-2, 0x1.54e5f19e5cp-2, -0x1.0e0062p-45f},
    {0x1.633p+0, 0x1.8ccp-2, 0x1.4f53de9d24p-2, 0x1.63014ep-43f},
    {0x1.615p+0, 0x1.854p-2, 0x1.49e85f23bcp-2, -0x1.9b66e4p-48f},
    {0x1.5f6p+0, 0x1.7d8p-2, 0x1.4446dddb98p-2, -0x1.1430e6p-43f},
    {0x1.5d8p+0, 0x1.76p-2, 0x1.3ecc460ef4p-2, 0x1.f4febcp-42f},
    {0x1.5bbp+0, 0x1.6ecp-2, 0x1.3979434698p-2, -0x1.8d1b88p-44f},
    {0x1.59dp+0, 0x1.674p-2, 0x1.33efc101dcp-2, -0x1.07ffd6p-44f},
    {0x1.58p+0, 0x1.6p-2, 0x1.2e8e2bae1p-2, 0x1.d309c2p-42f},
    {0x1.564p+0, 0x1.59p-2, 0x1.29552f82p-2, -0x1.5b968p-43f},
    {0x1.547p+0, 0x1.51cp-2, 0x1.23e5398b94p-2, -0x1.c5f166p-43f},
    {0x1.52bp+0, 0x1.4acp-2, 0x1.1e9e367888p-2, 0x1.1f4548p-42f},
    {0x1.50fp+0, 0x1.43cp-2, 0x1.195033b44p-2, -0x1.59a39ap-44f},
    {0x1.4f4p+0, 0x1.3dp-2, 0x1.142bfeb9ap-2, 0x1.1ce618p-44f},
    {0x1.4d8p+0, 0x1.36p-2, 0x1.0ed005f658p-2, -0x1.2dc752p-45f},
    {0x1.4bdp+0, 0x1.2f4p-2, 0x1.099e371c0cp-2, -0x1.bf067cp-45f},
    {0x1.4a2p+0, 0x1.288p-2, 0x1.0465a08154p-2, 0x1.ff37dp-43f},
    {0x1.488p+0, 0x1.22p-2, 0x1.feb0233e6p-3, 0x1.f316e4p-45f},
    {0x1.46ep+0, 0x1.1b8p-2, 0x1.f488311d18p-3, 0x1.a495f4p-42f},
    {0x1.454p+0, 0x1.15p-2, 0x1.ea5349e238p-3, 0x1.606e4ep-42f},
    {0x1.43ap+0, 0x1.0e8p-2, 0x1.e0114c533p-3, 0x1.97eeb6p-43f},
    {0x1.421p+0, 0x1.084p-2, 0x1.d627d7c1bp-3, 0x1.6d357cp-42f},
    {0x1.408p+0, 0x1.02p-2, 0x1.cc320c0178p-3, -0x1.afdbf2p-43f},
    {0x1.3efp+0, 0x1.f78p-3, 0x1.c22fca3188p-3, 0x1.f7402cp-45f},
    {0x1.3d6p+0, 0x1.ebp-3, 0x1.b820f2fc8p-3, -0x1.af7a22p-43f},
    {0x1.3bdp+0, 0x1.de8p-3, 0x1.ae05669628p-3, 0x1.04a6c2p-44f},
    {0x1.3a5p+0, 0x1.d28p-3, 0x1.a4454820dp-3, 0x1.9f9cecp-43f},
    {0x1.38dp+0, 0x1.c68p-3, 0x1.9a7938d208p-3, 0x1.94758ep-43f},
    {0x1.375p+0, 0x1.ba8p-3, 0x1.90a11b46b8p-3, 0x1.b5601p-43f},
    {0x1.35ep+0, 0x1.afp-3, 0x1.8726935ac8p-3, 0x1.6312ecp-42f},
    {0x1.346p+0, 0x1.a3p-3, 0x1.7d36832b9p-3, -0x1.e3a5d4p-44f},
    {0x1.32fp+0, 0x1.978p-3, 0x1.73a4d0172p-3, 0x1.72dcd8p-42f},
    {0x1.318p+0, 0x1.8cp-3, 0x1.6a079d0f78p-3, 0x1.568fe2p-42f},
    {0x1.302p+0, 0x1.81p-3, 0x1.60ca8fe888p-3, -0x1.3a85bap-42f},
    {0x1.2ebp+0, 0x1.758p-3, 0x1.57168c4bp-3, -0x1.e344bap-44f},
    {0x1.2d5p+0, 0x1.6a8p-3, 0x1.4dc3789698p-3, 0x1.8e09aep-42f},
    {0x1.2bfp+0, 0x1.5f8p-3, 0x1.446579dc2p-3, 0x1.1eec7ap-42f},
    {0x1.2a9p+0, 0x1.548p-3, 0x1.3afc766c2p-3, -0x1.df0258p-43f},
    {0x1.293p+0, 0x1.498p-3, 0x1.3188543c08p-3, 0x1.8a12a4p-43f},
    {0x1.27ep+0, 0x1.3fp-3, 0x1.2877bbc0b8p-3, -0x1.45a0bap-43f},
    {0x1.269p+0, 0x1.348p-3, 0x1.1f5cd21a1p-3, -0x1.363dd6p-42f},
    {0x1.254p+0, 0x1.2ap-3, 0x1.16377fb128p-3, -0x1.f370f2p-42f},
    {0x1.23fp+0, 0x1.1f8p-3, 0x1.0d07ac9dc8p-3, 0x1.e7bd88p-42f},
    {0x1.22ap+0, 0x1.15p-3, 0x1.03cd40a518p-3, 0x1.606a5ep-42f},
    {0x1.215p+0, 0x1.0a8p-3, 0x1.f510466fep-4, -0x1.fd0246p-42f},
    {0x1.201p+0, 0x1.008p-3, 0x1.e353fec9ap-4, 0x1.34c7dp-43f},
    {0x1.1edp+0, 0x1.edp-4, 0x1.d183f87eap-4, 0x1.cdf146p-42f},
    {0x1.1d9p+0, 0x1.d9p-4, 0x1.bfa007673p-4, -0x1.577574p-42f},
    {0x1.1c5p+0, 0x1.c5p-4, 0x1.ada7fec6bp-4, -0x1.bff6fep-43f},
    {0x1.1b1p+0, 0x1.b1p-4, 0x1.9b9bb1495p-4, -0x1.ba64e6p-42f},
    {0x1.19ep+0, 0x1.9ep-4, 0x1.8a6377a91p-4, 0x1.70a2eep-42f},
    {0x1.18bp+0, 0x1.8bp-4, 0x1.7918a1bfap-4, -0x1.f8a778p-42f},
    {0x1.178p+0, 0x1.78p-4, 0x1.67bb0726fp-4, -0x1.f8236ep-43f},
    {0x1.165p+0, 0x1.65p-4, 0x1.564a7ef51p-4, 0x1.0c44cap-42f},
    {0x1.152p+0, 0x1.52p-4, 0x1.44c6dfb9bp-4, 0x1.d81976p-42f},
    {0x1.13fp+0, 0x1.3fp-4, 0x1.332fff7bdp-4, 0x1.f18282p-44f},
    {0x1.12dp+0, 0x1.2dp-4, 0x1.22743457bp-4, -0x1.8dc94cp-42f},
    {0x1.11ap+0, 0x1.1ap-4, 0x1.10b75afd6p-4, 0x1.83185cp-42f},
    {0x1.108p+0, 0x1.08p-4, 0x1.ffae9119cp-5, -0x1.b3f322p-43f},
    {0x1.0f6p+0, 0x1.ecp-5, 0x1.ddcaadb46p-5, 0x1.de361p-42f},
    {0x1.0e4p+0, 0x1.c8p-5, 0x1.bbc2bfc44p-5, 0x1.e82e7ap-42f},
    {0x1.0d2p+0, 0x1.a4p-5, 0x1.99967a4f2p-5, 0x1.6390ccp-42f},
    {0x1.0c1p+0, 0x1.82p-5, 0x1.792e93e52p-5, -0x1.984da8p-43f},
    {0x1.0afp+0, 0x1.5ep-5, 0x1.56bac43eep-5, -0x1.00cc2cp-42f},
    {0x1.09ep+0, 0x1.3cp-5, 0x1.360ebf5d8p-5, 0x1.bb2b26p-44f},
    {0x1.08dp+0, 0x1.1ap-5, 0x1.15413ca0ep-5, 0x1.ca9e4ep-43f},
    {0x1.07cp+0, 0x1.fp-6, 0x1.e8a3ee30cp-6, 0x1.b95818p-43f},
    {0x1.06bp+0, 0x1.acp-6, 0x1.a68151fb4p-6, 0x1.c049fcp-42f},
    {0x1.05ap+0, 0x1.68p-6, 0x1.641a17628p-6, -0x1.e5213ap-43f},
    {0x1.049p+0, 0x1.24p-6, 0x1.216daf6d8p-6, 0x1.32199ep-42f},
    {0x1.0388p+0, 0x1.c4p-7, 0x1.c0e9338cp-7, 0x1.210b9ap-42f},
    {0x1.0p+0, 0x0.0p+0, 0x0.0p+0, 0x0.0p+0f},
    {0x1.0p+0, 0x0.0p+0, 0x0.0p+0, 0x0.0p+0f},
    {0x1.0p+0, 0x0.0p+0, 0x0.0p+0, 0x0.0p+0f},
};

// x = k ln2/128 + r + r_lo with |r| <= ln2/256 + the rounding of the FP32
// quotient, r exact and r_lo the remainder of k ln2/128; for x below 6.5 ln2/128
// (0.035) k = 0 and r = x.
struct Reduced {
  int k;
  double r;
  float r_lo;
};
RT_FN Reduced reduce(double x) {
  float kf = rintf(cut(x) * 184.664965f);  // 128 / ln 2
  kf = kf < 7.0f ? 0.0f : fminf(kf, 131071.0f);  // 2^1024 is no double
  return Reduced{(int)kf, fma(-widen(kf), kLn2Over128, x), -kf * kLn2Over128Lo};
}

// 1 - exp(-x) for x >= 0 (finite).  With T = 2^(-k/128) and p = 1 - exp(-r -
// r_lo): 1 - exp(-x) = (1 - T) + T p.  1 - T is the exact difference of 1 and T's
// leading 13 bits, plus the remainder, which joins T p: from k = 7 on that is
// small enough against the result for its rounding not to count (below, k = 0
// and the result is p, rounded once).  With T < 2^-5 all of it is small.  From 54
// ln 2 on the result rounds to 1.
RT_FN double one_minus_exp(double x) {
  const bool big = bits_of(x) > 0x4042b5c28f5c28f6ll;  // x > 37.42
  const Reduced R = reduce(big ? 0.0 : x);
  const double r = R.r;
  // p = r + r (-r/2 + r^2/6 - r^3/24 + r^4/120 - r^5 (1/720 - r/5040 + ...)) + r_lo (1 - r)
  const float rf = cut(r);
  const float tail = fmaf(rf, fmaf(rf, fmaf(rf, 1.0f / 362880.0f, -1.0f / 40320.0f), 1.0f / 5040.0f), -1.0f / 720.0f);
  double q = fma(r, widen(tail), 1.0 / 120.0);
  q = fma(r, q, -1.0 / 24.0);
  q = fma(r, q, 1.0 / 6.0);
  q = fma(r, q, -0.5);
  const double r_lo = widen(R.r_lo);
  const double v = fma(r, fma(r, q, -r_lo), r_lo);
  const ExpEntry e = kExpTable[R.k & 127];
  const int m = R.k >> 7;
  const long long scale = (long long)m << 52;
  const bool far = m > 5;
  const double T = double_of(bits_of(e.t) - scale);
  const double hi = far ? 0.0 : double_of(bits_of(e.hi) - scale);
  const double lo = far ? -T : ((R.k & 127) ? double_of(bits_of(e.lo) - scale) : 0.0);
  const double w = fma(T, r, fma(T, v, lo));
  return big ? 1.0 : (1.0 - hi) + w;
}

// exp(x) - 1 for 0 <= x <= 709.78 (the largest with a finite result), in the
// same way: T = 2^(k/128), exp(x) - 1 = (T - 1) + T p, p = exp(r + r_lo) - 1; from
// T = 2^53 on the 1 is one of the small terms.
RT_FN double exp_minus_one(double x) {
  const Reduced R = reduce(x);
  const double r = R.r;
  // p = r + r (r/2 + r^2/6 + r^3/24 + r^4/120 + r^5 (1/720 + r/5040 + ...)) + r_lo (1 + r)
  const float rf = cut(r);
  const float tail = fmaf(rf, fmaf(rf, fmaf(rf, 1.0f / 362880.0f, 1.0f / 40320.0f), 1.0f / 5040.0f), 1.0f / 720.0f);
  double q = fma(r, widen(tail), 1.0 / 120.0);
  q = fma(r, q, 1.0 / 24.0);
  q = fma(r, q, 1.0 / 6.0);
  q = fma(r, q, 0.5);
  const double r_lo = widen(R.r_lo);
  const double v = fma(r, fma(r, q, r_lo), r_lo);
  const ExpEntry e = kExpUpTable[R.k & 127];
  const int m = R.k >> 7;
  const long long scale = (long long)m << 52;
  const double T = double_of(bits_of(e.t) + scale);
  const double hi = double_of(bits_of(e.hi) + scale);
  double lo = (R.k & 127) ? double_of(bits_of(e.lo) + scale) : 0.0;
  if (m > 52) lo -= 1.0;
  const double w = fma(T, r, fma(T, v, lo));
  return (hi - (m > 52 ? 0.0 : 1.0)) + w;
}

// a / (exp(x) - 1) for x > 0; zero above 709.78, where exp(x) - 1 overflows.
RT_FN double bose(double x, double a = 1.0) {
  return bits_of(x) > 0x40862e42fefa39efll ? 0.0 : a / exp_minus_one(x);
}

// -ln(1 - v) for 0 <= v < 1.  y = 1 - v = 2^-m z with z in (1/2, 1], z rc = 1 +
// r, |r| <= 2^-8 (3/256 on the last three intervals, where rc = 1): -ln(1 - v) =
// m ln 2 + ln rc - ln(1 + r).  r = (rc - 1) - rc (1 - z), where 1 - z is v for m =
// 0 (v < 1/2) and exact above; the product's rounding error is kept.  m ln 2 + ln
// rc to a multiple of 2^-40 is exact; its remainder joins ln(1 + r).  Below 3/256
// the result is that, rounded once.
RT_FN double neg_log_one_minus(double v) {
  const bool low = bits_of(v) < 0x3fe0000000000000ll;  // v < 1/2
  long long by = bits_of(1.0 - v);
  if (low && by <= 0x3fe0000000000000ll) by = 0x3fe0000000000001ll;  // y rounded down to 1/2
  const long long b = by - 1;  // 1 and the other powers of two end their interval
  const int m = 1022 - (int)(b >> 52);
  const LogEntry e = kLogTable[(int)(b >> 45) & 127];
  const double z = double_of(by + ((long long)m << 52));
  const double w = low ? v : 1.0 - z;
  const double P = e.rc * w, pe = fma(e.rc, w, -P);
  const double r = e.c - P;  // exact; 1 + r - pe = z rc
  // -ln(1 + r) = -r + r (r/2 - r^2/3 + r^3/4 - r^4/5 + r^5 (1/6 - r/7 + ...))
  const float rf = cut(r);
  const float tail = fmaf(rf, fmaf(rf, fmaf(rf, -1.0f / 9.0f, 1.0f / 8.0f), -1.0f / 7.0f), 1.0f / 6.0f);
  double q = fma(r, widen(tail), -0.2);
  q = fma(r, q, 0.25);
  q = fma(r, q, -1.0 / 3.0);
  q = fma(r, q, 0.5);
  const float mf = (float)m;
  const float lo = cut(pe) + fmaf(mf, kLn2Lo, e.ln_lo);
  return fma(widen(mf), kLn2, e.ln) + (fma(r, r * q, widen(lo)) - r);
}

}  // namespace rtk
