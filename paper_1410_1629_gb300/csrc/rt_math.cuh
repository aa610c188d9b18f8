// Double-precision exponential and logarithm of the forced-scattering
// inversion (Sect. 1), written for a device whose FP64 pipe issues one warp
// instruction per 16 cycles of an SM, whatever its active lanes: 1 - exp(-x)
// in 9 FP64 instructions and -ln(1 - v) in 14, table-driven (P. T. P. Tang,
// "Table-driven implementation of the exponential function in IEEE
// floating-point arithmetic", ACM TOMS 15, 1989, and "... of the logarithm
// function ...", ACM TOMS 16, 1990).  The range reduction and the high-order
// terms of the series use integer and FP32 instructions; where an FP32 value
// enters an FP64 sum its weight there is below 2^-29, so its rounding stays
// below 2^-53 of the result.  Against extended precision (2e7 arguments): 1 -
// exp(-x) within 1.6 ulp, 0.34 ulp rms; -ln(1 - v) within 1.4 ulp, 0.36 ulp
// rms, i.e. 1e-16 of results that carry the 1e-7 of FP32 geometry.
// Measured with the CUDA library's expm1 and log1p in their place: a launch of
// 1e5 packets in a 32^3 cube issued 7.15e6 FP64 warp instructions against
// 3.04e6 now, 32 batched models 6.30e8 against 3.05e8 (57.2 against 53.1 ms,
// FP64 pipe 63 against 39 % busy), the taped forward launch 3.21e7 against
// 1.29e7 (4.07 against 3.87 ms).
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

// 2^(-j/128), and 1 - 2^(-j/128) as a double and its remainder
struct ExpEntry {
  double t, a, a_lo;
};
// a reciprocal of the middle of [1/2 + j/256, 1/2 + (j + 1)/256] to 13 bits
// (1 for the last interval), and its logarithm as a double and its remainder
struct LogEntry {
  double rc, ln, ln_lo;
};

constexpr double kLn2Over128Hi = 0x1.62e42fefa39efp-8, kLn2Over128Lo = 0x1.abc9e3b39803fp-63;
constexpr double kLn2 = 0x1.62e42fefa39efp-1, kLn2Lo = 0x1.abc9e3b39803fp-56;
RT_TABLE ExpEntry kExpTable[128] = {
    {0x1.0000000000000p+0, 0x0.0p+0, 0x0.0p+0},
    {0x1.fd3c22b8f71f1p-1, 0x1.61eea3847077bp-8, 0x1.148b699a8618bp-62},
    {0x1.fa7c1819e90d8p-1, 0x1.60f9f985bc9f4p-7, 0x1.6f5818b4d9c3ep-61},
    {0x1.f7bfdad9cbe14p-1, 0x1.0804a4c683d8fp-6, -0x1.13b4bfe72bd96p-61},
    {0x1.f50765b6e4540p-1, 0x1.5f134923757f3p-6, 0x1.60f6913af3a8ap-62},
    {0x1.f252b376bba97p-1, 0x1.b5a991288ad16p-6, 0x1.796903c9c6f2bp-61},
    {0x1.efa1bee615a27p-1, 0x1.05e4119ea5d89p-5, -0x1.c7f486a4b6b08p-59},
    {0x1.ecf482d8e67f1p-1, 0x1.30b7d271980f7p-5, 0x1.27e768235b188p-60},
    {0x1.ea4afa2a490dap-1, 0x1.5b505d5b6f268p-5, -0x1.63dce863d76ccp-59},
    {0x1.e7a51fbc74c83p-1, 0x1.85ae0438b37cbp-5, 0x1.2add35f3721e6p-59},
    {0x1.e502ee78b3ff6p-1, 0x1.afd11874c009ep-5, -0x1.cf44c054e647ap-59},
    {0x1.e264614f5a129p-1, 0x1.d9b9eb0a5ed76p-5, -0x1.2761fa17ada64p-61},
    {0x1.dfc97337b9b5fp-1, 0x1.01b466423250ap-4, 0x1.a5cd4f184b5b9p-59},
    {0x1.dd321f301b460p-1, 0x1.166f067f25cfep-4, -0x1.6d2bbc780c614p-58},
    {0x1.da9e603db3285p-1, 0x1.2b0cfe1266bd4p-4, 0x1.ee7fcb492566dp-58},
    {0x1.d80e316c98398p-1, 0x1.3f8e749b3e342p-4, 0x1.1ec18beddfe82p-59},
    {0x1.d5818dcfba487p-1, 0x1.53f391822dbc7p-4, -0x1.76816bad9b837p-59},
    {0x1.d2f87080d89f2p-1, 0x1.683c7bf93b074p-4, -0x1.5bc247313d440p-58},
    {0x1.d072d4a07897cp-1, 0x1.7c695afc3b424p-4, -0x1.a1e45e4342b1cp-58},
    {0x1.cdf0b555dc3fap-1, 0x1.907a55511e032p-4, -0x1.13e2563eb1470p-59},
    {0x1.cb720dcef9069p-1, 0x1.a46f918837cb7p-4, 0x1.5f8685c2d6c49p-58},
    {0x1.c8f6d9406e7b5p-1, 0x1.b84935fc8c257p-4, 0x1.ca6876eff4778p-58},
    {0x1.c67f12e57d14bp-1, 0x1.cc0768d4175a6p-4, -0x1.4426ffa41e566p-58},
    {0x1.c40ab5fffd07ap-1, 0x1.dfaa500017c2dp-4, -0x1.a29bf041e3051p-58},
    {0x1.c199bdd85529cp-1, 0x1.f332113d56b1fp-4, -0x1.1065895048dd3p-60},
    {0x1.bf2c25bd71e09p-1, 0x1.034f690a387dep-3, -0x1.0235c094638d1p-59},
    {0x1.bcc1e904bc1d2p-1, 0x1.0cf85bed0f8b7p-3, 0x1.b845f0ba4c2f7p-57},
    {0x1.ba5b030a1064ap-1, 0x1.1693f3d7be6dap-3, -0x1.032cf1abd6d20p-59},
    {0x1.b7f76f2fb5e47p-1, 0x1.20224341286e4p-3, 0x1.5584f7e54ac3bp-57},
    {0x1.b59728de5593ap-1, 0x1.29a35c86a9b1ap-3, -0x1.c7102222c90e8p-58},
    {0x1.b33a2b84f15fbp-1, 0x1.331751ec3a814p-3, 0x1.2805e3084d708p-58},
    {0x1.b0e07298db666p-1, 0x1.3c7e359c9266ap-3, -0x1.0842acdfc6f6dp-57},
    {0x1.ae89f995ad3adp-1, 0x1.45d819a94b14bp-3, -0x1.e8734d1773206p-57},
    {0x1.ac36bbfd3f37ap-1, 0x1.4f25100b03219p-3, -0x1.b72cd4624cbf9p-62},
    {0x1.a9e6b5579fdbfp-1, 0x1.58652aa180903p-3, -0x1.f5921deffa626p-60},
    {0x1.a799e1330b358p-1, 0x1.61987b33d329ep-3, 0x1.0d204d4ea70e5p-57},
    {0x1.a5503b23e255dp-1, 0x1.6abf137076a8ep-3, -0x1.684892395f0f8p-58},
    {0x1.a309bec4a2d33p-1, 0x1.73d904ed74b33p-3, -0x1.8c171f770daadp-57},
    {0x1.a0c667b5de565p-1, 0x1.7ce6612886a6dp-3, 0x1.aca4ae8e6a997p-58},
    {0x1.9e86319e32323p-1, 0x1.85e7398737374p-3, -0x1.824ca78e64c6ep-57},
    {0x1.9c49182a3f090p-1, 0x1.8edb9f5703dc0p-3, -0x1.c7c46b071f2bep-57},
    {0x1.9a0f170ca07bap-1, 0x1.97c3a3cd7e119p-3, 0x1.73bd91cee6321p-59},
    {0x1.97d829fde4e50p-1, 0x1.a09f58086c6c2p-3, -0x1.73d241f23d17bp-58},
    {0x1.95a44cbc8520fp-1, 0x1.a96ecd0deb7c4p-3, 0x1.64b7c96a5f039p-57},
    {0x1.93737b0cdc5e5p-1, 0x1.b23213cc8e86cp-3, 0x1.75fc781b57ebcp-58},
    {0x1.9145b0b91ffc6p-1, 0x1.bae93d1b800eap-3, -0x1.14c368d3ed6e2p-58},
    {0x1.8f1ae99157736p-1, 0x1.c39459baa2327p-3, 0x1.467d8ba38d128p-57},
    {0x1.8cf3216b5448cp-1, 0x1.cc337a52aedd0p-3, 0x1.0d55e32e9e3aap-57},
    {0x1.8ace5422aa0dbp-1, 0x1.d4c6af7557c93p-3, -0x1.ba7c55a192c9cp-57},
    {0x1.88ac7d98a6699p-1, 0x1.dd4e099d6659ap-3, 0x1.9acf4320d2b16p-57},
    {0x1.868d99b4492edp-1, 0x1.e5c9992edb44ep-3, -0x1.c83b21584a2e1p-62},
    {0x1.8471a4623c7adp-1, 0x1.ee396e770e14dp-3, -0x1.ca5ed72f8c813p-58},
    {0x1.82589994cce13p-1, 0x1.f69d99accc7b6p-3, -0x1.59f115f566940p-58},
    {0x1.80427543e1a12p-1, 0x1.fef62af0797b9p-3, 0x1.3e433136cb956p-58},
    {0x1.7e2f336cf4e62p-1, 0x1.03a199261633cp-2, -0x1.05d02ba15797ep-57},
    {0x1.7c1ed0130c132p-1, 0x1.07c25fd9e7d9bp-2, 0x1.db665dd36454fp-60},
    {0x1.7a11473eb0187p-1, 0x1.0bdd71829fcf2p-2, 0x1.41577ee04992fp-56},
    {0x1.780694fde5d3fp-1, 0x1.0ff2d60434581p-2, 0x1.e651fd7f7a74dp-57},
    {0x1.75feb564267c9p-1, 0x1.14029537b306fp-2, -0x1.fb74d519d2459p-56},
    {0x1.73f9a48a58174p-1, 0x1.180cb6eb4fd19p-2, -0x1.eae4d27345589p-56},
    {0x1.71f75e8ec5f74p-1, 0x1.1c1142e274118p-2, 0x1.16e4786887a99p-56},
    {0x1.6ff7df9519484p-1, 0x1.201040d5cd6f8p-2, 0x1.83c0f25860ef6p-56},
    {0x1.6dfb23c651a2fp-1, 0x1.2409b8735cba2p-2, 0x1.bbe3a683c88abp-58},
    {0x1.6c012750bdabfp-1, 0x1.27fdb15e84a82p-2, 0x1.2895667ff0b0dp-57},
    {0x1.6a09e667f3bcdp-1, 0x1.2bec333018867p-2, -0x1.08b2fb1366ea9p-57},
    {0x1.68155d44ca973p-1, 0x1.2fd545766ad1ap-2, -0x1.038ae44f73e65p-58},
    {0x1.6623882552225p-1, 0x1.33b8efb55bbb7p-2, -0x1.127d9e29b8f31p-57},
    {0x1.6434634ccc320p-1, 0x1.37973966679c0p-2, 0x1.c483c759d8933p-56},
    {0x1.6247eb03a5585p-1, 0x1.3b7029f8b54f7p-2, -0x1.8f87d037e96d2p-56},
    {0x1.605e1b976dc09p-1, 0x1.3f43c8d1247efp-2, -0x1.83b7ac9524372p-56},
    {0x1.5e76f15ad2148p-1, 0x1.43121d4a5bd6fp-2, 0x1.1641b3dfc668ap-57},
    {0x1.5c9268a5946b7p-1, 0x1.46db2eb4d7292p-2, -0x1.c4b1b816986a2p-61},
    {0x1.5ab07dd485429p-1, 0x1.4a9f0456f57adp-2, 0x1.39b67f57370a6p-56},
    {0x1.58d12d497c7fdp-1, 0x1.4e5da56d07006p-2, -0x1.295e15b9a1de8p-56},
    {0x1.56f4736b527dap-1, 0x1.521719295b04bp-2, 0x1.9134ffb89b14cp-57},
    {0x1.551a4ca5d920fp-1, 0x1.55cb66b44dbe2p-2, 0x1.d689cefede59bp-56},
    {0x1.5342b569d4f82p-1, 0x1.597a952c560fcp-2, 0x1.07abe1db13cadp-56},
    {0x1.516daa2cf6642p-1, 0x1.5d24aba61337cp-2, 0x1.f768569bd93efp-56},
    {0x1.4f9b2769d2ca7p-1, 0x1.60c9b12c5a6b3p-2, -0x1.699ec5b4d503ap-56},
    {0x1.4dcb299fddd0dp-1, 0x1.6469acc0445e5p-2, 0x1.c4c910e561f34p-57},
    {0x1.4bfdad5362a27p-1, 0x1.6804a5593abb2p-2, -0x1.d4397afec42e2p-57},
    {0x1.4a32af0d7d3dep-1, 0x1.6b9aa1e505843p-2, 0x1.8d27430b906a8p-57},
    {0x1.486a2b5c13cd0p-1, 0x1.6f2ba947d8660p-2, -0x1.3c1a3b69062f0p-57},
    {0x1.46a41ed1d0057p-1, 0x1.72b7c25c5ff51p-2, 0x1.b5da174dbac4dp-58},
    {0x1.44e086061892dp-1, 0x1.763ef3f3ceda6p-2, -0x1.89b7a04ef80d0p-60},
    {0x1.431f5d950a897p-1, 0x1.79c144d5eaed2p-2, 0x1.1c7dde35f7999p-56},
    {0x1.4160a21f72e2ap-1, 0x1.7d3ebbc11a3acp-2, 0x1.ef3691c309278p-59},
    {0x1.3fa4504ac801cp-1, 0x1.80b75f6a6ffc9p-2, -0x1.05fb80d520c19p-56},
    {0x1.3dea64c123422p-1, 0x1.842b367db97bcp-2, -0x1.ada0911f09ebcp-56},
    {0x1.3c32dc313a8e5p-1, 0x1.879a479d8ae37p-2, -0x1.0007c8a2d63cep-59},
    {0x1.3a7db34e59ff7p-1, 0x1.8b0499634c012p-2, 0x1.5e436d661f5e3p-57},
    {0x1.38cae6d05d866p-1, 0x1.8e6a325f44f35p-2, -0x1.6a72c366fb432p-59},
    {0x1.371a7373aa9cbp-1, 0x1.91cb1918aac6bp-2, -0x1.38a2a817a2a3dp-56},
    {0x1.356c55f929ff1p-1, 0x1.9527540dac01ep-2, 0x1.b5cee5c4e4628p-56},
    {0x1.33c08b26416ffp-1, 0x1.987ee9b37d201p-2, 0x1.9b1bcf7934cb5p-56},
    {0x1.32170fc4cd831p-1, 0x1.9bd1e07664f9ep-2, -0x1.a9ce78e18047cp-56},
    {0x1.306fe0a31b715p-1, 0x1.9f203eb9c91d6p-2, -0x1.6f46ad23182e4p-56},
    {0x1.2ecafa93e2f56p-1, 0x1.a26a0ad83a154p-2, -0x1.1ca0f45d52383p-57},
    {0x1.2d285a6e4030bp-1, 0x1.a5af4b237f9e9p-2, 0x1.ffb7156497c56p-56},
    {0x1.2b87fd0dad990p-1, 0x1.a8f005e4a4ce0p-2, 0x1.10adcd6381aa4p-60},
    {0x1.29e9df51fdee1p-1, 0x1.ac2c415c0423ep-2, -0x1.612e8afad1255p-56},
    {0x1.284dfe1f56381p-1, 0x1.af6403c1538ffp-2, -0x1.6cf15cf03ca09p-57},
    {0x1.26b4565e27cddp-1, 0x1.b2975343b0646p-2, -0x1.2bd339940e9d9p-56},
    {0x1.251ce4fb2a63fp-1, 0x1.b5c63609ab382p-2, -0x1.ac155bef4f4a4p-56},
    {0x1.2387a6e756238p-1, 0x1.b8f0b23153b8fp-2, 0x1.93e0524e3ea35p-57},
    {0x1.21f49917ddc96p-1, 0x1.bc16cdd0446d4p-2, -0x1.2a97e9494a5eep-56},
    {0x1.2063b88628cd6p-1, 0x1.bf388ef3ae654p-2, -0x1.dc775814a8495p-56},
    {0x1.1ed5022fcd91dp-1, 0x1.c255fba064dc7p-2, -0x1.c40cffb0890e9p-56},
    {0x1.1d4873168b9aap-1, 0x1.c56f19d2e8cabp-2, 0x1.fe91ff5d9bc3ep-59},
    {0x1.1bbe084045cd4p-1, 0x1.c883ef7f74659p-2, -0x1.ab1e72b4427e3p-57},
    {0x1.1a35beb6fcb75p-1, 0x1.cb94829206916p-2, -0x1.e5b4c7b4968e4p-56},
    {0x1.18af9388c8deap-1, 0x1.cea0d8ee6e42dp-2, -0x1.ddfb85cd1e128p-56},
    {0x1.172b83c7d517bp-1, 0x1.d1a8f87055d0ap-2, 0x1.19041b9d78a76p-56},
    {0x1.15a98c8a58e51p-1, 0x1.d4ace6eb4e35ep-2, -0x1.2406ab9eeab0ap-56},
    {0x1.1429aaea92de0p-1, 0x1.d7acaa2ada441p-2, -0x1.9a080ca1d92c3p-56},
    {0x1.12abdc06c31ccp-1, 0x1.daa847f279c68p-2, 0x1.1b514b36ca5c7p-59},
    {0x1.11301d0125b51p-1, 0x1.dd9fc5fdb495fp-2, -0x1.275df8d76c98cp-56},
    {0x1.0fb66affed31bp-1, 0x1.e0932a00259cap-2, 0x1.b9bedc44ebd7bp-58},
    {0x1.0e3ec32d3d1a2p-1, 0x1.e38279a585cbcp-2, -0x1.03a1727c57b53p-60},
    {0x1.0cc922b7247f7p-1, 0x1.e66dba91b7011p-2, 0x1.fc247d23b611dp-56},
    {0x1.0b5586cf9890fp-1, 0x1.e954f260cede1p-2, 0x1.d6746d48e7bd5p-57},
    {0x1.09e3ecac6f383p-1, 0x1.ec3826a7218f9p-2, 0x1.d6f0fcf9d3d95p-56},
    {0x1.0874518759bc8p-1, 0x1.ef175cf14c870p-2, -0x1.186be4bb284ffp-58},
    {0x1.0706b29ddf6dep-1, 0x1.f1f29ac441244p-2, 0x1.c91dfe2b13c27p-56},
    {0x1.059b0d3158574p-1, 0x1.f4c9e59d4f518p-2, -0x1.d73e2a475b465p-56},
    {0x1.04315e86e7f85p-1, 0x1.f79d42f2300f7p-2, -0x1.eb9c7cd106d24p-56},
    {0x1.02c9a3e778061p-1, 0x1.fa6cb8310ff3ep-2, 0x1.19083535b085dp-57},
    {0x1.0163da9fb3335p-1, 0x1.fd384ac099995p-2, 0x1.27b59951cc923p-57},
};
RT_TABLE LogEntry kLogTable[128] = {
    {0x1.fe00000000000p+0, 0x1.60e32f44788d9p-1, -0x1.ac1bb52fa589bp-56},
    {0x1.fa10000000000p+0, 0x1.5ceb4e16f11bdp-1, 0x1.a652604e75b1fp-55},
    {0x1.f630000000000p+0, 0x1.58fbcdcdb80c2p-1, -0x1.6d76d00f74961p-58},
    {0x1.f260000000000p+0, 0x1.5514efdbb2d63p-1, -0x1.b881274f6c64ep-56},
    {0x1.eea0000000000p+0, 0x1.5136f66336c97p-1, -0x1.0ed19cb7418c6p-55},
    {0x1.eaf0000000000p+0, 0x1.4d62242e94aa0p-1, -0x1.1e2cd982e8e53p-55},
    {0x1.e740000000000p+0, 0x1.4985ece016ba9p-1, 0x1.6122cbf70330cp-55},
    {0x1.e3b0000000000p+0, 0x1.45c414576a743p-1, 0x1.aa159b817c01bp-55},
    {0x1.e020000000000p+0, 0x1.41fb1f8350d6ep-1, -0x1.29f84c02e1e3dp-56},
    {0x1.dca0000000000p+0, 0x1.3e3c23918e76cp-1, 0x1.56bc923ba0df5p-55},
    {0x1.d930000000000p+0, 0x1.3a8766721ed12p-1, 0x1.1d0616c506bbbp-55},
    {0x1.d5d0000000000p+0, 0x1.36dd2e951ecccp-1, 0x1.58f1381bb2247p-58},
    {0x1.d270000000000p+0, 0x1.332c33125536fp-1, 0x1.62bd6dc6a5299p-55},
    {0x1.cf20000000000p+0, 0x1.2f860b54da12ap-1, 0x1.eadaea9e32d97p-55},
    {0x1.cbe0000000000p+0, 0x1.2beaff89b89ecp-1, -0x1.5a84b5cf90a51p-58},
    {0x1.c8b0000000000p+0, 0x1.285b5840fbf6ap-1, -0x1.5ffa7477ed891p-55},
    {0x1.c590000000000p+0, 0x1.24d75e6134bdbp-1, 0x1.0fb9e400963f8p-57},
    {0x1.c270000000000p+0, 0x1.214d2b9d6c05cp-1, -0x1.b6177df738c6bp-55},
    {0x1.bf60000000000p+0, 0x1.1dcef9ca55ce8p-1, 0x1.e883889132394p-57},
    {0x1.bc50000000000p+0, 0x1.1a4aa38b77f3cp-1, 0x1.61930171c9940p-55},
    {0x1.b950000000000p+0, 0x1.16d2a38adf5edp-1, -0x1.fc87e81d5af1dp-55},
    {0x1.b660000000000p+0, 0x1.1367452acf872p-1, -0x1.c7872efe848c0p-55},
    {0x1.b370000000000p+0, 0x1.0ff6041a2bfaep-1, -0x1.767c084f41340p-58},
    {0x1.b090000000000p+0, 0x1.0c91bc8186ce8p-1, 0x1.0d79be1dc3d80p-55},
    {0x1.adc0000000000p+0, 0x1.093abae514ea2p-1, 0x1.188f43b1000b1p-56},
    {0x1.aaf0000000000p+0, 0x1.05de1c19707f8p-1, 0x1.c2c7e152fcf60p-58},
    {0x1.a830000000000p+0, 0x1.028f1d69a5ffep-1, 0x1.933550a2d9e40p-56},
    {0x1.a570000000000p+0, 0x1.fe7538ded33fdp-2, 0x1.649258eaeec49p-58},
    {0x1.a2c0000000000p+0, 0x1.f7e82e660f5c1p-2, 0x1.a763b39986482p-57},
    {0x1.a020000000000p+0, 0x1.f177b7dfd4080p-2, -0x1.4d936740c5ae6p-56},
    {0x1.9d80000000000p+0, 0x1.eafcd2cea9d71p-2, 0x1.3a8c72437300dp-57},
    {0x1.9ae0000000000p+0, 0x1.e4775d2ec473fp-2, -0x1.16029eac3a8d7p-56},
    {0x1.9850000000000p+0, 0x1.de0f55682c86bp-2, -0x1.c03c0f9354e02p-56},
    {0x1.95d0000000000p+0, 0x1.d7c55acb1f74cp-2, 0x1.b67b2817dbb6ap-56},
    {0x1.9350000000000p+0, 0x1.d1716d3f8bfacp-2, -0x1.1c903b5713a63p-56},
    {0x1.90d0000000000p+0, 0x1.cb136d18feba4p-2, 0x1.c5d503d7e47e9p-58},
    {0x1.8e60000000000p+0, 0x1.c4d45b6e800bap-2, 0x1.b1a023082ae78p-57},
    {0x1.8c00000000000p+0, 0x1.beb4d9da71b7cp-2, -0x1.0f3c590a887cap-59},
    {0x1.89a0000000000p+0, 0x1.b88bea5879dfap-2, 0x1.f36db6aa702b0p-57},
    {0x1.8740000000000p+0, 0x1.b2596fb0c4ad3p-2, -0x1.fc0536ca18103p-56},
    {0x1.84f0000000000p+0, 0x1.ac476d020486fp-2, 0x1.bc43bed40898ap-61},
    {0x1.82a0000000000p+0, 0x1.a62c25e7fae87p-2, 0x1.69d2877705027p-58},
    {0x1.8060000000000p+0, 0x1.a0321ed14dda4p-2, 0x1.ea523f7a6025ep-56},
    {0x1.7e20000000000p+0, 0x1.9a2f1c2edb668p-2, 0x1.ae627419bc9f0p-56},
    {0x1.7bf0000000000p+0, 0x1.944e23354ad21p-2, -0x1.6a8bdf829d320p-57},
    {0x1.79c0000000000p+0, 0x1.8e64799901f7cp-2, -0x1.735f3a17be3a7p-56},
    {0x1.7790000000000p+0, 0x1.88720582eb4cep-2, 0x1.79a0604205e40p-60},
    {0x1.7570000000000p+0, 0x1.82a28d34904c8p-2, -0x1.05ecc5a735397p-59},
    {0x1.7350000000000p+0, 0x1.7cca97da6a214p-2, -0x1.6643e0faa0e68p-56},
    {0x1.7130000000000p+0, 0x1.76ea0c82cdd9cp-2, 0x1.65a91a2d284fep-56},
    {0x1.6f20000000000p+0, 0x1.712d738157b5dp-2, 0x1.d319a44184d74p-59},
    {0x1.6d20000000000p+0, 0x1.6b9574b0f8913p-2, 0x1.39be626b95702p-58},
    {0x1.6b10000000000p+0, 0x1.65c878c015543p-2, 0x1.94f3b885f2422p-57},
    {0x1.6910000000000p+0, 0x1.6020689b1c74dp-2, 0x1.e0e33042ec134p-58},
    {0x1.6720000000000p+0, 0x1.5a9ded96bc650p-2, -0x1.c04ec2e48f4d5p-57},
    {0x1.6520000000000p+0, 0x1.54e5f19e5bde4p-2, -0x1.8a73613f800ddp-63},
    {0x1.6330000000000p+0, 0x1.4f53de9d24b18p-2, 0x1.4d4cd2cc035d4p-59},
    {0x1.6150000000000p+0, 0x1.49e85f23bbf99p-2, 0x1.3239056cd3892p-57},
    {0x1.5f60000000000p+0, 0x1.4446dddb9775ep-2, 0x1.e34224b4e750fp-56},
    {0x1.5d80000000000p+0, 0x1.3ecc460ef5f50p-2, -0x1.4313e09807affp-58},
    {0x1.5bb0000000000p+0, 0x1.39794346979ccp-2, -0x1.b871970264e26p-56},
    {0x1.59d0000000000p+0, 0x1.33efc101dbbe0p-2, 0x1.4ce40ae6e981dp-63},
    {0x1.5800000000000p+0, 0x1.2e8e2bae11d31p-2, -0x1.8f4cdb95ebdf9p-56},
    {0x1.5640000000000p+0, 0x1.29552f81ff523p-2, 0x1.301771c407dbfp-56},
    {0x1.5470000000000p+0, 0x1.23e5398b931d0p-2, 0x1.d3331000bcafep-56},
    {0x1.52b0000000000p+0, 0x1.1e9e3678891f4p-2, 0x1.51d6e1f04c8fbp-56},
    {0x1.50f0000000000p+0, 0x1.195033b43fa99p-2, 0x1.c666783d93b26p-56},
    {0x1.4f40000000000p+0, 0x1.142bfeb9a0474p-2, -0x1.9e7a4a75619eep-56},
    {0x1.4d80000000000p+0, 0x1.0ed005f657da4p-2, 0x1.c56bd2abfe82ap-56},
    {0x1.4bd0000000000p+0, 0x1.099e371c0bc82p-2, -0x1.9f2684d93ab38p-59},
    {0x1.4a20000000000p+0, 0x1.0465a08154ffap-2, -0x1.05f0ad83878e2p-56},
    {0x1.4880000000000p+0, 0x1.feb0233e607ccp-3, 0x1.6e32d5e8c707fp-57},
    {0x1.46e0000000000p+0, 0x1.f488311d1b493p-3, -0x1.058a0d0c0c448p-57},
    {0x1.4540000000000p+0, 0x1.ea5349e23ac0ep-3, -0x1.b2ce30cd2d061p-58},
    {0x1.43a0000000000p+0, 0x1.e0114c533197fp-3, -0x1.4990bcaac412fp-59},
    {0x1.4210000000000p+0, 0x1.d627d7c1b2da7p-3, -0x1.41d2fa017c9e1p-57},
    {0x1.4080000000000p+0, 0x1.cc320c0176502p-3, 0x1.039a653793a85p-57},
    {0x1.3ef0000000000p+0, 0x1.c22fca31887ddp-3, 0x1.58817bad161d4p-64},
    {0x1.3d60000000000p+0, 0x1.b820f2fc7e508p-3, 0x1.77bcc3821db0fp-57},
    {0x1.3bd0000000000p+0, 0x1.ae05669628825p-3, 0x1.b09879b60e908p-58},
    {0x1.3a50000000000p+0, 0x1.a4454820d19fap-3, -0x1.89c33fab39712p-58},
    {0x1.38d0000000000p+0, 0x1.9a7938d209947p-3, 0x1.63756352dcf6dp-57},
    {0x1.3750000000000p+0, 0x1.90a11b46b9b56p-3, 0x1.01375545b6e9ap-63},
    {0x1.35e0000000000p+0, 0x1.8726935acac62p-3, 0x1.764c6465f6264p-57},
    {0x1.3460000000000p+0, 0x1.7d36832b8f0e3p-3, -0x1.74cf74e521faap-58},
    {0x1.32f0000000000p+0, 0x1.73a4d01722e5cp-3, -0x1.9403e4d3a5052p-57},
    {0x1.3180000000000p+0, 0x1.6a079d0f7aad2p-3, -0x1.eedcbac2a7f18p-62},
    {0x1.3020000000000p+0, 0x1.60ca8fe8858afp-3, 0x1.2287fa61504f0p-57},
    {0x1.2eb0000000000p+0, 0x1.57168c4aff0e6p-3, -0x1.2e7b6fdae802cp-58},
    {0x1.2d50000000000p+0, 0x1.4dc378969b1c1p-3, 0x1.ad9bb79187618p-58},
    {0x1.2bf0000000000p+0, 0x1.446579dc223dep-3, -0x1.c2a5423d9a9f7p-57},
    {0x1.2a90000000000p+0, 0x1.3afc766c1e210p-3, -0x1.2bf469fab63cap-58},
    {0x1.2930000000000p+0, 0x1.3188543c098a1p-3, 0x1.51c0051368273p-58},
    {0x1.27e0000000000p+0, 0x1.2877bbc0b6ba6p-3, -0x1.7205e9247dde8p-60},
    {0x1.2690000000000p+0, 0x1.1f5cd21a0d938p-3, 0x1.14d5ddc4da66ep-57},
    {0x1.2540000000000p+0, 0x1.16377fb124192p-3, -0x1.e540be89c1eaap-59},
    {0x1.23f0000000000p+0, 0x1.0d07ac9dcbcf8p-3, -0x1.3bdf113483a79p-57},
    {0x1.22a0000000000p+0, 0x1.03cd40a51ac0dp-3, 0x1.2f3828ce0d1ffp-57},
    {0x1.2150000000000p+0, 0x1.f510466fd80bfp-4, 0x1.b95ae75fde97ep-58},
    {0x1.2010000000000p+0, 0x1.e353fec9a2699p-4, -0x1.84447930b489ep-62},
    {0x1.1ed0000000000p+0, 0x1.d183f87ea737cp-4, 0x1.46a84404a2c41p-58},
    {0x1.1d90000000000p+0, 0x1.bfa007672aa23p-4, -0x1.745a21d1323b7p-58},
    {0x1.1c50000000000p+0, 0x1.ada7fec6ac801p-4, 0x1.01a5d7c4daf48p-59},
    {0x1.1b10000000000p+0, 0x1.9b9bb14949167p-4, -0x1.cdb2f79dfe743p-59},
    {0x1.19e0000000000p+0, 0x1.8a6377a915c29p-4, -0x1.1296e6f9d7a43p-58},
    {0x1.18b0000000000p+0, 0x1.7918a1bf981d6p-4, 0x1.11d0f40e35710p-59},
    {0x1.1780000000000p+0, 0x1.67bb0726ec0fcp-4, -0x1.b692c214ddbecp-58},
    {0x1.1650000000000p+0, 0x1.564a7ef514311p-4, 0x1.9517cbf107190p-59},
    {0x1.1520000000000p+0, 0x1.44c6dfb9b7606p-4, 0x1.75f0688514f9bp-58},
    {0x1.13f0000000000p+0, 0x1.332fff7bd1f18p-4, 0x1.41527a4ec5456p-59},
    {0x1.12d0000000000p+0, 0x1.22743457a9c8ep-4, -0x1.4bdf5146181b1p-58},
    {0x1.11a0000000000p+0, 0x1.10b75afd660c6p-4, 0x1.7330e591f5790p-60},
    {0x1.1080000000000p+0, 0x1.ffae9119b9303p-5, 0x1.ba13162a9c446p-60},
    {0x1.0f60000000000p+0, 0x1.ddcaadb46ef1bp-5, 0x1.09ab6f79cf161p-62},
    {0x1.0e40000000000p+0, 0x1.bbc2bfc44f417p-5, 0x1.e5bafa0943c21p-60},
    {0x1.0d20000000000p+0, 0x1.99967a4f2b1c8p-5, 0x1.976b97544edd3p-59},
    {0x1.0c10000000000p+0, 0x1.792e93e5199edp-5, -0x1.a883781558c79p-59},
    {0x1.0af0000000000p+0, 0x1.56bac43ed7f9ap-5, -0x1.5c8202e48debep-61},
    {0x1.09e0000000000p+0, 0x1.360ebf5d83765p-5, 0x1.9281d2d2c97b2p-59},
    {0x1.08d0000000000p+0, 0x1.15413ca0e72a8p-5, -0x1.b1d2c1c45ef5ep-59},
    {0x1.07c0000000000p+0, 0x1.e8a3ee30cdcacp-6, 0x1.7086b1c00b395p-63},
    {0x1.06b0000000000p+0, 0x1.a68151fb5c04ap-6, -0x1.080ed414e3611p-64},
    {0x1.05a0000000000p+0, 0x1.641a176270d6fp-6, 0x1.8ca45dca6d9e5p-60},
    {0x1.0490000000000p+0, 0x1.216daf6d9321ap-6, -0x1.87ca4f815f331p-60},
    {0x1.0390000000000p+0, 0x1.c4db352e6d472p-7, -0x1.f0d97312e07a1p-61},
    {0x1.0280000000000p+0, 0x1.3e7295d25a7d9p-7, -0x1.ff29a11443a06p-65},
    {0x1.0180000000000p+0, 0x1.7ee11ebd82e94p-8, -0x1.61e96e2fc5d90p-62},
    {0x1.0000000000000p+0, 0x0.0p+0, 0x0.0p+0},
};

// 1 - exp(-x) for x >= 0 (finite).  x = k ln2/128 + r, |r| <= ln2/256 + the
// rounding of the FP32 quotient: 1 - exp(-x) = (1 - T) + T (1 - exp(-r)), T =
// 2^(-k/128).  For x > 64 the result rounds to 1.
RT_FN double one_minus_exp(double x) {
  const bool big = bits_of(x) > 0x4050000000000000ll;  // x > 64
  const float xf = big ? 64.0f : cut(x);
  const float kf = rintf(xf * 184.664965f);  // 128 / ln 2
  const int k = (int)kf;
  const double kd = widen(kf);
  const double r = fma(-kd, kLn2Over128Lo, fma(-kd, kLn2Over128Hi, x));
  // p = 1 - exp(-r) = r + r (-r/2 + r^2/6 - r^3 (1/24 - r/120 + r^2/720))
  const float rf = cut(r);
  const float tail = fmaf(rf, fmaf(rf, -1.0f / 720.0f, 1.0f / 120.0f), -1.0f / 24.0f);
  double q = fma(r, widen(tail), 1.0 / 6.0);
  q = fma(r, q, -0.5);
  const double p = fma(r, r * q, r);
  const ExpEntry e = kExpTable[k & 127];
  const int m = k >> 7;
  const double T = double_of(bits_of(e.t) - ((long long)m << 52));
  const double A = m > 0 ? 1.0 - T : e.a;
  return big ? 1.0 : A + fma(T, p, m > 0 ? 0.0 : e.a_lo);
}

// exp(-x) / (1 - exp(-x)) = 1 / (exp(x) - 1) for x > 0 (zero above 709.78, where
// exp(x) - 1 overflows), with the reduction of one_minus_exp.
RT_FN double bose(double x) {
  if (bits_of(x) > 0x40862e42fefa39efll) return 0.0;
  const float kf = rintf(cut(x) * 184.664965f);
  const int k = (int)kf;
  const double kd = widen(kf);
  const double r = fma(-kd, kLn2Over128Lo, fma(-kd, kLn2Over128Hi, x));
  const float rf = cut(r);
  const float tail = fmaf(rf, fmaf(rf, -1.0f / 720.0f, 1.0f / 120.0f), -1.0f / 24.0f);
  double q = fma(r, widen(tail), 1.0 / 6.0);
  q = fma(r, q, -0.5);
  const double p = fma(r, r * q, r);
  const ExpEntry e = kExpTable[k & 127];
  const int m = k >> 7, big = m > 960 ? m - 960 : 0;  // 2^-m in two normal factors
  const double T = double_of(bits_of(e.t) - ((long long)(m - big) << 52));
  const double A = m > 0 ? 1.0 - T : e.a;
  const double one_minus = m > 64 ? 1.0 : A + fma(T, p, m > 0 ? 0.0 : e.a_lo);
  const double z = fma(-T, p, T) / one_minus;
  return big ? z * double_of((long long)(1023 - big) << 52) : z;
}

// -ln(1 - v) for 0 <= v < 1.  y = 1 - v rounded, its rounding error kept; y =
// 2^-m z with z in (1/2, 1]; z rc = 1 + r, |r| <= 2^-8: -ln(1 - v) = m ln 2 +
// ln rc - ln(1 + r).  On the last interval of z with m = 0, rc = 1 and r = -v
// exactly, so small v keep their relative precision.
RT_FN double neg_log_one_minus(double v) {
  const double y = 1.0 - v;
  const double err = (1.0 - y) - v;  // exact; zero for v >= 1/2
  const long long b = bits_of(y) - 1;  // 1 and the other powers of two end their interval
  const int m = 1022 - (int)(b >> 52);
  const LogEntry e = kLogTable[(int)(b >> 45) & 127];
  const double z = double_of(bits_of(y) + ((long long)m << 52));
  const double r = fma(err, e.rc, fma(z, e.rc, -1.0));
  // -ln(1 + r) = -r + r (r/2 - r^2/3 + r^3/4 - r^4 (1/5 - r/6 + r^2/7))
  const float rf = cut(r);
  const float tail = fmaf(rf, fmaf(rf, -1.0f / 7.0f, 1.0f / 6.0f), -1.0f / 5.0f);
  double q = fma(r, widen(tail), 0.25);
  q = fma(r, q, -1.0 / 3.0);
  q = fma(r, q, 0.5);
  const double md = widen((float)m);
  const double L = fma(md, kLn2, e.ln);
  return L + (fma(r, r * q, -r) + fma(md, kLn2Lo, e.ln_lo));
}

}  // namespace rtk
