// Exponential and logarithm in 64-bit fixed point, for the rate constants.
//
// GB300 retires one FP64 warp instruction per 64 clocks on a sub-partition and a 64 x 64 -> high
// 64 bit integer multiply in 17-20 (measured), so the exponentials and the logarithm of the rate
// evaluation, most of its FP64 instructions, run on the integer pipe.  Logarithms are base 2 and
// kept as int64 with 52 fraction bits ("fx", range +-2048): ln k = ln A + b ln T - E/T is a sum
// of terms of size 10-100, whose FP64 rounding errors are 2^-50..2^-47 absolute.  In fx, in units of 2^-52:
// log2 A is rounded (1/2), the products with b and with 1/T are truncated (below 1 each), and the error of
// log2 T (below 0.9) counts |b| times: for |b| <= 2 the sum is within 4.5 units, 2^-49.8, of the exact
// one.  In a species' g/RT the term a_6/T is doubled after its truncation (below 2).
// Everything here also compiles for the host.
#pragma once
#include <cstdint>
#include <cstring>
#ifdef __CUDACC__
#define CHEM_FX_FN __device__ __forceinline__
#define CHEM_FX_TABLE static __device__ const  // global memory: the lanes of a warp read different entries
#else
#define CHEM_FX_FN inline
#define CHEM_FX_TABLE static const
#endif

namespace chemgpu {

typedef int64_t fx_t;  // value * 2^52
constexpr int kFxBits = 52;
constexpr fx_t kFxOne = (fx_t)1 << kFxBits;
constexpr double kLog2e = 1.4426950408889634074;

CHEM_FX_FN int64_t fx_bits(double v) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(v);
#else
  int64_t b;
  std::memcpy(&b, &v, 8);
  return b;
#endif
}
CHEM_FX_FN double fx_from_bits(int64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double v;
  std::memcpy(&v, &b, 8);
  return v;
#endif
}
// The bits of |v|, ordered like the magnitudes, NaN above infinity.  Not fx_bits(v) & 0x7ff..f: the compiler
// may make that an fabs, and abs.f64 passes a NaN through with its sign, so that CUDA's own NaN
// (0xfff8...) compares as a negative integer.
CHEM_FX_FN uint64_t fx_mag(double v) {
#ifdef __CUDA_ARCH__
  unsigned hi;
  asm("and.b32 %0, %1, 0x7fffffff;" : "=r"(hi) : "r"(__double2hiint(v)));
  return (uint64_t)hi << 32 | (unsigned)__double2loint(v);
#else
  return (uint64_t)fx_bits(v) & 0x7fffffffffffffffULL;
#endif
}
// high 64 bits of the signed product
CHEM_FX_FN int64_t fx_mulhi(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (int64_t)(((__int128)a * b) >> 64);
#endif
}
CHEM_FX_FN int32_t fx_mulhi32(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int32_t)(((int64_t)a * b) >> 32);
#endif
}

CHEM_FX_FN uint64_t fx_umulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// 1/a outside the normal range of fx_rcp (kept out of line)
#ifdef __CUDACC__
static __device__ __noinline__ double fx_rcp_wide(double a) { return 1.0 / a; }
#else
inline double fx_rcp_wide(double a) { return 1.0 / a; }
#endif

// 1/a of a normal a (exponent field 3 .. 2043) by Newton's iteration r <- r + r (1 - m r) on the significand
// m in [1, 2) as integers: two steps from a seed with an error below 2^-22 reach 2^-62, so the
// rounded result is within 0.51 units in the last place.  No FP64 instruction (a Newton iteration in
// FP64 takes four).  seed: the bits of a float next to 1/m in [1/2, 1].  r: the reciprocal of the significand
// before rounding, in (1/2, 1], unit 2^-64.
CHEM_FX_FN double fx_rcp_from(double a, uint32_t seed, uint64_t& r) {
  const int64_t b = fx_bits(a);
  const int ef = (int)((b >> 52) & 0x7ff);
  const uint64_t m = ((uint64_t)b << 11) | 0x8000000000000000ULL;  // unit 2^-63
  // the seed as a 32-bit fraction (1 itself as 1 - 2^-24, inside its error).  Its leading bit is added, not set: for
  // m next to 2 the seed may come out below 1/2, as 0x3effffff, whose shifted bits carry out and leave 2^31 - 2^8
  const uint32_t r0 = seed >= 0x3f800000u ? 0xffffff00u : (seed << 8) + 0x80000000u;
  r = (uint64_t)r0 << 32;  // unit 2^-64
  int64_t e = (int64_t)(0x8000000000000000ULL - fx_umulhi(m, r));  // 1 - m r, unit 2^-63, below 2^42
  r += (uint64_t)((int64_t)((uint64_t)fx_mulhi((int64_t)(r >> 1), e << 21)) >> 19);
  e = (int64_t)(0x8000000000000000ULL - fx_umulhi(m, r));          // below 2^21
  r += (uint64_t)(fx_mulhi((int64_t)(r >> 1), e << 42) >> 40);
  // round r in (1/2, 1] to 53 bits; its leading bit adds one to the exponent field.  A power of two
  // (m = 1) leaves r next to 1: set the result directly
  const uint64_t mant = (r >> 11) + ((r >> 10) & 1);
  const int64_t res = (b & 0xfffffffffffffLL) == 0 ? (int64_t)(2046 - ef) << 52 : ((int64_t)(2044 - ef) << 52) + (int64_t)mant;
  return fx_from_bits(res | (b & (int64_t)0x8000000000000000ULL));
}

// 1/a from the FP32 approximate reciprocal (rcp.approx, documented within one unit in the last place: 2^-23).
// Zero, subnormal, very large, infinite and NaN arguments take the division (r = 0).
CHEM_FX_FN double fx_rcp(double a, uint64_t& r) {
  const int64_t b = fx_bits(a);
  const int ef = (int)((b >> 52) & 0x7ff);
  if (ef < 3 || ef > 2043) {
    r = 0;
    return fx_rcp_wide(a);
  }
  const uint32_t mf = 0x3f800000u | ((uint32_t)(b >> 29) & 0x7fffffu);
  uint32_t rf;
#ifdef __CUDA_ARCH__
  float s;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(__uint_as_float(mf)));
  rf = __float_as_uint(s);
#else
  float x;
  std::memcpy(&x, &mf, 4);
  x = 1.0f / x;
  std::memcpy(&rf, &x, 4);
#endif
  return fx_rcp_from(a, rf, r);
}
CHEM_FX_FN double fx_rcp(double a) {
  uint64_t r;
  return fx_rcp(a, r);
}

// 2^((2 j + 1) / 256) * 2^62
CHEM_FX_TABLE uint64_t c_fx_exp2[128] = {
    0x402c6be96af2fb58ULL, 0x4085a050ec0a036aULL, 0x40df50b846ef302bULL, 0x41397dcbd952c4a6ULL,
    0x41942838f07e22a3ULL, 0x41ef50adcaa0d899ULL, 0x424af7d9981f7e98ULL, 0x42a71e6c7ce464afULL,
    0x4303c51791b21550ULL, 0x4360ec8ce577ae44ULL, 0x43be957f7ea712b6ULL, 0x441cc0a35c8cf8eaULL,
    0x447b6ead78aad636ULL, 0x44daa053c812abd2ULL, 0x453a564d3cc4b723ULL, 0x459a9151c70f0819ULL,
    0x45fb521a56ef0042ULL, 0x465c9960dd74bd4bULL, 0x46be67e04e28717cULL, 0x4720be54a071ad01ULL,
    0x47839d7ad1009a90ULL, 0x47e70610e3393241ULL, 0x484af8d5e2a06536ULL, 0x48af7689e44b44eaULL,
    0x49147fee085028d6ULL, 0x497a15c47b39d53eULL, 0x49e038d0777ca5e0ULL, 0x4a46e9d646edbf6aULL,
    0x4aae299b443c4a6bULL, 0x4b15f8e5dc6cbab0ULL, 0x4b7e587d905625d1ULL, 0x4be7492af621abd6ULL,
    0x4c50cbb7bacbf4cbULL, 0x4cbae0eea3a8c63cULL, 0x4d25899b8fe8b365ULL, 0x4d90c68b7a20eb1eULL,
    0x4dfc988c79d52661ULL, 0x4e69006dc503ba65ULL, 0x4ed5feffb1b3d155ULL, 0x4f439513b785cc80ULL,
    0x4fb1c37c7145d328ULL, 0x50208b0d9e8090dfULL, 0x508fec9c251a267cULL, 0x50ffe8fe12e750c4ULL,
    0x5170810a9f48c7cfULL, 0x51e1b59a2cc8da3eULL, 0x525387864abb4762ULL, 0x52c5f7a9b6df5b77ULL,
    0x533906e05f045106ULL, 0x53acb60762affaaeULL, 0x542105fd14c7b869ULL, 0x5495f7a0fd3bbb8eULL,
    0x550b8bd3dab49cbdULL, 0x5581c377a44346f0ULL, 0x55f89f6f8b133af4ULL, 0x5670209ffc1f2e82ULL,
    0x56e847eea1e80a49ULL, 0x57611642662e4a33ULL, 0x57da8c8373adc331ULL, 0x5854ab9b37dbd1e5ULL,
    0x58cf747464a7f584ULL, 0x594ae7faf23eda52ULL, 0x59c7071c20cfd70cULL, 0x5a43d2c67a54e0c0ULL,
    0x5ac14be9d45cf869ULL, 0x5b3f737751d915c8ULL, 0x5bbe4a6164eb92f4ULL, 0x5c3dd19bd0ba1c1aULL,
    0x5cbe0a1bab4226dfULL, 0x5d3ef4d75f2ff504ULL, 0x5dc092c6adb825b8ULL, 0x5e42e4e2b073d935ULL,
    0x5ec5ec25db3f6a41ULL, 0x5f49a98bfe1bc11cULL, 0x5fce1e124712437cULL, 0x60534ab7441b6546ULL,
    0x60d9307ae507dd9aULL, 0x615fd05e7d6c83e4ULL, 0x61e72b64c690d8afULL, 0x626f4291e1603dd5ULL,
    0x62f816eb585de1edULL, 0x6381a978219b628fULL, 0x640bfb40a0b22959ULL, 0x64970d4ea8bf8766ULL,
    0x6522e0ad7e639312ULL, 0x65af7669d9c2cbe4ULL, 0x663ccf91e88a8873ULL, 0x66caed354ff83222ULL,
    0x6759d0652ee352afULL, 0x67e97a341fca775bULL, 0x6879ebb63ae2edc6ULL, 0x690b2601182b5e56ULL,
    0x699d2a2bd181482aULL, 0x6a2ff94f04b962b0ULL, 0x6ac39484d5bae8c5ULL, 0x6b57fce8f09dd17fULL,
    0x6bed33988bcbfab5ULL, 0x6c8339b26a25494eULL, 0x6d1a1056dd26c382ULL, 0x6db1b8a7c714a92bULL,
    0x6e4a33c89d278e49ULL, 0x6ee382de69bc7bf8ULL, 0x6f7da70fce881bf9ULL, 0x7018a18506ccf314ULL,
    0x70b47367e994ae92ULL, 0x71511de3ebec8913ULL, 0x71eea2262324cb0cULL, 0x728d015d47136b40ULL,
    0x732c3cb9b459d38bULL, 0x73cc556d6eadce5fULL, 0x746d4cac2325a155ULL, 0x750f23ab2a87593eULL,
    0x75b1dba18b9b4c20ULL, 0x765575c7fd81d5a0ULL, 0x76f9f358ea0c5249ULL, 0x779f559070195e36ULL,
    0x78459dac65f45bb5ULL, 0x78ecccec5bb84661ULL, 0x7994e4919db5d74eULL, 0x7a3de5df36dcfeefULL,
    0x7ae7d219f329b948ULL, 0x7b92aa886214411cULL, 0x7c3e7072d904a6ceULL, 0x7ceb252375c9cf9bULL,
    0x7d98c9e62113e1faULL, 0x7e47600890f223deULL, 0x7ef6e8da4b544f9aULL, 0x7fa765aca88f6453ULL};
// round(2^15 / (1 + (2 i + 1) / 256)): reciprocals of the midpoints of the 128 significand intervals
CHEM_FX_TABLE uint16_t c_fx_rcp[128] = {
    32640, 32388, 32140, 31896, 31655, 31418, 31184, 30954, 30728, 30504, 30284, 30067, 29853, 29642, 29434, 29229,
    29026, 28827, 28630, 28436, 28244, 28056, 27869, 27685, 27504, 27324, 27148, 26973, 26801, 26631, 26462, 26297,
    26133, 25971, 25811, 25653, 25497, 25343, 25191, 25041, 24892, 24745, 24600, 24457, 24315, 24175, 24036, 23899,
    23764, 23630, 23498, 23367, 23237, 23109, 22982, 22857, 22733, 22611, 22490, 22370, 22251, 22134, 22017, 21902,
    21789, 21676, 21565, 21454, 21345, 21237, 21130, 21024, 20919, 20815, 20713, 20611, 20510, 20410, 20311, 20214,
    20117, 20021, 19925, 19831, 19738, 19645, 19554, 19463, 19373, 19284, 19196, 19108, 19022, 18936, 18851, 18766,
    18683, 18600, 18518, 18437, 18356, 18276, 18197, 18118, 18040, 17963, 17886, 17810, 17735, 17660, 17586, 17513,
    17440, 17368, 17296, 17225, 17155, 17085, 17015, 16947, 16878, 16811, 16744, 16677, 16611, 16546, 16481, 16416};
// -log2 of those reciprocals * 2^56
CHEM_FX_TABLE int64_t c_fx_log2[128] = {
    0x001720d9c06a836LL, 0x0044edafb0d43e5LL, 0x007259d23b43df1LL, 0x009f624dfe13bd6LL,
    0x00cc33f19777050LL, 0x00f89ca86eb0ea5LL, 0x0124c9ea8884545LL, 0x015088dbb155c07LL,
    0x017bd662dcb6237LL, 0x01a7128f47ca26aLL, 0x01d1d87c3ec9f6fLL, 0x01fc574cd45dc84LL,
    0x02268ce274ce83bLL, 0x025077186dbc4b2LL, 0x027a13c41651106LL, 0x02a360b4fa779b2LL,
    0x02cc8fd2ffca26cLL, 0x02f53702d667fdfLL, 0x031dbc9c04ea157LL, 0x0345ea3a657f893LL,
    0x036df3223fd8093LL, 0x03956a41000db47LL, 0x03bcef04f2fc203LL, 0x03e413f5f59c5a7LL,
    0x040ad6b5fd9f331LL, 0x0431a39ca8efefaLL, 0x0457d3411c6d12dLL, 0x047e0a648af1faaLL,
    0x04a3d7ddfffcd5bLL, 0x04c97208d295078LL, 0x04ef10add311e30LL, 0x051406e752ddd7cLL,
    0x0538fecc1dec987LL, 0x055dbdc4a55d260LL, 0x05824260877ea3dLL, 0x05a68b2bf45543aLL,
    0x05ca96afc449047LL, 0x05ee637190365f4LL, 0x0611eff3cae6d95LL, 0x06353ab5dbf71b1LL,
    0x06587ef9f40e32fLL, 0x067b7f2c3853ed7LL, 0x069e39c312719a7LL, 0x06c0ad3240bdb14LL,
    0x06e31621ddec30cLL, 0x070535819f94db7LL, 0x072748ad0479d61LL, 0x07490fd5d45902dLL,
    0x076a89628fb1fc8LL, 0x078bf3bc482d90bLL, 0x07ad0df8735ff99LL, 0x07ce1733e3203efLL,
    0x07ef0ee0bce160cLL, 0x080fb2f88b3ffdaLL, 0x083043a6a6c1e98LL, 0x08507e274da9cb8LL,
    0x0870a35a79e65e3LL, 0x08906fbfb015534LL, 0x08b024eb6f10ab3LL, 0x08cfc240ec921a1LL,
    0x08ef4721a605e89LL, 0x090e6e945a73d31LL, 0x092dc04c2ec6d7dLL, 0x094cb296e5f3470LL,
    0x096b43b99fd4ba5LL, 0x0989fd8c6363327LL, 0x09a8542dd4dbb82LL, 0x09c6d2e3be56488LL,
    0x09e4ec581b8a9ceLL, 0x0a02e603729babcLL, 0x0a20bf360ef3d65LL, 0x0a3e773ebaa4b8bLL,
    0x0a5c0d6ac384986LL, 0x0a798106009be36LL, 0x0a9688516a077ecLL, 0x0ab3b44c4e36211LL,
    0x0ad0bb915e0b561LL, 0x0aed9d66d58e0b8LL, 0x0b0a59119a0eaadLL, 0x0b26a2fe40e0a83LL,
    0x0b430fc0b7d6a29LL, 0x0b5f541f8190a53LL, 0x0b7bbb46668d13cLL, 0x0b97acf85bbb7bbLL,
    0x0bb3740298efe1aLL, 0x0bcf5ca277e7143LL, 0x0beacc6d2e4120fLL, 0x0c065cfb5b75fa9LL,
    0x0c21c084e13b786LL, 0x0c3cf6418ecd595LL, 0x0c57fd683c3caf0LL, 0x0c732459c24e08eLL,
    0x0c8dcc50f556aa4LL, 0x0ca893341d425deLL, 0x0cc3290afbea499LL, 0x0cdddda3b7b2df0LL,
    0x0cf80f5297ffc91LL, 0x0d125edcc87f98bLL, 0x0d2c7ad4e55fedeLL, 0x0d46626926c2a08LL,
    0x0d6067305aa7abeLL, 0x0d7a36a5ed76f7aLL, 0x0d93cff55caa3e3LL, 0x0dad85c7f5c48e7LL,
    0x0dc7048198bb61fLL, 0x0de04b4b391265dLL, 0x0df9ade0f354586LL, 0x0e12d78f049181bLL,
    0x0e2bc77c0c3262cLL, 0x0e44d277034f9b2LL, 0x0e5da2b4b7ac3bfLL, 0x0e763759afc2ad0LL,
    0x0e8ee647894157aLL, 0x0ea7589c240f10bLL, 0x0ebfe4f049faa5eLL, 0x0ed833a7ceaa2abLL,
    0x0ef043e3bbf09ffLL, 0x0f086d4fc64089bLL, 0x0f20b020dfeed0aLL, 0x0f385a023747319LL,
    0x0f5075df5b5ad70LL, 0x0f67f708d3673aeLL, 0x0f7f9039c915ed4LL, 0x0f9741a3907c380LL,
    0x0faeb0654925d4bLL, 0x0fc5db9a742ba0cLL, 0x0fdd1e2847c5705LL, 0x0ff4783e007ac55LL};

// the value of an fx (one conversion, exact scaling)
CHEM_FX_FN double fx_value(fx_t x) { return (double)x * (1.0 / 4503599627370496.0); }

// v as fx, |v| < 1024 (the caller's condition; v is rounded to nearest on the last bit)
CHEM_FX_FN fx_t fx_of(double v) {
  const int64_t b = fx_bits(v);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;
  const int64_t m = (b & 0xfffffffffffffLL) | 0x10000000000000LL;
  int64_t r;
  if (e >= 0) r = m << (e & 15);
  else r = (e < -60) ? 0 : ((m >> (-1 - e)) + 1) >> 1;
  return b < 0 ? -r : r;
}

// exp2 of a double outside the fixed-point path (rare, kept out of line)
#ifdef __CUDACC__
static __device__ __noinline__ double fx_exp2_wide(double v) { return exp2(v); }
#else
inline double fx_exp2_wide(double v) { return __builtin_exp2(v); }
#endif

// 2^x of an fx.  x = n + (j + 1/2) / 128 + r, |r| <= 2^-8: 2^x = 2^n t_j 2^r with t_j from a table
// (62 fraction bits) and 2^r = 1 + z + z^2/2 + z^3 (1/6 + z/24 + z^2/120), z = r ln 2, |z| <= 2^-8.5
// (the next term is below 2^-60); z and z^2 as 64-bit products, the cubic and up (below 2^-28) as
// 32-bit ones.  The error before the final rounding to double is below 2^-56.5 relative.
// Outside |x| < 1020 the result is exp2 of the value (overflow, subnormals and zero as there).
CHEM_FX_FN double fx_exp2(fx_t x) {
  const int64_t lim = 1020LL << kFxBits;
  if (x >= lim || x <= -lim) {
    const double v = fx_value(x);
    return fx_exp2_wide(v);
  }
  const int n = (int)(x >> kFxBits);
  const int j = (int)(x >> 45) & 127;
  const int64_t r = (x & ((1LL << 45) - 1)) - (1LL << 44);  // unit 2^-52
  const int64_t z = fx_mulhi(r << 13, 0x58b90bfbe8e7bcd6LL);   // ln 2 * 2^63: z in units 2^-64
  const int64_t z2 = fx_mulhi(z << 7, z << 7);                 // unit 2^-78
  const int32_t zh = (int32_t)(z >> 25);                       // unit 2^-39
  const int32_t z2h = (int32_t)(z2 >> 31);                     // unit 2^-47
  const int32_t q1 = 1431655765 + fx_mulhi32(zh, 2236962);     // 1/24 + z/120, unit 2^-35
  const int32_t q = 1431655765 + (fx_mulhi32(zh, q1) >> 9);    // 1/6 + z q1, unit 2^-33
  const int32_t z3 = (int32_t)(((int64_t)z2h * zh) >> 30);     // unit 2^-56
  const int64_t p = z + (z2 >> 15) + (((int64_t)z3 * q) >> 25);  // unit 2^-64
  const int64_t t = (int64_t)c_fx_exp2[j];
  const int64_t m = t + fx_mulhi(t, p);                        // unit 2^-62, in [2^62, 2^63)
  // round to 53 bits; the implicit bit adds one to the exponent field
  return fx_from_bits(((int64_t)(n + 1022) << 52) + ((m + 512) >> 10));
}

// log2 of a positive normal double as fx.  m = the significand in [1, 2), c = a 15-bit reciprocal
// of the midpoint of its interval: r = m c - 1 is exact (|r| < 2^-7.9), and
// ln(1 + r) = r - r^2/2 + r^3 (1/3 - r/4 + r^2/5 - r^3/6 + r^4/7), the cubic and up in 32-bit
// products.  Absolute error below 2^-52 with the rounding to fx.
CHEM_FX_FN fx_t fx_log2(double x) {
  const int64_t b = fx_bits(x);
  const int e = (int)(b >> 52) - 1023;
  const int i = (int)(b >> 45) & 127;
  const int64_t m = (b & 0xfffffffffffffLL) | 0x10000000000000LL;
  const int64_t r = (int64_t)((uint64_t)m * (uint64_t)c_fx_rcp[i]);  // mod 2^64: (m c - 1), unit 2^-67
  const int64_t r2 = fx_mulhi(r << 3, r << 3);                 // unit 2^-76
  const int32_t rh = (int32_t)((r + (1LL << 28)) >> 29);                     // unit 2^-38
  const int32_t r2h = (int32_t)(r2 >> 30);                     // unit 2^-46
  int32_t q = -715827883 + fx_mulhi32(rh, 9586981);            // -1/6 + r/7, unit 2^-32
  q = 858993459 + (fx_mulhi32(rh, q) >> 6);                    // 1/5 + r q
  q = -1073741824 + (fx_mulhi32(rh, q) >> 6);                  // -1/4 + r q
  q = 1431655765 + (fx_mulhi32(rh, q) >> 6);                   // 1/3 + r q
  const int32_t r3 = (int32_t)(((int64_t)r2h * rh) >> 30);     // unit 2^-54
  const int64_t l = r - (r2 >> 10) + (((int64_t)r3 * q) >> 19);  // ln(1 + r), unit 2^-67
  const int64_t l2 = fx_mulhi(l << 3, 0x5c551d94ae0bf85eLL);   // / ln 2: unit 2^-70 2^-62 2^64 = 2^-68
  return ((int64_t)e << kFxBits) + (((int64_t)c_fx_log2[i] + (l2 >> 12) + 8) >> 4);
}

// 2^v of any double
CHEM_FX_FN double fx_exp2_of(double v) {
  return fx_mag(v) < 0x408fe00000000000ULL ? fx_exp2(fx_of(v)) : fx_exp2_wide(v);  // |v| < 1020
}

// whether fx_log2 takes x: positive and normal
CHEM_FX_FN bool fx_log2_takes(double x) {
  const int64_t b = fx_bits(x);
  return b >= 0x0010000000000000LL && b < 0x7ff0000000000000LL;
}

}  // namespace chemgpu
