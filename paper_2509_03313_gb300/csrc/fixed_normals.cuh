// The pieces of the FP64 mode's Box-Muller transform in 64-bit fixed point.
//
// The FP64 pipe of this part issues two lanes per clock and SM, so a logarithm, a square
// root and a sine-cosine pair in double precision cost a warp some two thousand cycles,
// while the integer multipliers run 32 to 64 lanes per clock. The arguments are 53-bit
// integers (the uniforms of the Philox block), which suits fixed point: no argument
// reduction is rounded, and every result carries at least 58 correct bits before its one
// rounding to double, so the errors stay below those of the double-precision functions.
// An FP64 evaluation of the transform rounds the angle 2 pi u and the logarithm to double before
// it goes on, and so do these: the angle's difference from 2 pi u is formed exactly from the
// integers and added to the folded angle to first order, the logarithm is rounded before the
// root. (Positions after 1,000 steps of 2,000 species are 4.7e-17 from an FP64 evaluation's,
// 2.0e-16 with the logarithm unrounded or with double-precision functions, 6.9e-16 with the
// angle unrounded too; the roundings cost the FP64 mode's passes 1 to 3 %.) The diffusion of 1e6 FP64
// species, with the cells and offsets taken on the FP32 pipe (cell_index_split), went from
// 313 to some 65 us.
//
// Methods, from the mathematics: octant folding and the Taylor polynomials of sine and
// cosine on [0, pi/4] by Horner's rule; the logarithm by a table of ln(R_i / 512), R_i =
// floor(2^17 / (129 + i)), and the series of -ln(1 - t), 0 <= t < 0.01; the square root by
// two Newton steps from a single-precision reciprocal square root. The constants are
// 2^64 / n!, 2^64 pi / 4, 2^58 ln 2 and the table 2^64 ln(R_i / 512), rounded to nearest.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define FN_FN __device__ __forceinline__
#define FN_TABLE static __device__ const
#else  // the same arithmetic on the host, for its tests
#include <cmath>
#define FN_FN inline
#define FN_TABLE static const
#endif

namespace chem {
namespace fixedn {

FN_FN uint32_t hi32(uint64_t a) { return static_cast<uint32_t>(a >> 32); }
FN_FN uint32_t lo32(uint64_t a) { return static_cast<uint32_t>(a); }
FN_FN uint64_t mul_wide(uint32_t a, uint32_t b) { return static_cast<uint64_t>(a) * b; }
FN_FN uint32_t mh32(uint32_t a, uint32_t b) {
#ifdef __CUDACC__
  return __umulhi(a, b);
#else
  return hi32(mul_wide(a, b));
#endif
}
// High half of a 64 x 64 bit product without the low x low term: at most 3 too small.
FN_FN uint64_t mh64(uint64_t a, uint64_t b) {
  return mul_wide(hi32(a), hi32(b)) + mh32(hi32(a), lo32(b)) + mh32(lo32(a), hi32(b));
}
FN_FN int clz64(uint64_t v) {  // v != 0
#ifdef __CUDACC__
  return __clzll(static_cast<long long>(v));
#else
  return __builtin_clzll(v);
#endif
}

// v 2^-e rounded to double (0 for v = 0; the results here are normal numbers).
FN_FN double to_double(uint64_t v, int e) {
  const int lz = clz64(v | 1u);
  v <<= lz;
  // 53 bits, rounded; a carry out of the fraction moves the exponent by itself
  const uint64_t r = (v >> 11) + ((v >> 10) & 1u);
  const uint64_t bits = v ? r + (static_cast<uint64_t>(1023 + 63 - lz - e - 1) << 52) : 0u;
#ifdef __CUDACC__
  return __longlong_as_double(static_cast<long long>(bits));
#else
  double d;
  std::memcpy(&d, &bits, 8);
  return d;
#endif
}

// The folded angle x = 2 pi m / 2^53 modulo the octants, 0 <= x <= pi/4.
struct Folded {
  uint64_t xn;  // x 2^se, its leading bits kept however small x is
  int se;
  uint64_t z;   // x^2 2^64
  int64_t d;    // what the rounding of 2 pi u to double adds to x, 2^103 units
  bool swap, neg_s, neg_c;  // sine and cosine change places; their signs
};

// fl(fl(2 pi) fl(m / 2^53)) - 2 pi m / 2^53 in units of 2^-103, below 2^53 in magnitude.
FN_FN int64_t angle_rounding(uint64_t m) {
  constexpr uint64_t TWO_PI = 0x1921fb54442d18ull;  // the double nearest 2 pi, 2^50 units
  const uint64_t lo = TWO_PI * m;
#ifdef __CUDACC__
  const uint64_t hi = __umul64hi(TWO_PI, m);
#else
  const uint64_t hi = static_cast<uint64_t>((static_cast<unsigned __int128>(TWO_PI) * m) >> 64);
#endif
  const int n = hi ? 128 - clz64(hi) : 64 - clz64(lo | 1u);  // bits of the product
  const int drop = n > 53 ? n - 53 : 0;                      // at most 53 go, to nearest, ties to even
  const uint64_t one = 1ull << drop, rem = lo & (one - 1u), half = one >> 1;
  const bool up = drop > 0 && (rem > half || (rem == half && (lo & one) != 0u));
  const int64_t e = static_cast<int64_t>(up ? rem - one : rem);
  // (2 pi minus its double) u: 2^103 units
  return -e - static_cast<int64_t>(mh64(m << 11, 0x8d313198a2e03ull));
}

FN_FN Folded fold(uint64_t m) {
  Folded f;
  const uint32_t q = static_cast<uint32_t>(m >> 50);
  uint64_t r = m & ((1ull << 50) - 1u);
  if (q & 1u) r = (1ull << 50) - r;
  r <<= 13;
  const int sh = clz64(r | 1u);
  f.xn = mh64(r << sh, 0xc90fdaa22168c235ull);
  f.se = 63 + sh;
  const uint64_t x = f.xn >> sh;  // 2^63 units
  f.z = mh64(x, x) << 2;
  const int64_t d = angle_rounding(m);
  f.d = (q & 1u) ? -d : d;
  f.swap = ((q + 1u) >> 1) & 1u;
  f.neg_s = q >= 4u;
  f.neg_c = ((q + 2u) >> 2) & 1u;
  return f;
}

// sin(x + d) from v = sin x in 2^f.se units: v + d cos x.
FN_FN double sine_at(const Folded& f, uint64_t v) {
  const int sh = f.se - 63;
  // (below 2^-45, two draws in 2^45, in double: d may be as large as x)
  if (sh > 45) return to_double(v, f.se) + static_cast<double>(f.d) * 0x1p-103;
  const uint64_t a = static_cast<uint64_t>(f.d < 0 ? -f.d : f.d);
  uint64_t D = sh <= 40 ? a >> (40 - sh) : a << (sh - 40);
  const uint32_t zh = hi32(f.z);
  if (zh >= 16u) {  // cos x to z^3 / 6!, 2^31 units
    const uint32_t z2 = mh32(zh, zh);
    const uint32_t c = 0x80000000u - (zh >> 2) + mh32(z2, 0x05555555u) - mh32(mh32(z2, zh), 0x002d82d8u);
    D = mh64(D, static_cast<uint64_t>(c) << 33);
  }
  return to_double(f.d < 0 ? v - D : v + D, f.se);
}

// cos(x + d) from v = cos x in 2^63 units: v - d sin x.
FN_FN double cosine_at(const Folded& f, uint64_t v) {
  const uint64_t a = static_cast<uint64_t>(f.d < 0 ? -f.d : f.d) >> 40;  // 2^63 units, below 2^13
  const uint32_t zh = hi32(f.z), x = hi32(f.xn >> (f.se - 63));         // 2^31 units
  const uint32_t sn = x - mh32(x, mh32(zh, 0x2aaaaaabu) - mh32(mh32(zh, zh), 0x02222222u));
  const uint64_t D = mul_wide(static_cast<uint32_t>(a), sn) >> 31;
  return to_double(f.d < 0 ? v + D : v - D, 63);
}

// sin x = x (1 - z/3! + z^2/5! - ...), to z^8 / 17!.
FN_FN double sine(const Folded& f) {
  const uint32_t zh = hi32(f.z);
  uint32_t t = 0x00d73f9fu - mh32(zh, 0x0000ca96u);
  t = 0xb092309du - mh32(zh, t);
  uint64_t s = 0x6b99159fd5ull - mh32(zh, t);
  s = 0x2e3bc74aad8eull - mh64(f.z, s);
  s = 0x000d00d00d00d00dull - mh64(f.z, s);
  s = 0x0222222222222222ull - mh64(f.z, s);
  s = 0x2aaaaaaaaaaaaaabull - mh64(f.z, s);
  s = mh64(f.z, s);
  return sine_at(f, f.xn - mh64(f.xn, s));
}

// cos x = 1 - (z/2! - z^2/4! + ...), to z^9 / 18!.
FN_FN double cosine(const Folded& f) {
  const uint32_t zh = hi32(f.z);
  uint32_t t = 0x000d73fau - mh32(zh, 0x00000b41u);
  t = 0x0c9cba54u - mh32(zh, t);
  uint64_t c = 0x8f76c77fcull - mh32(zh, t);
  c = 0x049f93edde28ull - mh64(f.z, c);
  c = 0x0001a01a01a01a02ull - mh64(f.z, c);
  c = 0x005b05b05b05b05bull - mh64(f.z, c);
  c = 0x0aaaaaaaaaaaaaabull - mh64(f.z, c);
  c = 0x8000000000000000ull - mh64(f.z, c);
  c = mh64(f.z, c);
  return cosine_at(f, 0x8000000000000000ull - (c >> 1));
}

FN_FN double with_sign(double v, bool neg) { return neg ? -v : v; }

// sin and cos of 2 pi m / 2^53 (rounded to double).
FN_FN void sincos_2pi(uint64_t m, double& s, double& c) {
  const Folded f = fold(m);
  const double a = sine(f), b = cosine(f);
  s = with_sign(f.swap ? b : a, f.neg_s);
  c = with_sign(f.swap ? a : b, f.neg_c);
}

// cos of 2 pi m / 2^53 (rounded to double): one polynomial, the coefficients chosen by the octant.
FN_FN double cos_2pi(uint64_t m) {
  const Folded f = fold(m);
  const uint32_t zh = hi32(f.z);
  const bool w = f.swap;  // the sine's
  uint32_t t = (w ? 0x00d73f9fu : 0x000d73fau) - mh32(zh, w ? 0x0000ca96u : 0x00000b41u);
  t = (w ? 0xb092309du : 0x0c9cba54u) - mh32(zh, t);
  uint64_t s = (w ? 0x6b99159fd5ull : 0x8f76c77fcull) - mh32(zh, t);
  s = (w ? 0x2e3bc74aad8eull : 0x049f93edde28ull) - mh64(f.z, s);
  s = (w ? 0x000d00d00d00d00dull : 0x0001a01a01a01a02ull) - mh64(f.z, s);
  s = (w ? 0x0222222222222222ull : 0x005b05b05b05b05bull) - mh64(f.z, s);
  s = (w ? 0x2aaaaaaaaaaaaaabull : 0x0aaaaaaaaaaaaaabull) - mh64(f.z, s);
  s = w ? s : 0x8000000000000000ull - mh64(f.z, s);
  s = mh64(f.z, s);
  const uint64_t v = w ? f.xn - mh64(f.xn, s) : 0x8000000000000000ull - (s >> 1);
  return with_sign(w ? sine_at(f, v) : cosine_at(f, v), f.neg_c);
}

struct alignas(16) LogRow {
  uint64_t ln;  // 2^64 ln(R / 512)
  uint32_t R, pad;
};

FN_TABLE LogRow LOG_TABLE[128] = {
    {0xaf70154920b3ab87ull, 1016u, 0u}, {0xad6a0261acf967d9ull, 1008u, 0u}, {0xab5fcead9f9cca09ull, 1000u, 0u},
    {0xa9516932de2d5774ull, 992u, 0u}, {0xa78151e9817830bfull, 985u, 0u}, {0xa5adeb4ab7139c6full, 978u, 0u},
    {0xa393a1f99d55698dull, 970u, 0u}, {0xa1b8fa4f11ece85dull, 963u, 0u}, {0x9fdadc268b7a12daull, 956u, 0u},
    {0x9df93a785d38659bull, 949u, 0u}, {0x9c1407f2c3cbf5fdull, 942u, 0u}, {0x9a7144ece70e98b7ull, 936u, 0u},
    {0x98854ec423189149ull, 929u, 0u}, {0x96dcaab906f11632ull, 923u, 0u}, {0x94e9bff615845643ull, 916u, 0u},
    {0x933b1009a186fe69ull, 910u, 0u}, {0x9140fd9a330cfa7full, 903u, 0u}, {0x8f8c1514d7ed8360ull, 897u, 0u},
    {0x8dd43de4c760d5c8ull, 891u, 0u}, {0x8c196de51316c6c5ull, 885u, 0u}, {0x8a5b9abbcce6889cull, 879u, 0u},
    {0x889ab9d893140c1full, 873u, 0u}, {0x87224c2e8e645fb7ull, 868u, 0u}, {0x855bb5f670a68e03ull, 862u, 0u},
    {0x8391f2e0e6fa0273ull, 856u, 0u}, {0x821205cb2f2a610cull, 851u, 0u}, {0x80425294db9c2f47ull, 845u, 0u},
    {0x7ebd623de3cc7b67ull, 840u, 0u}, {0x7ce796f204796f34ull, 834u, 0u}, {0x7b5d8165d998ed42ull, 829u, 0u},
    {0x79d109875a1e1f8eull, 824u, 0u}, {0x784227e89745a0fbull, 819u, 0u}, {0x76b0d4f8b165508cull, 814u, 0u},
    {0x751d0902fb77562aull, 809u, 0u}, {0x7386bc2e17cfadeeull, 804u, 0u}, {0x71ede67b0dbabe07ull, 799u, 0u},
    {0x70527fc457c09ab3ull, 794u, 0u}, {0x6eb47fbcea4595caull, 789u, 0u}, {0x6d13ddef323d8a33ull, 784u, 0u},
    {0x6bc4a4c91de1ac45ull, 780u, 0u}, {0x6a1f305976c66479ull, 775u, 0u}, {0x68cc100813e98dcdull, 771u, 0u},
    {0x6721ac0b70218a6full, 766u, 0u}, {0x65ca8d044d4561a6ull, 762u, 0u}, {0x641b1b88711d4e7aull, 757u, 0u},
    {0x62bfe569985dffa4ull, 753u, 0u}, {0x610b47687a2c5d25ull, 748u, 0u}, {0x5fabe0ee0abf0d93ull, 744u, 0u},
    {0x5e4a957f751e89f0ull, 740u, 0u}, {0x5ce75fdaef401a74ull, 736u, 0u}, {0x5b823aa8ae878e30ull, 732u, 0u},
    {0x5a1b207a6c52bb11ull, 728u, 0u}, {0x58b20bcae71e54beull, 724u, 0u}, {0x5746f6fd60272942ull, 720u, 0u},
    {0x55d9dc5d1569b152ull, 716u, 0u}, {0x546ab61cb7e0b427ull, 712u, 0u}, {0x52f97e55dde2836dull, 708u, 0u},
    {0x51862f08717b09f4ull, 704u, 0u}, {0x5010c21a1a9f8ef4ull, 700u, 0u}, {0x4ef7493ac52da84bull, 697u, 0u},
    {0x4d7e19724ca4f822ull, 693u, 0u}, {0x4c02bab418d42f57ull, 689u, 0u}, {0x4ae4c0eae2749277ull, 686u, 0u},
    {0x496580437dd8e7bcull, 682u, 0u}, {0x4844956618582e79ull, 679u, 0u}, {0x46c15e47c1ed22baull, 675u, 0u},
    {0x459d72aeae98380eull, 672u, 0u}, {0x44162fe6b92b5462ull, 668u, 0u}, {0x42ef336c3492f32dull, 665u, 0u},
    {0x4163cf1c0faf1799ull, 661u, 0u}, {0x4039b116b540731aull, 658u, 0u}, {0x3f0e36512aa08a03ull, 655u, 0u},
    {0x3de15b97b8b26ca4ull, 652u, 0u}, {0x3c4e0edc55e5cbd4ull, 648u, 0u}, {0x3b1df235e63abbe8ull, 645u, 0u},
    {0x39ec6a9c138bb892ull, 642u, 0u}, {0x38b974a875c8494full, 639u, 0u}, {0x37850ce85b19ac54ull, 636u, 0u},
    {0x364f2fdc8c641775ull, 633u, 0u}, {0x3517d9f9105e3186ull, 630u, 0u}, {0x33df07a4ed3467a4ull, 627u, 0u},
    {0x32a4b539e8ad68edull, 624u, 0u}, {0x3168df0446c4b67dull, 621u, 0u}, {0x302b814286afd5adull, 618u, 0u},
    {0x2eec98251e424e92ull, 615u, 0u}, {0x2dac1fce33a4391bull, 612u, 0u}, {0x2c6a1451554eaf60ull, 609u, 0u},
    {0x2b2671b330410ba7ull, 606u, 0u}, {0x2a4dcbc743686f46ull, 604u, 0u}, {0x29077999cdc7ba95ull, 601u, 0u},
    {0x27bf8561d98c5395ull, 598u, 0u}, {0x2675eaeaee1c9ecdull, 595u, 0u}, {0x259941ebebe4a10eull, 593u, 0u},
    {0x244cde3214b596fbull, 590u, 0u}, {0x22fec8b1f94c21fdull, 587u, 0u}, {0x221f1c844a736264ull, 585u, 0u},
    {0x20ce2a2594b2dc54ull, 582u, 0u}, {0x1f7b79fec37ddecfull, 579u, 0u}, {0x1e98b54967146775ull, 577u, 0u},
    {0x1d4313d66cb35d5eull, 574u, 0u}, {0x1c5e548f5bc74316ull, 572u, 0u}, {0x1b05b49bee43fe46ull, 569u, 0u},
    {0x1a1ef1d8061cd417ull, 567u, 0u}, {0x18c345d6319b20f6ull, 564u, 0u}, {0x17da766d7b12cc84ull, 562u, 0u},
    {0x16f0d28ae56b4b9cull, 560u, 0u}, {0x1590cafdf01c284full, 557u, 0u}, {0x14a50d3aa1b0400full, 555u, 0u},
    {0x13b87598b1b6edf5ull, 553u, 0u}, {0x1253f62f0a1416f9ull, 550u, 0u}, {0x116536eea37ae0e8ull, 548u, 0u},
    {0x1075983598e47130ull, 546u, 0u}, {0x0f0c838613b00addull, 543u, 0u}, {0x0e1aaee8490f9666ull, 541u, 0u},
    {0x0d27f4ffd1e91a7bull, 539u, 0u}, {0x0c34541841fb6771ull, 537u, 0u}, {0x0ac52dd7e4726a46ull, 534u, 0u},
    {0x09cf43dcff5eafd5ull, 532u, 0u}, {0x08d86cc491ecbfe1ull, 530u, 0u}, {0x07e0a6c39e0cc013ull, 528u, 0u},
    {0x06e7f009ebe465ffull, 526u, 0u}, {0x05ee46c1f56c46aaull, 524u, 0u}, {0x04f3a910d1a95d3cull, 522u, 0u},
    {0x03f815161f807c7aull, 520u, 0u}, {0x02fb88ebf0214edcull, 518u, 0u}, {0x01fe02a6b1067890ull, 516u, 0u},
    {0x00ff805515885e02ull, 514u, 0u}, {0x0000000000000000ull, 512u, 0u},
};

// -ln((m + 1) / 2^53) = v 2^-e, 0 <= m < 2^53 (m = 2^53 - 1: v = 0).
FN_FN uint64_t neg_log(uint64_t m, int& e) {
  const uint64_t M = m + 1u;
  const int lz = clz64(M);                  // 10 only for M = 2^53
  const uint64_t y = M << lz;               // w 2^64: (m + 1) / 2^53 = w 2^(11 - lz), 1/2 <= w < 1
  const uint32_t i = static_cast<uint32_t>(y >> 56) & 127u;
#ifdef __CUDACC__
  const uint4 row4 = __ldg(reinterpret_cast<const uint4*>(LOG_TABLE) + i);
  const uint64_t ln_r = (static_cast<uint64_t>(row4.y) << 32) | row4.x;
  const uint32_t R = row4.z;
#else
  const uint64_t ln_r = LOG_TABLE[i].ln;
  const uint32_t R = LOG_TABLE[i].R;
#endif
  // t = 1 - w R / 512, exact (2^64 units)
  const uint64_t t = ((1ull << 62) - (y >> 11) * R) << 2;
  const uint32_t th = hi32(t);
  // -ln(1 - t) = t + t q, q = t (1/2 + t (1/3 + ... + t/9))
  uint32_t h = 0x20000000u + mh32(th, 0x1c71c71cu);
  h = 0x24924925u + mh32(th, h);
  h = 0x2aaaaaabu + mh32(th, h);
  h = 0x33333333u + mh32(th, h);
  uint64_t g = 0x4000000000000000ull + mul_wide(th, h) + mh32(lo32(t), h);
  g = 0x5555555555555555ull + mh64(t, g);
  g = 0x8000000000000000ull + mh64(t, g);
  const uint64_t q = mh64(t, g);
  // -ln u = (lz - 11) ln 2 + ln(R / 512) + t + t q. Close to u = 1 it is t (1 + q) alone:
  // its leading bits are kept
  const int k = lz - 11;
  const int sh = (k == 0 && ln_r == 0u) ? clz64(t | 1u) - 1 : 0;
  const uint64_t tn = t << sh;
  const uint64_t frac = ln_r + tn + mh64(tn, q);  // 2^(64 + sh) units, below 2^64
  const bool big = k > 0;
  e = big ? 58 : 64 + sh;
  return k < 0 ? 0u : (big ? static_cast<uint64_t>(k) * 0x02c5c85fdf473de7ull + (frac >> 6) : frac);
}

// sqrt(2 v 2^-e).
FN_FN double root_of_twice(uint64_t v, int e) {
  // 2 v 2^-e = a 2^ea, 1/4 <= a < 1, ea even
  const int lv = clz64(v | 1u);
  uint64_t a = v << lv;
  int ea = 65 - lv - e;
  if (ea & 1) { a >>= 1; ++ea; }
  // sqrt(a): s0 = a / sqrt(a) to 21 bits, then two Newton steps s += (a - s^2) / (2 sqrt(a))
#ifdef __CUDACC__
  const float y0 = rsqrtf(static_cast<float>(hi32(a)) * 2.3283064365386963e-10f);
#else
  const float y0 = 1.0f / std::sqrt(static_cast<float>(hi32(a)) * 2.3283064365386963e-10f);
#endif
  const uint32_t Y = static_cast<uint32_t>(y0 * 1073741824.0f);  // 2^30 units, at most 2^31
  uint64_t s0 = mul_wide(hi32(a), Y) >> 30;
  s0 = s0 > 0xFFFFFFFFull ? 0xFFFFFFFFull : s0;
  const int64_t d0 = static_cast<int64_t>(a - s0 * s0);
  const uint64_t s1 = (s0 << 32) + static_cast<uint64_t>((d0 * static_cast<int64_t>(Y >> 12)) >> 19);
  const int64_t d1 = static_cast<int64_t>(a - mh64(s1, s1));
  const int64_t c1 = (d1 * static_cast<int64_t>(Y)) >> 32;
  const uint64_t s2 = (s1 >> 1) + static_cast<uint64_t>(c1);  // 2^63 units
  return v == 0u ? 0.0 : to_double(s2, 63 - (ea >> 1));
}

// sqrt(-2 ln((m + 1) / 2^53)), its logarithm and its root each rounded to double, as an FP64
// evaluation has them (with the root's rounding alone positions lay 3 to 20 % farther from
// one, root mean square, than with double-precision functions).
FN_FN double radius_fp64(uint64_t m) {
  int e;
  const uint64_t v = neg_log(m, e);
  const int drop = 11 - clz64(v | 1u);  // bits past 53 (v is far from its type's limit)
  const uint64_t unit = 1ull << (drop > 0 ? drop : 0);
  return root_of_twice((v + (unit >> 1)) & ~(unit - 1u), e);
}
// The same with one rounding.
FN_FN double radius(uint64_t m) {
  int e;
  const uint64_t v = neg_log(m, e);
  return root_of_twice(v, e);
}

}  // namespace fixedn
}  // namespace chem
