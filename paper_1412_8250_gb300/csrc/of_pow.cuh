// u^e for positive u in 64-bit fixed point: log2 u, times e, and 2 to that power, each to about
// 2^-60, so the result is the rounded one but for ties closer than that (0.51 units in the last
// place; pow() is specified to 2).
// GB300 does 2 FP64 operations per clock and SM but 60 32 x 32 -> 64-bit multiply-adds: a double
// pow() took 95 FP64 operations' time, one of these the time of about 8.  k_powers (two powers of
// 96^3 amplitudes): 294 -> 23.5 us.
// One table, 2^{j/128}, serves both directions.  Logarithm: m in [1, 2) times 2^{-j/128} is 1 + r,
// |r| <= 2^-8.4, and log2(1 + r) is log2(e) times the series of ln(1 + r) to r^7; exponential:
// 2^{j/128} times the series of e^y to y^6, 0 <= y < 2^-7.5.  The remainders are below 2^-62.
// Compiles for the host too.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define OF_HD __host__ __device__ __forceinline__
#else
#define OF_HD inline
#endif

namespace of {

// 2^63 2^{j/128}, rounded
#define OF_POW2_TABLE \
    0x8000000000000000ull, 0x80b1ed4fd999ab6cull, 0x8164d1f3bc030773ull, 0x8218af4373fc25ecull, \
    0x82cd8698ac2ba1d7ull, 0x8383594eefb6ee37ull, 0x843a28c3acde4046ull, 0x84f1f656379c1a29ull, \
    0x85aac367cc487b15ull, 0x8664915b923fba04ull, 0x871f61969e8d1010ull, 0x87db357ff698d792ull, \
    0x88980e8092da8527ull, 0x8955ee03618e5fddull, 0x8a14d575496efd9aull, 0x8ad4c6452c728924ull, \
    0x8b95c1e3ea8bd6e7ull, 0x8c57c9c4646f4ddeull, 0x8d1adf5b7e5ba9e6ull, 0x8ddf042022e69cd6ull, \
    0x8ea4398b45cd53c0ull, 0x8f6a8117e6c8e5c4ull, 0x9031dc431466b1dcull, 0x90fa4c8beee4b12bull, \
    0x91c3d373ab11c336ull, 0x928e727d9531f9acull, 0x935a2b2f13e6e92cull, 0x9426ff0fab1c04b6ull, \
    0x94f4efa8fef70961ull, 0x95c3fe86d6cc7fefull, 0x96942d3720185a00ull, 0x97657d49f17ab08eull, \
    0x9837f0518db8a96full, 0x990b87e266c189aaull, 0x99e0459320b7fa65ull, 0x9ab62afc94ff864aull, \
    0x9b8d39b9d54e5539ull, 0x9c6573682ec32c2dull, 0x9d3ed9a72cffb751ull, 0x9e196e189d472420ull, \
    0x9ef5326091a111aeull, 0x9fd228256400dd06ull, 0xa0b0510fb9714fc2ull, 0xa18faeca8544b6e4ull, \
    0xa27043030c496819ull, 0xa3520f68e802bb93ull, 0xa43515ae09e6809eull, 0xa5195786be9ef339ull, \
    0xa5fed6a9b15138eaull, 0xa6e594cfeee86b1eull, 0xa7cd93b4e965356aull, 0xa8b6d5167b320e09ull, \
    0xa9a15ab4ea7c0ef8ull, 0xaa8d2652ec907629ull, 0xab7a39b5a93ed337ull, 0xac6896a4be3fe929ull, \
    0xad583eea42a14ac6ull, 0xae493452ca35b80eull, 0xaf3b78ad690a4375ull, 0xb02f0dcbb6e04584ull, \
    0xb123f581d2ac2590ull, 0xb21a31a66618fe3bull, 0xb311c412a9112489ull, 0xb40aaea2654b9841ull, \
    0xb504f333f9de6484ull, 0xb60093a85ed5f76cull, 0xb6fd91e328d17791ull, 0xb7fbefca8ca41e7cull, \
    0xb8fbaf4762fb9ee9ull, 0xb9fcd2452c0b9debull, 0xbaff5ab2133e45fbull, 0xbc034a7ef2e9fb0dull, \
    0xbd08a39f580c36bfull, 0xbe0f6809860993e2ull, 0xbf1799b67a731083ull, 0xc0213aa1f0d08db0ull, \
    0xc12c4cca66709456ull, 0xc238d2311e3d6673ull, 0xc346ccda24976407ull, 0xc4563ecc5334cb33ull, \
    0xc5672a115506daddull, 0xc67990b5aa245f79ull, 0xc78d74c8abb9b15dull, 0xc8a2d85c8ffe2c45ull, \
    0xc9b9bd866e2f27a3ull, 0xcad2265e4290774eull, 0xcbec14fef2727c5dull, 0xcd078b86503dcdd2ull, \
    0xce248c151f8480e4ull, 0xcf4318cf191918c1ull, 0xd06333daef2b2595ull, 0xd184df6251699ac6ull, \
    0xd2a81d91f12ae45aull, 0xd3ccf099859ac379ull, 0xd4f35aabcfedfa1full, 0xd61b5dfe9f9bce07ull, \
    0xd744fccad69d6af4ull, 0xd870394c6db32c84ull, 0xd99d15c278afd7b6ull, 0xdacb946f2ac9cc72ull, \
    0xdbfbb797daf23755ull, 0xdd2d818508324c20ull, 0xde60f4825e0e9124ull, 0xdf9612deb8f04420ull, \
    0xe0ccdeec2a94e111ull, 0xe2055afffe83d369ull, 0xe33f8972be8a5a51ull, 0xe47b6ca0373da88dull, \
    0xe5b906e77c8348a8ull, 0xe6f85aaaee1fce22ull, 0xe8396a503c4bdc68ull, 0xe97c38406c4f8c57ull, \
    0xeac0c6e7dd24392full, 0xec0718b64c1cbddcull, 0xed4f301ed9942b84ull, 0xee990f980da3025bull, \
    0xefe4b99bdcdaf5cbull, 0xf13230a7ad094509ull, 0xf281773c59ffb13aull, 0xf3d28fde3a641a5bull, \
    0xf5257d152486cc2cull, 0xf67a416c733f846eull, 0xf7d0df730ad13bb9ull, 0xf92959bb5dd4ba74ull, \
    0xfa83b2db722a033aull, 0xfbdfed6ce5f09c49ull, 0xfd3e0c0cf486c175ull, 0xfe9e115c7b8f884cull,

#ifdef __CUDACC__
__device__ const unsigned long long pow2_table_device[128] = {OF_POW2_TABLE};
#endif
static const unsigned long long pow2_table_host[128] = {OF_POW2_TABLE};
OF_HD unsigned long long pow2_entry(int j) {
#ifdef __CUDA_ARCH__
    return __ldg(pow2_table_device + j);
#else
    return pow2_table_host[j];
#endif
}
OF_HD unsigned long long mulhi_u(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}
OF_HD long long mulhi_s(long long a, long long b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (long long)(((__int128)a * b) >> 64);
#endif
}
OF_HD unsigned long long bits_of(double v) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(v);
#else
    unsigned long long b;
    std::memcpy(&b, &v, 8);
    return b;
#endif
}
OF_HD double of_bits(unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double v;
    std::memcpy(&v, &b, 8);
    return v;
#endif
}

// An exponent with its value times 2^58, or 0 where that is not exact or does not fit (pow() then)
struct PowExp {
    double e;
    long long fixed;
};
inline PowExp pow_exp(double e) {
    const double s = std::ldexp(e, 58);
    const bool fits = std::fabs(e) < 16.0 && s == std::floor(s);
    return {e, fits ? (long long)s : 0};
}

// log2 u = k + f 2^-63; false outside 2^-60 <= u < 2^60 (and for NaN)
OF_HD bool log2_fixed(double u, int& k, long long& f) {
    const unsigned long long b = bits_of(u);
    k = (int)(b >> 52) - 1023;          // a negative u has a large k
    if (k < -60 || k >= 60) return false;
    const unsigned long long m = (1ull << 63) | ((b & 0xfffffffffffffull) << 11);   // 2^63 m
    // j = 128 log2 m rounded, log2(1 + x) by a least-squares polynomial (128 times its error: 0.01)
    const float x = (float)(unsigned)(m >> 40) * (1.f / 8388608.f) - 1.f;   // m - 1, 23 bits
    int j = (int)(x * (184.6444518f + x * (-91.9082996f + x * (58.5162395f + x * (-35.4997307f + x * (15.5485374f + x * -3.3014202f))))) + 0.5f);
    // 1 + r = m 2^{-j/128}: half the table's entry 128 - j, or m and m / 2 at the ends
    const unsigned long long c = pow2_entry((128 - j) & 127);
    const unsigned long long p = j == 0 ? m : mulhi_u(m, c), lo = j == 0 ? 0ull : m * c;
    const long long s = (long long)(((p - (1ull << 63)) << 8) | (lo >> 56));   // 2^71 r
    if (j >= 128) {
        j = 0;
        ++k;
    }
    long long h = 1537228672809129301ll - (mulhi_s(s, 1317624576693539401ll) >> 7);             // 1/6 - r/7, times 2^63
    h = 1844674407370955162ll - (mulhi_s(s, h) >> 7);                          // 1/5 - r (...)
    h = 2305843009213693952ll - (mulhi_s(s, h) >> 7);
    h = 3074457345618258603ll - (mulhi_s(s, h) >> 7);
    h = 4611686018427387904ll - (mulhi_s(s, h) >> 7);
    // ln(1 + r) = r - r^2 (1/2 - r (1/3 - ...)), times 2^70
    const long long r2 = mulhi_s(s, mulhi_s(s, h));           // 2^(71 + 71 + 63 - 128) = 2^77 r^2 (...)
    const long long ln = (s >> 1) - (r2 >> 7);
    f = ((long long)j << 56) + ((mulhi_s(ln, 6653256548922161246ll) + 16) >> 5);
    return true;
}

// v = u^e from k and f; false where the result is not a normal number
OF_HD bool exp2_fixed(const PowExp& e, int k, long long f, double& v) {
    // e f = 2^-121 (xh 2^64 + xl) and e k = 2^-58 (yh 2^64 + yl): integer part and 2^64 times the rest
    const long long xh = mulhi_s(e.fixed, f), yh = mulhi_s(e.fixed, (long long)k);
    const unsigned long long xl = (unsigned long long)e.fixed * (unsigned long long)f;
    const unsigned long long yl = (unsigned long long)e.fixed * (unsigned long long)(long long)k;
    const unsigned long long fx = ((unsigned long long)xh << 7) | (xl >> 57);
    const unsigned long long g = fx + (yl << 6);
    const long long n = (xh >> 57) + (long long)(((unsigned long long)yh << 6) | (yl >> 58)) + (g < fx ? 1 : 0);
    if (n < -1000 || n > 1000) return false;
    const int j = (int)(g >> 57);
    const unsigned long long y = mulhi_u(g & ((1ull << 57) - 1), 12786308645202655660ull);       // the remainder times ln 2
    unsigned long long h = 153722867280912930ull + mulhi_u(y, 25620477880152155ull);                          // 1/120 + y / 720
    h = 768614336404564651ull + mulhi_u(y, h);
    h = 3074457345618258603ull + mulhi_u(y, h);
    h = (1ull << 63) + mulhi_u(y, h);
    const unsigned long long t = pow2_entry(j);
    const unsigned long long w = t + mulhi_u(t, y + mulhi_u(y, mulhi_u(y, h)));   // 2^63 .. 2^64
    // to 53 bits, nearest; a carry moves the exponent
    const unsigned long long r = (w >> 11) + ((w >> 10) & 1ull);
    v = of_bits(((unsigned long long)(n + 1022) << 52) + r);
    return true;
}

}  // namespace of
