// vamp_soft64.cuh -- products of positive numbers with 64-bit mantissas on the
// integer pipe, for the FP64 form of the channel loop (Eq. 30).
//
// Why: the FP64 pipe of sm_103a retires 1.7 lanes per SM and cycle
// (vamp_measure_peaks), about 1/75 of the 32-bit lane rate, and the FP64
// channel loop is products all the way: d bin densities, the Jacobians, the
// peak's factors.  A product of two 64-bit mantissas is three 32 x 32 -> 64
// multiplies and a few adds, so a factor costs about eight issue slots
// instead of the 75 its DMUL occupies; it is short by less than 2^-60 instead
// of rounded at 2^-53.
//
// A number is m 2^e with m > 0.  "Normalised" means bit 63 of m is set.
// Products of normalised numbers are not renormalised at once: each loses at
// most one leading bit.  The kernels chain eight at most, which are short of
// the true product by less than 2^-52.4 together (largest seen on the GPU:
// 2^-53.4 for mantissas spread over 1 to 2, 2^-52.8 for mantissas below 1.01;
// eight products of doubles: 2^-50.9 and 2^-50.5, to either side).
//
// The errors below are the largest seen on the GPU over each function's range.
//
// A packed number (one 64-bit word, the form of the density rows and of the
// per-call tables) is the double's 53-bit significand in the high bits and its
// biased exponent in the low eleven: value = (w & ~2047) 2^((w & 2047) - 1086).
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define VAMP_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#define VAMP_HD inline
#endif

namespace vamp {

struct Sf {
    uint64_t m;
    int e;
};

constexpr int SF_BIAS = 1086;  // exponent field of a double + 63 bits of mantissa below the leading one

VAMP_HD uint64_t sf_bits(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    std::memcpy(&b, &x, 8);
    return b;
#endif
}

VAMP_HD double sf_from_bits(uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double x;
    std::memcpy(&x, &b, 8);
    return x;
#endif
}

// Normalises m 2^e whose leading bit is among the upper 32.
VAMP_HD void sf_norm(uint64_t& m, int& e)
{
    const uint32_t hi = (uint32_t)(m >> 32), lo = (uint32_t)m;
#ifdef __CUDA_ARCH__
    const int z = __clz((int)hi);
    m = ((uint64_t)__funnelshift_l(lo, hi, z) << 32) | (lo << z);
#else
    const int z = __builtin_clz(hi);
    m <<= z;
    (void)lo;
#endif
    e -= z;
}

// High 64 bits of a b without the low halves' product: short of the true
// value by at most three units of 2^-64.
VAMP_HD uint64_t sf_mulhi(uint64_t a, uint64_t b)
{
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    return (uint64_t)ah * bh + (((uint64_t)ah * bl) >> 32) + (((uint64_t)al * bh) >> 32);
}

VAMP_HD Sf sf_norm(Sf a)
{
    sf_norm(a.m, a.e);
    return a;
}

VAMP_HD Sf sf_mul(Sf a, Sf b) { return Sf{sf_mulhi(a.m, b.m), a.e + b.e + 64}; }

// A positive normal double (a subnormal or zero reads as its exponent's
// smallest normal, as the FP64 inverse fifth root reads it).
VAMP_HD Sf sf_from_double(double x)
{
    const uint64_t b = sf_bits(x);
    return Sf{(b << 11) | (1ull << 63), (int)((uint32_t)(b >> 52) & 0x7ffu) - SF_BIAS};
}

// Any finite x >= 0: subnormal numbers as they are, 0 as 2^-65536 (whose
// reciprocal is beyond a double, as 1 / 0).
VAMP_HD Sf sf_from_any(double x)
{
    const Sf a = sf_from_double(x);
    if (a.e != -SF_BIAS) return a;
    const uint64_t m = sf_bits(x) << 11;
    if (m == 0ull) return Sf{1ull << 63, -65536};
#ifdef __CUDA_ARCH__
    const int z = __clzll((long long)m);
#else
    const int z = __builtin_clzll(m);
#endif
    return Sf{m << z, 1 - SF_BIAS - z};
}

// Nearest double of a normalised number; 0 below the normal range, infinity above.
VAMP_HD double sf_to_double(Sf a)
{
    const int x = a.e + SF_BIAS;
    const uint64_t r = (a.m >> 11) + ((a.m >> 10) & 1u);  // [2^52, 2^53]
    uint64_t b = ((uint64_t)(uint32_t)(x - 1) << 52) + r;
    b = x >= 1 ? b : 0ull;
    b = x <= 2046 ? b : 0x7ff0000000000000ull;
    return sf_from_bits(b);
}

VAMP_HD Sf sf_unpack(uint64_t w) { return Sf{w & ~2047ull, (int)((uint32_t)w & 2047u) - SF_BIAS}; }

VAMP_HD uint64_t sf_pack_double(double x)
{
    const uint64_t b = sf_bits(x);
    return (b << 11) | (1ull << 63) | ((b >> 52) & 2047u);
}

VAMP_HD double sf_unpack_double(uint64_t w) { return sf_from_bits(((w & 2047u) << 52) | ((w >> 11) & 0xFFFFFFFFFFFFFull)); }

// Packs a normalised number, rounded to 53 bits (exponents beyond a double's
// range are clamped: no table entry gets there).
VAMP_HD uint64_t sf_pack(Sf a)
{
    const uint64_t r = (a.m >> 11) + ((a.m >> 10) & 1u);  // [2^52, 2^53]
    int x = a.e + SF_BIAS + (int)(r >> 53);
    x = x < 0 ? 0 : (x > 2047 ? 2047 : x);
    return (r << 11) | (1ull << 63) | (uint32_t)x;
}

// x in FP32, truncated; 0 below the normal range.
VAMP_HD float sf_to_float(double x)
{
    const uint64_t b = sf_bits(x);
    const uint32_t hi = (uint32_t)(b >> 32), e = (hi >> 20) & 0x7ffu;
    uint32_t r = (hi & 0x80000000u) | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | ((uint32_t)b >> 29);
    r = e < 897u ? 0u : (e > 1150u ? (hi & 0x80000000u) | 0x7f7fffffu : r);
#ifdef __CUDA_ARCH__
    return __uint_as_float(r);
#else
    float f;
    std::memcpy(&f, &r, 4);
    return f;
#endif
}

VAMP_HD float sf_lg2f(float v)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
#else
    return std::log2(v);
#endif
}

VAMP_HD float sf_ex2f(float v)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
#else
    return std::exp2(v);
#endif
}

VAMP_HD float sf_rcpf(float v)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
#else
    return 1.0f / v;
#endif
}

VAMP_HD uint32_t sf_f2u(float v)  // v >= 0, saturating
{
#ifdef __CUDA_ARCH__
    return __float2uint_rz(v);
#else
    return v >= 4294967296.0f ? 0xffffffffu : (uint32_t)v;
#endif
}

// c a >> 31 and c a >> 30 of a 32-bit number c and a signed a below 2^44 in size
VAMP_HD int64_t sf_scale(uint32_t c, int64_t a, int sh)
{
    const uint64_t lo = (uint64_t)c * (uint32_t)a;
    const int64_t hi = (int64_t)(int32_t)(a >> 32) * (int64_t)(uint64_t)c;
    return (hi << (32 - sh)) + (int64_t)(lo >> sh);
}

// 1 / a of a normalised number, to 2^-60.7: an FP32 reciprocal y0 of x =
// m 2^-64 in [1/2, 1), then one step of third order (Householder's method),
// y = y0 (1 + r + r^2) with r = 1 - x y0 taken in 63-bit fixed point (|r| <=
// 2^-22, so the next term is below 2^-66).
VAMP_HD Sf sf_rcp(Sf a)
{
    const float xf = (float)(uint32_t)(a.m >> 40) * 0x1p-24f;
    const uint32_t y0 = sf_f2u(sf_rcpf(xf) * 0x1p31f);  // Q1.31
    const uint64_t p = (a.m >> 32) * (uint64_t)y0 + (((a.m & 0xffffffffull) * (uint64_t)y0) >> 32);  // x y0, Q1.63
    const int64_t r = (int64_t)((1ull << 63) - p) - 3;  // |r| < 2^43, never above the true residual
    const int32_t rh = (int32_t)(r >> 14);
    const int64_t c = r + (int64_t)(((int64_t)rh * rh) >> 35);  // r + r^2
    const uint64_t y = ((uint64_t)y0 << 32) + (uint64_t)sf_scale(y0, c, 31);
    return Sf{y, -127 - a.e};
}

// v^(-4/5) of a positive normal double, normalised, to 2^-55.  With v = X
// 2^(5a), X in [2^-4, 2): an FP32 seed s of X^(-1/5) in (0.87, 1.75), s^2, s^4
// and s^5 in fixed point, the residual r = 1 - X s^5 (|r| <= 2^-20), and the
// binomial series (1 - r)^(-4/5) = 1 + (4/5) r + (18/25) r^2 + ... cut after r^2:
// X^(-4/5) = s^4 (1 - r)^(-4/5).
VAMP_HD Sf sf_powm08(double v)
{
    const uint64_t b = sf_bits(v);
    const uint64_t m = (b << 11) | (1ull << 63);            // v = m 2^-64 2^ex
    const int ex = (int)((uint32_t)(b >> 52) & 0x7ffu) - 1022;
    // ex = 5 a + h with h in -3..1
    const int a = (int)(((uint32_t)(ex + 5003) * 52429u) >> 18) - 1000;  // floor((ex + 3) / 5), ex + 5003 < 2^14
    const int h = ex - 5 * a;
    const float l = sf_lg2f((float)(uint32_t)(m >> 40)) + (float)(h - 24);
    const uint32_t s = sf_f2u(sf_ex2f(-0.2f * l) * 0x1p31f);  // Q1.31
    const uint64_t s2 = (uint64_t)s * s;                      // Q2.62
    const uint64_t s4 = sf_mulhi(s2, s2);                     // Q4.60
    const uint64_t s5 = (s4 >> 32) * (uint64_t)s + (((s4 & 0xffffffffull) * (uint64_t)s) >> 32);  // Q5.59
    const uint64_t q = sf_mulhi(m, s5);                       // X s^5 2^-h, Q5.59
    const int64_t d = (int64_t)((1ull << (59 - h)) - q);
    const int64_t r = (int64_t)((uint64_t)d << (3 + h));      // Q0.62, |r| < 2^43
    // c = 0.8 r + 0.72 r^2 in Q0.64 (|c| < 2^45): 0.8 r = r - r / 5 with 2^34 / 5, r^2 from the upper bits
    const uint32_t rl = (uint32_t)r;
    const int32_t rh = (int32_t)(r >> 32), rm = (int32_t)(r >> 20);
    const int64_t r5 = (int64_t)(((uint64_t)rl * 3435973837u >> 32) + (uint64_t)((int64_t)rh * 3435973837ll));  // 4 r / 5
    const uint32_t r2 = (uint32_t)(((int64_t)rm * rm) >> 20);
    const int64_t c = 4 * r - r5 + (int64_t)(((uint64_t)r2 * 3092376453u) >> 32);
    const int32_t ch = (int32_t)(c >> 32);
    const uint32_t zh = (uint32_t)(s4 >> 32), zl = (uint32_t)s4;
    const uint64_t z = s4 + (uint64_t)((int64_t)ch * (int64_t)(uint64_t)zh) + (((uint64_t)zh * (uint32_t)c) >> 32) +
                       (uint64_t)((int64_t)((int64_t)ch * (int64_t)(uint64_t)zl) >> 32);
    return sf_norm(Sf{z, -60 - 4 * a});
}

// High 64 bits of a b, exact.
VAMP_HD uint64_t sf_mulhi_exact(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// 2^(n + f 2^-64), to 2^-60, normalised: the fraction's leading two bits
// pick 2^(i/4), the rest goes through the series of 2^t = sum (t ln 2)^k / k!
// for t in [0, 1/4), whose terms from t^7 on (below 2^-30) are summed in 32 bits.
VAMP_HD Sf sf_exp2_fixed(int n, uint64_t f)
{
    const uint32_t i = (uint32_t)(f >> 62);
    const uint64_t t = f & 0x3fffffffffffffffull;  // Q0.64, below 1/4
    const uint32_t th = (uint32_t)(t >> 32);
    // (ln 2)^k / k!: 47-bit fractions for k = 12..7, 64-bit ones for k = 6..1
    uint32_t w = 3614u;
    w = 62565u + (uint32_t)(((uint64_t)w * th) >> 32);
    w = 992891u + (uint32_t)(((uint64_t)w * th) >> 32);
    w = 14324383u + (uint32_t)(((uint64_t)w * th) >> 32);
    w = 185991442u + (uint32_t)(((uint64_t)w * th) >> 32);
    w = 2146631446u + (uint32_t)(((uint64_t)w * th) >> 32);
    uint64_t v = 0xa184897c363c4ull + sf_mulhi(t, (uint64_t)w << 17);
    v = 0x5761ff9e299cc4ull + sf_mulhi(t, v);
    v = 0x276556df749cee5ull + sf_mulhi(t, v);
    v = 0xe35846b82505fc6ull + sf_mulhi(t, v);
    v = 0x3d7f7bff058b1d51ull + sf_mulhi(t, v);
    v = 0xb17217f7d1cf79acull + sf_mulhi(t, v);
    v = (1ull << 63) + (sf_mulhi(t, v) >> 1);  // 2^t, Q1.63
    const uint64_t k01 = (i & 1u) ? 0x9837f0518db8a96full : 0x8000000000000000ull;
    const uint64_t k23 = (i & 1u) ? 0xd744fccad69d6af4ull : 0xb504f333f9de6484ull;
    return Sf{sf_mulhi_exact(v, (i & 2u) ? k23 : k01) << 1, n - 63};
}

// 2^(±m 2^(ex - 63)), m normalised (from 2^20 on as 2^±(2^20)).
VAMP_HD Sf sf_exp2_parts(bool neg, uint64_t m, int ex)
{
    // integer part and 64-bit fraction of the size
    int n = 0;
    uint64_t f;
    if (ex >= 20) {
        n = 1 << 20;
        f = 0ull;
    } else if (ex >= 0) {
        n = (int)(m >> (63 - ex));
        f = m << (ex + 1);
    } else {
        f = ex >= -64 ? m >> (-1 - ex) : 0ull;
    }
    if (neg) {  // 2^-(n + f) = 2^(-n-1) 2^(1-f)
        n = f ? -n - 1 : -n;
        f = 0ull - f;
    }
    return sf_exp2_fixed(n, f);
}

// 2^x of a double; beyond a double's range for NaN, of either sign, so that what
// it enters is not finite.
VAMP_HD Sf sf_exp2(double x)
{
    const uint64_t b = sf_bits(x);
    const bool nan = (b << 1) > 0xffe0000000000000ull;
    return sf_exp2_parts(!nan && (b >> 63), (b << 11) | (1ull << 63), (int)((uint32_t)(b >> 52) & 0x7ffu) - 1023);
}

// |log2 a| of a normalised number, normalised (zero: m = 0), and its sign: an
// FP32 logarithm y of the significand s in [1, 2) in 32-bit fixed point, then
// log2 (s 2^-y) = (d - d^2/2 + ...) / ln 2 of d = s 2^-y - 1 (|d| < 2^-21, the
// next term below 2^-64).  Integer part and fraction stay apart until the end:
// error about 2^-60 below 1, relative above.
VAMP_HD Sf sf_log2(Sf a, bool& neg)
{
    const float yf = sf_lg2f((float)(uint32_t)(a.m >> 40) * 0x1p-23f);  // in [0, 1]
    const uint64_t y = (uint64_t)sf_f2u(yf > 0.f ? yf * 0x1p31f : 0.f) << 1;  // Q0.32, up to 2^32
    const Sf t = y ? sf_exp2_fixed(-1, 0ull - (y << 32)) : Sf{1ull << 63, -63};  // 2^-y
    const uint64_t p = sf_mulhi_exact(a.m, t.m);  // s 2^-y 2^(62 + (0 or 1)): t's exponent is -63 or -64
    const int64_t d = (int64_t)((p << (t.e == -63 ? 1 : 0)) - (1ull << 63));  // Q1.63
    const int64_t dh = d >> 14;
    const int64_t c = d - ((dh * dh) >> 36);
    // c / ln 2 in Q0.64
#ifdef __CUDA_ARCH__
    const int64_t r = __mul64hi(c << 20, 0x5c551d94ae0bf85ell) >> 17;
#else
    const int64_t r = (int64_t)(((__int128)(c << 20) * 0x5c551d94ae0bf85ell) >> 64) >> 17;
#endif
    // n + f 2^-64 = exponent + y + r
    const uint64_t f0 = y << 32, f1 = f0 + (uint64_t)r;
    int n = a.e + 63 + (int)(y >> 32) + (r < 0 ? -1 : 0) + (f1 < f0 ? 1 : 0);
    uint64_t f = f1;
    neg = n < 0;
    if (neg) {  // size of a negative number
        n = f ? -n - 1 : -n;
        f = 0ull - f;
    }
    // normalise (n < 2^31)
    if (n) {
#ifdef __CUDA_ARCH__
        const int z = __clz(n);
#else
        const int z = __builtin_clz((unsigned)n);
#endif
        return Sf{((uint64_t)(uint32_t)n << (32 + z)) | (f >> (32 - z)), -32 - z};
    }
    if (f == 0ull) return Sf{0ull, 0};
#ifdef __CUDA_ARCH__
    const int z = __clzll((long long)f);
#else
    const int z = __builtin_clzll(f);
#endif
    return Sf{f << z, -64 - z};
}

// a^y of a normalised number and a finite normal double, normalised: the
// logarithm, the product and its fraction are carried in 64 bits, so that the
// error is about |y log2 a| 2^-63 and max(1, |y|) 2^-59.
VAMP_HD Sf sf_pow(Sf a, double y)
{
    bool neg;
    const Sf l = sf_log2(a, neg), b = sf_from_double(y);
    if (l.m == 0ull) return Sf{1ull << 63, -63};
    uint64_t m = sf_mulhi_exact(l.m, b.m);
    int e = l.e + b.e + 64;
    sf_norm(m, e);
    return sf_exp2_parts(neg != (sf_bits(y) >> 63 != 0ull), m, e + 63);
}

// tan of a double |th| < pi/2, to about 2^-58: the ninth convergent of Lambert's
// continued fraction, tan z = z N(z^2) / D(z^2) within 6e-19 for z <= pi/4, with
// tan = D / (z N) of z = pi/2 - |th| above.  N and D are taken in 64-bit fixed
// point (each inner sum is positive), z with its own exponent.
VAMP_HD double sf_tan(double th)
{
    const uint64_t b = sf_bits(th) & 0x7fffffffffffffffull;
    const bool far = b >= 0x3fe921fb54442d18ull;  // above pi/4
    Sf z = sf_from_double(sf_from_bits(b));
    if (b < 0x0010000000000000ull) return th;
    if (far) {
        // pi/2 - |th| (whose 53 bits lie above 2^-63) in Q1.63 and 64 bits more
        uint64_t m = 0xc90fdaa22168c234ull - (z.m >> (-63 - z.e)), lo = 0xc4c6628b80dc1cd1ull;
        int e = -63;
        if (!(m >> 32)) { m = (m << 32) | (lo >> 32); lo <<= 32; e -= 32; }
        if (!(m >> 32)) { m = (m << 32) | (lo >> 32); lo <<= 32; e -= 32; }
#ifdef __CUDA_ARCH__
        const int s = __clz((int)(m >> 32)) & 31;
#else
        const int s = __builtin_clz((uint32_t)(m >> 32) | 1u) & 31;
#endif
        m = (m << s) | (uint64_t)((uint32_t)(lo >> 32) >> 1 >> (31 - s));
        e -= s;
        z = Sf{m, e};
    }
    const int sh = -64 - z.e;  // z < 1
    const uint64_t q = sh < 64 ? z.m >> sh : 0ull, v = sf_mulhi(q, q);  // z^2, Q0.64
    uint64_t N = 0x1e20001e20002ull - sf_mulhi(v, 0x7ca36d9c30ull);
    N = 0x101010101010101ull - sf_mulhi(v, N);
    N = 0x2323232323232323ull - sf_mulhi(v, N);
    N = ~sf_mulhi(v, N);  // 1 - ..., Q0.64 (short of it by 2^-64)
    uint64_t d = 0x1a5c001a5c001aull - sf_mulhi(v, 0x15e8ba44745dull);
    d = 0x707070707070707ull - sf_mulhi(v, d);
    d = 0x7878787878787878ull - sf_mulhi(v, d);
    d = ~sf_mulhi(v, d);
    const Sf zn = sf_mul(z, Sf{N, -64}), dd{d, -64};
    const Sf t = far ? sf_mul(dd, sf_rcp(sf_norm(zn))) : sf_mul(zn, sf_rcp(sf_norm(dd)));
    const double r = sf_to_double(sf_norm(t));
    return sf_bits(th) >> 63 ? -r : r;
}

// a / b of doubles, b > 0 normal and a / b not below the normal range, to about
// 2^-53: the reciprocal above (0 / b = 0).
VAMP_HD double sf_div(double a, double b)
{
    const uint64_t ua = sf_bits(a);
    if ((ua << 1) < (1ull << 53)) return a * 0.0;  // zero or subnormal
    const double q = sf_to_double(sf_norm(sf_mul(sf_from_double(a), sf_rcp(sf_from_double(b)))));
    return ua >> 63 ? -q : q;
}

// n 2^-33 of a 33-bit integer, exact: the fraction of 1.xxx less 1.
VAMP_HD double sf_frac33(uint64_t n) { return sf_from_bits(0x3ff0000000000000ull | (n << 19)) - 1.0; }

}  // namespace vamp
