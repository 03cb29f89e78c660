// fp64_int.cuh -- FP64 operations of the stokeslet evaluation on the integer
// pipe, correctly rounded, for a GPU whose FP64 pipe is the bottleneck.
//
// GB300 issues one FP64 warp instruction per scheduler in 64 clocks (fused
// multiply-add; 76 for a plain add or multiply), and __dsqrt_rn and __ddiv_rn
// take 572 and 344; 32 x 32 + 64 bit multiply-adds, shifts and logic take 2
// clocks each and run beside the FP64 pipe.  So the products, the square root
// and the reciprocal of a stokeslet term are formed here from 53-bit integer
// significands, and only the additions stay on the FP64 pipe.  Every result is
// the correctly rounded one (round to nearest, ties to even), the same bits
// as __dmul_rn, __dsqrt_rn and __ddiv_rn give:
//  * a product's 106 bits are formed exactly except for the lowest 32, which
//    matter only where the bits after the last kept one read exactly one half
//    (a tie, or a hair above one): `tie` reports that and the caller evaluates
//    the term on the FP64 pipe instead;
//  * the square root and the reciprocal are approximated to a fraction of an
//    ulp and rounded by the exact sign of (operand - midpoint^2) or
//    (1 - midpoint x operand), formed modulo 2^64 (Markstein's remainder test
//    in integers; no midpoint is ever hit).
// Operands are normal numbers whose results stay normal; the callers check
// the exponents.  The functions compile for the host too (the CPU test).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define NRS_HD __host__ __device__ __forceinline__
#else
#define NRS_HD inline
#endif

namespace nrs {

// A positive 53-bit significand with its sign and biased exponent field:
// value = +-(m / 2^52) 2^(exponent - 1023); m = 2^53 (a rounding carry) is
// allowed.  f: sign and exponent, the bits of a double's high word.
struct Sig {
    uint64_t m;
    uint32_t f;
};

NRS_HD uint32_t hi32(uint64_t v) { return (uint32_t)(v >> 32); }
NRS_HD uint32_t lo32(uint64_t v) { return (uint32_t)v; }
NRS_HD uint64_t wide(uint32_t a, uint32_t b, uint64_t c) { return (uint64_t)a * b + c; }

NRS_HD uint64_t double_bits(double v)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    uint64_t u;
    memcpy(&u, &v, 8);
    return u;
#endif
}

NRS_HD double bits_double(uint64_t u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double v;
    memcpy(&v, &u, 8);
    return v;
#endif
}

NRS_HD float bits_float(uint32_t u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float v;
    memcpy(&v, &u, 4);
    return v;
#endif
}

// the 64 bits of (hi : lo) << n from its high word, 0 <= n < 32
NRS_HD uint32_t funnel_l(uint32_t lo, uint32_t hi, uint32_t n)
{
#ifdef __CUDA_ARCH__
    return __funnelshift_l(lo, hi, n);
#else
    return hi32((((uint64_t)hi << 32) | lo) << n);
#endif
}

// approximate 1/sqrt of a float, and its absolute error's sign does not matter
NRS_HD uint32_t rsqrt_bits(uint32_t b)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(b)));
    return __float_as_uint(r);
#else
    float f, r;
    memcpy(&f, &b, 4);
    r = 1.0f / sqrtf(f);
    uint32_t u;
    memcpy(&u, &r, 4);
    return u;
#endif
}

NRS_HD Sig unpack(double v)
{
    const uint64_t u = double_bits(v);
    return Sig{(u & 0xfffffffffffffULL) | 0x10000000000000ULL, hi32(u) & 0xfff00000u};
}

NRS_HD double pack(const Sig &s)
{
    // the implicit bit of m adds one to the exponent field, and so does a carry
    return bits_double(s.m + ((uint64_t)(s.f - (1u << 20)) << 32));
}

// a b rounded: a.m shifted left by 10 (63 bits), b given shifted left by 1, so
// that the top 64 bits of the 128-bit product hold 52 or 53 bits of it and
// every partial sum fits 64 bits.  At most one of the significands is 2^53.
NRS_HD Sig mul_sig(const Sig &a, uint64_t b2, uint32_t bf, bool &tie)
{
    const uint64_t A = a.m << 10;
    const uint32_t al = lo32(A), ah = hi32(A), bl = lo32(b2), bh = hi32(b2);
    const uint64_t t0 = wide(al, bl, 0);
    const uint64_t t1 = wide(ah, bl, hi32(t0));
    const uint64_t t2 = wide(al, bh, t1);
    const uint64_t h = wide(ah, bh, hi32(t2));
    const uint32_t n = (hi32(h) >> 20) ^ 1u;  // 1: the product of the significands is below 2
    const uint32_t rh = funnel_l(lo32(h), hi32(h), n), rl = funnel_l(lo32(t2), lo32(h), n);
    const uint32_t rest = lo32(t2) << n;  // the 32 bits after the last kept one
    tie |= rest == 0x80000000u;
    Sig r;
    r.m = (((uint64_t)rh << 32) | rl) + (rest >> 31);
    r.f = a.f + bf - (1022u << 20) - (n << 20);
    return r;
}

// 1/sqrt of rho in [2^-100, 2^100) to 2^-28: rho = m' 2^(2k) with m' in [1, 4).
struct RsqrtSeed {
    uint64_t M;    // m' 2^62
    uint32_t Y;    // 2^30 / sqrt(m'), about
    uint32_t ex;   // rho's biased exponent, 1024 + 2k - par
    uint32_t par;  // 1: m' below 2
};

NRS_HD RsqrtSeed rsqrt_seed(double rho_d)
{
    const uint64_t rb = double_bits(rho_d);
    const uint32_t rhi = hi32(rb), rlo = lo32(rb);
    RsqrtSeed r;
    r.ex = rhi >> 20;
    r.par = r.ex & 1u;
    r.M = unpack(rho_d).m << (11 - r.par);
    const uint32_t Mh = hi32(r.M);
    // y0 = 1/sqrt(m') to 16 bits, truncated: the seed's operand is rounded to
    // mid-interval at 2^-20 so that y stays inside (1/2, 1)
    const uint32_t fb = (funnel_l(rlo, rhi - (896u << 20), 3) & ~0x1fu) | 0x10u;
    const uint32_t Y0 = ((rsqrt_bits(fb) >> 8) & 0x7fffu) | 0x8000u;
    // e0 = 1 - m' y0^2 (2^-14 at most) in units of 2^-44; y = y0 (1 + e0/2 + 3/8 e0^2)
    const uint64_t W = wide(Mh, Y0 * Y0, 0);
    const int32_t e = (int32_t)(0u - (uint32_t)(W >> 18));
    const uint32_t e2 = hi32((uint64_t)((int64_t)e * e));  // e0^2 2^56
    const int32_t c = e + (int32_t)((e2 * 3u) >> 14);      // in units of 2^-45
    r.Y = (Y0 << 14) + (uint32_t)(((int64_t)(int32_t)Y0 * c) >> 31);
    return r;
}

// y^2 and y^3, rounded, for one y within 2^-28 of 1/sqrt(rho), rho in
// [2^-100, 2^100): with e = 1 - rho y^2, rho^(-3/2) = y^3 (1 + 3/2 e) to 2^-54.
NRS_HD void rsqrt_powers(double rho, double &y2, double &y3)
{
    const RsqrtSeed r = rsqrt_seed(rho);
    const uint32_t Y = r.Y < 0x3fffffffu ? r.Y : 0x3fffffffu;  // below 2^30
    const uint64_t v = wide(Y, Y, 0);                          // y^2 2^60, 59 or 60 bits
    const uint32_t top = hi32(v) >> 27;
    const uint32_t k2 = r.ex + r.par;                          // 1024 + 2k
    y2 = bits_double(((v + (32ull << top)) >> (6u + top)) + ((uint64_t)(1021u + 1024u - 1u + top - k2) << 52));
    const uint64_t h = wide(hi32(v), Y, hi32(wide(lo32(v), Y, 0)));  // y^3 2^58, 56 to 58 bits
    const uint32_t n = (hi32(h) >> 25) ? 2u : (hi32(h) >> 24) ? 1u : 0u;  // bits above 56
    // 2^52 of the significand is bit 55 + n of h: value m 2^(3 + n - 58 - 3k)
    y3 = bits_double(((h + (4ull << n)) >> (3u + n)) +
                     ((uint64_t)(1023u + 52u + 3u + n - 58u - 1u - (3 * (k2 - 1024u)) / 2) << 52));
}

// s = RN(1 / RN(rho RN(sqrt(rho)))) for rho in [2^-100, 2^100); `tie` as above.
NRS_HD Sig inv_rho_sqrt(double rho_d, bool &tie)
{
    const RsqrtSeed seed = rsqrt_seed(rho_d);
    const Sig rho = unpack(rho_d);
    const uint64_t M = seed.M;
    const uint32_t Mh = hi32(M), Y = seed.Y, ex = seed.ex, par = seed.par;
    // g = sqrt(m') to about 2^-28, then one step g + (m' - g^2) y / 2
    const uint32_t G = (uint32_t)(wide(Mh, Y, 0) >> 29);  // g 2^31
    const int64_t d = (int64_t)(M - wide(G, G, 0));       // (m' - g^2) 2^62
    const int32_t d6 = (int32_t)(d >> 6);
    const int32_t corr = (int32_t)hi32((uint64_t)((int64_t)d6 * (int32_t)Y)) >> 3;
    uint64_t q = ((uint64_t)G << 21) + (uint64_t)(int64_t)corr;  // floor(sqrt 2^52), about
    {
        // up if m' 2^104 > (q + 1/2)^2, that is m' 2^104 - q (q + 1) - 1 >= 0
        const uint64_t q1 = q + 1;
        const uint64_t t = wide(lo32(q), lo32(q1), 1);
        const uint32_t th = hi32(t) + lo32(q) * hi32(q1) + hi32(q) * lo32(q1);
        const uint32_t dh = (lo32(M) << 10) - th - (lo32(t) != 0u);
        q += (dh >> 31) ^ 1u;
    }
    // p = rho q
    const uint32_t qf = ((ex + 1022u + par) >> 1) << 20;
    const Sig p = mul_sig(rho, q << 1, qf, tie);
    // z = y^3 2^j approximates 1 / (p's significand), j = 0, 1, 2
    const uint32_t np = (rho.f + qf - (1022u << 20) - p.f) >> 20;
    const uint32_t y2 = (uint32_t)(wide(Y, Y, 0) >> 30);
    uint32_t z = (uint32_t)(wide(y2, Y, 0) >> (27u + np + par));  // z 2^31
    z = z < 0x7fffffffu ? z : 0x7fffffffu;
    // r = 1 - p z (2^-25 at most) in units of 2^-56; z (1 + r + r^2)
    const uint64_t t = wide(lo32(p.m), z, 0);
    const uint32_t hl = lo32(wide(hi32(p.m), z, hi32(t)));
    const int64_t rr = (int64_t)(0ull - (((uint64_t)hl << 32) | lo32(t)));  // r 2^83
    const int32_t r = (int32_t)(rr >> 27);
    const int32_t r2 = r + (int32_t)(hi32((uint64_t)((int64_t)r * r)) >> 24);
    const int32_t zc = (int32_t)hi32((uint64_t)((int64_t)r2 * (int32_t)z)) >> 2;
    uint64_t s = ((uint64_t)z << 22) + (uint64_t)(int64_t)zc;  // floor(2^53 / significand), about
    {
        // up if 2^106 > (2 s + 1) m
        const uint64_t m2 = 2 * s + 1;
        const uint32_t th = hi32(wide(lo32(m2), lo32(p.m), 0)) + lo32(m2) * hi32(p.m) +
                            hi32(m2) * lo32(p.m);
        s += th >> 31;
    }
    // 2^53 (p a power of two) becomes 2^52 and one more in the exponent: a product
    // with it may meet another factor of 2^53
    const uint32_t carry = hi32(s) >> 21;
    return Sig{s - ((uint64_t)carry << 52), (2045u << 20) - p.f + (carry << 20)};
}

// 1/x from y within 2^-19 of it (relative): one step of the hyperpower iteration
// of order three, y (1 + e + e^2) with e = 1 - x y (Altman, "An optimum cubically
// convergent iterative method of inverting a linear bounded operator in Hilbert
// space", 1960).  The step leaves e^3, and its last operation rounds once: within
// 0.57 units in the last place.
NRS_HD double rcp_refined(double x, double y)
{
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// v = hi + lo as two floats: hi the nearest float (a tie away from zero), lo
// the rest rounded to nearest.  On the integer pipe, because a conversion
// between FP64 and FP32 takes the FP64 pipe 68 clocks.  False (nothing
// written) for |v| outside [2^-70, 2^100).
NRS_HD bool split_pair(double v, float &hi, float &lo)
{
    const uint64_t u = double_bits(v);
    const uint32_t ex = (hi32(u) >> 20) & 0x7ffu;
    if (ex - 953u >= 170u) return false;
    const uint32_t sign = hi32(u) & 0x80000000u;
    const uint64_t m = (u & 0xfffffffffffffULL) | 0x10000000000000ULL;
    const uint32_t h = (uint32_t)((m + (1ull << 28)) >> 29);  // 24 bits, or 2^24
    const int32_t rest = (int32_t)(lo32(m) - (h << 29));      // m - h 2^29, at most 2^28
    hi = bits_float(sign | (((ex - 897u) << 23) + h));
    lo = (float)rest * bits_float(sign | ((ex - 948u) << 23));
    return true;
}

// ---- exact products placed in a 192-bit integer (the exact residual) ----------
// A double as the factor of many products: |v| = m 2^(max(ex, 1) - 1075) with
// ex its exponent field, and s = max(ex, 1) - 1075 - c the part of the
// product's place that it settles; f: its high word.
struct FxFactor {
    uint64_t m;
    int32_t s;
    uint32_t f;
};

// |x v| 2^-L in three words, little-endian
struct FxPlaced {
    uint64_t z0, z1, z2;
};

NRS_HD FxFactor fx_factor(double v, int c)
{
    const uint64_t u = double_bits(v);
    const uint32_t ex = (hi32(u) >> 20) & 0x7ffu, e1 = ex > 1u ? ex : 1u;
    return FxFactor{(u & 0xfffffffffffffULL) | ((uint64_t)(ex < 1u ? ex : 1u) << 52),
                    (int32_t)e1 - 1075 - c, hi32(u)};
}

// a 106-bit product
struct FxWords {
    uint32_t w0, w1, w2, w3;
};

NRS_HD FxWords fx_product(uint64_t x, uint64_t v)
{
    const uint64_t p = wide(lo32(x), lo32(v), 0);
    const uint64_t q = wide(lo32(x), hi32(v), hi32(p));
    const uint64_t r = wide(hi32(x), lo32(v), lo32(q));
    const uint64_t t = wide(hi32(x), hi32(v), (uint64_t)hi32(q) + hi32(r));
    return FxWords{lo32(p), lo32(r), lo32(t), hi32(t)};
}

// A product whose place s is outside [0, 86], moved so that it is inside: down,
// dropping what falls below bit 0, or (a short product, of a subnormal factor)
// up.  False if it has no room.
NRS_HD bool fx_move(FxWords &w, int32_t &s)
{
    if ((w.w0 | w.w1 | w.w2 | w.w3) == 0) s = 0;
    if (s < -127) w = FxWords{0, 0, 0, 0}, s = 0;
    while (s < 0) {
        const uint32_t k = s < -31 ? 31u : (uint32_t)-s;
        w = FxWords{funnel_l(w.w0, w.w1, 32u - k), funnel_l(w.w1, w.w2, 32u - k),
                    funnel_l(w.w2, w.w3, 32u - k), w.w3 >> k};
        s += (int32_t)k;
    }
    while (s > 86) {
        if (w.w3 >> 9) return false;  // 106 bits already
        w = FxWords{w.w0 << 1, funnel_l(w.w0, w.w1, 1), funnel_l(w.w1, w.w2, 1),
                    funnel_l(w.w2, w.w3, 1)};
        --s;
    }
    return true;
}

// The product placed s bits up, 0 <= s <= 86 (its 106 bits fit): five words of
// 32 bits from a shift by s mod 32, moved up by s / 32 words.
NRS_HD FxPlaced fx_place(const FxWords &w, uint32_t s)
{
    const uint32_t b = s & 31u;
    const uint32_t y0 = w.w0 << b, y1 = funnel_l(w.w0, w.w1, b), y2 = funnel_l(w.w1, w.w2, b);
    const uint32_t y3 = funnel_l(w.w2, w.w3, b), y4 = funnel_l(w.w3, 0u, b);
    const bool q1 = s >= 32u, q2 = s >= 64u;
    const uint32_t z0 = q1 ? 0u : y0, z1 = q1 ? (q2 ? 0u : y0) : y1;
    const uint32_t z2 = q1 ? (q2 ? y0 : y1) : y2, z3 = q1 ? (q2 ? y1 : y2) : y3;
    const uint32_t z4 = q1 ? (q2 ? y2 : y3) : y4, z5 = q1 ? (q2 ? y3 : y4) : 0u;
    return FxPlaced{((uint64_t)z1 << 32) | z0, ((uint64_t)z3 << 32) | z2,
                    ((uint64_t)z5 << 32) | z4};
}

}  // namespace nrs
