// stokeslet_int.cuh -- the six terms S_jk w of one (force point, quadrature
// point) pair with the products, the square root and the reciprocal on the
// integer pipe (fp64_int.cuh): the integer form of the FP64 assembly
// (assemble.cu).  It compiles for the host too (the CPU test).
#pragma once

#include <math.h>

#include "fp64_int.cuh"

namespace nrs {

struct Acc6 {
    double xx, xy, xz, yy, yz, zz;
};

// FP64 additions and products as fused multiply-adds: GB300 issues an FP64
// fused multiply-add every 64 clocks per scheduler, a plain add or multiply
// every 76.  `one` is 1.0 and `nz` is -0.0, passed at run time so that the
// compiler does not turn them back; a 1 + b and a b + (-0.0) round exactly as
// a + b and a b do (signed zeros included).
struct FmaOps {
    double one, nz;
    NRS_HD double add(double a, double b) const { return fma(a, one, b); }
    NRS_HD double sub(double a, double b) const { return fma(b, -one, a); }
    NRS_HD double mul(double a, double b) const { return fma(a, b, nz); }
};

// Components of r below the first count as zero in terms_int; from the second
// on, infinities and NaN among them, the pair is left to the general path
// (rho leaves the integer path's range there, but a square formed from wrapped
// exponents need not).
constexpr uint32_t kTinyHi = 873u << 20;  // 2^-150
constexpr uint32_t kFarHi = 1073u << 20;  // 2^50

// A quadrature point staged for the pair loop: its weight also as a
// significand for the integer products (shifted left by one, sign and
// exponent field), and the high word from which a component of r sends the pair
// to the general path: kFarHi, or zero (every pair) if the weight is outside the
// integer path's range.
struct alignas(16) StagedX {
    double x, y, z, w;
    uint64_t w2;
    uint32_t wf, far_hi;
};

NRS_HD StagedX stage_weighted(double x, double y, double z, double w)
{
    StagedX v;
    v.x = x;
    v.y = y;
    v.z = z;
    v.w = w;
    const Sig sw = unpack(w);
    v.w2 = sw.m << 1;
    v.wf = sw.f;
    // 2^-200 <= |w| < 2^200 (zero, subnormal and non-finite weights excluded)
    const uint32_t ex = (sw.f >> 20) & 0x7ffu;
    v.far_hi = ex - 823u < 400u ? kFarHi : 0u;
    return v;
}

NRS_HD uint32_t magnitude_hi(double r) { return hi32(double_bits(r)) & 0x7fffffffu; }
NRS_HD bool tiny(double r) { return magnitude_hi(r) < kTinyHi; }

// The terms of one pair, without a branch.  The FP64 pipe bounds the assembly,
// so it is left the 16 additions and subtractions; the square root, the
// reciprocal and the 18 products r_j r_k, s and w run beside it on the integer
// pipe, rounded identically (fp64_int.cuh).  A component of r below 2^-150 is
// taken as zero (then a product with it is a zero, whose sign does not matter:
// a sum starts at +0).  odd = 1: some component was; 2 and more: the general
// path is needed.  (The components' range and the weight's in one comparison:
// 2000 x 20000 points 1748 us, 1737 without the components'; in two, 1781, with
// spills.)
NRS_HD Acc6 terms_int(double mx, double my, double mz, const StagedX &X, double eps2, double two_e2,
                      const FmaOps &op, int &odd)
{
    const double rx = op.sub(mx, X.x), ry = op.sub(my, X.y), rz = op.sub(mz, X.z);
    const uint32_t hx = magnitude_hi(rx), hy = magnitude_hi(ry), hz = magnitude_hi(rz);
    const bool tx = hx < kTinyHi, ty = hy < kTinyHi, tz = hz < kTinyHi;
    const Sig ux = unpack(rx), uy = unpack(ry), uz = unpack(rz);
    const uint32_t hxy = hx > hy ? hx : hy;
    bool bad = (hxy > hz ? hxy : hz) >= X.far_hi;
    const Sig pxx = mul_sig(ux, ux.m << 1, ux.f, bad);
    const Sig pyy = mul_sig(uy, uy.m << 1, uy.f, bad);
    const Sig pzz = mul_sig(uz, uz.m << 1, uz.f, bad);
    const double xx = tx ? 0.0 : pack(pxx), yy = ty ? 0.0 : pack(pyy), zz = tz ? 0.0 : pack(pzz);
    const double r2 = op.add(op.add(xx, yy), zz);
    const double rho = op.add(r2, eps2);
    const double dg = op.add(r2, two_e2);
    // rho in [2^-100, 2^100)
    bad |= (hi32(double_bits(rho)) - (923u << 20)) >= (200u << 20);
    const Sig s = inv_rho_sqrt(rho, bad);
    const uint64_t s2 = s.m << 1;
    auto term = [&](const Sig &p) {
        return pack(mul_sig(mul_sig(p, s2, s.f, bad), X.w2, X.wf, bad));
    };
    Acc6 v;
    v.xx = term(unpack(op.add(xx, dg)));
    v.yy = term(unpack(op.add(yy, dg)));
    v.zz = term(unpack(op.add(zz, dg)));
    const double xy = term(mul_sig(ux, uy.m << 1, uy.f, bad));
    const double xz = term(mul_sig(ux, uz.m << 1, uz.f, bad));
    const double yz = term(mul_sig(uy, uz.m << 1, uz.f, bad));
    v.xy = tx || ty ? 0.0 : xy;
    v.xz = tx || tz ? 0.0 : xz;
    v.yz = ty || tz ? 0.0 : yz;
    odd = (bad ? 2 : 0) | (tx || ty || tz ? 1 : 0);
    return v;
}

}  // namespace nrs
