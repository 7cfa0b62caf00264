// fp64.cuh -- correctly rounded FP64 division and square root for the face
// kernels, with the parts that several quotients share computed once.
//
// GB300 issues one FP64 warp instruction per 64 cycles and SM quadrant (595 G
// fused multiply-adds per second on the whole chip against 35 T in FP32), so a
// face kernel costs its count of FP64 instructions: a __ddiv_rn measures 558
// cycles, about 9 of them, a __dsqrt_rn 671.  Here the reciprocal (square
// root) starts from a float-float value of about 44 bits, made on the FP32 and
// integer pipes from the operand's bits, and one FP64 Newton step brings it
// within half a unit of 1/b (to 2^-34 of a unit).  The quotient follows
// Markstein (P. W. Markstein, "Computation of elementary functions on the IBM
// RISC System/6000 processor", IBM J. Res. Dev. 34, 1990): with y = 1/b rounded
// and q next to a/b, RN(q + RN(a - b q) y) = RN(a/b).  The slack of y against
// that theorem: the sum misses a/b by |a/b - q| |b y - 1|, and a/b (b in [1, 2))
// stays 2^-53/b units from a midpoint, so a y within 1/2 + s units serves every
// b with b^2 (1 + 2 s) < 4: for s = 2^-34 all but the b within 2^-33 of 2.  There,
// b = 2 - k 2^-52, 1/b lies k^2 2^-54 units from a multiple of half a unit, so y is
// 1/b rounded from k = 2^10 on; divisor_ok refuses the k up to 2^12 (a/b =
// 0x1.6666666666663p+0 / 0x1.ffffffffffffbp+0 fails without).  A reciprocal takes
// 3 FP64 instructions, each quotient by the same divisor 3 more; a square root
// with its reciprocal takes 8.  Operands outside the stated ranges (zeros,
// infinities, NaN, very large or small values, those divisors) take the built-in
// operations.  Times: at the face kernels that use them.
#pragma once
#include <cuda_runtime.h>

namespace spuma {

__device__ __forceinline__ int exp_bits(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
// 2^-300 <= |v| < 2^300: products and quotients of such values, and the
// remainders a - b q, stay normal
__device__ __forceinline__ bool mid_range(double v) { return (unsigned)(exp_bits(v) - (1023 - 300)) < 600u; }

// A divisor for the forms below: positive, mid_range, mantissa not among the 2^12
// below all ones.
__device__ __forceinline__ bool divisor_ok(double b)
{
    const int hi = __double2hiint(b);
    return hi > 0 && mid_range(b) && !((hi & 0xfffff) == 0xfffff && (unsigned)__double2loint(b) >= 0xfffff000u);
}

// A float's value times 2^e as a double, by its bits (|v| from 2^-126 up; a
// zero gives 2^(e-127), far below what the callers keep).
__device__ __forceinline__ double widen(float v, int e)
{
    const unsigned b = __float_as_uint(v);
    const int hi = (int)(b & 0x80000000u) | (int)(((b & 0x7fffffffu) >> 3) + ((unsigned)(1023 - 127 + e) << 20));
    return __hiloint2double(hi, (int)(b << 29));
}

// The mantissa of v > 0 in [1, 2) as a float pair (46 bits): h + l 2^-23.
__device__ __forceinline__ void mantissa_pair(double v, float& h, float& l)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    h = __uint_as_float(0x3f800000u | ((hi & 0xfffffu) << 3) | (lo >> 29));
    l = __fsub_rn(__uint_as_float(0x3f800000u | ((lo & 0x1fffffffu) >> 6)), 1.0f);
}

// 1/b within half a unit (to 2^-34 of it), for divisor_ok(b).
__device__ __forceinline__ double recip(double b)
{
    float h, l, y;
    mantissa_pair(b, h, l);
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(h));
    float e = __fmaf_rn(-h, y, 1.0f);
    e = __fmaf_rn(-l, __fmul_rn(y, 1.1920928955078125e-7f), e);
    const float c = __fmul_rn(y, __fmaf_rn(e, e, e));
    const int s = 1023 - exp_bits(b);
    const double y0 = __dadd_rn(widen(y, s), widen(c, s));
    return __fma_rn(__fma_rn(-b, y0, 1.0), y0, y0);
}

// RN(a/b) with y = recip(b), a zero or in mid_range.
__device__ __forceinline__ double div_by(double a, double b, double y)
{
    const double q = __dmul_rn(a, y);
    const double r = __fma_rn(__fma_rn(-b, q, a), y, q);
    // a zero quotient keeps a's sign (the sum above would make it +0)
    return __double2hiint(a) << 1 == 0 && __double2loint(a) == 0 ? a : r;
}

// RN(1/b) for divisor_ok(b): one more step of the same kind.
__device__ __forceinline__ double recip_rn(double b)
{
    const double y = recip(b);
    return __fma_rn(__fma_rn(-b, y, 1.0), y, y);
}

// RN(sqrt(v)), and its reciprocal as recip() gives it, for v > 0 in mid_range.
__device__ __forceinline__ double sqrt_rn(double v, double& inv)
{
    float h, l;
    mantissa_pair(v, h, l);
    const int e2 = exp_bits(v) - 1023;
    if (e2 & 1) {           // mantissa in [1, 4) with an even exponent
        h = __fadd_rn(h, h);
        l = __fadd_rn(l, l);
    }
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(h));
    // e = 1 - m y^2 in float-float
    const float t = __fmul_rn(y, y), tl = __fmaf_rn(y, y, -t);
    const float p = __fmul_rn(h, t), pl = __fmaf_rn(h, t, -p);
    float e = __fsub_rn(__fsub_rn(1.0f, p), pl);
    e = __fmaf_rn(-h, tl, e);
    e = __fmaf_rn(-l, __fmul_rn(t, 1.1920928955078125e-7f), e);
    const float c = __fmul_rn(__fmul_rn(y, e), __fmaf_rn(0.375f, e, 0.5f));
    const int s = -(e2 >> 1);
    const double y0 = __dadd_rn(widen(y, s), widen(c, s));
    const double half = __hiloint2double(__double2hiint(y0) - (1 << 20), __double2loint(y0));
    double g = __dmul_rn(v, y0);
    g = __fma_rn(__fma_rn(-g, g, v), half, g);              // within half a unit plus 2^-86
    const double y1 = __fma_rn(__fma_rn(-g, y0, 1.0), y0, y0);
    const double h1 = __hiloint2double(__double2hiint(y1) - (1 << 20), __double2loint(y1));
    const double root = __fma_rn(__fma_rn(-g, g, v), h1, g);
    // y1 is 1/g: of use for the root unless this last step moved it (sqrt(v)
    // within 2^-34 of a unit of a midpoint)
    inv = __double2loint(root) == __double2loint(g) ? y1 : recip(root);
    return root;
}

// |S|, its reciprocal, and whether quotients by |S| may use it.
struct FaceNorm {
    double mag, inv;
    bool fast;
};

__device__ __forceinline__ double sum_sq(double x, double y, double z)
{
    return __dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z));
}
__device__ __forceinline__ double dot3(double ax, double ay, double az, double bx, double by, double bz)
{
    return __dadd_rn(__dadd_rn(__dmul_rn(ax, bx), __dmul_rn(ay, by)), __dmul_rn(az, bz));
}

// a / |S| (correctly rounded)
__device__ __forceinline__ double over_norm(double a, const FaceNorm& n)
{
    if (n.fast && (mid_range(a) || a == 0.0)) return div_by(a, n.mag, n.inv);
    return __ddiv_rn(a, n.mag);
}

__device__ __forceinline__ FaceNorm face_norm(double sx, double sy, double sz)
{
    const double s2 = sum_sq(sx, sy, sz);
    FaceNorm n;
    n.fast = s2 > 0.0 && mid_range(s2);
    if (n.fast) {
        n.mag = sqrt_rn(s2, n.inv);
        n.fast = divisor_ok(n.mag);
    } else {
        n.mag = __dsqrt_rn(s2);
        n.inv = 0.0;
    }
    return n;
}

// A float near v (20 bits, |v| in float range), by its bits.
__device__ __forceinline__ float near_float(double v)
{
    const unsigned hi = (unsigned)__double2hiint(v);
    return __uint_as_float((hi & 0x80000000u) | (((hi & 0x7fffffffu) - ((1023u - 127u) << 20)) << 3));
}

// max(n.d, 0.05 |d|) with n.d = (S.d)/|S|.  Where the face is far from the
// limit (n.d above 0.06 |d| in 20-bit arithmetic; the limit is 0.05), which
// is nearly everywhere, |d| and its square root are not computed: the maximum
// is n.d itself.
__device__ __forceinline__ double limited_ndotd(double sx, double sy, double sz, double dx, double dy, double dz,
                                                const FaceNorm& n)
{
    const double dot = dot3(sx, sy, sz, dx, dy, dz);
    const double ndotd = over_norm(dot, n);
    auto ok = [](double v) { return (unsigned)(exp_bits(v) - (1023 - 40)) < 60u || exp_bits(v) == 0; };
    auto f = [](double v) { return exp_bits(v) == 0 ? 0.0f : near_float(v); };
    if (exp_bits(ndotd) != 0 && ok(ndotd) && ok(dx) && ok(dy) && ok(dz)) {
        const float nd = near_float(ndotd), fx = f(dx), fy = f(dy), fz = f(dz);
        if (nd > 0.0f && nd * nd > 0.0036f * (fx * fx + fy * fy + fz * fz)) return ndotd;
    }
    return fmax(ndotd, __dmul_rn(0.05, __dsqrt_rn(sum_sq(dx, dy, dz))));
}

// a = (gamma |S|) / max(n.d, 0.05 |d|), no contraction, every operation
// correctly rounded (bit-identical to the sequential definition).
__device__ __forceinline__ double face_coeff(double sx, double sy, double sz, double dx, double dy, double dz,
                                             double gamma)
{
    const FaceNorm n = face_norm(sx, sy, sz);
    const double denom = limited_ndotd(sx, sy, sz, dx, dy, dz, n);
    const double a = __dmul_rn(gamma, n.mag);
    if (divisor_ok(denom) && mid_range(a)) return div_by(a, denom, recip(denom));
    return __ddiv_rn(a, denom);
}

}  // namespace spuma
