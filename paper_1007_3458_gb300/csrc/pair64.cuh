// pair64.cuh -- separations, r^-1 and r^-3 of a pair to FP64 accuracy on the
// FP32 pipes.
//
// An SM of this GPU retires one FP64 warp instruction per ~19 cycles, the time
// of 76 FP32 ones, so the ~22 FP64 instructions of a pair force (separations,
// r^2, reciprocal square root, products, sums) cost more than the same
// arithmetic on unevaluated sums of three floats (24 + 24 + 24 bits). The
// building blocks are the error-free transformations of floating-point sums
// and products (Dekker 1971; Knuth's two-sum): a float sum or product together
// with its rounding error, itself a float. A reciprocal square root starts from
// the FP32 approximation y0 and is corrected by the binomial series of
// (1 - e)^(-1/2) or (1 - e)^(-3/2) in e = 1 - r^2 y0^2 (|e| < 2^-20: e^3 is
// below 2^-60). Every dropped term is below 2^-56 of the result, so what is
// left are the two roundings of its assembly as a double: at most 1 ulp over
// 4e6 pairs against 113-bit arithmetic, where the FP64 form's ten roundings
// reach 9.9 ulp.
//
// Range: one of the two positions has coordinates below 2 in magnitude (Scale),
// and r^2, the weight and the result leave room in FP32's range for their low
// parts (r2_fits, g_fits, kMinResult); r >= 2^-25 also keeps the separation's
// leading parts apart. The callers evaluate the pairs outside in FP64.
//
// Written with explicit roundings (no contraction), so host and device give
// the same bits but for the approximation y0.
#pragma once
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define P64_HD __host__ __device__ __forceinline__
#else
#define P64_HD inline
#include <cmath>
#endif

namespace qym {
namespace p64 {

#ifdef __CUDA_ARCH__
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ uint32_t bits(float a) { return __float_as_uint(a); }
__device__ __forceinline__ float from_bits(uint32_t a) { return __uint_as_float(a); }
__device__ __forceinline__ int32_t to_int(float a) { return __float2int_rn(a); }
__device__ __forceinline__ uint64_t bits64(double a) { return (uint64_t)__double_as_longlong(a); }
__device__ __forceinline__ double from_bits64(uint64_t a) { return __longlong_as_double((long long)a); }
#else
P64_HD float add(float a, float b) { return a + b; }
P64_HD float sub(float a, float b) { return a - b; }
P64_HD float mul(float a, float b) { return a * b; }
P64_HD float fma_(float a, float b, float c) { return fmaf(a, b, c); }
P64_HD uint32_t bits(float a) { uint32_t u; memcpy(&u, &a, 4); return u; }
P64_HD float from_bits(uint32_t u) { float a; memcpy(&a, &u, 4); return a; }
P64_HD int32_t to_int(float a) { return (int32_t)lrintf(a); }
P64_HD uint64_t bits64(double a) { uint64_t u; memcpy(&u, &a, 8); return u; }
P64_HD double from_bits64(uint64_t u) { double a; memcpy(&a, &u, 8); return a; }
#endif

struct F3 {
    float h, m, l;  // h + m + l, each below half an ulp of the one before
};

// s + e = a + b exactly
P64_HD void two_sum(float a, float b, float &s, float &e) {
    s = add(a, b);
    const float bb = sub(s, a);
    e = add(sub(a, sub(s, bb)), sub(b, bb));
}
// the same for |a| >= |b| (or a = 0)
P64_HD void fast_two_sum(float a, float b, float &s, float &e) {
    s = add(a, b);
    e = sub(b, sub(s, a));
}
// p + e = a b exactly
P64_HD void two_prod(float a, float b, float &p, float &e) {
    p = mul(a, b);
    e = fma_(a, b, -p);
}

// x as h + m + l, exact for 2^-88 <= |x| < 2^128 (zero below, h infinite above
// or NaN), by moving its bits: the leading 24 in place, the next 15 and the last
// 14 under the exponents they stand for, each less its implicit one. No FP64
// instruction (a conversion holds the FP64 pipe like an addition).
P64_HD F3 split3(double x) {
    const uint64_t u = bits64(x);
    const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
    const uint32_t e = (hi >> 20) & 0x7ffu, sign = hi & 0x80000000u;
    const uint32_t a = ((((hi << 3) | (lo >> 29)) & 0x7fffffffu) ^ 0x40000000u) | sign;
    const uint32_t b1 = (a & 0xff800000u) - (23u << 23), b2 = b1 - (15u << 23);
    // rounded to nearest part by part: each stays under half the last place of
    // the one before
    F3 r;
    float t, v;
    fast_two_sum(from_bits(a), sub(from_bits(b1 | ((lo >> 6) & 0x7fff00u)), from_bits(b1)), t, v);
    two_sum(v, sub(from_bits(b2 | ((lo << 9) & 0x7ffe00u)), from_bits(b2)), v, r.l);
    fast_two_sum(t, v, r.h, r.m);
    if (e - (1023u - 88u) > 88u + 127u) {
        const bool small = e < 1023u - 88u;
        r.h = small ? 0.0f : from_bits(0x7f800000u | sign);
        r.m = r.l = small ? 0.0f : r.h;
    }
    return r;
}

// a - b: exact where a and b are near each other, else to 2^-70 of |a| + |b|
P64_HD F3 diff(const F3 &a, const F3 &b) {
    float s, e, t, f, v, g, r;
    two_sum(a.h, -b.h, s, e);
    two_sum(a.m, -b.m, t, f);
    two_sum(e, t, v, g);
    const float low = add(g, add(f, sub(a.l, b.l)));
    F3 d;
    fast_two_sum(s, v, d.h, r);
    two_sum(r, low, d.m, d.l);
    return d;
}

// Sum of small terms: an accumulator started at a value `big` above every
// partial sum, so that each addition's error is the three-operation form
struct Biased {
    float big, t, err;
    P64_HD explicit Biased(float b) : big(b), t(b), err(0.0f) {}
    P64_HD void operator+=(float z) {
        const float n = add(t, z);
        err = add(err, sub(z, sub(n, t)));
        t = n;
    }
    P64_HD float sum() const { return sub(t, big); }
};

// |d|^2 = r.h + r.m + r.l, error below 2^-60 relative
P64_HD F3 norm2(const F3 &x, const F3 &y, const F3 &z) {
    float px, ex, py, ey, pz, ez, qx, fx, qy, fy, qz, fz;
    const float x2 = add(x.h, x.h), y2 = add(y.h, y.h), z2 = add(z.h, z.h);
    two_prod(x.h, x.h, px, ex);
    two_prod(y.h, y.h, py, ey);
    two_prod(z.h, z.h, pz, ez);
    two_prod(x2, x.m, qx, fx);
    two_prod(y2, y.m, qy, fy);
    two_prod(z2, z.m, qz, fz);
    // second-order parts: m^2 + 2 h l + the products' errors
    const float ox = fma_(x.m, x.m, fma_(x2, x.l, fx));
    const float oy = fma_(y.m, y.m, fma_(y2, y.l, fy));
    const float oz = fma_(z.m, z.m, fma_(z2, z.l, fz));
    float s, e1, S, e2;
    two_sum(px, py, s, e1);
    two_sum(s, pz, S, e2);
    // eight first-order terms, each below 2^-23 S
    Biased a(mul(S, 0x1p-16f));
    a += qx;
    a += qy;
    a += qz;
    a += ex;
    a += ey;
    a += ez;
    a += e1;
    a += e2;
    F3 r;
    r.h = S;
    r.m = a.sum();
    r.l = add(a.err, add(ox, add(oy, oz)));
    return r;
}

// e = 1 - r2 y0^2 as E0 + E1 (|e| < 2^-20, error below 2^-62; E0 a multiple
// of 2^-39), and w = y0^2 = w0 + w1 exactly
struct Residual {
    float w0, w1, E0, E1;
};
P64_HD Residual residual(const F3 &r2, float y0) {
    Residual R;
    two_prod(y0, y0, R.w0, R.w1);
    float p, pe, q1, f1, q2, f2;
    two_prod(r2.h, R.w0, p, pe);
    two_prod(r2.m, R.w0, q1, f1);
    two_prod(r2.h, R.w1, q2, f2);
    const float o = fma_(r2.m, R.w1, fma_(r2.l, R.w0, add(f1, f2)));
    Biased a(0x1p-16f);
    a += sub(1.0f, p);  // exact: p lies within 2^-20 of 1
    a += -pe;
    a += -q1;
    a += -q2;
    R.E0 = a.sum();
    R.E1 = sub(a.err, o);
    return R;
}

// (h + m + l) 2^k as a double, for h >= kMinResult, m below 2^-22 h and l below
// 2^-42 h (bias: k << 52): the bits of h shifted into FP64 place, then the rest
// added to the mantissa as an integer in units of the last place (of the
// binade below h when the rest is negative and h is a power of two). No FP64
// instruction; two roundings of half a unit.
constexpr float kMinResult = 0x1p-70f;
P64_HD double to_double(float h, float m, float l, uint64_t bias) {
    float s, r;
    fast_two_sum(h, m, s, r);
    const uint32_t b = bits(s);
    const uint32_t tb = b + (uint32_t)((int32_t)bits(add(r, l)) >> 31);
    // 2^(52 - exponent)
    const float K = from_bits((306u << 23) - (tb & 0x7f800000u));
    const int32_t i = to_int(mul(r, K)) +
                      (int32_t)(bits(fma_(l, K, 12582912.0f)) - 0x4b400000u);
    return from_bits64((((uint64_t)b << 29) + (0x3800000000000000ull + bias)) + (uint64_t)(int64_t)i);
}

// r^2 (its leading part) and the weight's leading part inside the range where
// every low part is a normal float; false for NaN
P64_HD bool r2_fits(float r2) { return r2 >= 0x1p-50f && r2 <= 0x1p+40f; }
P64_HD bool g_fits(float g) { return g >= 0x1p-60f && g <= 0x1p+40f; }

// three-part product with a float pair (w0, w1), w1 below 2^-24 w0
P64_HD F3 mul_pair(const F3 &a, float w0, float w1) {
    float p, pe, q1, f1, q2, f2, s, e, t, u;
    two_prod(a.h, w0, p, pe);
    two_prod(a.h, w1, q1, f1);
    two_prod(a.m, w0, q2, f2);
    two_sum(pe, q1, s, e);
    two_sum(s, q2, t, u);
    return F3{p, t, add(fma_(a.m, w1, fma_(a.l, w0, add(f1, f2))), add(e, u))};
}

// out = g r^-3 2^k (bias: k << 52); false where it is below kMinResult
P64_HD bool g_over_r3(const F3 &g, const F3 &r2, float y0, uint64_t bias, double &out) {
    const Residual R = residual(r2, y0);
    // (1 - e)^(-3/2) = 1 + T, T = 3/2 e + 15/8 e^2; 3/2 E0 is exact
    const float T0 = mul(1.5f, R.E0);
    const float T1 = fma_(mul(1.875f, R.E0), R.E0, mul(1.5f, R.E1));
    float p, pe, q, qe, k1, k2;
    two_prod(g.h, y0, p, pe);
    two_prod(g.m, y0, q, qe);
    two_sum(pe, q, k1, k2);
    const F3 s = mul_pair(F3{p, k1, fma_(g.l, y0, add(qe, k2))}, R.w0, R.w1);
    float z0, z0e, z, ze;
    two_prod(s.h, T0, z0, z0e);
    two_sum(z0, s.m, z, ze);
    const float lo = add(fma_(s.h, T1, fma_(s.m, T0, z0e)), add(s.l, ze));
    out = to_double(s.h, z, lo, bias);
    return s.h >= kMinResult;
}

// 1 / r 2^k (bias: k << 52) as a double
P64_HD double inv_r(const F3 &r2, float y0, uint64_t bias) {
    const Residual R = residual(r2, y0);
    // (1 - e)^(-1/2) = 1 + e / 2 + 3/8 e^2
    const float C0 = mul(0.5f, R.E0);
    const float C1 = fma_(mul(0.375f, R.E0), R.E0, mul(0.5f, R.E1));
    float z, ze;
    two_prod(y0, C0, z, ze);
    return to_double(y0, z, fma_(y0, C1, ze), bias);
}

#ifdef __CUDACC__
// Powers of two that bring a CTA's lengths (by its largest coordinate) and
// weights (by the largest weight of its first tile) near 1. Only the float
// parts are scaled; results come back unscaled through `bias`.
struct Scale {
    double len, wt;  // 2^-kb, 2^-ka
    int ka, kb;
    bool ok;         // exponents in the range where biased results are normal doubles
    // largest |coordinate| and |weight| as their high words
    __device__ __forceinline__ Scale(int hi_len, int hi_wt) {
        kb = (hi_len >> 20) - 1023;
        ka = (hi_wt >> 20) - 1023;
        ok = kb >= -200 && kb <= 200 && ka >= -200 && ka <= 200;
        len = ok ? __hiloint2double((1023 - kb) << 20, 0) : 1.0;
        wt = ok ? __hiloint2double((1023 - ka) << 20, 0) : 1.0;
    }
    // bias of weight / length^n
    __device__ __forceinline__ uint64_t bias(int n) const {
        return (uint64_t)(int64_t)(ok ? ka - n * kb : 0) << 52;
    }
};
__device__ __forceinline__ int hi_abs(double x) { return __double2hiint(x) & 0x7fffffff; }

// x 2^-k by its exponent field: zero below the normal range, infinite above it;
// infinities and NaN as they are
__device__ __forceinline__ double scale2(double x, int k) {
    const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
    if (e == 0x7ff) return x;
    if (e == 0 || e - k <= 0) return 0.0;
    if (e - k >= 0x7ff) return __hiloint2double(0x7ff00000, 0);
    return __hiloint2double(hi - k * (1 << 20), __double2loint(x));
}

// the leading 24 bits of x 2^-k as a float, truncated (zero below FP32's normal
// range, infinite above it)
__device__ __forceinline__ float lead(double x, int k) {
    const int hi = __double2hiint(x), field = (hi >> 20) & 0x7ff, e = field - k - 896;
    const unsigned b = ((unsigned)hi << 3 | (unsigned)__double2loint(x) >> 29) & 0x7fffffu;
    const unsigned f = field == 0 || e <= 0 ? 0u : (e >= 255 ? 0x7f800000u : ((unsigned)e << 23 | b));
    return __uint_as_float(f | ((unsigned)hi & 0x80000000u));
}

// |x| as an integer that orders like it
__device__ __forceinline__ long long abs_bits(double x) {
    return __double_as_longlong(x) & 0x7fffffffffffffffll;
}
// any finite or infinite double as an integer that orders like it (-0 below +0)
__device__ __forceinline__ long long order_bits(double x) {
    const long long u = __double_as_longlong(x);
    return u ^ ((u >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ bool finite_bits(double x) { return hi_abs(x) < 0x7ff00000; }
// x 2^k by its exponent field, for a normal result; zero, infinities and NaN (and
// denormals) stay as they are
__device__ __forceinline__ double mul_pow2(double x, int k) {
    return (unsigned)(hi_abs(x) - 0x00100000) >= 0x7fe00000u ? x : __hiloint2double(__double2hiint(x) + k * (1 << 20), __double2loint(x));
}
// a normal float as a double
__device__ __forceinline__ double to_double(float x) {
    const unsigned b = __float_as_uint(x);
    return __hiloint2double((int)((((b & 0x7fffffffu) >> 3) + 0x38000000u) | (b & 0x80000000u)), (int)(b << 29));
}

// Reciprocal, quotient, reciprocal square root and square root of positive normal
// numbers: one third-order step from the FP32 approximation (Householder's method:
// the binomial series in the residual e = 1 - x y or 1 - x y^2, |e| < 2^-20, to e^2;
// the next term is below 2^-61) gives y within an ulp, and one step with the exact
// residual of a multiply-add the rounded value (Markstein 1990): 1/x, a/b, sqrt(x)
// and 1/sqrt(x)'s rounded root are what the library's correctly rounded forms return,
// for five to nine FP64 instructions where those take ten and more. Outside the
// exponents [-1000, 1000] (quotient and root, whose residuals are the operands'
// size: [-500, 500]) the library forms.
__device__ __forceinline__ bool mid_range(double x) {
    const int hi = __double2hiint(x);
    return hi > (23 << 20) && hi < (2023 << 20);
}
__device__ __forceinline__ bool near_one(double x) {
    const int hi = hi_abs(x);
    return hi > (523 << 20) && hi < (1523 << 20);
}
__device__ __forceinline__ double rcp(double x) {
    if (!mid_range(x)) return 1.0 / x;
    const int k = (__double2hiint(x) >> 20) - 1023;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(lead(x, k)));
    double y = mul_pow2(to_double(r), -k);
    const double e = fma(-x, y, 1.0);
    y = fma(y, fma(e, e, e), y);
    return fma(y, fma(-x, y, 1.0), y);
}
// a / b from ib = rcp(b)
__device__ __forceinline__ double div(double a, double b, double ib) {
    if (!near_one(a) || !near_one(b)) return a / b;
    const double q = a * ib;
    return fma(ib, fma(-b, q, a), q);
}
// within an ulp of 1 / sqrt(x)
__device__ __forceinline__ double rsqrt_mid(double x) {
    const int k = ((__double2hiint(x) >> 20) - 1023) & ~1;  // even
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(lead(x, k)));
    const double y = mul_pow2(to_double(r), -(k >> 1));
    const double e = fma(-x, y * y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}
__device__ __forceinline__ double rsqrt64(double x) { return mid_range(x) ? rsqrt_mid(x) : rsqrt(x); }
// square root and the reciprocal of that rounded root
__device__ __forceinline__ double sqrt_rcp(double x, double &ir) {
    if (!mid_range(x) || !near_one(x)) {
        const double r = sqrt(x);
        ir = 1.0 / r;
        return r;
    }
    const double y = rsqrt_mid(x), s = x * y;
    const double r = fma(mul_pow2(y, -1), fma(-s, s, x), s);
    ir = fma(y, fma(-r, y, 1.0), y);
    // (the one mantissa that the step can miss: all ones)
    if (__double2loint(r) == -1 && (__double2hiint(r) & 0xfffff) == 0xfffff) ir = 1.0 / r;
    return r;
}

// x rounded to the nearest float, by its bits where the result is normal
__device__ __forceinline__ float to_float(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7ff) - 896;
    if (e <= 0 || e >= 254) return (float)x;  // (the conversion holds the FP64 pipe)
    const unsigned b = ((unsigned)e << 23) | ((hi << 3 | lo >> 29) & 0x7fffffu);
    const unsigned rest = (lo << 3) | (b & 1u);  // above half, or at half with an odd b
    return __uint_as_float((b + (rest > 0x80000000u ? 1u : 0u)) | (hi & 0x80000000u));
}

// an upper bound of |(x, y, z)| within 1e-6, without an FP64 instruction (an
// FP64 square root is ten); NaN or infinite for such inputs
__device__ __forceinline__ float norm_up(double x, double y, double z) {
    const int hm = max(hi_abs(x), max(hi_abs(y), hi_abs(z)));
    if (hm >= 0x7ff00000) return (float)x + (float)y + (float)z;
    const int k = (hm >> 20) - 1023;
    const float a = lead(x, k), b = lead(y, k), c = lead(z, k);
    const float n = sqrtf(fmaf(a, a, fmaf(b, b, c * c))) * (1.0f + 0x1p-21f);
    if (k > 127) return INFINITY;
    return k < -125 ? n * 0x1p-125f : n * __int_as_float((127 + k) << 23);
}

// x as hi + lo, each the nearest float (of x, and of x - hi)
__device__ __forceinline__ float2 split2(double x) {
    const F3 s = split3(x);
    const float hi = to_float(x);  // s.h but for ties between floats
    return make_float2(hi, add(add(sub(s.h, hi), s.m), s.l));
}
#endif

}  // namespace p64
}  // namespace qym
