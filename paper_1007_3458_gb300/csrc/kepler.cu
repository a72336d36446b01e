// kepler.cu -- E_Kep: universal-variable Kepler drift of every body about its
// star (Sec. 2 and the Appendix: f and g functions, Stumpff C and S, the
// universal Kepler equation F(x) = 0 solved by Laguerre's method, n = 5).
//
// One thread per body, the state and the solve in FP64. Structure-of-arrays
// loads are coalesced; q0, v0 are kept and the result goes to separate buffers
// because the encounter test needs both ends of the step (Sec. 2.3 item 4).
//
// The kernel is bound by the FP64 pipe: one warp instruction per ~19 cycles and
// SM, whatever the number of active lanes. So (1) only arithmetic on the state
// goes there: comparisons, scalings by powers of two and conversions work on the
// bits, the residual's scale and (until it matters) the root's bracket are FP32
// with the margins stated at each, square roots, reciprocals and quotients are rounded
// from FP32 approximations (pair64.cuh); (2) F' and F'' are formed only where a step
// follows; (3) a warp iterates while at least kPackBelow of its lanes do, then the
// CTA's unfinished bodies are packed into full warps (some 5% of bodies need another
// evaluation, that is four of five warps). 1,048,576 test particles with NEWTON32: 235 FP64
// warp instructions per warp, 369 before (0.772 -> 0.564 ms).
//
// With the learned guess (MLP = true) each warp first evaluates the guess
// network for its 32 bodies on the tensor cores (mlp.cuh); the iteration then
// starts from x_std (1 + sigma t) instead of x_std = sqrt(mu) dt / r0 for the
// bodies on bound orbits (the network's domain). With a log buffer every
// solve on a bound orbit also writes its training row (u1..u4, t) with
// t = (x / x_std - 1) / sigma at the converged root x.
#include "mlp.cuh"

namespace qym {

// Stumpff functions C = c2(y), S = c3(y) (Appendix, Eqs. 2.40) by quartering
// the argument: y is scaled by 4^-k into |y| < 1 (exactly, a power of two),
// where the series C = sum_n (-y)^n / (2n+2)!, S = sum_n (-y)^n / (2n+3)! to
// the y^8 term is exact to rounding (the first omitted term is below 1e-18),
// and k doublings of s = sqrt(y) then follow from the double-angle formulas
// of sin and cos:  c2(4y) = c1(y)^2 / 2,  c3(4y) = (c3(y) + c1(y) c2(y)) / 4,
// with c1(y) = 1 - y c3(y) = sin(s) / s formed afresh at each level. Only
// multiply-adds, no division, square root or transcendental call, and the
// same instructions for bound and unbound orbits. Past 4^64 (s > 2^64) C and
// S are NaN, which the iteration treats as a point beyond the root.
__device__ __forceinline__ void stumpff(double y, double &C, double &S) {
    int k = 0;
    const int hi = p64::hi_abs(y);
    if (hi >= 0x3ff00000) {
        // |y| in [2^e, 2^(e+1)): k = floor(e/2) + 1 puts y / 4^k in [1/4, 1)
        const int e = (hi >> 20) - 1023;
        k = e / 2 + 1;
        if (k > 64) {
            C = S = __longlong_as_double(0x7ff8000000000000ll);
            return;
        }
        y = p64::mul_pow2(y, -2 * k);
    }
    // 1/(2n+2)! and 1/(2n+3)! for n = 0..8, alternating signs
    C = 1.0 / 2.0 + y * (-1.0 / 24.0 + y * (1.0 / 720.0 + y * (-1.0 / 40320.0 +
        y * (1.0 / 3628800.0 + y * (-1.0 / 479001600.0 + y * (1.0 / 87178291200.0 +
        y * (-1.0 / 20922789888000.0 + y * (1.0 / 6402373705728000.0))))))));
    S = 1.0 / 6.0 + y * (-1.0 / 120.0 + y * (1.0 / 5040.0 + y * (-1.0 / 362880.0 +
        y * (1.0 / 39916800.0 + y * (-1.0 / 6227020800.0 + y * (1.0 / 1307674368000.0 +
        y * (-1.0 / 355687428096000.0 + y * (1.0 / 121645100408832000.0))))))));
    for (int i = 0; i < k; ++i) {
        const double c1 = fma(-y, S, 1.0);
        S = p64::mul_pow2(fma(c1, C, S), -2);
        C = p64::mul_pow2(c1 * c1, -1);
        y = p64::mul_pow2(y, 2);
    }
}

// F, F', F'' of the universal Kepler equation (Appendix), sig = r0.v0/sqrt(mu).
// Sums and products that a compiler may fuse in one place and not in another are
// written out with their roundings, here and at the state's dot products: the root
// and the drifted state are the same bits whatever is compiled around them (a last
// place here grows to 1e-8 of a velocity in an ensemble's encounters).
struct KepEq {
    double sqmu_dt, r0, sig, alpha, b;  // b = 1 - r0 alpha
    // F at x with C, S; sc: the sum of F's terms' magnitudes in FP32 (within
    // 1e-6; NaN or out of FP32's range where a term is)
    __device__ __forceinline__ double value(double x, double &C, double &S, float &sc) const {
        const double x2 = x * x;
        stumpff(alpha * x2, C, S);
        const double t1 = sig * x2, t2 = b * x2 * x;
        sc = fabsf(p64::lead(sqmu_dt, 0)) + fabsf(p64::lead(t1, 0) * p64::lead(C, 0)) +
             fabsf(p64::lead(t2, 0) * p64::lead(S, 0)) + p64::lead(r0, 0) * fabsf(p64::lead(x, 0));
        return fma(r0, x, __dadd_rn(__dmul_rn(t1, C), __dmul_rn(t2, S))) - sqmu_dt;
    }
    __device__ __forceinline__ double scale(double x, double C, double S) const {
        const double x2 = x * x;
        return fabs(sqmu_dt) + fabs(sig * x2 * C) + fabs(b * x2 * x * S) + r0 * fabs(x);
    }
    __device__ __forceinline__ void slopes(double x, double C, double S, double &Fp, double &Fpp) const {
        const double x2 = x * x, y = alpha * x2, oyS = 1.0 - y * S;
        Fp = __dadd_rn(fma(b * x2, C, __dmul_rn(sig * x, oyS)), r0);
        Fpp = fma(sig, fma(-y, C, 1.0), __dmul_rn(b * x, oyS));
    }
};

// Stumpff functions in FP32 for the first iterations of QYM_SOLVER_NEWTON32:
// the series to the y^6 term for |y| < 1 (its truncation below 1e-11, so
// only FP32 rounding remains), the closed forms beyond (s - sin s and
// sinh s - s lose at most about three bits there)
__device__ __forceinline__ void stumpff_f32(float y, float &C, float &S) {
    if (fabsf(y) < 1.0f) {
        C = 0.5f + y * (-1.0f / 24.0f + y * (1.0f / 720.0f + y * (-1.0f / 40320.0f +
            y * (1.0f / 3628800.0f + y * (-1.0f / 479001600.0f + y * (1.0f / 87178291200.0f))))));
        S = 1.0f / 6.0f + y * (-1.0f / 120.0f + y * (1.0f / 5040.0f + y * (-1.0f / 362880.0f +
            y * (1.0f / 39916800.0f + y * (-1.0f / 6227020800.0f + y * (1.0f / 1307674368000.0f))))));
    } else if (y > 0.0f) {
        const float s = sqrtf(y);
        float sh, ch;
        sincosf(0.5f * s, &sh, &ch);
        C = 2.0f * sh * sh / y;
        S = (s - 2.0f * sh * ch) / (y * s);
    } else {
        const float s = sqrtf(-y);
        C = (coshf(s) - 1.0f) / (-y);
        S = (sinhf(s) - s) / ((-y) * s);
    }
}

// The iteration of one body between two evaluations of F
struct KepIter {
    double x, lo, hi;      // the point to evaluate next; the root's bracket
    bool rough;            // its outer bound is the FP32 one (kep_bracket), then
    float inside;          // a magnitude below the FP64 form's
    double dx_old;         // last step
    double x_prev, res_prev;  // settle: the point the last step started from, its relative residual
    double C, S;           // Stumpff values of the last evaluation
    int it, iters;         // evaluations of this pass; iterations counted in all
    bool settle;           // the last step was at the rounding level
    bool conv, cs_at_x;    // C, S hold the Stumpff values at the final x
};

// Root bracket: F(0) = -sqrt(mu) dt and F' = r >= r_p (periapsis distance), so
// the root lies between 0 and the outer bound sqrt(mu) dt / r_p; for an unbound
// orbit also |x| <= 700 / sqrt(-alpha), past which C and S overflow. Widened by
// 1e-12 for the rounding of r_p = p / (1 + e).
// Returns the outer bound (of dt's sign; infinite where there is none). Out of
// line, by value: the body's iteration stays in registers.
__device__ __noinline__ double kep_outer_exact(const double *q, const double *v, int64_t ld, double imu,
                                               double alpha, double sqmu_dt, bool forward) {
    const double qx = q[0], qy = q[ld], qz = q[2 * ld];
    const double vx = v[0], vy = v[ld], vz = v[2 * ld];
    const double hx = qy * vz - qz * vy, hy = qz * vx - qx * vz, hz = qx * vy - qy * vx;
    const double p = (hx * hx + hy * hy + hz * hz) * imu;
    const double ecc = sqrt(fmax(0.0, 1.0 - p * alpha));
    double out = forward ? INFINITY : -INFINITY;
    if (p > 0.0) out = sqmu_dt * (1.0 + ecc) / p * (1.0 + 1e-12);
    if (alpha < 0.0) {
        // rsqrt within 2 ulp: the bound is widened by 1e-12
        const double xm = 700.0 * (1.0 + 1e-12) * rsqrt(-alpha);
        out = forward ? fmin(out, xm) : fmax(out, -xm);
    }
    return out;
}

// both bounds by the FP64 form
__device__ __forceinline__ void kep_exact_bracket(const KeplerArgs &a, int64_t r, double imu, const KepEq &eq,
                                                  KepIter &s) {
    const bool forward = a.dt >= 0.0;
    const double out = kep_outer_exact(a.q0 + r, a.v0 + r, a.ld, imu, eq.alpha, eq.sqmu_dt, forward);
    // (a radial bound orbit has no outer bound, and then no inner one either)
    const double in = p64::finite_bits(out) || out != out ? 0.0 : -out;
    s.lo = forward ? in : out;
    s.hi = forward ? out : in;
    s.rough = false;
}

// The outer bound of an iteration by the FP64 form, where a decision may depend
// on it (`rough` says that neither bound there has been replaced by a point)
__device__ __forceinline__ void kep_refine_bracket(const KeplerArgs &a, int64_t r, double imu, const KepEq &eq,
                                                   KepIter &s) {
    if (!s.rough) return;
    const bool forward = a.dt >= 0.0;
    const double out = kep_outer_exact(a.q0 + r, a.v0 + r, a.ld, imu, eq.alpha, eq.sqmu_dt, forward);
    if (forward) s.hi = out; else s.lo = out;
    s.rough = false;
}

// whether x, reached by a step dx of 2^-10 or more, may lie beyond the FP64 form's
// outer bound (the rough one is at or above it, s.inside below)
__device__ __forceinline__ bool kep_near_outer(const KepIter &s, double x, double dx) {
    return !(fabsf(p64::lead(x, 0)) <= s.inside) && p64::abs_bits(dx) > p64::abs_bits(x) - (10ll << 52);
}

// The bracket of a bound orbit in FP32: the angular momentum is within 1e-6 |q||v|
// of the FP64 one, so where it is above |q||v| / 4, p is within 1e-5, and the bound
// is known from both sides: within 0.4% for e below 0.01, 1e-4 and less above 0.1.
// The upper side serves until a step of 2^-10 or more may end beyond the FP64 bound
// or would be bisected, which is rare; then the FP64 form takes its place and the
// decision is that form's. (A smaller step that ends a hair beyond the FP64 bound, on
// a near-circular orbit, is kept where that form would bisect.) Other orbits take the
// FP64 form at once.
__device__ __forceinline__ void kep_bracket(const KeplerArgs &a, int64_t r, double imu, const KepEq &eq,
                                            double qx, double qy, double qz, double vx, double vy,
                                            double vz, double r0sq, double vv, KepIter &s) {
    const float x = p64::lead(qx, 0), y = p64::lead(qy, 0), z = p64::lead(qz, 0);
    const float u = p64::lead(vx, 0), v = p64::lead(vy, 0), w = p64::lead(vz, 0);
    const float hx = y * w - z * v, hy = z * u - x * w, hz = x * v - y * u;
    const float h2 = fmaf(hx, hx, fmaf(hy, hy, hz * hz));
    const float qv = p64::lead(r0sq, 0) * p64::lead(vv, 0), al = p64::lead(eq.alpha, 0);
    const float p = h2 * p64::lead(imu, 0), pa = p * al, num = p64::lead(eq.sqmu_dt, 0);
    s.rough = false;
    if (al > 0.0f && h2 > 0x1p-4f * qv && h2 > 1e-25f && qv < 1e30f && p > 1e-25f && p < 1e25f &&
        pa < 1e20f && fabsf(num) > 1e-15f && fabsf(num) < 1e10f) {
        // e = sqrt(1 - p alpha), raised by the error of p alpha
        const float E = 1.0f - pa, xp = num / p;
        const float b = xp * (1.0f + sqrtf(fmaxf(0.0f, E) + 1.2e-5f)) * (1.0f + 2e-5f);
        s.inside = fabsf(xp) * (1.0f + sqrtf(fmaxf(0.0f, E - 1.2e-5f))) * (1.0f - 2e-5f);
        s.rough = fabsf(b) < 1e37f && fabsf(b) > 1e-35f;
        const double xb = p64::to_double(b);
        s.lo = a.dt >= 0.0 ? 0.0 : xb;
        s.hi = a.dt >= 0.0 ? xb : 0.0;
    }
    if (!s.rough) kep_exact_bracket(a, r, imu, eq, s);
}

// standard: x is the standard guess sqrt(mu) dt / r0, inside the bracket as r0 >= r_p
__device__ __forceinline__ void kep_start(const KeplerArgs &a, int64_t r, double imu, const KepEq &eq,
                                          KepIter &s, double x, bool standard) {
    if (s.rough && !standard &&
        !(p64::finite_bits(x) && !kep_near_outer(s, x, x) && (x >= 0.0) == (a.dt >= 0.0)))
        kep_refine_bracket(a, r, imu, eq, s);
    s.x = x;
    if (!s.rough && p64::finite_bits(s.lo) && p64::finite_bits(s.hi) && !(x >= s.lo && x <= s.hi))
        s.x = 0.5 * (s.lo + s.hi);
    s.dx_old = INFINITY;
    s.settle = s.conv = s.cs_at_x = false;
    s.x_prev = s.x;
    s.res_prev = INFINITY;
    s.it = 0;
}

// QYM_SOLVER_NEWTON32: Newton's method on F in FP32 from x while it stays in
// the bracket [lo, hi] (at most 12 steps), until a step falls below 1e-5 |x|;
// x then holds the FP32 root (relative error about 1e-7, more where F's terms
// cancel) and the FP64 iteration finishes from there under the unchanged
// residual test. Returns
// the FP32 steps taken, and leaves x unchanged (0 steps counted) when the FP32
// form fails (a step leaves the bracket, F or F' is not finite).
__device__ __forceinline__ int newton_f32(const KeplerArgs &a, int64_t r, double imu, const KepEq &eq,
                                          KepIter &s, double &x) {
    const float sq = p64::to_float(eq.sqmu_dt), r0 = p64::to_float(eq.r0), sig = p64::to_float(eq.sig);
    const float al = p64::to_float(eq.alpha), b = p64::to_float(eq.b);
    float lof = p64::to_float(s.lo), hif = p64::to_float(s.hi);
    float xf = p64::to_float(x);
    for (int it = 0; it < 12; ++it) {
        const float x2 = xf * xf, y = al * x2;
        float C, S;
        stumpff_f32(y, C, S);
        const float F = sig * x2 * C + b * x2 * xf * S + r0 * xf - sq;
        const float Fp = sig * xf * (1.0f - y * S) + b * x2 * C + r0;
        if (!isfinite(F) || !(Fp > 0.0f) || !isfinite(Fp)) return 0;
        const float dx = F / Fp;
        const float xn = xf - dx;
        if (s.rough && !(fabsf(xn) <= s.inside || fabsf(dx) < 0x1p-10f * fabsf(xn))) {
            kep_refine_bracket(a, r, imu, eq, s);
            lof = p64::to_float(s.lo);
            hif = p64::to_float(s.hi);
        }
        if (!(xn >= lof && xn <= hif)) return 0;
        xf = xn;
        if (fabsf(dx) <= 1e-5f * fabsf(xf)) {
            x = fabsf(xf) >= 1.1754944e-38f ? p64::to_double(xf) : (double)xf;
            return it + 1;
        }
    }
    return 0;
}

// One evaluation and the step from it; true when the iteration has ended
// (converged, or max_iter evaluations made)
__device__ __forceinline__ bool kep_iterate(const KeplerArgs &a, int64_t r, double imu, const KepEq &eq,
                                            bool laguerre, KepIter &s) {
    if (s.it >= a.max_iter) return true;
    ++s.it;
    ++s.iters;
    const double x = s.x;
    float sc;
    const double F = eq.value(x, s.C, s.S, sc);
    const bool F_ok = p64::finite_bits(F);
    double scale = 0.0;
    if (F_ok) {
        // |F| <= 1e-14 sum |terms|, in FP32 where its range holds and the two sides
        // differ by more than the FP32 sum's error: the decision is the FP64 one
        bool small = false;
        const float Fa = fabsf(p64::lead(F, 0)), lim = 1e-14f * sc;
        if (sc > 1e-18f && sc < 1e30f && !(fabsf(Fa - lim) <= 4e-6f * lim)) {
            small = Fa < lim;
        } else {
            scale = eq.scale(x, s.C, s.S);
            small = fabs(F) <= 1e-14 * scale;
        }
        if (small) {
            --s.iters;
            s.conv = s.cs_at_x = true;
            return true;
        }
        if (s.settle) {
            // evaluated after a rounding-level step and still above 1e-14: the
            // better of the last two points is the root
            if (scale == 0.0) scale = eq.scale(x, s.C, s.S);
            --s.iters;
            s.conv = true;
            if (fabs(F) / scale <= s.res_prev) s.cs_at_x = true; else s.x = s.x_prev;
            return true;
        }
    }
    double Fp = 0.0, Fpp = 0.0;
    if (F_ok) eq.slopes(x, s.C, s.S, Fp, Fpp);
    if (!F_ok || !p64::finite_bits(Fp) || !p64::finite_bits(Fpp)) {
        if (x > 0.0) s.hi = x; else s.lo = x;
        if ((x > 0.0) == (a.dt >= 0.0)) s.rough = false;
        kep_refine_bracket(a, r, imu, eq, s);
        s.x = 0.5 * (s.lo + s.hi);
        return false;
    }
    if (F < 0.0) s.lo = x; else s.hi = x;
    if ((F < 0.0) == (a.dt < 0.0)) s.rough = false;  // the outer bound is a point now
    double dx;
    const double iFp = Fp > 0.0 ? p64::rcp(Fp) : 1.0 / Fp;
    if (laguerre) {
        // Laguerre, n = 5: dx = n F / (F' + sgn(F') sqrt|(n-1)^2 F'^2 - n(n-1) F F''|),
        // with F' taken out of the root so that F'^2 never overflows:
        // dx = rf 5 / (1 + sqrt|16 - 20 z|), rf = F / F', z = rf F'' / F'.
        // Near the root (|z| < 1e-6) the factor is its series
        // 1 + z / 2 + 13 z^2 / 32 (next term 0.38 z^3 < 4e-19): the same
        // step to rounding without the square root and the division
        const double rf = F * iFp, z = rf * (Fpp * iFp);
        if (p64::hi_abs(z) < 0x3eb0c6f7) {  // 1e-6
            dx = rf * fma(z, fma(13.0 / 32.0, z, 0.5), 1.0);
        } else {
            double irt;
            const double den = 1.0 + p64::sqrt_rcp(fabs(16.0 - 20.0 * z), irt);
            dx = p64::div(5.0 * rf, den, p64::rcp(den));
        }
    } else {
        dx = p64::div(F, Fp, iFp);
    }
    double xn = x - dx;
    // bisect when the step is not finite, leaves the bracket, or fails
    // to halve the previous step (slow approach along exp(sqrt(-alpha) x))
    if (s.rough && (!p64::finite_bits(dx) || kep_near_outer(s, xn, dx) ||
                    p64::abs_bits(dx) > p64::abs_bits(s.dx_old) - (1ll << 52) ||
                    p64::order_bits(xn) < p64::order_bits(s.lo) || p64::order_bits(xn) > p64::order_bits(s.hi)))
        kep_refine_bracket(a, r, imu, eq, s);
    const bool have_br = p64::finite_bits(s.lo) && p64::finite_bits(s.hi);
    if (have_br) {
        const long long xo = p64::order_bits(xn);
        if (!p64::finite_bits(dx) || xo < p64::order_bits(s.lo) || xo > p64::order_bits(s.hi) ||
            p64::abs_bits(dx) > p64::abs_bits(s.dx_old) - (1ll << 52)) {
            xn = 0.5 * (s.lo + s.hi);
            dx = x - xn;
        }
    }
    s.dx_old = dx;
    const long long small = p64::abs_bits(xn) - (50ll << 52);  // 2^-50 |xn|
    const double wd = s.hi - s.lo;
    if (p64::abs_bits(dx) <= small || p64::abs_bits(dx) == 0 ||
        (have_br && (p64::abs_bits(wd) <= small || p64::abs_bits(wd) == 0 || __double2hiint(wd) < 0))) {
        s.settle = true;
        s.x_prev = x;
        s.res_prev = fabs(F) / eq.scale(x, s.C, s.S);
    }
    s.x = xn;
    return false;
}

constexpr int kPackBelow = 12;  // lanes still iterating below which a warp's bodies are packed

// an unfinished body on its way to another thread of the CTA
struct KepPacked {
    KepEq eq;
    KepIter s;
    int64_t r;
    double imu;
};

template <bool MLP, int T>
__global__ void __launch_bounds__(T, 512 / T) k_kepler(const __grid_constant__ KeplerArgs a) {
    chain_wait();
    __shared__ KepPacked s_body[T];
    __shared__ int s_list[T];
    __shared__ int s_n;
    const int tid = threadIdx.x;
    if (tid == 0) s_n = 0;
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + tid;
    const bool act = k < a.n;
    const int64_t r = act ? (a.rows ? a.rows[k] : a.row0 + k) : 0;
    const int64_t ld = a.ld;
    double qx = 0.0, qy = 0.0, qz = 0.0, vx = 0.0, vy = 0.0, vz = 0.0;
    // sqrt(mu) and 1/mu of mu = G m0, formed once per system on the host
    // (correctly rounded, as sqrt and the division here would give them)
    double sqmu = 1.0, imu = 1.0;
    if (act) {
        qx = a.q0[r]; qy = a.q0[ld + r]; qz = a.q0[2 * ld + r];
        vx = a.v0[r]; vy = a.v0[ld + r]; vz = a.v0[2 * ld + r];
        if (a.kmu) {
            const double *km = a.kmu + 3 * (int64_t)a.sys_of[r];
            sqmu = km[1]; imu = km[2];
        } else {
            sqmu = a.sqmu; imu = a.imu;
        }
    }
    const double dt = a.dt;
    const double r0sq = fma(qz, qz, fma(qy, qy, qx * qx));
    double ir0 = 0.0;
    const double r0 = p64::sqrt_rcp(r0sq, ir0);
    const bool body = act && !(r0 == 0.0);
    const double vv = fma(vz, vz, fma(vy, vy, vx * vx));
    const double rv = fma(qz, vz, fma(qy, vy, qx * vx));
    float u[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    double sigma = 0.0;
    bool bound = false;  // in the learned guess's domain
    if (act && r0 > 0.0 && dt != 0.0 && (MLP || a.log))
        bound = mlp::features(rv, vv, r0, ir0, sqmu, imu, dt, u, sigma);
    double x_mlp = 0.0;
    bool have_mlp = false;
    if (MLP) {
        // every lane of the warp takes part, active or not
        float fn[4];
        mlp::normalise(a.mlp_w, u, fn);
        const float y = mlp::warp_forward(a.mlp_w, fn);
        const float tn = a.mlp_w[mlp::OM] + a.mlp_w[mlp::OSD] * y;
        x_mlp = sqmu * dt * ir0 * (1.0 + sigma * (double)tn);
        have_mlp = bound && isfinite(x_mlp);
    }
    // the FP64 pipe bounds this kernel: divisions by mu, sqrt(mu) and r0
    // become products with reciprocals formed once (within an ulp of the
    // quotients)
    const double isqmu = sqmu * imu;
    KepEq eq;
    KepIter s;
    s.iters = 0;
    bool laguerre = a.solver != QYM_SOLVER_NEWTON;
    bool busy = body;
    if (body) {
        eq.sqmu_dt = sqmu * dt;
        eq.r0 = r0;
        eq.alpha = 2.0 * ir0 - vv * imu;
        eq.sig = rv * isqmu;
        eq.b = 1.0 - r0 * eq.alpha;
        double x;
        const bool standard = a.guess != QYM_GUESS_R0 && !(MLP && have_mlp);
        if (standard)
            x = eq.sqmu_dt * ir0;
        else
            x = a.guess == QYM_GUESS_R0 ? r0 : x_mlp;
        if (a.x0_out) a.x0_out[k] = x;
        kep_bracket(a, r, imu, eq, qx, qy, qz, vx, vy, vz, r0sq, vv, s);
        // FP32 Newton steps first, then the FP64 iteration in Laguerre's
        // form: from the FP32 root (about 1e-7) one cubic step reaches
        // the rounding level, so the evaluation after it meets the
        // residual test
        if (a.solver == QYM_SOLVER_NEWTON32) s.iters = newton_f32(a, r, imu, eq, s, x);
        kep_start(a, r, imu, eq, s, x, standard && s.iters == 0);
    }
    // (a warp below the threshold from the start iterates once all the same)
    do {
        if (busy) busy = !kep_iterate(a, r, imu, eq, laguerre, s);
    } while (__popc(__ballot_sync(0xffffffffu, busy)) >= kPackBelow);
    __syncthreads();  // s_n = 0
    int slot = -1;
    if (busy) {
        slot = atomicAdd(&s_n, 1);
        s_list[slot] = tid;
        s_body[tid].eq = eq;
        s_body[tid].s = s;
        s_body[tid].r = r;
        s_body[tid].imu = imu;
    }
    __syncthreads();
    if (tid < s_n) {
        KepPacked &b = s_body[s_list[tid]];
        const KepEq e = b.eq;
        KepIter t = b.s;
        while (!kep_iterate(a, b.r, b.imu, e, laguerre, t)) {}
        b.s = t;
    }
    __syncthreads();
    if (body) {
        if (slot >= 0) s = s_body[tid].s;
        // learned guess only: Laguerre from the standard guess if the iteration
        // from it did not converge
        if (MLP && !s.conv) {
            kep_exact_bracket(a, r, imu, eq, s);
            kep_start(a, r, imu, eq, s, eq.sqmu_dt * ir0, true);
            while (!kep_iterate(a, r, imu, eq, true, s)) {}
        }
        const double x = s.x;
        // f and g functions at the root (Appendix); r before fdot, gdot. The
        // last evaluation left C, S at this x unless the iteration kept the
        // point before it, or ran out of iterations after a step
        const double x2 = x * x, y = eq.alpha * x2;
        double C = s.C, S = s.S;
        if (!s.cs_at_x) stumpff(y, C, S);
        const double x2C = x2 * C;
        const double f = 1.0 - x2C * ir0;
        const double g = dt - x2 * x * S * isqmu;
        const double nx = f * qx + g * vx, ny = f * qy + g * vy, nz = f * qz + g * vz;
        double irr;
        p64::sqrt_rcp(nx * nx + ny * ny + nz * nz, irr);
        const double fd = sqmu * x * (y * S - 1.0) * irr * ir0;
        const double gd = 1.0 - x2C * irr;
        const double ux = fd * qx + gd * vx, uy = fd * qy + gd * vy, uz = fd * qz + gd * vz;
        a.q1[r] = nx; a.q1[ld + r] = ny; a.q1[2 * ld + r] = nz;
        a.v1[r] = ux; a.v1[ld + r] = uy; a.v1[2 * ld + r] = uz;
        if (a.x_out) a.x_out[k] = x;
        if (a.iters) a.iters[k] = s.iters;
        if (a.log && bound) {
            // training row of this solve: slot (steps logged so far) * n + k
            const int64_t base = a.log_step ? (int64_t)(*a.log_base + *a.log_step) * a.n : 0;
            const int64_t row_i = base + k;
            if (row_i < a.log_cap) {
                const double t = (x * r0 / eq.sqmu_dt - 1.0) / sigma;
                float *row = a.log + 5 * row_i;
                row[0] = u[0]; row[1] = u[1]; row[2] = u[2]; row[3] = u[3];
                row[4] = (float)t;
            }
        }
        if (a.status) {
            int bits = 0;
            if (!s.conv) bits |= QYM_ST_KEPLER_NOCONV;
            if (!(p64::finite_bits(nx) && p64::finite_bits(ny) && p64::finite_bits(nz) &&
                  p64::finite_bits(ux) && p64::finite_bits(uy) && p64::finite_bits(uz)))
                bits |= QYM_ST_NAN;
            if (bits) atomicOr(a.status, bits);
        }
    } else if (act) {
        // a star row (held at Q = v = 0): stays at the origin
        a.q1[r] = 0.0; a.q1[ld + r] = 0.0; a.q1[2 * ld + r] = 0.0;
        a.v1[r] = 0.0; a.v1[ld + r] = 0.0; a.v1[2 * ld + r] = 0.0;
        if (a.x_out) a.x_out[k] = 0.0;
        if (a.x0_out) a.x0_out[k] = 0.0;
        if (a.iters) a.iters[k] = 0;
    }
    if (a.iter_sum) {
        const unsigned sum = __reduce_add_sync(0xffffffffu, body ? (unsigned)s.iters : 0u);
        if ((tid & 31) == 0 && sum) atomicAdd(a.iter_sum, (unsigned long long)sum);
    }
}

template <bool MLP>
static cudaError_t launch_kepler_t(const KeplerArgs &a, cudaStream_t st) {
    // A warp issues an FP64 instruction every 64 cycles, an SM one every 19: the
    // fewest bodies spread best as two warps a CTA, one or two CTAs on every SM
    // (16384 test particles 64 us in CTAs of 256, on 64 of the SMs); large inputs
    // pack their unfinished bodies over eight warps.
    if (a.n <= 4 * 64 * 152)
        return launch_chain(k_kepler<MLP, 64>, (unsigned)((a.n + 63) / 64), 64, 0, st, a);
    return launch_chain(k_kepler<MLP, 256>, (unsigned)((a.n + 255) / 256), 256, 0, st, a);
}

cudaError_t launch_kepler(const KeplerArgs &a, cudaStream_t st) {
    if (a.n <= 0) return cudaSuccess;
    return a.guess == QYM_GUESS_MLP && a.mlp_w ? launch_kepler_t<true>(a, st) : launch_kepler_t<false>(a, st);
}

}  // namespace qym
