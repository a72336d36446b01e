// hermite.cu -- the close-encounter branch of the hybrid step (Sec. 2.2 and
// Sec. 2.3 items 5-8), one CTA per encounter set, or a thread-block cluster
// (2, 4 or 8 CTAs) for each of the large sets predicted to take longest:
//   1. remove the (1-K) part of the first kick at q0 (item 5),
//   2. integrate the set for tau with a 4th-order Hermite predictor /
//      evaluate / corrector (Makino & Aarseth, no Ahmad-Cohen) under H'_Kep:
//      the star, fixed at the origin, plus the members' pair forces weighted
//      by [1 - K(s) + s K'(s)], jerks with the K'' term (item 6),
//   3. pre-remove the (1-K) part of the coming kick at q1 (item 7),
//   4. write the members' q1, v1 over their Kepler result (item 8).
// Members carry individual block time steps (Makino & Aarseth): time runs in
// integer ticks of |tau| / 2^48, member i steps with |tau| 2^-k_i from the
// Aarseth criterion (eta; eta_s at start-up) rounded down to a power of two,
// and a step doubles only on a commensurate block time. At each block time
// the members whose step ends there are evaluated and corrected, against
// their partners predicted to that time; a partner farther than r_crit
// exerts no force (K = 1), so an FP32 prediction with a bound on its error
// first rules out the pairs that are surely that far, and only the others
// are predicted and evaluated in FP64 (the result is the same as evaluating
// every pair). FP64 instructions issue at one per 64 cycles per warp here, so
// each block step is split by instruction stream across warps: items
// (member, coordinate) for predictor and corrector, each pair item on three or
// two warps, the star's pull on its own warp, fixed-order sums (a cluster's CTAs
// send their parts to each other and add them in rank order, so every copy of
// the set stays bit-identical). Every loop has a cap and reports through the status
// word.
//
// A set's result is the same bits whatever the work is spread over: products and
// sums that could be grouped in several ways are written out, lanes' parts are added
// in one order. Close passages amplify a last place by up to 1e9 within a few steps,
// so another grouping moves some velocity of an ensemble of a million bodies by 1e-7.
#include <climits>

#include <cooperative_groups.h>

#include "hermite_plan.cuh"
#include "pair64.cuh"
#include "qym_internal.cuh"

namespace qym {
namespace cg = cooperative_groups;

constexpr int HCAP = 320;       // members per set held in shared memory
constexpr int HTHREADS = 256;

// Comparisons by the bits of a double: an FP64 comparison holds the warp like an
// addition. y <= 0, y >= 1 and y > 1/2 of the transition's argument (finite), and
// a >= b for a, b >= 0 (false where a is NaN)
__device__ __forceinline__ bool y_at_most_0(double y) {
    return __double_as_longlong(y) <= 0;
}
__device__ __forceinline__ bool y_at_least_1(double y) {
    return (unsigned)(__double2hiint(y) - 0x3ff00000) <= 0x40000000u;  // (not NaN)
}
__device__ __forceinline__ bool y_above_half(double y) {
    return __double_as_longlong(y) > 0x3fe0000000000000ll;
}
__device__ __forceinline__ bool at_least(double a, double b) {
    const long long ua = __double_as_longlong(a);
    return ua >= __double_as_longlong(b) && ua <= 0x7ff0000000000000ll;
}

// sin and cos of (pi/2) y for y in [0, 1]: y > 1/2 is folded onto 1 - y
// (sin and cos swap), so the argument w = (pi/2) y' stays in [0, pi/4], where
// the Taylor series of sin to w^15 and of cos to w^16 leave truncation errors
// below 7e-17 and 3e-18 (the next terms, w^17/17! and w^18/18!, at pi/4).
struct HalfPi {
    double w, x, x2, x4;  // w = (pi/2) y', y' = y or 1 - y; x = w^2, x^2, x^4
    bool fold;            // y' = 1 - y: sin and cos swap
};
__device__ __forceinline__ HalfPi half_pi_arg(double y) {
    HalfPi a;
    a.fold = y_above_half(y);
    a.w = 1.5707963267948966 * (a.fold ? 1.0 - y : y);
    a.x = a.w * a.w;
    a.x2 = a.x * a.x;
    a.x4 = a.x2 * a.x2;
    return a;
}
// both polynomials in x = w^2 by Estrin's scheme
// sin w = w (1 - x/3! + x^2/5! - ... - x^7/15!)
__device__ __forceinline__ double sin_w(const HalfPi &a) {
    const double s01 = fma(-1.0 / 6.0, a.x, 1.0);
    const double s23 = fma(-1.0 / 5040.0, a.x, 1.0 / 120.0);
    const double s45 = fma(-1.0 / 39916800.0, a.x, 1.0 / 362880.0);
    const double s67 = fma(-1.0 / 1307674368000.0, a.x, 1.0 / 6227020800.0);
    const double ps = fma(fma(s67, a.x2, s45), a.x4, fma(s23, a.x2, s01));
    return a.w * ps;
}
// cos w = 1 - x/2! + x^2/4! - ... + x^8/16!
__device__ __forceinline__ double cos_w(const HalfPi &a) {
    const double c01 = fma(-0.5, a.x, 1.0);
    const double c23 = fma(-1.0 / 720.0, a.x, 1.0 / 24.0);
    const double c45 = fma(-1.0 / 3628800.0, a.x, 1.0 / 40320.0);
    const double c67 = fma(-1.0 / 87178291200.0, a.x, 1.0 / 479001600.0);
    const double c8 = (1.0 / 20922789888000.0) * (a.x4 * a.x4);
    return fma(fma(c67, a.x2, c45), a.x4, fma(c23, a.x2, c01)) + c8;
}
__device__ __forceinline__ void sincos_half_pi(double y, double &sn, double &cs) {
    const HalfPi a = half_pi_arg(y);
    const double sw = sin_w(a), pc = cos_w(a);
    sn = a.fold ? pc : sw;
    cs = a.fold ? sw : pc;
}

// Constants of the transition function of one set: K(y) = sin(pi y / 2) with
// y = 1.1 s / r_crit - 0.1 (Sec. 2.1), so y = a s - 0.1 and dy/ds = a.
struct TransC {
    double rc2;  // r_crit^2: K = 1 (and K' = K'' = 0) beyond
    double a;    // 1.1 / r_crit
    double c;    // (pi / 2) a: K' = c cos, K'' = -c^2 sin
    double nc2;  // -c^2
    __device__ __forceinline__ explicit TransC(double rc)
        : rc2(rc * rc), a(1.1 / rc), c(0.5 * kPi * a), nc2(-c * c) {}
};

// the transition's argument y = 1.1 s / r_crit - 0.1
__device__ __forceinline__ double trans_y(double s, const TransC &tc) { return fma(tc.a, s, -0.1); }

// K and its first and second derivatives with respect to s
__device__ __forceinline__ void transition(double s, const TransC &tc, double &K, double &Kp,
                                           double &Kpp) {
    const double y = trans_y(s, tc);
    if (y_at_most_0(y)) {
        K = 0.0; Kp = 0.0; Kpp = 0.0;
    } else if (y_at_least_1(y)) {
        K = 1.0; Kp = 0.0; Kpp = 0.0;
    } else {
        double sn, cs;
        sincos_half_pi(y, sn, cs);
        K = sn;
        Kp = tc.c * cs;
        Kpp = tc.nc2 * sn;
    }
}

__global__ void k_transition(int64_t n, const double *s, double rc, double *K, double *Kp,
                             double *Kpp) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const TransC tc(rc);
    double k0, k1, k2;
    transition(s[i], tc, k0, k1, k2);
    K[i] = k0;
    Kp[i] = k1;
    Kpp[i] = k2;
}

cudaError_t launch_transition(int64_t n, const double *s, double rc, double *K, double *Kp,
                              double *Kpp, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_transition<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, s, rc, K, Kp, Kpp);
    return cudaGetLastError();
}

// shared memory of k_hermite, at file scope so that every array of a set's
// state is a constant offset (no base pointers held in registers or passed
// through the stack of the per-set function)
extern __shared__ __align__(16) unsigned char g_hsmem[];

// CTAs of a cluster sharing one large set: 2, 4 or 8 (one lane group of 8
// pushes), chosen per context at launch; buffers are sized for the largest
constexpr int CLMAX = 8;
#ifndef QYM_HERM_F32MIN
#define QYM_HERM_F32MIN 64
#endif
// partners of a CTA plus active members above which the FP32 prediction
// screens the partners before the FP64 one
constexpr int F32MIN = QYM_HERM_F32MIN;
constexpr int ACH = 64;    // active members per force round (exchange, correction)
constexpr int RSL = 16;    // members per force round on a cluster (receive buffer slots)

constexpr int KMAX = 48;

// corrector constants of a level's step h (signed), rows of HermSmem::lvt:
// a2 = (-6 d - h (4 j0 + 2 j1)) / h^2 = A2D d + A2J0 j0 + A2J1 j1,
// a3 = (12 d + 6 h (j0 + j1)) / h^3 = A3D d + A3J (j0 + j1),
// x1 = x_p + h^4/24 a2 + h^5/120 a3, v1 = v_p + h^3/6 a2 + h^4/24 a3,
// and a2 at the end of the step, a2 + h a3 (d = a0 - a1)
enum LvConst : int { LV_H = 0, LV_A2D, LV_A2J0, LV_A2J1, LV_A3D, LV_A3J, LV_H4, LV_H5, LV_H3, LV_N };
// what a warp of the corrector forms from a2 and a3
enum LvForm : int { LF_X = 0, LF_V, LF_A2, LF_A3 };

struct HermSmem {
    double *ex, *ey, *ez, *eu, *ev, *ew;      // evaluation point of every member
    double *gm;                               // -G m of every member
    double *x, *y, *z, *u, *v, *w;            // state at the member's own time
    double *ax, *ay, *az, *jx, *jy, *jz;      // a, adot at the member's own time
    double *pr;                               // per-lane partial a, adot [6][HTHREADS]
    double *rb;                               // partials received from each CTA [2][CL][6][RSL]
    double *a1s;                              // a, adot of the round's active members [6][ACH]
    double *lvt;                              // corrector constants per level [LV_N][KMAX + 1]
    long long *ti;                            // member time in ticks
    float *f;                                 // x..z, u..w, ax..az, jx..jz cut to FP32 [12][HCAP]
    float *px, *py, *pz, *pd;                 // FP32 prediction and its error bound
    float *cf;                                // step criterion inputs [12][ACH]
    int32_t *lev;                             // member level: step = tau 2^-lev
    uint16_t *act;                            // members whose step ends now, and at the next
                                              // block time [2][HCAP]
    int32_t *ids;
    int32_t *need;                            // member needed in FP64 at this block time
    int32_t *nl;                              // those members [HCAP], 2 HCAP - 64 spare
                                              // (need and nl also hold the two-warp force's
                                              // exchange slots, [2][3][96] doubles)
};

__device__ __forceinline__ HermSmem carve(void *base) {
    double *p = (double *)base;
    HermSmem s;
    s.ex = p; p += HCAP; s.ey = p; p += HCAP; s.ez = p; p += HCAP;
    s.eu = p; p += HCAP; s.ev = p; p += HCAP; s.ew = p; p += HCAP;
    s.gm = p; p += HCAP;
    s.x = p; p += HCAP; s.y = p; p += HCAP; s.z = p; p += HCAP;
    s.u = p; p += HCAP; s.v = p; p += HCAP; s.w = p; p += HCAP;
    s.ax = p; p += HCAP; s.ay = p; p += HCAP; s.az = p; p += HCAP;
    s.jx = p; p += HCAP; s.jy = p; p += HCAP; s.jz = p; p += HCAP;
    s.pr = p; p += 6 * HTHREADS;
    s.rb = p; p += 2 * CLMAX * 6 * RSL;
    s.a1s = p; p += 6 * ACH;
    s.lvt = p; p += LV_N * (KMAX + 1);
    s.ti = (long long *)p; p += HCAP;
    float *fp = (float *)p;
    s.f = fp; fp += 12 * HCAP;
    s.px = fp; fp += HCAP; s.py = fp; fp += HCAP; s.pz = fp; fp += HCAP; s.pd = fp; fp += HCAP;
    s.cf = fp; fp += 12 * ACH;
    int32_t *ip = (int32_t *)fp;
    s.lev = ip; ip += HCAP;
    s.act = (uint16_t *)ip; ip += HCAP;
    s.ids = ip; ip += HCAP;
    s.need = ip; ip += HCAP;
    s.nl = ip;
    return s;
}
constexpr size_t kHermSmem =
    sizeof(double) * (HCAP * 20 + 6 * HTHREADS + 2 * CLMAX * 6 * RSL + 6 * ACH + LV_N * (KMAX + 1)) +
    sizeof(float) * (16 * HCAP + 12 * ACH) + sizeof(int32_t) * (HCAP * 7 - 64);
static_assert(2 * 3 * 96 * sizeof(double) <= (4 * HCAP - 64) * sizeof(int32_t),
              "the two-warp force's exchange slots overlay need and nl");
// two CTAs per SM (228 KB of shared memory, 1 KB of it per CTA reserved, 128 bytes
// for the variables below)
static_assert(2 * (kHermSmem + 128 + 1024) <= 228 * 1024, "Hermite shared memory above two CTAs per SM");

// The start-up level, the smallest k in [0, KMAX] with T 2^-k <= eta_s |a| / |adot|,
// from the squares (no square root and one reciprocal): T^2 4^-k <= d2 with
// T^2 = fT 2^eT and d2 = fd 2^ed (fT, fd in [1/2, 1)) holds exactly when
// 2 k >= eT - ed + (fT > fd). T when the jerk is zero.
__device__ __forceinline__ int first_level(const double *aj, double eta_s, double T2, double T) {
    const double a2 = fma(aj[0], aj[0], fma(aj[1], aj[1], aj[2] * aj[2]));
    const double j2 = fma(aj[3], aj[3], fma(aj[4], aj[4], aj[5] * aj[5]));
    if (!(j2 > 0.0)) return 0;
    const double d2 = (eta_s * eta_s) * (a2 * p64::rcp(j2));
    if (!p64::mid_range(d2) || !p64::mid_range(T2)) {
        // (out of the squares' range)
        const double dt = eta_s * sqrt(a2) / sqrt(j2);
        if (!(dt > 0.0)) return KMAX;
        int eT, ed;
        const double fT = frexp(T, &eT), fd = frexp(dt, &ed);
        return dt >= T ? 0 : min(max(eT - ed + (fT > fd ? 1 : 0), 0), KMAX);
    }
    int eT, ed;
    const double fT = frexp(T2, &eT), fd = frexp(d2, &ed);
    const int k2 = eT - ed + (fT > fd ? 1 : 0);
    return min(max((k2 + 1) >> 1, 0), KMAX);
}

// Work split inside a CTA: each member of a group of n is handled by P
// consecutive lanes (P a power of two, P * n <= HTHREADS when possible); lane
// l of a member's group takes the partners lo + l, lo + l + P, ... below hi;
// the group's partial sums are combined with warp shuffles in a fixed tree.
__device__ __forceinline__ int lanes_per_member(int n, int partners) {
    int p = 32;
    while (p > 1 && (p * n > HTHREADS || p >= 2 * partners)) p >>= 1;
    return p;
}

__device__ __forceinline__ void group_sum(double *v, int cnt, int P) {
    #pragma unroll 1
    for (int off = P >> 1; off > 0; off >>= 1)
        for (int c = 0; c < cnt; ++c) v[c] += __shfl_xor_sync(0xffffffffu, v[c], off);
}

// partial (1-K)-weighted pair acceleration of member k at the evaluation
// point, unsmoothed (the kick used the bare separation):
// sum_l -G m_l q_kl / q^3 [1 - K + q K'] over the partners of this lane
__device__ __forceinline__ void kcorr_part(const HermSmem &S, int lo, int hi, int k, int l0, int P,
                           const TransC &tc, double *c) {
    c[0] = c[1] = c[2] = 0.0;
    #pragma unroll 1
    for (int l = lo + l0; l < hi; l += P) {
        if (l == k) continue;
        double qx = S.ex[k] - S.ex[l], qy = S.ey[k] - S.ey[l], qz = S.ez[k] - S.ez[l];
        double q2 = qx * qx + qy * qy + qz * qz;
        if (at_least(q2, tc.rc2)) continue;  // K = 1 beyond r_crit: no (1-K) part
        const double qi = rsqrt(q2);
        const double q = q2 * qi;
        double K, Kp, Kpp;
        transition(q, tc, K, Kp, Kpp);
        double wgt = S.gm[l] * (qi * qi * qi) * (1.0 - K + q * Kp);
        c[0] += wgt * qx;
        c[1] += wgt * qy;
        c[2] += wgt * qz;
    }
}

// the star's pull on member k at the evaluation point, fixed at the origin: a, adot
__device__ __forceinline__ void star_pull(const HermSmem &S, int k, double gm0, double eps2,
                                          double *aj) {
    const double xk = S.ex[k], yk = S.ey[k], zk = S.ez[k];
    const double uk = S.eu[k], vk = S.ev[k], wk = S.ew[k];
    const double s2 = xk * xk + yk * yk + zk * zk + eps2;
    const double si = rsqrt(s2);
    const double si2 = si * si;
    const double rv = xk * uk + yk * vk + zk * wk;
    const double c = gm0 * (si2 * si);
    const double t = 3.0 * rv * si2;
    aj[0] += c * xk; aj[1] += c * yk; aj[2] += c * zk;
    aj[3] += c * (uk - t * xk); aj[4] += c * (vk - t * yk); aj[5] += c * (wk - t * zk);
}

// partial Hermite acceleration and jerk of member k at the evaluation point
// (Sec. 2.2): the star's term on lane 0 of the group, then the pair terms with the
// transition bracket over this lane's partners (one reciprocal square root per
// pair: q = q2 / sqrt(q2), 1/q^3, 1/q^2)
__device__ __forceinline__ void herm_part(const HermSmem &S, int lo, int hi, int k, int l0, int P,
                                          double gm0, const TransC &tc, double eps2, double *aj) {
    const double xk = S.ex[k], yk = S.ey[k], zk = S.ez[k];
    const double uk = S.eu[k], vk = S.ev[k], wk = S.ew[k];
    for (int c = 0; c < 6; ++c) aj[c] = 0.0;
    if (l0 == 0) star_pull(S, k, gm0, eps2, aj);
    #pragma unroll 1
    for (int l = lo + l0; l < hi; l += P) {
        if (l == k) continue;
        double qx = xk - S.ex[l], qy = yk - S.ey[l], qz = zk - S.ez[l];
        double q2 = qx * qx + qy * qy + qz * qz + eps2;
        if (at_least(q2, tc.rc2)) continue;  // K = 1, K' = K'' = 0: no force, no jerk
        double px = uk - S.eu[l], py = vk - S.ev[l], pz = wk - S.ew[l];
        const double qi = rsqrt(q2);
        const double qi2 = qi * qi;
        const double sq = q2 * qi;
        double K, Kp, Kpp;
        transition(sq, tc, K, Kp, Kpp);
        double br = 1.0 - K + sq * Kp;
        double rvl = qx * px + qy * py + qz * pz;
        double cl = S.gm[l] * (qi2 * qi);
        double tl = 3.0 * rvl * qi2;
        aj[0] += cl * br * qx; aj[1] += cl * br * qy; aj[2] += cl * br * qz;
        aj[3] += cl * (rvl * qx * Kpp + (px - tl * qx) * br);
        aj[4] += cl * (rvl * qy * Kpp + (py - tl * qy) * br);
        aj[5] += cl * (rvl * qz * Kpp + (pz - tl * qz) * br);
    }
}

// 2^e as a double, -1022 <= e <= 1023 (from the bits: no FP64 instruction)
__device__ __forceinline__ double pow2d(int e) {
    return __longlong_as_double((long long)(e + 1023) << 52);
}

// v 2^s as a float, the mantissa truncated, by integer operations on the bits
// (no FP64 instruction): signed zero below the float normal range, +-FLT_MAX
// above it. Used only for the step-size criterion.
__device__ __forceinline__ float to_float_scaled(double v, int s) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    const int eb = (int)((b >> 52) & 0x7ff);
    if (eb == 0) return __uint_as_float(sign);
    const int e = eb - 1023 + s;
    if (e < -126) return __uint_as_float(sign);
    if (e > 127) return __uint_as_float(sign | 0x7f7fffffu);
    return __uint_as_float(sign | ((unsigned)(e + 127) << 23) | (unsigned)((b >> 29) & 0x7fffffu));
}

// Step levels by the Aarseth criterion,
// dt_c^2 = eta (|a| |a2| + |j|^2) / (|j| |a3| + |a2|^2), with a, j the new
// acceleration and jerk and a2, a3 the corrector's derivatives: the new level
// is the smallest k with T 2^-k <= dt_c. With g = 2^-lv (lv the level of the
// step just taken), j g, a2 g^2 and a3 g^3 are accelerations scaled alike and
// r = eta (|a||a2 g^2| + |j g|^2) / (|j g||a3 g^3| + |a2 g^2|^2) =
// (dt_c / (T g))^2 T^2, so T 2^-k <= dt_c is T^2 4^(lv - k) <= r. The powers
// of g are applied exactly through the exponents when the inputs are cut to
// FP32, and the criterion runs in FP32 (an FP64 operation costs about fifteen
// FP32 ones here). It only picks a power of two: a level different from an
// FP64 evaluation needs dt_c within ~1e-7 of a level boundary.
// level_from: that level from the criterion's inputs as floats f[c * ACH]
// (stride ACH): a (3), j g (3), a2 g^2 (3), a3 g^3 (3)
// T^2 split for level_from: T2 = ft 2^et, ft in [1/2, 1)
struct T2Split {
    int et;
    float ft;
    __device__ __forceinline__ explicit T2Split(float T2) { ft = frexpf(T2, &et); }
};
__device__ __forceinline__ int level_from(const float *f, int lv, float eta, const T2Split &T2) {
    float q[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const float x = f[(3 * g) * ACH], y = f[(3 * g + 1) * ACH], z = f[(3 * g + 2) * ACH];
        q[g] = sqrtf(fmaf(x, x, fmaf(y, y, z * z)));
    }
    const float num = eta * fmaf(q[0], q[2], q[1] * q[1]);
    const float den = fmaf(q[1], q[3], q[2] * q[2]);
    const float r = num / den;
    // r = fr 2^er with fr in [1/2, 1)
    const int br = __float_as_int(r);
    int er = (br >> 23) - 126;
    float fr = __int_as_float((br & 0x7fffff) | 0x3f000000);
    if (br < 0x00800000) fr = frexpf(r, &er);
    const int dd = er - T2.et;
    const int m = (dd & 1) ? (dd - 1) >> 1 : ((T2.ft <= fr) ? dd >> 1 : (dd >> 1) - 1);
    int k = min(max(lv - m, 0), KMAX);
    if (!(r < INFINITY)) k = 0;
    if (!(num > 0.0f)) k = KMAX;
    return den > 0.0f ? k : 0;
}

// A time in ticks (below 2^52) times a factor f in one FP64 operation: the bits of
// 2^52 + dt are dt's under the exponent, and the product with f less 2^52 f is rounded
// once, as (double)dt * f is. (b = -2^52 f, exact.)
struct TickF {
    double f, b;
    __device__ __forceinline__ explicit TickF(double v) : f(v), b(v * -0x1p52) {}
};
__device__ __forceinline__ double ticks_times(long long dt, const TickF &s) {
    return fma(__longlong_as_double(0x4330000000000000ll | dt), s.f, s.b);
}
// v / 2 from the bits (v / 2 normal), else by the multiplication
__device__ __forceinline__ double half_of(double v) {
    const int hi = __double2hiint(v);
    if ((hi & 0x7fe00000) == 0) return 0.5 * v;
    return __hiloint2double(hi - 0x00100000, __double2loint(v));
}
// Coordinate c of member k predicted from its own time to tn: the position
// x + h (u + h (a/2 + h/6 j)) or the velocity u + h (a + h/2 j)
__device__ __forceinline__ double predict_x(const HermSmem &S, int k, int c, long long tn,
                                            const TickF &stick) {
    const int o = c * HCAP + k;
    const double hs = ticks_times(tn - S.ti[k], stick);
    const double h6 = hs * (1.0 / 6.0);
    return fma(hs, fma(hs, fma(0.5, S.ax[o], __dmul_rn(h6, S.jx[o])), S.u[o]), S.x[o]);
}
__device__ __forceinline__ double predict_v(const HermSmem &S, int k, int c, long long tn,
                                            const TickF &stick) {
    const int o = c * HCAP + k;
    const double hs = ticks_times(tn - S.ti[k], stick);
    return fma(hs, fma(half_of(hs), S.jx[o], S.ax[o]), S.u[o]);
}

// FP32 copies of member k's state (truncated: within 2^-23 of the FP64
// values, relative), kept beside the FP64 state for the FP32 prediction
__device__ __forceinline__ void store_f32(const HermSmem &S, int k) {
    const double *src[12] = {S.x, S.y, S.z, S.u, S.v, S.w, S.ax, S.ay, S.az, S.jx, S.jy, S.jz};
#pragma unroll
    for (int q = 0; q < 12; ++q) S.f[q * HCAP + k] = to_float_scaled(src[q][k], 0);
}

// Member k's position predicted to tn in FP32 from the copies, by the
// Horner form x + h (u + h (a/2 + (h/6) j)), and a bound pd on its distance from the
// FP64 prediction. Each input is within 2^-23 of its FP64 value (hs within
// 3 2^-24), and each of the three fmaf roundings adds 2^-24 relative to the
// magnitude of what it rounds, so every term of the polynomial is within
// 15 2^-24 < 2^-20 of its FP64 value, relative to the sum M of the terms'
// magnitudes; pd = 2^-18 (M_x + M_y + M_z) (plus 1e-30 for inputs flushed
// to zero) keeps a factor 4 to spare.
__device__ __forceinline__ void predict_f32(const HermSmem &S, int k, long long tn, float stickf) {
    const float hs = (float)(tn - S.ti[k]) * stickf;
    const float ah = fabsf(hs);
    const float h6 = hs * (1.0f / 6.0f), ah6 = ah * (1.0f / 6.0f);
    float *out[3] = {S.px, S.py, S.pz};
    float m = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float xk = S.f[c * HCAP + k], uk = S.f[(3 + c) * HCAP + k];
        const float ak = S.f[(6 + c) * HCAP + k], jk = S.f[(9 + c) * HCAP + k];
        out[c][k] = fmaf(hs, fmaf(hs, fmaf(h6, jk, 0.5f * ak), uk), xk);
        m += fmaf(ah, fmaf(ah, fmaf(ah6, fabsf(jk), 0.5f * fabsf(ak)), fabsf(uk)), fabsf(xk));
    }
    S.pd[k] = fmaf(m, 0x1p-18f, 1e-30f);
}

// One item (active slot, coordinate) of the corrector's form f: everything but
// the new acceleration and jerk, read while those are on their way.
struct CorrItem {
    double a2d, a2j0, a2j1, a3d, a3j, f2, f3;  // a2 and a3; the form f2 a2 + f3 a3 + base
    double a, j, base;
    int o, s, lv;  // coordinate and member, coordinate and slot, the member's level
    __device__ __forceinline__ void fetch(const HermSmem &S, int f, const uint16_t *act, int it) {
        constexpr int LS = KMAX + 1;
        const int sl = it / 3, c = it - 3 * sl;
        const int k = act[sl];
        o = c * HCAP + k;
        s = c * ACH + sl;
        lv = S.lev[k];
        const double *L = S.lvt + lv;
        a2d = L[LV_A2D * LS];
        a2j0 = L[LV_A2J0 * LS];
        a2j1 = L[LV_A2J1 * LS];
        a3d = L[LV_A3D * LS];
        a3j = L[LV_A3J * LS];
        f2 = L[(f == LF_X ? LV_H4 : LV_H3) * LS];
        f3 = L[(f == LF_X ? LV_H5 : (f == LF_V ? LV_H4 : LV_H)) * LS];
        a = S.ax[o];
        j = S.jx[o];
        base = f < LF_A2 ? S.ex[3 * f * HCAP + o] : 0.0;
    }
    __device__ __forceinline__ double value(const HermSmem &S, int f) const {
        const double d = a - S.a1s[s], j1 = S.a1s[3 * ACH + s];
        const double a3 = fma(a3d, d, a3j * (j + j1));
        if (f == LF_A3) return a3;
        const double a2 = fma(a2d, d, fma(a2j0, j, a2j1 * j1));
        if (f == LF_A2) return fma(f3, a3, a2);  // at the end of the step
        return fma(f2, a2, fma(f3, a3, base));
    }
};

// false only when members k and l, both predicted in FP32 to the same time,
// are surely farther apart than r_crit in their FP64 predictions: then the
// FP64 pair test (q^2 + eps^2 >= r_crit^2) rejects the pair as well. The
// separation is within 2^-21 (relative) of that of the FP32 positions, which
// differ from the FP64 ones by at most pd_k + pd_l; rcf >= r_crit (1 + 2^-20).
// Written with explicit roundings so that every call gives the same answer.
__device__ __forceinline__ bool maybe_near(const HermSmem &S, int k, int l, float rcf) {
    const float dx = __fsub_rn(S.px[k], S.px[l]);
    const float dy = __fsub_rn(S.py[k], S.py[l]);
    const float dz = __fsub_rn(S.pz[k], S.pz[l]);
    const float q = __fsqrt_rn(__fmaf_rn(dx, dx, __fmaf_rn(dy, dy, __fmul_rn(dz, dz))));
    return __fmul_rn(q, 1.0f - 0x1p-20f) <= __fadd_rn(rcf, __fadd_rn(S.pd[k], S.pd[l]));
}

// Pieces of the pair force shared by the one-lane form (herm_item) and the
// two-warp form of the block step, written with explicit fused operations
// so that both give the same bits: q^2 + eps^2; q . p; cl = -G m_l / q^3;
// br = 1 - K + q K'; the acceleration cl br q and the jerk cl br p + cq q
// with cq = cl (q . p) (K'' - 3 br / q^2)
__device__ __forceinline__ double pair_q2(double qx, double qy, double qz, double eps2) {
    return fma(qx, qx, fma(qy, qy, fma(qz, qz, eps2)));
}
__device__ __forceinline__ double pair_rv(double qx, double qy, double qz, double px, double py,
                                          double pz) {
    return fma(qx, px, fma(qy, py, qz * pz));
}
__device__ __forceinline__ double pair_cl(double gml, double qi, double qi2) {
    return gml * (qi2 * qi);
}
__device__ __forceinline__ double pair_br(double sq, double K, double Kp) {
    return fma(sq, Kp, 1.0 - K);
}
// m3qi2 = -3 / q^2
__device__ __forceinline__ double pair_cq(double cl, double rvl, double m3qi2, double br,
                                          double Kpp) {
    return (cl * rvl) * fma(m3qi2, br, Kpp);
}

// Hermite a, adot of member k from one item: partner mlo + item of this
// CTA's range (with f32, skipped at once when maybe_near rules it out), or
// the star for item == npart (with `star`)
__device__ __forceinline__ void herm_item(const HermSmem &S, int k, int item, int mlo, int npart,
                                          bool star, double gm0, const TransC &tc, double eps2,
                                          bool f32, float rcf, double *aj) {
    if (item < npart && (mlo + item == k || (f32 && !maybe_near(S, k, mlo + item, rcf)))) return;
    if (item == npart) {
        if (star) star_pull(S, k, gm0, eps2, aj);
        return;
    }
    const double xk = S.ex[k], yk = S.ey[k], zk = S.ez[k];
    const double uk = S.eu[k], vk = S.ev[k], wk = S.ew[k];
    const int l = mlo + item;
    const double qx = xk - S.ex[l], qy = yk - S.ey[l], qz = zk - S.ez[l];
    const double q2 = pair_q2(qx, qy, qz, eps2);
    if (at_least(q2, tc.rc2)) return;  // K = 1, K' = K'' = 0: no force, no jerk
    const double px = uk - S.eu[l], py = vk - S.ev[l], pz = wk - S.ew[l];
    const double qi = rsqrt(q2);
    const double qi2 = qi * qi;
    const double sq = q2 * qi;
    double K, Kp, Kpp;
    transition(sq, tc, K, Kp, Kpp);
    const double rvl = pair_rv(qx, qy, qz, px, py, pz);
    const double cl = pair_cl(S.gm[l], qi, qi2), br = pair_br(sq, K, Kp);
    const double cb = cl * br;
    const double cq = pair_cq(cl, rvl, -3.0 * qi2, br, Kpp);
    aj[0] = fma(cb, qx, aj[0]); aj[1] = fma(cb, qy, aj[1]); aj[2] = fma(cb, qz, aj[2]);
    aj[3] = fma(cb, px, fma(cq, qx, aj[3]));
    aj[4] = fma(cb, py, fma(cq, qy, aj[4]));
    aj[5] = fma(cb, pz, fma(cq, qz, aj[5]));
}

// the pair barrier of warps 2p and 2p + 1 (named barrier 1 + p, 64 threads)
__device__ __forceinline__ void pair_bar(int p) {
    asm volatile("bar.sync %0, 64;" ::"r"(1 + p) : "memory");
}

// A cluster's exchange of force sums: every CTA stores its sums into the others'
// receive buffers by st.async, which counts the bytes on the receiver's mbarrier
// (g_rbar, one per receive buffer; a phase ends when the bytes of all CTAs' sums,
// announced by one thread, are there). A cluster barrier instead waits for the
// stores' round trip and then for the barrier's own.
__shared__ __align__(8) unsigned long long g_rbar[2];
__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void rbar_init() {
    for (int b = 0; b < 2; ++b)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&g_rbar[b])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void rbar_expect(int b, int bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&g_rbar[b])),
                 "r"(bytes)
                 : "memory");
}
// v into CTA r's copy of *p, counted on its g_rbar[b]
__device__ __forceinline__ void rbar_send(double *p, double v, int r, int b) {
    unsigned pa, ba;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(pa) : "r"(smem_addr(p)), "r"(r));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ba) : "r"(smem_addr(&g_rbar[b])), "r"(r));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(pa),
                 "l"(__double_as_longlong(v)), "r"(ba)
                 : "memory");
}
// waits for the phase of the given parity; false when it does not end in a second or so
__device__ __forceinline__ bool rbar_wait(int b, int parity) {
    #pragma unroll 1
    for (int i = 0; i < (1 << 20); ++i) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(smem_addr(&g_rbar[b])), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

struct HermArgs {
    double G, eps2, eta, eta_s, tau;
    int64_t max_steps;
};

__shared__ int g_next_small;
__shared__ long long g_tn;
__shared__ int g_na;
__shared__ int g_nneed;  // members of the FP32-screened list

// The earliest end of a member's step later than `after`, and the members whose step
// ends then, listed in member order in act, by one warp (LLONG_MAX and none when no
// step ends later). The minimum (below 2^49) is taken as the minimum of the high words,
// then of the low words among the lanes that hold it.
struct Block {
    long long t;
    int na;
};
__device__ __forceinline__ long long step_end(const int32_t *lev, const long long *ti, int k,
                                              int n, long long after) {
    const long long te = k < n ? ti[k] + (1ll << (KMAX - lev[k])) : LLONG_MAX;
    return te > after ? te : LLONG_MAX;
}
__device__ __forceinline__ Block next_block(const int32_t *lev, const long long *ti,
                                            uint16_t *act, int n, long long after) {
    const int wl = threadIdx.x & 31;
    const long long t0 = step_end(lev, ti, wl, n, after);
    long long t = t0;
#pragma unroll 1
    for (int k = 32 + wl; k - wl < n; k += 32) t = min(t, step_end(lev, ti, k, n, after));
    const unsigned hi = __reduce_min_sync(0xffffffffu, (unsigned)(t >> 32));
    const unsigned lo =
        __reduce_min_sync(0xffffffffu, (unsigned)(t >> 32) == hi ? (unsigned)t : 0xffffffffu);
    Block b;
    b.t = (long long)(((unsigned long long)hi << 32) | lo);
    b.na = 0;
    if (b.t == LLONG_MAX) return b;
    t = t0;
#pragma unroll 1
    for (int k = wl;;) {
        const unsigned m = __ballot_sync(0xffffffffu, t == b.t);
        if (t == b.t) act[b.na + __popc(m & ((1u << wl) - 1u))] = (uint16_t)k;
        b.na += __popc(m);
        k += 32;
        if (k - wl >= n) return b;
        t = step_end(lev, ti, k, n, after);
    }
}

// Copy the member range [lo, hi) of arrays a..: from CTA `r` of the cluster
// into this CTA's shared memory.
__device__ __forceinline__ void pull_range(cg::cluster_group &cl, const HermSmem &S, int r,
                                           int lo, int hi, double *const *arrs, int narr) {
    #pragma unroll 1
    for (int q = 0; q < narr; ++q) {
        const double *src = cl.map_shared_rank(arrs[q], r);
        #pragma unroll 1
        for (int k = lo + threadIdx.x; k < hi; k += blockDim.x) arrs[q][k] = src[k];
    }
}

// One set through items 5-7 of the step (Sec. 2.3): K correction at q0,
// Hermite over tau with individual block steps, K correction at q1. With
// COOP the cs CTAs of a cluster share the set: every CTA keeps a full copy of
// the members' state; CTA `rank` evaluates the start-up forces and the K
// corrections of its member range, exchanged once; in each block step it sums
// the forces on the active members from its partner range, sends its sums
// to every CTA's receive buffer, adds all CTAs' sums in rank order and applies
// the same corrector, so the copies stay identical.
template <bool COOP, int CLT>
__device__ __noinline__ void hermite_set(const Dev &d, const HermArgs h, int set, int rank,
                                         int cs) {
    const HermSmem S = carve(g_hsmem);
    cg::cluster_group cl = cg::this_cluster();
    const int64_t R = d.rows;
    const int tid = threadIdx.x;
    const int st = d.set_start[set];
    const int n = d.set_start[set + 1] - st;
    if (n < 1) return;
    if (n > HCAP || st + n > d.max_members) {
        if (tid == 0 && rank == 0) atomicOr(d.status, QYM_ST_SET_OVERFLOW);
        if (rank == 0)
            #pragma unroll 1
            for (int k = tid; k < n && st + k < d.max_members; k += blockDim.x)
                d.uf[d.set_mem[st + k]] = -1;
        return;
    }
    // a system integrated whole by the Hermite this step (whole.cu): its
    // members only leave the union-find
    if (d.wh_flag && d.wh_flag[d.sys_of[d.set_mem[st]]]) {
        if (rank == 0)
            #pragma unroll 1
            for (int k = tid; k < n; k += blockDim.x) d.uf[d.set_mem[st + k]] = -1;
        return;
    }
    // (the first cluster barrier below comes before the first exchange; a cluster
    // integrates one set)
    if (COOP && tid == 0) rbar_init();
    // this CTA's member range (COOP) or all members
    const int mlo = n * rank / cs, mhi = n * (rank + 1) / cs;
    const int P = lanes_per_member(mhi - mlo, n);
    const int NG = HTHREADS / P;
    const int grp = tid / P, lane = tid % P;
    const int64_t star_row = d.offsets[d.sys_of[d.set_mem[st]]];
    const double gm0 = -h.G * d.m[star_row], rcrit = d.rcrit[set];
    const TransC tc(rcrit);
    // members in ascending row order (rank sort)
    __syncthreads();
    #pragma unroll 1
    for (int k = tid; k < n; k += blockDim.x) S.ids[k] = d.set_mem[st + k];
    __syncthreads();
    int myid[HCAP / HTHREADS], myrank[HCAP / HTHREADS];
    for (int c = 0; c < HCAP / HTHREADS; ++c) {
        int k = tid + c * blockDim.x;
        myid[c] = k < n ? S.ids[k] : 0;
        int rk = 0;
        if (k < n)
            #pragma unroll 4
            for (int l = 0; l < n; ++l) rk += S.ids[l] < myid[c];
        myrank[c] = rk;
    }
    __syncthreads();
    for (int c = 0; c < HCAP / HTHREADS; ++c) {
        int k = tid + c * blockDim.x;
        if (k < n) S.ids[myrank[c]] = myid[c];
    }
    __syncthreads();
    const double tau = h.tau;
    // state entering the Kepler drift (after the first kick)
    #pragma unroll 1
    for (int k = tid; k < n; k += blockDim.x) {
        int64_t r = S.ids[k];
        S.ex[k] = S.x[k] = d.q[r];
        S.ey[k] = S.y[k] = d.q[R + r];
        S.ez[k] = S.z[k] = d.q[2 * R + r];
        S.u[k] = d.v[r];
        S.v[k] = d.v[R + r];
        S.w[k] = d.v[2 * R + r];
        S.gm[k] = -h.G * d.m[r];
    }
    __syncthreads();
    // item 5: remove the (1-K) part of the first kick (own members)
    #pragma unroll 1
    for (int k0 = mlo; k0 < mhi; k0 += NG) {
        int k = k0 + grp;
        double c[3] = {0.0, 0.0, 0.0};
        if (k < mhi) kcorr_part(S, 0, n, k, lane, P, tc, c);
        group_sum(c, 3, P);
        if (k < mhi && lane == 0) {
            S.u[k] -= 0.5 * tau * c[0];
            S.v[k] -= 0.5 * tau * c[1];
            S.w[k] -= 0.5 * tau * c[2];
        }
    }
    if (COOP) {
        cl.sync();
        double *const arr[3] = {S.u, S.v, S.w};
        #pragma unroll 1
        for (int r = 0; r < cs; ++r)
            if (r != rank) pull_range(cl, S, r, n * r / cs, n * (r + 1) / cs, arr, 3);
        cl.sync();
    } else {
        __syncthreads();
    }
    #pragma unroll 1
    for (int k = tid; k < n; k += blockDim.x) {
        S.eu[k] = S.u[k]; S.ev[k] = S.v[k]; S.ew[k] = S.w[k];
    }
    __syncthreads();
    // start-up: a, adot at t = 0 and the levels from eta_s |a| / |adot|
    const double sgn = tau >= 0.0 ? 1.0 : -1.0;
    const double T = fabs(tau);
    const long long TT = 1ll << KMAX;
    const double tick = T / (double)TT;
    const double T2d = T * T;
    // (warp 7 first sets up the corrector's constants per level, products with powers
    // of two: scalars that every warp computes take the sub-partitions' FP64 units
    // eight times)
    const int warp = tid >> 5, wl = tid & 31;
    if (warp == 7) {
        const double inv_T = 1.0 / T, iT2 = inv_T * inv_T, iT3 = iT2 * inv_T;
        const double T3 = T2d * T, T4 = T3 * T;
#pragma unroll 1
        for (int lv = wl; lv <= KMAX; lv += 32) {
            constexpr int LS = KMAX + 1;
            double *L = S.lvt + lv;
            const double ih = sgn * inv_T * pow2d(lv), ih2 = iT2 * pow2d(2 * lv);
            L[LV_H * LS] = sgn * T * pow2d(-lv);
            L[LV_A2D * LS] = -6.0 * ih2;
            L[LV_A2J0 * LS] = -4.0 * ih;
            L[LV_A2J1 * LS] = -2.0 * ih;
            L[LV_A3D * LS] = 12.0 * (sgn * iT3 * pow2d(3 * lv));
            L[LV_A3J * LS] = 6.0 * ih2;
            L[LV_H4 * LS] = (T4 * pow2d(-4 * lv)) * (1.0 / 24.0);
            L[LV_H5 * LS] = (sgn * T4 * T * pow2d(-5 * lv)) * (1.0 / 120.0);
            L[LV_H3 * LS] = (sgn * T3 * pow2d(-3 * lv)) * (1.0 / 6.0);
        }
    }
#pragma unroll 1
    for (int k0 = mlo; k0 < mhi; k0 += NG) {
        const int k = k0 + grp;
        double aj[6] = {0, 0, 0, 0, 0, 0};
        if (k < mhi) herm_part(S, 0, n, k, lane, P, gm0, tc, h.eps2, aj);
        group_sum(aj, 6, P);
        if (k < mhi && lane == 0) {
            S.ax[k] = aj[0]; S.ay[k] = aj[1]; S.az[k] = aj[2];
            S.jx[k] = aj[3]; S.jy[k] = aj[4]; S.jz[k] = aj[5];
            S.lev[k] = first_level(aj, h.eta_s, T2d, T);
            S.ti[k] = 0;
        }
    }
    if (COOP) {
        cl.sync();
        double *const arr[6] = {S.ax, S.ay, S.az, S.jx, S.jy, S.jz};
        #pragma unroll 1
        for (int r = 0; r < cs; ++r) {
            if (r == rank) continue;
            const int lo = n * r / cs, hi = n * (r + 1) / cs;
            pull_range(cl, S, r, lo, hi, arr, 6);
            const int32_t *pl = cl.map_shared_rank(S.lev, r);
            #pragma unroll 1
            for (int k = lo + tid; k < hi; k += blockDim.x) {
                S.lev[k] = pl[k];
                S.ti[k] = 0;
            }
        }
        cl.sync();
    }
    // Block steps. FP64 instructions are issued at about one warp-instruction
    // per 64 cycles per SM sub-partition here, whatever the number of active
    // lanes, so the work is split by instruction stream across warps (which
    // the sub-partitions serve in parallel): items (member, coordinate) of
    // the predictor and of each of the corrector's forms on warps of their own,
    // several warps per pair for the forces, lane groups for the sums.
    const double stick = sgn * tick;
    const T2Split T2s((float)T2d);
    const float etaf = (float)h.eta;
    const float stickf = (float)stick;
    const TickF tick1(stick);
    const float rcf = __double2float_ru(rcrit * (1.0 + 0x1p-20));
    const int npart = mhi - mlo;
    // the largest range of the cluster: every CTA derives its lane layout and
    // its round count from it, so all CTAs pass the same cluster barriers and
    // lay out their partial sums alike
    const int npmax = (n + cs - 1) / cs;
    // lanes per active member of the pair forces, LA = 2^las, and the members of a
    // round in either form (constants of the set: a division in every block step is
    // latency on its only chain)
    int las = 0;
    while ((1 << las) < npmax && las < 6) ++las;
    const int LA = 1 << las;
    const int NU = min(COOP ? RSL : 32, (HTHREADS - 32) >> las);
    const int NP = min(COOP ? RSL : 32, 96 >> las);
    const int N3 = min(COOP ? RSL : 32, 32 >> las);
    // FP32 copies of the start-up state
    __syncthreads();
    #pragma unroll 1
    for (int k = tid; k < n; k += blockDim.x) store_f32(S, k);
    const bool with_star = rank == 0;
    int64_t steps = 0;
    bool capped = false, lost = false;
    int buf = 0, par = 0;  // receive buffer and its barrier's parity
    // The first block time. Later ones are found by warp 6, which writes every level
    // and time: over the members that do not move now while the other warps evaluate
    // the forces, and over those that do right after it sets their levels; one barrier
    // per block step publishes them. (One scan of all members after the levels took
    // 550 of a block step's 10000 cycles.)
    if (warp == 6) {
        const Block b = next_block(S.lev, S.ti, S.act, n, -1);
        if (wl == 0) {
            g_tn = b.t;
            g_na = b.na;
        }
    }
    // chunk of 32 prediction items this warp takes first: positions (even) and
    // velocities (odd) on all four sub-partitions
    const int pq0 = warp ^ (warp >> 2);
    for (;;) {
        __syncthreads();
        const long long tn = g_tn;
        if (tn > TT) break;  // every member has reached tau
        if (steps >= h.max_steps) { capped = true; break; }
        const int na = g_na;
        const uint16_t *act = S.act + (steps & 1) * HCAP;
        // Predict this CTA's partners and the active members to tn: items
        // (member, coordinate), 32 to a warp, positions and velocities in chunks of
        // their own, so that a few members cost one warp's five FP64 instructions
        // instead of eleven on each of three warps. Up to F32MIN members FP64 passes
        // over them all; above that the FP32 prediction first rules out the partners
        // that are surely beyond r_crit of every active member.
        //
        // One CTA's set whose moving members' partners would not fit one warp
        // (na > N3) first lists the pairs that maybe_near leaves, by member and
        // partner: few of a set's pairs lie within r_crit, and an FP64 instruction
        // costs the same for one lane as for 32. Up to 96 pairs the block step then
        // predicts and evaluates the list alone, packed into lanes (sparse). One system's
        // sets only: a member's pulls are then added in another order, and a batch's
        // sums keep theirs.
        int32_t *plist = S.need + 640, *poff = S.need + 736, *pcnt = S.need + 800;
        bool sparse = false;
        int npair = 0;
        if (!COOP && d.nsys == 1 && na > N3 && na <= 32) {
#pragma unroll 1
            for (int k = tid; k < n; k += HTHREADS) predict_f32(S, k, tn, stickf);
            __syncthreads();
#pragma unroll 1
            for (int ia = warp; ia < na; ia += HTHREADS / 32) {
                const int k = act[ia];
                int m = 0;
#pragma unroll 1
                for (int l = wl; l - wl < n; l += 32)
                    m += __popc(__ballot_sync(0xffffffffu,
                                              l < n && l != k && maybe_near(S, k, l, rcf)));
                if (wl == 0) pcnt[ia] = m;
            }
            __syncthreads();
            int to = wl < na ? pcnt[wl] : 0;  // end of member wl's pairs
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, to, o);
                if (wl >= o) to += v;
            }
            npair = __shfl_sync(0xffffffffu, to, 31);
            sparse = npair <= 96;
            if (sparse) {
                if (warp == 0) poff[wl] = to;
#pragma unroll 1
                for (int ia = warp; ia < na; ia += HTHREADS / 32) {
                    const int k = act[ia];
                    int m = __shfl_sync(0xffffffffu, to, (ia + 31) & 31);
                    if (ia == 0) m = 0;
#pragma unroll 1
                    for (int l = wl; l - wl < n; l += 32) {
                        const bool f = l < n && l != k && maybe_near(S, k, l, rcf);
                        const unsigned b = __ballot_sync(0xffffffffu, f);
                        if (f) plist[m + __popc(b & ((1u << wl) - 1u))] = (ia << 16) | l;
                        m += __popc(b);
                    }
                }
            }
            __syncthreads();
        }
        const bool f32 = npmax + na > F32MIN && !sparse;
        const int32_t *list = nullptr;
        int np = sparse ? na + npair : npart + na;
        if (f32) {
            #pragma unroll 1
            for (int k = tid; k < n; k += HTHREADS) S.need[k] = 0;
            #pragma unroll 1
            for (int i = tid; i < npart + na; i += HTHREADS) {
                int k = mlo + i;
                if (i >= npart) {
                    k = act[i - npart];
                    if (k >= mlo && k < mhi) continue;
                }
                predict_f32(S, k, tn, stickf);
            }
            __syncthreads();
            // members needed in FP64: the active ones and the partners that
            // maybe_near does not rule out for some active member
            #pragma unroll 1
            for (int i = tid; i < na; i += HTHREADS) S.need[act[i]] = 1;
            #pragma unroll 1
            for (int p = tid; p < na * npart; p += HTHREADS) {
                const int ia = p / npart, l = mlo + (p - ia * npart);
                const int k = act[ia];
                if (l != k && maybe_near(S, k, l, rcf)) S.need[l] = 1;
            }
            __syncthreads();
            // listed in member order by one warp
            if (warp == 0) {
                int nn = 0;
                #pragma unroll 1
                for (int k0 = 0; k0 < n; k0 += 32) {
                    const int k = k0 + wl;
                    const bool f = k < n && S.need[k] != 0;
                    const unsigned b = __ballot_sync(0xffffffffu, f);
                    if (f) S.nl[nn + __popc(b & ((1u << wl) - 1u))] = k;
                    nn += __popc(b);
                }
                if (wl == 0) g_nneed = nn;
            }
            __syncthreads();
            list = S.nl;
            np = g_nneed;
        }
        #pragma unroll 1
        for (int pq = pq0; (pq >> 1) * 32 < 3 * np; pq += HTHREADS / 32) {
            const int it = (pq >> 1) * 32 + wl, i = it / 3, c = it - 3 * i;
            if (i >= np) continue;
            int k;
            double *to = S.ex + c * HCAP;
            if (f32) {
                k = list[i];
                to += k;
            } else if (sparse && i >= na) {
                // a listed partner, into the list's own copy ([6][96], in place of
                // the cluster's receive buffers)
                k = plist[i - na] & 0xffff;
                to = S.rb + c * 96 + (i - na);
            } else if (sparse) {
                k = act[i];
                to += k;
            } else {
                k = mlo + i;
                if (i >= npart) {
                    k = act[i - npart];
                    if (k >= mlo && k < mhi) continue;
                }
                to += k;
            }
            if (pq & 1)
                to[sparse && i >= na ? 3 * 96 : 3 * HCAP] = predict_v(S, k, c, tn, tick1);
            else
                to[0] = predict_x(S, k, c, tn, tick1);
        }
        __syncthreads();
        uint16_t *nact = S.act + (~steps & 1) * HCAP;
        Block nb;       // (warp 6)
        int lmax = -1;  // (warp 6) the deepest new level, and
        int mk = 0;     // the lane's member when at most 32 move
        if (warp == 6) nb = next_block(S.lev, S.ti, nact, n, tn);
        #pragma unroll 1
        for (int a0 = 0; a0 < na; a0 += ACH) {
            const int nc = min(ACH, na - a0);
            // pair items on warps 0-6 (LA lanes per member), the star's pull
            // (rank 0) on warp 7, so neither path diverges inside a warp
            // slots per round (warp 7 holds one star per slot; on a cluster at
            // most RSL, the receive buffer's width). When the round's members
            // fit three warps' worth of lanes, each pair item runs on two warps
            // of different sub-partitions (pair_bar): the even warp takes sin,
            // q . p and the acceleration, the odd warp cos and the jerk, which
            // shortens each warp's FP64 instruction stream by about a third.
            // When they fit one warp's worth (most block steps: one or two members
            // move), a pair item runs on three warps: sin, cos, and everything that
            // needs neither, then one coordinate each; its longest instruction stream
            // is 38 FP64 instructions against the pair's 51, with the star's pull on
            // the fourth sub-partition.
            const bool paired = sparse || nc <= NP;
            const int NR = paired ? nc : NU;
            CorrItem item;  // (warps 0-3)
            #pragma unroll 1
            for (int s0 = 0; s0 < nc; s0 += NR) {
                const int cnt = min(NR, nc - s0);
                double *prb = S.pr;
                if (!paired) {
                    double aj[6] = {0, 0, 0, 0, 0, 0};
                    if (warp < 7) {
                        const int slot = s0 + (tid >> las), la = tid & (LA - 1);
                        if (slot < s0 + cnt) {
                            const int k = act[a0 + slot];
                            #pragma unroll 1
                            for (int it = la; it < npart; it += LA)
                                herm_item(S, k, it, mlo, npart, false, gm0, tc, h.eps2, f32, rcf, aj);
                        }
                    } else if (with_star && wl < cnt) {
                        herm_item(S, act[a0 + s0 + wl], npart, mlo, npart, true, gm0, tc, h.eps2,
                                  f32, rcf, aj);
                    }
#pragma unroll
                    for (int c = 0; c < 6; ++c) prb[c * HTHREADS + tid] = aj[c];
                } else if (sparse ? npair <= 32 : nc <= N3) {
                    if (warp < 3) {
                        // (LA >= npart: one partner per lane)
                        const int role = warp;
                        int slot = wl >> las, l = mlo + (wl & (LA - 1));
                        bool valid = slot < cnt && l < mhi;
                        const double *pe = S.ex + l;  // the partner's x, y, z, u, v, w
                        int pst = HCAP;
                        if (sparse) {
                            valid = wl < npair;
                            const int e = valid ? plist[wl] : 0;
                            slot = e >> 16;
                            l = e & 0xffff;
                            pe = S.rb + wl;
                            pst = 96;
                        }
                        const int k = valid ? act[a0 + slot] : 0;
                        valid = valid && l != k && (!f32 || maybe_near(S, k, l, rcf));
                        // exchange slots [8][32] in place of the idle FP32 lists
                        double *xs = reinterpret_cast<double *>(S.need) + wl;
                        double qr = 0.0, sq = 0.0;
                        bool fold = false;
                        if (valid) {
                            const double qx = S.ex[k] - pe[0];
                            const double qy = S.ey[k] - pe[pst];
                            const double qz = S.ez[k] - pe[2 * pst];
                            const double q2 = pair_q2(qx, qy, qz, h.eps2);
                            valid = !at_least(q2, tc.rc2);  // beyond r_crit: no force, no jerk
                            if (valid) {
                                qr = role == 0 ? qx : (role == 1 ? qy : qz);
                                const double qi = rsqrt(q2);
                                sq = q2 * qi;
                                const double y = trans_y(sq, tc);
                                const bool zero = y_at_most_0(y), one = y_at_least_1(y);
                                fold = !zero && !one && y_above_half(y);
                                if (role < 2) {
                                    // K = 0 (sin 0, cos taken as 0) and 1 outside (0, 1)
                                    double p = one && role == 0 ? 1.0 : 0.0;
                                    if (!zero && !one) {
                                        const HalfPi arg = half_pi_arg(y);
                                        p = role == 0 ? sin_w(arg) : cos_w(arg);
                                    }
                                    xs[32 * role] = p;
                                } else {
                                    const double qi2 = qi * qi;
                                    const double px = S.eu[k] - pe[3 * pst];
                                    const double py = S.ev[k] - pe[4 * pst];
                                    const double pz = S.ew[k] - pe[5 * pst];
                                    const double cl = pair_cl(S.gm[l], qi, qi2);
                                    xs[32 * 2] = cl;
                                    xs[32 * 3] = cl * pair_rv(qx, qy, qz, px, py, pz);
                                    xs[32 * 4] = -3.0 * qi2;
                                    xs[32 * 5] = px;
                                    xs[32 * 6] = py;
                                    xs[32 * 7] = pz;
                                }
                            }
                        }
                        __syncwarp();
                        asm volatile("bar.sync 4, 96;" ::: "memory");
                        double ar = 0.0, jr = 0.0;
                        if (valid) {
                            const double sw = xs[0], pc = xs[32];
                            const double sn = fold ? pc : sw, cs = fold ? sw : pc;
                            const double br = pair_br(sq, sn, tc.c * cs);
                            const double cl = xs[32 * 2];
                            const double cq = xs[32 * 3] * fma(xs[32 * 4], br, tc.nc2 * sn);
                            const double cb = cl * br;
                            ar = cb * qr;
                            jr = fma(cb, xs[32 * (5 + role)], cq * qr);
                        }
                        prb[role * HTHREADS + wl] = ar;
                        prb[(3 + role) * HTHREADS + wl] = jr;
                    } else if (warp == 7) {
                        double aj[6] = {0, 0, 0, 0, 0, 0};
                        if (with_star && wl < cnt)
                            herm_item(S, act[a0 + s0 + wl], npart, mlo, npart, true, gm0, tc,
                                      h.eps2, f32, rcf, aj);
#pragma unroll
                        for (int c = 0; c < 6; ++c) prb[c * HTHREADS + tid] = aj[c];
                    }
                } else if (warp < 6) {
                    const int role = warp & 1, vl = (warp >> 1) * 32 + wl;
                    int slot = vl >> las;
                    const int la = vl & (LA - 1);
                    const int e = sparse && vl < npair ? plist[vl] : 0;
                    if (sparse) slot = e >> 16;
                    const bool sv = sparse ? vl < npair : slot < cnt;
                    const int k = sv ? act[a0 + slot] : 0;
                    // exchange slots [2][3][96] (sin, q . p, cos): the FP32
                    // pass's lists, which are idle until the next block time
                    double *xch = reinterpret_cast<double *>(S.need);
                    double acc[3] = {0.0, 0.0, 0.0};
                    int par = 0;
                    #pragma unroll 1
                    for (int it0 = 0; it0 < (sparse ? 1 : npart); it0 += LA) {
                        const int l = sparse ? e & 0xffff : mlo + it0 + la;
                        const double *pe = sparse ? S.rb + vl : S.ex + l;
                        const int pst = sparse ? 96 : HCAP;
                        double *xs = xch + par * (3 * 96);
                        bool valid = sv && (sparse || it0 + la < npart) && l != k &&
                                     (!f32 || maybe_near(S, k, l, rcf));
                        double qx = 0.0, qy = 0.0, qz = 0.0, qi2 = 0.0, sq = 0.0;
                        double y = 0.0, mine = 0.0, cl = 0.0, m3 = 0.0, px = 0.0, py = 0.0, pz = 0.0;
                        bool fold = false;
                        if (valid) {
                            qx = S.ex[k] - pe[0];
                            qy = S.ey[k] - pe[pst];
                            qz = S.ez[k] - pe[2 * pst];
                            const double q2 = pair_q2(qx, qy, qz, h.eps2);
                            valid = !at_least(q2, tc.rc2);  // beyond r_crit: no force, no jerk
                            if (valid) {
                                const double qi = rsqrt(q2);
                                qi2 = qi * qi;
                                sq = q2 * qi;
                                y = trans_y(sq, tc);
                                if (!y_at_most_0(y) && !y_at_least_1(y)) {
                                    const HalfPi arg = half_pi_arg(y);
                                    fold = arg.fold;
                                    mine = role == 0 ? sin_w(arg) : cos_w(arg);
                                    xs[2 * 96 * role + vl] = mine;
                                }
                                // what does not wait for the partner warp's
                                // polynomial is done before the barrier
                                cl = pair_cl(S.gm[l], qi, qi2);
                                px = S.eu[k] - pe[3 * pst];
                                py = S.ev[k] - pe[4 * pst];
                                pz = S.ew[k] - pe[5 * pst];
                                if (role == 0)
                                    xs[96 + vl] = pair_rv(qx, qy, qz, px, py, pz);
                                else
                                    m3 = -3.0 * qi2;
                            }
                        }
                        __syncwarp();
                        pair_bar(warp >> 1);
                        if (valid) {
                            double K = 0.0, Kp = 0.0, Kpp = 0.0;
                            if (y_at_least_1(y)) {
                                K = 1.0;
                            } else if (!y_at_most_0(y)) {
                                const double sw = role == 0 ? mine : xs[vl];
                                const double pc = role == 1 ? mine : xs[2 * 96 + vl];
                                const double sn = fold ? pc : sw, cs = fold ? sw : pc;
                                K = sn;
                                Kp = tc.c * cs;
                                Kpp = tc.nc2 * sn;
                            }
                            const double br = pair_br(sq, K, Kp);
                            const double cb = cl * br;
                            if (role == 0) {
                                acc[0] = fma(cb, qx, acc[0]);
                                acc[1] = fma(cb, qy, acc[1]);
                                acc[2] = fma(cb, qz, acc[2]);
                            } else {
                                const double cq = pair_cq(cl, xs[96 + vl], m3, br, Kpp);
                                acc[0] = fma(cb, px, fma(cq, qx, acc[0]));
                                acc[1] = fma(cb, py, fma(cq, qy, acc[1]));
                                acc[2] = fma(cb, pz, fma(cq, qz, acc[2]));
                            }
                        }
                        par ^= 1;
                    }
#pragma unroll
                    for (int c = 0; c < 3; ++c) prb[(3 * role + c) * HTHREADS + vl] = acc[c];
                } else if (warp == 7) {
                    double aj[6] = {0, 0, 0, 0, 0, 0};
                    if (with_star && wl < cnt)
                        herm_item(S, act[a0 + s0 + wl], npart, mlo, npart, true, gm0, tc, h.eps2,
                                  f32, rcf, aj);
#pragma unroll
                    for (int c = 0; c < 6; ++c) prb[c * HTHREADS + tid] = aj[c];
                }
                if (COOP) {
                    // This CTA's part of every (member, component): its LA lanes
                    // summed by a group of eight lanes in a fixed order (plus the
                    // star's pull on rank 0), sent by lane g into CTA g's
                    // receive buffer under this rank; when all CTAs' parts are
                    // there every CTA adds them in rank order. Receive buffers
                    // are double-buffered: a CTA sends into this one again only
                    // when it has the next round's parts of every CTA, which
                    // that CTA sends after it has read this one (and announced
                    // this round's bytes).
                    __syncthreads();
                    if (tid == HTHREADS - 1) rbar_expect(buf, CLT * 6 * cnt * (int)sizeof(double));
                    double *rbb = S.rb + buf * (CLT * 6 * RSL);
                    const int g = wl & 7;
                    #pragma unroll 1
                    for (int pi0 = warp * 4; pi0 < 6 * cnt; pi0 += HTHREADS / 8) {
                        const int pi = pi0 + (wl >> 3);
                        const bool live = pi < 6 * cnt;
                        const int sl = pi / 6, c = pi - 6 * sl;
                        const double *col = prb + c * HTHREADS + (sl << las);
                        double v = live && g < LA ? col[g] : 0.0;
                        if (live)
                            #pragma unroll 1
                            for (int m = g + 8; m < LA; m += 8) v += col[m];
                        v += __shfl_xor_sync(0xffffffffu, v, 1);
                        v += __shfl_xor_sync(0xffffffffu, v, 2);
                        v += __shfl_xor_sync(0xffffffffu, v, 4);
                        if (live && with_star) v += prb[c * HTHREADS + 224 + sl];
                        if (live && g < CLT) rbar_send(rbb + (rank * 6 + c) * RSL + sl, v, g, buf);
                    }
                    if (warp < 4 && wl < 3 * nc) item.fetch(S, warp, act + a0, wl);
                    if (!rbar_wait(buf, par)) lost = true;
                    // pairwise tree over CLT lanes: rank r with rank r + w, halving w
                    #pragma unroll 1
                    for (int t0 = warp * 32; t0 < 6 * cnt * CLT; t0 += HTHREADS) {
                        const int t = t0 + wl, pi = t / CLT, r = t % CLT;
                        const int sl = pi / 6, c = pi - 6 * sl;
                        double v = pi < 6 * cnt ? rbb[(r * 6 + c) * RSL + sl] : 0.0;
#pragma unroll
                        for (int w = CLT / 2; w >= 1; w >>= 1) v += __shfl_xor_sync(0xffffffffu, v, w);
                        if (pi < 6 * cnt && r == 0) S.a1s[c * ACH + s0 + sl] = v;
                    }
                    par ^= buf;
                    buf ^= 1;
                } else {
                    if (warp < 4 && wl < 3 * nc) item.fetch(S, warp, act + a0, wl);
                    __syncthreads();
                    // sparse: each (member, component) on one thread, the star's pull
                    // and its pairs in order
                    if (sparse && tid < 6 * cnt) {
                        const int sl = tid / 6, c = tid - 6 * sl;
                        double v = prb[c * HTHREADS + 224 + sl];
#pragma unroll 1
                        for (int m = sl ? poff[sl - 1] : 0; m < poff[sl]; ++m)
                            v += prb[c * HTHREADS + m];
                        S.a1s[c * ACH + sl] = v;
                    }
                    // sums over the LA lanes of each (member, component), one
                    // warp each, in a fixed order
                    #pragma unroll 1
                    for (int pi = sparse ? 6 * cnt : warp; pi < 6 * cnt; pi += HTHREADS / 32) {
                        const int sl = pi / 6, c = pi - 6 * sl;
                        const double *col = prb + c * HTHREADS + (sl << las);
                        double v = wl < LA ? col[wl] : 0.0;
                        #pragma unroll 1
                        for (int m = wl + 32; m < LA; m += 32) v += col[m];
                        #pragma unroll 1
                        for (int off = (LA < 32 ? LA : 32) >> 1; off > 0; off >>= 1)
                            v += __shfl_xor_sync(0xffffffffu, v, off);
                        if (wl == 0) S.a1s[c * ACH + s0 + sl] = v + prb[c * HTHREADS + 224 + sl];
                    }
                }
                __syncthreads();
            }
            // Corrector and step criterion (the same in every CTA): items (member,
            // coordinate), 32 to a warp, and each of the four forms on a warp of
            // its own sub-partition, which forms a2 and a3 for itself (four to nine FP64
            // instructions deep); warps 4 and 5 bring the new acceleration and jerk. Warp
            // 6 sets the new levels when the criterion's inputs are there, and finds the
            // next block time. (One warp per coordinate with a2 and a3 first took eight
            // instructions to the criterion and twelve to the state. With the forms
            // written out in the new and old derivatives every warp takes four, 300
            // cycles of a block step's 9000, but rounds differently.)
            if (warp < 4) {
                const int f = warp;
                #pragma unroll 1
                for (int it = wl; it < 3 * nc; it += 32) {
                    if (it >= 32) item.fetch(S, f, act + a0, it);
                    const double r = item.value(S, f);
                    if (f < LF_A2) {
                        S.x[3 * f * HCAP + item.o] = r;
                        S.f[3 * f * HCAP + item.o] = to_float_scaled(r, 0);
                    } else {
                        S.cf[3 * f * ACH + item.s] = to_float_scaled(r, -f * item.lv);
                    }
                }
                __syncwarp();
                asm volatile("bar.arrive 5, 224;" ::: "memory");
                // (levels, active list, a and adot are not read by these warps any more)
            } else if (warp < 6) {
                const int f = warp - 4;  // 0: a, 1: adot
                constexpr int NS = 3 * ACH / 32;
                int oo[NS];
                float fv[NS];
#pragma unroll
                for (int q = 0; q < NS; ++q) {
                    const int it = q * 32 + wl, sl = it / 3, c = it - 3 * sl;
                    oo[q] = -1;
                    if (it >= 3 * nc) continue;
                    const int k = act[a0 + sl];
                    const double r = S.a1s[(3 * f + c) * ACH + sl];
                    oo[q] = c * HCAP + k;
                    fv[q] = to_float_scaled(r, 0);
                    S.cf[(3 * f + c) * ACH + sl] = to_float_scaled(r, -f * S.lev[k]);
                }
                __syncwarp();
                asm volatile("bar.sync 5, 224;" ::: "memory");
                double *to = S.ax + 3 * f * HCAP;
#pragma unroll
                for (int q = 0; q < NS; ++q) {
                    if (oo[q] < 0) continue;
                    const int it = q * 32 + wl, sl = it / 3, c = it - 3 * sl;
                    to[oo[q]] = S.a1s[(3 * f + c) * ACH + sl];
                    S.f[(6 + 3 * f) * HCAP + oo[q]] = fv[q];
                }
            } else if (warp == 6) {
                // new time and level by the Aarseth criterion (FP32 on scaled
                // inputs); a larger step only by one level and on a commensurate time
                // (what does not wait for the inputs is read before they are there)
                int k = wl < nc ? act[a0 + wl] : 0;
                int lv = S.lev[k];
                bool up = (tn & ((1ll << (KMAX + 1 - lv)) - 1)) == 0;
                asm volatile("bar.sync 5, 224;" ::: "memory");
                #pragma unroll 1
                for (int sl = wl; sl < nc; sl += 32) {
                    if (sl >= 32) {
                        k = act[a0 + sl];
                        lv = S.lev[k];
                        up = (tn & ((1ll << (KMAX + 1 - lv)) - 1)) == 0;
                    }
                    int kn = level_from(S.cf + sl, lv, etaf, T2s);
                    if (kn < lv) kn = up ? lv - 1 : lv;
                    S.lev[k] = kn;
                    S.ti[k] = tn;
                    lmax = max(lmax, kn);
                }
                mk = k;
            }
            if (a0 + ACH < na) __syncthreads();  // the next round's sums and derivatives
        }
        // the next block time: the earliest of the others' and of the members that
        // moved now, the ends of whose steps are their levels' (every thread read
        // (tn, na) before the barriers above)
        if (warp == 6) {
            const int deep = __reduce_max_sync(0xffffffffu, lmax);
            const long long tm = tn + (1ll << (KMAX - deep));
            const long long t = min(tm, nb.t);
            int nn = nb.t == t ? nb.na : 0;
            if (tm == t && na <= 32) {
                const bool f = lmax == deep;
                const unsigned m = __ballot_sync(0xffffffffu, f);
                if (f) nact[nn + __popc(m & ((1u << wl) - 1u))] = (uint16_t)mk;
                nn += __popc(m);
            } else if (tm == t) {
                __syncwarp();
                #pragma unroll 1
                for (int b0 = 0; b0 < na; b0 += 32) {
                    const int k = b0 + wl < na ? act[b0 + wl] : -1;
                    const bool f = k >= 0 && S.lev[k] == deep;
                    const unsigned m = __ballot_sync(0xffffffffu, f);
                    if (f) nact[nn + __popc(m & ((1u << wl) - 1u))] = (uint16_t)k;
                    nn += __popc(m);
                }
            }
            if (wl == 0) {
                g_tn = lost ? LLONG_MAX : t;  // (ends the set)
                g_na = nn;
            }
        }
        ++steps;
    }
    // peers may still read this CTA's partial sums of the last round
    if (COOP) cl.sync(); else __syncthreads();
    if ((capped && tid == 0 && rank == 0) || lost) atomicOr(d.status, QYM_ST_HERMITE_CAP);
    // item 7: pre-remove the (1-K) part of the coming kick at q1 (own members)
    #pragma unroll 1
    for (int k = tid; k < n; k += blockDim.x) {
        S.ex[k] = S.x[k]; S.ey[k] = S.y[k]; S.ez[k] = S.z[k];
    }
    __syncthreads();
    #pragma unroll 1
    for (int k0 = mlo; k0 < mhi; k0 += NG) {
        int k = k0 + grp;
        double c[3] = {0.0, 0.0, 0.0};
        if (k < mhi) kcorr_part(S, 0, n, k, lane, P, tc, c);
        group_sum(c, 3, P);
        if (k < mhi && lane == 0) {
            int64_t r = S.ids[k];
            d.q1[r] = S.x[k];
            d.q1[R + r] = S.y[k];
            d.q1[2 * R + r] = S.z[k];
            d.v1[r] = S.u[k] - 0.5 * tau * c[0];
            d.v1[R + r] = S.v[k] - 0.5 * tau * c[1];
            d.v1[2 * R + r] = S.w[k] - 0.5 * tau * c[2];
            d.uf[r] = -1;
            d.hcost[r] = (int32_t)min(steps, (int64_t)INT_MAX);
        }
    }
    if (tid == 0 && rank == 0) {
        atomicAdd(d.ctr + C_SUM_HSTEPS, (unsigned long long)steps);
        atomicMax(d.ctr + C_MAX_HSET, (unsigned long long)steps);
    }
    // the next set reuses shared memory that peers read above
    if (COOP) cl.sync(); else __syncthreads();
}

__global__ void __launch_bounds__(1024) k_hermite_plan(Dev d, int ncl) {
    chain_wait();
    hermite_plan(d, ncl);
}

// Each cluster of CLT CTAs first integrates the set the plan gave it (all its
// CTAs on one set), then every CTA takes sets one at a time from the queue, in
// the order of a counter, so CTAs freed early take more.
template <int CLT>
__global__ void __cluster_dims__(CLT, 1, 1) __launch_bounds__(HTHREADS, 2) k_hermite(Dev d, HermArgs h) {
    chain_wait();
    static_assert(CLT == 2 || CLT == 4 || CLT == 8, "a cluster is 2, 4 or 8 CTAs");
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int cid = blockIdx.x / CLT;
    const int cset = cid < kHermMaxClusters ? d.hcl[cid] : -1;
    if (cset >= 0) hermite_set<true, CLT>(d, h, cset, rank, CLT);
    const int nq = (int)d.ctr[C_HNQ];
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) g_next_small = (int)atomicAdd(d.ctr + C_HSMALL, 1ull);
        __syncthreads();
        const int k = g_next_small;
        if (k >= nq) break;
        hermite_set<false, 2>(d, h, d.hq[k], 0, 1);
    }
}

// every member of every set leaves the union-find (-1) and, when this context
// integrated only its own sets, the other sets' members get their states and
// costs from the GPUs that did
__global__ void k_uf_clear_members(Dev d) {
    chain_wait();
    const unsigned long long n = min(d.ctr[C_NMEM], (unsigned long long)d.max_members);
    for (unsigned long long k = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (unsigned long long)gridDim.x * blockDim.x)
        d.uf[d.set_mem[k]] = -1;
}

cudaError_t hermite_prepare() {
    cudaError_t e = cudaFuncSetAttribute(k_hermite<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kHermSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_hermite<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kHermSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_hermite<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kHermSmem);
    return e;
}

// Cluster size for a batch (qym_params.hermite_cluster; 0 = automatic). One
// system holds a few sets, and its longest set gains most from spreading its
// partners over eight SMs (16384-body disk: 0.96 ms per step against 1.08 ms on
// two). A batch of many systems keeps thousands of sets in flight, and a set on
// eight CTAs keeps seven from the queue: two (512-system ensemble: 17.4 ms per
// step against 18.4 ms with eight). Either way two CTAs per SM: a CTA's chain
// keeps its SM's FP64 units busy a third of the time (the ensemble with one per
// SM: 18.4 ms).
int hermite_cluster_size(const Dev &d, const qym_params &p) {
    if (p.hermite_cluster == 2 || p.hermite_cluster == 4 || p.hermite_cluster == 8)
        return p.hermite_cluster;
    return d.nsys == 1 ? 8 : 2;
}

constexpr int kHermGrid = 2 * 152;  // CTAs per SM x SMs
// clusters that take a set of the plan (with two CTAs each, half of them: how many
// sets share their sums over a cluster is part of a batch's results)
int hermite_clusters(const Dev &d, const qym_params &p) {
    const int cls = hermite_cluster_size(d, p);
    return (cls == 2 ? 1 : 2) * 152 / cls;
}
static_assert(2 * 152 / 4 <= kHermMaxClusters && 152 / 2 <= kHermMaxClusters, "more clusters than plan entries");

cudaError_t launch_hermite(const Dev &d, const qym_params &p, double tau, cudaStream_t st) {
    HermArgs h;
    h.G = p.G;
    h.eps2 = p.eps_H * p.eps_H;
    h.eta = p.eta;
    h.eta_s = p.eta_s;
    h.tau = tau;
    h.max_steps = p.max_hermite_steps;
    const int cls = hermite_cluster_size(d, p);
    const int grid = kHermGrid;
    cudaError_t e;
    if (!sets_one(d)) {  // (else at the end of the set builder)
        launch_chain(k_hermite_plan, 1, 1024, 0, st, d, hermite_clusters(d, p));
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    switch (cls) {
    case 2: launch_chain(k_hermite<2>, grid, HTHREADS, kHermSmem, st, d, h); break;
    case 4: launch_chain(k_hermite<4>, grid, HTHREADS, kHermSmem, st, d, h); break;
    default: launch_chain(k_hermite<8>, grid, HTHREADS, kHermSmem, st, d, h); break;
    }
    e = cudaGetLastError();
    if (e != cudaSuccess || d.own_hi == 0) return e;
    launch_chain(k_uf_clear_members, 152, 256, 0, st, d);
    return cudaGetLastError();
}

}  // namespace qym
