// encounter.cu -- close-encounter identification after the Kepler drift
// (Sec. 2.3 item 4, Sec. 2.4) and the partition of the encounter pairs into
// non-intersecting sets with their transition radius r_crit (Eq. 9).
//
// The rigorous test is evaluated in FP64 with explicitly rounded operations
// (no contraction into FMA) in a fixed order, so that equal inputs give equal
// bits on any IEEE-754 machine evaluating the same sequence.
#include "hermite_plan.cuh"
#include "qym_internal.cuh"

namespace qym {

#define DM(a, b) __dmul_rn((a), (b))
#define DA(a, b) __dadd_rn((a), (b))
#define DS(a, b) __dsub_rn((a), (b))

// Minimum over [0, tau] of the cubic p(u), u = t / tau, that matches
// d^2 = |dQ|^2 and its slope at both ends (third-order interpolation of the
// minimum separation, Sec. 2.4); clamped at 0.
__device__ double dmin2_cubic(const double *dq0, const double *dv0, const double *dq1,
                              const double *dv1, double tau) {
    double d0 = DA(DA(DM(dq0[0], dq0[0]), DM(dq0[1], dq0[1])), DM(dq0[2], dq0[2]));
    double d1 = DA(DA(DM(dq1[0], dq1[0]), DM(dq1[1], dq1[1])), DM(dq1[2], dq1[2]));
    double g0 = DA(DA(DM(dq0[0], dv0[0]), DM(dq0[1], dv0[1])), DM(dq0[2], dv0[2]));
    double g1 = DA(DA(DM(dq1[0], dv1[0]), DM(dq1[1], dv1[1])), DM(dq1[2], dv1[2]));
    double s0 = DM(DM(2.0, g0), tau);
    double s1 = DM(DM(2.0, g1), tau);
    double c0 = d0, c1 = s0;
    double c2 = DS(DS(DM(3.0, DS(d1, d0)), DM(2.0, s0)), s1);
    double c3 = DA(DA(DM(2.0, DS(d0, d1)), s0), s1);
    double best = d0 < d1 ? d0 : d1;
    // stationary points of p: A u^2 + B u + Cc = 0 with A = 3 c3, B = 2 c2,
    // Cc = c1; roots w / A and Cc / w, w = -(B + sgn(B) sqrt(B^2 - 4 A Cc)) / 2
    double A = DM(3.0, c3), B = DM(2.0, c2), Cc = c1;
    double disc = DS(DM(B, B), DM(DM(4.0, A), Cc));
    if (disc >= 0.0) {
        double sq = __dsqrt_rn(disc);
        double w = DM(-0.5, DA(B, B >= 0.0 ? sq : -sq));
        double u[2];
        int nu = 0;
        if (A != 0.0) u[nu++] = __ddiv_rn(w, A);
        if (w != 0.0) u[nu++] = __ddiv_rn(Cc, w);
        for (int k = 0; k < nu; ++k) {
            double uk = u[k];
            if (uk > 0.0 && uk < 1.0) {
                double p = DA(c0, DM(uk, DA(c1, DM(uk, DA(c2, DM(uk, c3))))));
                if (p < best) best = p;
            }
        }
    }
    return best > 0.0 ? best : 0.0;
}

__device__ __forceinline__ double pair_test(const double *q0, const double *v0,
                                            const double *q1, const double *v1,
                                            const double *rH, int64_t R, int64_t i, int64_t j,
                                            double tau, double a_E, double &thr2) {
    double dq0[3], dv0[3], dq1[3], dv1[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        dq0[c] = DS(q0[c * R + i], q0[c * R + j]);
        dv0[c] = DS(v0[c * R + i], v0[c * R + j]);
        dq1[c] = DS(q1[c * R + i], q1[c * R + j]);
        dv1[c] = DS(v1[c * R + i], v1[c * R + j]);
    }
    double Rr = DM(a_E, DA(rH[i], rH[j]));
    thr2 = DM(Rr, Rr);
    return dmin2_cubic(dq0, dv0, dq1, dv1, tau);
}

// ---------------------------------------------------------------- public pair test
__global__ void k_pair_test(int64_t rows, const double *q0, const double *v0, const double *q1,
                            const double *v1, const double *rH, double tau, double a_E,
                            int64_t npairs, const int32_t *pairs, double *d2, int32_t *flag) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= npairs) return;
    int64_t i = pairs[2 * k], j = pairs[2 * k + 1];
    double thr2;
    double dm = pair_test(q0, v0, q1, v1, rH, rows, i, j, tau, a_E, thr2);
    if (d2) d2[k] = dm;
    if (flag) flag[k] = dm < thr2 ? 1 : 0;
}

cudaError_t launch_pair_test(int64_t rows, const double *q0, const double *v0, const double *q1,
                             const double *v1, const double *rH, double tau, double a_E,
                             int64_t npairs, const int32_t *pairs, double *d2, int32_t *flag,
                             cudaStream_t st) {
    if (npairs <= 0) return cudaSuccess;
    int tb = 256;
    k_pair_test<<<(unsigned)((npairs + tb - 1) / tb), tb, 0, st>>>(rows, q0, v0, q1, v1, rH, tau,
                                                                  a_E, npairs, pairs, d2, flag);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- refine
__device__ __forceinline__ void push_encounter(const Dev &d, int i, int j) {
    unsigned long long k = atomicAdd(d.ctr + C_NENC, 1ull);
    if (k < (unsigned long long)d.max_enc)
        d.enc[k] = make_int2(i, j);
    else
        atomicOr(d.status, QYM_ST_ENC_OVERFLOW);
    if (!d.log_refine) return;
    unsigned long long l = atomicAdd(d.ctr + C_LOG, 1ull);
    if (l < (unsigned long long)d.max_log) {
        d.log[3 * l] = (int64_t)d.ctr[C_STEP];
        d.log[3 * l + 1] = i;
        d.log[3 * l + 2] = j;
    } else {
        atomicOr(d.status, QYM_ST_LOG_OVERFLOW);
    }
}

// rigorous test of the crude candidates: (d.q, d.v) hold the state entering
// the Kepler drift, (d.q1, d.v1) the Kepler result; and, on the CTAs past
// kRefineCtas, the exact re-search of rows whose crude bounds were exceeded: the
// row against every other body of its system (one CTA per row; nearly always none)
constexpr int kRefineCtas = 2 * 152;
__global__ void __launch_bounds__(256) k_refine(Dev d, double tau, double a_E) {
    chain_wait();
    const int64_t R = d.rows;
    if (blockIdx.x < kRefineCtas) {
        unsigned long long n = d.ctr[C_NCAND];
        if (n > (unsigned long long)d.max_cand) n = d.max_cand;
        for (unsigned long long k = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; k < n;
             k += (unsigned long long)kRefineCtas * blockDim.x) {
            int2 p = d.cand[k];
            double thr2;
            double dm = pair_test(d.q, d.v, d.q1, d.v1, d.rH, R, p.x, p.y, tau, a_E, thr2);
            if (dm < thr2) push_encounter(d, p.x, p.y);
        }
        return;
    }
    unsigned long long n = d.ctr[C_NRESCAN];
    if (n > (unsigned long long)d.rows) n = d.rows;
    for (unsigned long long b = blockIdx.x - kRefineCtas; b < n; b += gridDim.x - kRefineCtas) {
        int64_t i = d.rescan[b];
        int sys = d.sys_of[i];
        int64_t lo = d.offsets[sys] + 1, hi = d.offsets[sys + 1];
        for (int64_t j = lo + threadIdx.x; j < hi; j += blockDim.x) {
            if (j == i) continue;
            int64_t a = i < j ? i : j, c = i < j ? j : i;
            double thr2;
            double dm = pair_test(d.q, d.v, d.q1, d.v1, d.rH, R, a, c, tau, a_E, thr2);
            if (dm < thr2) push_encounter(d, (int)a, (int)c);
        }
    }
}

cudaError_t launch_refine(const Dev &d, double tau, double a_E, cudaStream_t st) {
    return launch_chain(k_refine, kRefineCtas + 152, 256, 0, st, d, tau, a_E);
}

// ---------------------------------------------------------------- sets
// Union-find over the encounter pairs on uf[rows] (-1 = not in any pair):
// roots are the smallest row of each set. Hooking links the larger root under
// the smaller with compare-and-swap; every loop is capped.
constexpr int UF_CAP = 1 << 20;

// Parents are read with volatile (L1-bypassing) loads: links are made with
// atomics in L2, and a cached line could still show a node as unset (-1).
// A negative parent is never followed.
__device__ __forceinline__ int uf_find(int *uf, int x, int &guard) {
    volatile int *u = uf;
    int p = u[x];
    while (p != x && p >= 0 && guard < UF_CAP) {
        x = p;
        p = u[x];
        ++guard;
    }
    return x;
}

// join the sets of a pair
__device__ __forceinline__ void uf_hook(const Dev &d, int2 p) {
    int *uf = d.uf;
    atomicCAS(uf + p.x, -1, p.x);
    atomicCAS(uf + p.y, -1, p.y);
    int guard = 0;
    while (guard < UF_CAP) {
        int a = uf_find(uf, p.x, guard), b = uf_find(uf, p.y, guard);
        if (a == b) break;
        if (a > b) { int t = a; a = b; b = t; }
        if (atomicCAS(uf + b, b, a) == b) break;
        ++guard;
    }
    if (guard >= UF_CAP) atomicOr(d.status, QYM_ST_UF_CAP);
}

__global__ void k_uf_hook(Dev d) {
    chain_wait();
    unsigned long long n = d.ctr[C_NENC];
    if (n > (unsigned long long)d.max_enc) n = d.max_enc;
    for (unsigned long long k = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (unsigned long long)gridDim.x * blockDim.x)
        uf_hook(d, d.enc[k]);
}

// per-block counts of roots, for an ordered numbering of the sets
__global__ void __launch_bounds__(1024) k_uf_count(Dev d, int32_t *blk) {
    chain_wait();
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int isroot = 0;
    if (r < d.rows) {
        int p = d.uf[r];
        isroot = (p == (int)r);
    }
    int c = __syncthreads_count(isroot);
    if (threadIdx.x == 0) blk[blockIdx.x] = c;
}

// exclusive scan of the block counts (one CTA)
__global__ void __launch_bounds__(1024) k_scan_blocks(Dev d, int32_t *blk, int nblk) {
    chain_wait();
    __shared__ int32_t part[1024];
    int per = (nblk + 1023) / 1024;
    int b0 = threadIdx.x * per;
    int s = 0;
    for (int b = b0; b < b0 + per && b < nblk; ++b) s += blk[b];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        int t = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
        __syncthreads();
        part[threadIdx.x] += t;
        __syncthreads();
    }
    int run = threadIdx.x ? part[threadIdx.x - 1] : 0;
    for (int b = b0; b < b0 + per && b < nblk; ++b) {
        int c = blk[b];
        blk[b] = run;
        run += c;
    }
    if (threadIdx.x == 1023) d.ctr[C_NSETS] = (unsigned long long)part[1023];
}

// number the roots in row order: sid[root] = set index; members are counted
__global__ void __launch_bounds__(1024) k_uf_number(Dev d, const int32_t *blk, int32_t *sid,
                                                    int32_t *size) {
    chain_wait();
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int isroot = 0;
    if (r < d.rows) isroot = (d.uf[r] == (int)r);
    unsigned ball = __ballot_sync(0xffffffffu, isroot);
    __shared__ int wsum[32];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) wsum[w] = __popc(ball);
    __syncthreads();
    if (threadIdx.x < 32) {
        int x = wsum[threadIdx.x];
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        wsum[threadIdx.x] = x;  // inclusive
    }
    __syncthreads();
    if (isroot) {
        int before = (w ? wsum[w - 1] : 0) + __popc(ball & ((1u << lane) - 1u));
        int s = blk[blockIdx.x] + before;
        sid[r] = s;
        size[s] = 0;
        if (s < d.max_sets) d.set_root[s] = (int32_t)r;
    }
}

// each member finds its root, adds itself to its set size, raises the set's
// r_crit (a_H times the largest Hill radius) and the set's predicted Hermite cost
// (the block steps of the member's set in the previous step)
__device__ __forceinline__ void uf_member(const Dev &d, int64_t r, const int32_t *sid, int32_t *size,
                                          unsigned long long *rc_bits, double a_H) {
    int guard = 0;
    int root = uf_find(d.uf, (int)r, guard);
    int s = sid[root];
    if (s < 0 || s >= d.max_sets) return;
    atomicAdd(size + s, 1);
    double rc = a_H * d.rH[r];
    atomicMax(rc_bits + s, (unsigned long long)__double_as_longlong(rc));
    const int32_t hc = d.hcost[r];
    if (hc > 0) atomicMax(d.hsetcost + s, hc);
}

__global__ void __launch_bounds__(256) k_uf_members(Dev d, const int32_t *sid, int32_t *size,
                                                    unsigned long long *rc_bits, double a_H) {
    chain_wait();
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < d.rows && d.uf[r] >= 0) uf_member(d, r, sid, size, rc_bits, a_H);
}

// set_start = exclusive scan of set sizes (one CTA); the fill counters reset
// (sizes and r_crit come from atomics: read past L1, for callers that raised
// them in the same kernel)
__device__ __forceinline__ void scan_sets(const Dev &d, int n, const int32_t *size, int32_t *fill,
                                          unsigned long long *rc_bits) {
    __shared__ int32_t part[1024];
    if (n > d.max_sets) n = d.max_sets;
    int per = (n + 1023) / 1024;
    int b0 = threadIdx.x * per;
    int s = 0;
    for (int b = b0; b < b0 + per && b < n; ++b) s += __ldcg(size + b);
    part[threadIdx.x] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        int t = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
        __syncthreads();
        part[threadIdx.x] += t;
        __syncthreads();
    }
    int run = threadIdx.x ? part[threadIdx.x - 1] : 0;
    int mx = 0;
    for (int b = b0; b < b0 + per && b < n; ++b) {
        d.set_start[b] = run;
        run += __ldcg(size + b);
        mx = max(mx, __ldcg(size + b));
        fill[b] = 0;
        d.rcrit[b] = __longlong_as_double((long long)__ldcg(rc_bits + b));
        rc_bits[b] = 0ull;
    }
    // largest set
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    __shared__ int wmax[32];
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 1023) {
        d.set_start[n] = part[1023];
        d.ctr[C_NMEM] = (unsigned long long)part[1023];
        int m = 0;
        for (int k = 0; k < 32; ++k) m = max(m, wmax[k]);
        if ((unsigned long long)m > d.ctr[C_MAX_SET]) d.ctr[C_MAX_SET] = (unsigned long long)m;
        d.ctr[C_SUM_SETS] += (unsigned long long)n;
        if (part[1023] > d.max_members) atomicOr(d.status, QYM_ST_SET_OVERFLOW);
    }
}

__global__ void __launch_bounds__(1024) k_scan_sets(Dev d, const int32_t *size, int32_t *fill,
                                                    unsigned long long *rc_bits) {
    chain_wait();
    scan_sets(d, (int)d.ctr[C_NSETS], size, fill, rc_bits);
}

__device__ __forceinline__ void uf_place(const Dev &d, int64_t r, const int32_t *sid, int32_t *fill) {
    int guard = 0;
    int root = uf_find(d.uf, (int)r, guard);
    int s = sid[root];
    if (s < 0 || s >= d.max_sets) return;
    int pos = d.set_start[s] + atomicAdd(fill + s, 1);
    if (pos < d.max_members) d.set_mem[pos] = (int32_t)r;
}

__global__ void __launch_bounds__(256) k_uf_place(Dev d, const int32_t *sid, int32_t *fill) {
    chain_wait();
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= d.rows) return;
    d.hcost[r] = 0;  // uf_member has read the last step's; this step's sets write theirs
    if (d.uf[r] >= 0) uf_place(d, r, sid, fill);
}

// The whole set builder in one CTA for up to kSetsOneRows rows: the seven kernels
// below are a few microseconds of latency each (22 us a step, 10 us here for 260
// rows; at 16384 rows the one CTA's rounds take 3 us longer than the seven), while
// the pairs of a step are few. A thread takes the rows tid, tid + 1024, ...: whether they are
// members and roots stays in two bit masks; the roots' counts per (round, warp) are
// numbered by one scan of 1024 entries.
// The Hermite's plan follows in the same CTA (a launch of 3.7 us less: 16 steps of
// 260 bodies 1636 -> 1618 us).
constexpr int kSetsRounds = 8;
constexpr int64_t kSetsOneRows = kSetsRounds * 1024;
__global__ void __launch_bounds__(1024) k_sets_one(Dev d, SetScratch s, double a_H, int ncl) {
    chain_wait();
    __shared__ int s_cnt[32][32], s_warp[32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int rows = (int)d.rows, rounds = (rows + 1023) >> 10;
    const unsigned long long n = min(d.ctr[C_NENC], (unsigned long long)d.max_enc);
    for (unsigned long long k = tid; k < n; k += 1024) uf_hook(d, d.enc[k]);
    __syncthreads();
    unsigned member = 0, root = 0;
#pragma unroll
    for (int it = 0; it < kSetsRounds; ++it) {
        const int r = it * 1024 + tid;
        if (r >= rows) break;
        const int p = n ? __ldcg(d.uf + r) : -1;
        if (p >= 0) member |= 1u << it;
        if (p == r) root |= 1u << it;
    }
    if (w >= kSetsRounds) s_cnt[w][lane] = 0;
    for (int it = 0; it < kSetsRounds; ++it) {
        const unsigned b = __ballot_sync(0xffffffffu, (root >> it) & 1u);
        if (lane == 0) s_cnt[it][w] = __popc(b);
    }
    __syncthreads();
    // exclusive scan of the 1024 counts in row order
    const int c = s_cnt[w][lane];
    int inc = c;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) s_warp[w] = inc;
    __syncthreads();
    const int ws = s_warp[lane];
    const int nsets = __reduce_add_sync(0xffffffffu, ws);
    s_cnt[w][lane] = __reduce_add_sync(0xffffffffu, lane < w ? ws : 0) + inc - c;
    __syncthreads();
    for (int it = 0; it < rounds; ++it) {
        const bool mine = (root >> it) & 1u;
        const unsigned b = __ballot_sync(0xffffffffu, mine);
        if (mine) {
            const int k = s_cnt[it][w] + __popc(b & ((1u << lane) - 1u));
            s.sid[it * 1024 + tid] = k;
            s.size[k] = 0;
            if (k < d.max_sets) d.set_root[k] = it * 1024 + tid;
        }
    }
    if (tid == 0) d.ctr[C_NSETS] = (unsigned long long)nsets;
    __threadfence();  // the cleared sizes before the members' atomics on them
    __syncthreads();
    for (unsigned m = member; m; m &= m - 1)
        uf_member(d, (int64_t)(__ffs(m) - 1) * 1024 + tid, s.sid, s.size, s.rc_bits, a_H);
    __syncthreads();
    scan_sets(d, nsets, s.size, s.fill, s.rc_bits);
    __threadfence();
    __syncthreads();
    for (int it = 0; it < rounds; ++it) {
        const int r = it * 1024 + tid;
        if (r < rows) d.hcost[r] = 0;
    }
    for (unsigned m = member; m; m &= m - 1)
        uf_place(d, (int64_t)(__ffs(m) - 1) * 1024 + tid, s.sid, s.fill);
    __syncthreads();
    hermite_plan(d, ncl);
}

// A batch can have a pair for nearly every row (swarms about its planets), and one CTA
// takes them in more rounds then: 1980 rows 240 us a step either way, 4320 rows 409
// against 394 in the seven kernels, 6600 rows 309 against 287.
bool sets_one(const Dev &d) { return d.rows <= (d.nsys == 1 ? kSetsOneRows : 2048); }
int sets_launches(const Dev &d) { return sets_one(d) ? 1 : 8; }

cudaError_t launch_sets_impl(const Dev &d, const qym_params &p, const SetScratch &s, cudaStream_t st) {
    const double a_H = p.a_H;
    if (sets_one(d))
        return launch_chain(k_sets_one, 1, 1024, 0, st, d, s, a_H, hermite_clusters(d, p));
    int nblk = (int)((d.rows + 1023) / 1024);
    launch_chain(k_uf_hook, 152, 256, 0, st, d);
    launch_chain(k_uf_count, nblk, 1024, 0, st, d, s.blk);
    launch_chain(k_scan_blocks, 1, 1024, 0, st, d, s.blk, nblk);
    launch_chain(k_uf_number, nblk, 1024, 0, st, d, s.blk, s.sid, s.size);
    int tb = 256;
    unsigned g = (unsigned)((d.rows + tb - 1) / tb);
    launch_chain(k_uf_members, g, tb, 0, st, d, s.sid, s.size, s.rc_bits, a_H);
    launch_chain(k_scan_sets, 1, 1024, 0, st, d, s.size, s.fill, s.rc_bits);
    launch_chain(k_uf_place, g, tb, 0, st, d, s.sid, s.fill);
    return cudaGetLastError();
}

}  // namespace qym
