// energy.cu -- total energy of each system (Sec. 2, Eqs. 2-4), FP64:
//   E = |S|^2 / (2 m0) + sum_i [m_i v_i^2 / 2 - G m0 m_i / |Q_i|]
//       - sum_{i < j} G m_i m_j / |Q_i - Q_j|        (i, j bodies),
// each pair once (the paper's kernel takes both orders and halves the sum),
// with the star mass restored for the star terms.
//
// The pair sum is bound by issue: a pair's separation, r^2 and 1 / r run to
// FP64 accuracy on the FP32 pipes (pair64.cuh), FP64 multiplies by G m and adds
// (one instruction). A CTA takes 128 rows against a range of later
// rows; the range's length (energy_plan) gives the GPU about 16 CTAs per SM
// whatever the sizes, where one CTA per 256 rows against all rows left 16384
// bodies on 64 of the 152 SMs with 15 FP64 instructions per ordered pair
// (16.6 ms).
#include <algorithm>

#include "pair64.cuh"
#include "qym_internal.cuh"

namespace qym {

constexpr int ET = 128;  // rows of an i-block = threads of a CTA = rows of a j tile

// 1 / r of a pair in FP64, where the float form does not hold (0 for r = 0)
__device__ __noinline__ double inv_r_fp64(double dx, double dy, double dz) {
    const double r2 = dx * dx + dy * dy + dz * dz;
    return (r2 > 0.0) ? rsqrt(r2) : 0.0;
}

// CTA (I, c): rows of i-block I against the rows j > i of its c-th range;
// writes -sum_i m_i sum_j G m_j / r_ij, and for c = 0 adds the rows' kinetic
// and star terms and writes their momentum to ps[I]
__global__ void __launch_bounds__(ET) k_energy_pairs(EnergyPlan pl, int64_t R, const double *m,
                                                     const double *q, const double *v, double G,
                                                     double *pe, double *ps) {
    chain_wait();
    __shared__ D4 s_q[ET];
    __shared__ float4 s_a[ET], s_b[ET];  // (x, y, z) in three parts: x.h y.h z.h x.m, y.m z.m x.l y.l
    __shared__ float s_c[ET];            // z.l
    __shared__ int s_hi[ET / 32];
    __shared__ double red[4][ET / 32];
    const int2 it = pl.items ? pl.items[blockIdx.x]
                             : make_int2((int)(blockIdx.x / pl.nranges), (int)(blockIdx.x % pl.nranges));
    const int64_t I = it.x;
    const int c = it.y;
    const int4 bk = pl.blocks ? pl.blocks[I]
                              : make_int4((int)(1 + I * ET), (int)min(1 + (I + 1) * (int64_t)ET, R), (int)R, 0);
    const int64_t jb = bk.x + (int64_t)c * pl.range;
    if (jb >= bk.z) {
        if (threadIdx.x == 0) pe[blockIdx.x] = 0.0;
        return;
    }
    const int j0 = (int)jb, j1 = (int)min(jb + pl.range, (int64_t)bk.z);
    const int i = bk.x + threadIdx.x;
    const int r = min(i, bk.y - 1);  // an idle lane repeats the last row
    const double xi = q[r], yi = q[R + r], zi = q[2 * R + r];
    int hl = __reduce_max_sync(0xffffffffu, max(p64::hi_abs(xi), max(p64::hi_abs(yi), p64::hi_abs(zi))));
    if ((threadIdx.x & 31) == 0) s_hi[threadIdx.x >> 5] = hl;
    __syncthreads();
    for (int w = 0; w < ET / 32; ++w) hl = max(hl, s_hi[w]);
    const p64::Scale sc(hl, 0x3ff00000);
    const uint64_t bias = sc.bias(1);
    const p64::F3 px = p64::split3(xi * sc.len), py = p64::split3(yi * sc.len);
    const p64::F3 pz = p64::split3(zi * sc.len);
    double phi = 0.0;
    for (int jt = j0; jt < j1; jt += ET) {
        const int n = min(ET, j1 - jt);
        __syncthreads();
        if ((int)threadIdx.x < n) {
            const int j = jt + threadIdx.x, t = threadIdx.x;
            const D4 p{q[j], q[R + j], q[2 * R + j], G * m[j]};
            const p64::F3 x = p64::split3(p.x * sc.len), y = p64::split3(p.y * sc.len);
            const p64::F3 z = p64::split3(p.z * sc.len);
            s_q[t] = p;
            s_a[t] = make_float4(x.h, y.h, z.h, x.m);
            s_b[t] = make_float4(y.m, z.m, x.l, y.l);
            s_c[t] = z.l;
        }
        __syncthreads();
#pragma unroll 2
        for (int t = 0; t < n; ++t) {
            const float4 A = s_a[t], B = s_b[t];
            const p64::F3 r2 = p64::norm2(p64::diff(px, p64::F3{A.x, A.w, B.z}),
                                          p64::diff(py, p64::F3{A.y, B.x, B.w}),
                                          p64::diff(pz, p64::F3{A.z, B.y, s_c[t]}));
            double y = p64::inv_r(r2, rsqrt_ftz(r2.h), bias);
            const bool later = jt + t > i;
            if (later && !(sc.ok && p64::r2_fits(r2.h))) {
                const D4 p = s_q[t];
                y = inv_r_fp64(xi - p.x, yi - p.y, zi - p.z);
            }
            if (later) phi = fma(s_q[t].w, y, phi);
        }
    }
    const bool act = i < bk.y;
    double e[4] = {0.0, 0.0, 0.0, 0.0};
    if (act) {
        const double mi = m[i];
        e[0] = -mi * phi;
        if (c == 0) {
            const double vx = v[i], vy = v[R + i], vz = v[2 * R + i];
            const double d = sqrt(xi * xi + yi * yi + zi * zi);
            e[0] += 0.5 * mi * (vx * vx + vy * vy + vz * vz) - G * m[bk.w] * mi / d;
            e[1] = mi * vx;
            e[2] = mi * vy;
            e[3] = mi * vz;
        }
    }
    const int nq = c == 0 ? 4 : 1;
    for (int k = 0; k < nq; ++k) {
        e[k] = warp_sum(e[k]);
        if ((threadIdx.x & 31) == 0) red[k][threadIdx.x >> 5] = e[k];
    }
    __syncthreads();
    if ((int)threadIdx.x < nq) {
        double s = 0.0;
        for (int k = 0; k < ET / 32; ++k) s += red[threadIdx.x][k];
        if (threadIdx.x == 0)
            pe[blockIdx.x] = s;
        else
            ps[3 * I + threadIdx.x - 1] = s;
    }
}

// per system (one CTA each): its CTAs' sums in a fixed order plus |S|^2 / (2 m0)
__global__ void __launch_bounds__(256) k_energy_final(EnergyPlan pl, const int64_t *offsets,
                                                      const double *m, const double *pe,
                                                      const double *ps, double *E) {
    chain_wait();
    const int s = blockIdx.x;
    const int64_t b0 = pl.block0 ? pl.block0[s] : 0, b1 = pl.block0 ? pl.block0[s + 1] : pl.nblocks;
    const int64_t i0 = pl.item0 ? pl.item0[s] : 0, i1 = pl.item0 ? pl.item0[s + 1] : pl.nitems;
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t k = i0 + threadIdx.x; k < i1; k += blockDim.x) t[0] += pe[k];
    for (int64_t k = b0 + threadIdx.x; k < b1; k += blockDim.x)
        for (int c = 0; c < 3; ++c) t[1 + c] += ps[3 * k + c];
    __shared__ double sh[4][8];
    for (int c = 0; c < 4; ++c) {
        t[c] = warp_sum(t[c]);
        if ((threadIdx.x & 31) == 0) sh[c][threadIdx.x >> 5] = t[c];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int c = 0; c < 4; ++c) {
            t[c] = 0.0;
            for (int k = 0; k < 8; ++k) t[c] += sh[c][k];
        }
        E[s] = t[0] + (t[1] * t[1] + t[2] * t[2] + t[3] * t[3]) / (2.0 * m[offsets ? offsets[s] : 0]);
    }
}

// host: i-blocks of at most 128 rows of each system and the ranges' length: about 16
// CTAs per SM over the batch's pairs, ranges of 8 (a small system's walk is latency)
// to 4096 rows. A batch's items are its non-empty ranges: one count of ranges for all
// i-blocks, the largest system's, made a million systems of two bodies beside one of
// 3000 launch 1.9e8 CTAs and hold 1.5 GB of partial sums.
EnergyPlan energy_plan(const int64_t *offsets, int32_t nsys, EnergyTables *t) {
    EnergyPlan pl;
    double pairs = 0.0;
    for (int32_t s = 0; s < nsys; ++s) {
        const int64_t nb = offsets[s + 1] - offsets[s] - 1;
        pairs += 0.5 * (double)nb * (double)nb;
        pl.nblocks += (int32_t)((nb + ET - 1) / ET);
    }
    const double want = pairs / (16.0 * 152.0 * ET);
    pl.range = (int32_t)std::min(4096.0, std::max(8.0, 8.0 * (double)(int64_t)(want / 8.0 + 1.0)));
    if (!t) {
        pl.nranges = (int32_t)((offsets[1] - offsets[0] - 1 + pl.range - 1) / pl.range);
        pl.nitems = pl.nblocks * pl.nranges;
        return pl;
    }
    for (int32_t s = 0; s < nsys; ++s) {
        t->block0.push_back((int32_t)t->blocks.size());
        t->item0.push_back((int32_t)t->items.size());
        const int64_t b1 = offsets[s + 1];
        for (int64_t i0 = offsets[s] + 1; i0 < b1; i0 += ET) {
            for (int64_t j0 = i0; j0 < b1; j0 += pl.range)
                t->items.push_back(make_int2((int)t->blocks.size(), (int)((j0 - i0) / pl.range)));
            t->blocks.push_back(make_int4((int)i0, (int)std::min<int64_t>(i0 + ET, b1), (int)b1, (int)offsets[s]));
        }
    }
    t->block0.push_back((int32_t)t->blocks.size());
    t->item0.push_back((int32_t)t->items.size());
    pl.nitems = (int32_t)t->items.size();
    return pl;
}

int64_t energy_partials(const EnergyPlan &pl) { return (int64_t)pl.nitems + 3 * (int64_t)pl.nblocks; }

cudaError_t launch_energy(const EnergyPlan &pl, int32_t nsys, const int64_t *offsets, int64_t R,
                          const double *m, const double *q, const double *v, double G, double *part,
                          double *E, cudaStream_t st) {
    double *ps = part + pl.nitems;
    launch_chain(k_energy_pairs, (unsigned)pl.nitems, ET, 0, st, pl, R, m, q, v, G, part, ps);
    launch_chain(k_energy_final, nsys, 256, 0, st, pl, offsets, m, part, ps, E);
    return cudaGetLastError();
}

}  // namespace qym
