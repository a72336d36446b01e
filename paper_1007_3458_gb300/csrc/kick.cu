// kick.cu -- E_Int: all-pairs interaction accelerations (Sec. 2, Eq. 4),
//   a_i = -sum_{j >= 1, j != i} G m_j (Q_i - Q_j) / |Q_i - Q_j|^3,
// the star's mass zeroed (its row is simply not in any tile), fused with the
// crude close-encounter search of the first kick of a step (Sec. 2.4).
//
// Work decomposition: one CTA per work item (system, i-block, j-range). The
// i rows of the block live in registers (IPT per thread); j rows stream
// through shared memory in tiles of TILE. Each item writes its partial sums to
// its own slot of apart[slot][3][rows]; the finisher adds the slots in a fixed
// order, so results are deterministic.
//
// Mixed precision (QYM_KICK_MIXED): positions are split into float hi + lo
// parts, the separation is formed as (hi_i - hi_j) + (lo_i - lo_j) (a
// double-single difference, accurate to ~1e-7 relative even for close pairs
// far from the star), the pair force is FP32 with rsqrt, and the FP32 tile sums
// are folded every FOLD pairs into a float two-sum (hi, lo) accumulator that
// is returned as a double. The FP32 arithmetic runs on Blackwell's packed
// FP32x2 instructions, two j rows per instruction.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "pair64.cuh"
#include "qym_internal.cuh"

namespace qym {

constexpr int TILE = kKickTile;
constexpr int FOLD = 64;
#ifndef QYM_KICK_UNROLL
#define QYM_KICK_UNROLL 4
#endif
constexpr int kPairUnroll = QYM_KICK_UNROLL;  // j pairs per unrolled step

struct KickArgs {
    const int4 *items;      // NULL: one system of `rows` rows, items by kick_item
    const int32_t *slots;
    int32_t chunk = 0;      // j rows per split (items == NULL)
    int32_t parts = 1;      // splits per chunk, of FOLD rows each (items == NULL; 1: whole chunks)
    const float4 *pos;      // (x_hi, y_hi, z_hi, G m)
    const float4 *lo;       // (x_lo, y_lo, z_lo, c = 2 rho^2 of the crude reach rho)
    const double *q;        // [3][rows] (FP64 path)
    const double *m;        // [rows] (FP64 path)
    double G;
    double *apart;
    int64_t rows;
    int2 *cand;
    int64_t max_cand;
    unsigned long long *ncand;
    int4 *fchunk;
    int64_t max_fchunk;
    unsigned long long *nfchunk;
    int32_t *status;
    int32_t far_tiles;      // 1: tiles far from a warp's rows take the one-add separation
    const int32_t *perm;    // row of each position of the packs (NULL: row order)
    const float4 *far;      // (o_x, o_y, o_z, G m): offset from the tile's reference point
    const float4 *tile;     // per tile: (c_x, c_y, c_z, R), box min (x, y, z, -), box max
    SymShape sym;           // pair-symmetric form (k_kick_sym)
    int32_t *blk_cnt = nullptr;  // arrivals per i-block (NULL: each slot stays for the finisher)
    int32_t splits = 1;          // items (slots) per i-block
    int32_t uniform = 1;         // windows of one G m multiply by it once per sum
};

// The item of CTA b: its rows [x, y), its j-range [z, w) and its slot; for one
// system (items == NULL) i-blocks of `ti` rows times `splits` ranges of `chunk`, or
// of the `parts` parts of FOLD rows of each
__device__ __forceinline__ int4 kick_item(const KickArgs &a, int ti, int &slot) {
    if (a.items) {
        slot = a.slots[blockIdx.x];
        return a.items[blockIdx.x];
    }
    const int64_t ib = blockIdx.x / a.splits;
    slot = (int)(blockIdx.x - ib * a.splits);
    const int64_t i0 = 1 + ib * ti, c = slot / a.parts;
    const int64_t j0 = 1 + c * a.chunk + (slot - c * a.parts) * FOLD;
    const int64_t j1 = a.parts == 1 ? j0 + a.chunk : min(j0 + FOLD, 1 + (c + 1) * a.chunk);
    return make_int4((int)i0, (int)min(i0 + ti, a.rows), (int)min(j0, a.rows), (int)min(j1, a.rows));
}

// The last CTA of an i-block to finish (arrivals counted per i-block, the
// counter reset by that CTA for the next launch) adds the block's `splits`
// slots into slot 0, in the order a reader of the slots used (lane q of
// four summing slots q, q + 4, ..., the four parts added as (0 + 1) + (2 + 3)),
// and discards the other slots' lines from L2 (PTX discard.global.L2): they
// are dead, and discarded lines are not written back, so the partial sums of
// all splits stay on chip and HBM sees only slot 0. Lines shared with a
// neighbouring i-block's rows are kept.
// (not inlined: as a call it leaves the register allocation of the kick's
// tile loop as it is without this epilogue)
template <int IPT>
__device__ __noinline__ void sum_block_slots(const KickArgs &a, const int (&gi)[IPT], int i_lo,
                                             int i_hi) {
    __shared__ int s_last;
    __syncthreads();  // every thread's slot stores issued
    if (threadIdx.x == 0) {
        // release: the block's slot stores (ordered before by the barrier)
        // precede the arrival; acquire: the last arrival sees every slot
        const int blk = (int)(blockIdx.x / a.splits);
        int old;
        asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;"
                     : "=r"(old)
                     : "l"(a.blk_cnt + blk)
                     : "memory");
        s_last = old == a.splits - 1;
        if (s_last) a.blk_cnt[blk] = 0;
    }
    __syncthreads();
    if (!s_last) return;
    const int64_t rows = a.rows;
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        if (gi[k] < i_hi) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double *p = a.apart + (int64_t)c * rows + gi[k];
                const int64_t st = 3 * rows;
                double p0 = 0.0, p1 = 0.0, p2 = 0.0, p3 = 0.0;
                int s = 0;
                for (; s + 3 < a.splits; s += 4) {
                    p0 += __ldcg(p + s * st);
                    p1 += __ldcg(p + (s + 1) * st);
                    p2 += __ldcg(p + (s + 2) * st);
                    p3 += __ldcg(p + (s + 3) * st);
                }
                if (s < a.splits) p0 += __ldcg(p + s * st);
                if (s + 1 < a.splits) p1 += __ldcg(p + (s + 1) * st);
                if (s + 2 < a.splits) p2 += __ldcg(p + (s + 2) * st);
                a.apart[(int64_t)c * rows + gi[k]] = (p0 + p1) + (p2 + p3);
            }
        }
    }
    __syncthreads();  // every read done before a line goes
    // whole 128-byte lines inside this block's rows of slots 1 .. splits-1:
    // per slot-component row sc, the lines from the first 128-byte boundary
    // at or after row i_lo to the last one at or before row i_hi
    const int L = (int)(((int64_t)(i_hi - i_lo) * 8 + 127) >> 7);  // lines a row range can span
    const int tot = (a.splits - 1) * 3 * L;
    for (int t = threadIdx.x; t < tot; t += blockDim.x) {
        const int sc = 3 + t / L;
        const uintptr_t base = (uintptr_t)(a.apart + (int64_t)sc * rows);
        const uintptr_t l0 = (base + (uintptr_t)i_lo * 8 + 127) & ~(uintptr_t)127;
        const uintptr_t l1 = (base + (uintptr_t)i_hi * 8) & ~(uintptr_t)127;
        const uintptr_t line = l0 + ((uintptr_t)(t % L) << 7);
        if (line < l1)  // [line, line + 128) inside [start, end)
            asm volatile("discard.global.L2 [%0], 128;" ::"l"(line) : "memory");
    }
}

// a + b + c for |c| far below |a + b|, rounded once: the rounding error of
// a + b (Knuth's two-sum) joins c before the last rounding
__device__ __forceinline__ float ds_add(float a, float b, float c) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return __fadd_rn(s, __fadd_rn(e, c));
}

// min(a, b, c) in one instruction (the three-input form of sm_100 and later)
__device__ __forceinline__ float fmin3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// append candidate (i, j) from a divergent branch, warp-aggregated
__device__ __forceinline__ void push_candidate(const KickArgs &a, int i, int j) {
    unsigned mask = __activemask();
    int lane = threadIdx.x & 31;
    int leader = __ffs(mask) - 1;
    unsigned long long base = 0;
    if (lane == leader) base = atomicAdd(a.ncand, (unsigned long long)__popc(mask));
    base = __shfl_sync(mask, base, leader);
    unsigned long long idx = base + __popc(mask & ((1u << lane) - 1u));
    if (idx < (unsigned long long)a.max_cand)
        a.cand[idx] = make_int2(i, j);
    else if (lane == leader)
        atomicOr(a.status, QYM_ST_CAND_OVERFLOW);
}

// j rows of a tile sit in shared memory in pairs (j = 2p, 2p+1), each pair as
// four float4: (xh0, xh1, yh0, yh1), (zh0, zh1, Gm0, Gm1), (xl0, xl1, yl0,
// yl1), (zl0, zl1, -c0, -c1). A float4's halves are float2 operands of the
// packed FP32 instructions (FADD2 / FMUL2 / FFMA2), so one instruction serves
// both j of a pair for an i row; the i operands are per-thread constants,
// negated and duplicated once. Each lane computes exactly what the scalar
// form (Q_i - Q_j, r^2, rsqrt, m r^-3, force) computes, with the sign of
// the separation flipped: d = Q_j - Q_i, a_i += (G m_j / r^3) d.
struct JPairs {
    float4 *a, *b, *c, *d;
};

// Pair forces of the j pairs [p0, p1) for the IPT rows of a thread. With
// FLAG, each i keeps the minimum over the chunk of r^2 - c_j, c_j = 2 rho_j^2
// (no branch); since (rho_i + rho_j)^2 <= c_i + c_j, a chunk without a
// candidate of i has that minimum >= c_i and needs no further look; a chunk
// with a smaller minimum is recorded and re-tested exactly by k_flag_chunks.
// In a chunk of the diagonal tile the row's own j (r^2 = 0) is left out of
// the minimum. Without FORCE only the search runs (the same separations and
// r^2). With UNI every j has the same G m, which the caller multiplies the sums
// by: one product a pair less on the FMA pipe that bounds the kick (planetesimals
// of one mass fill nearly every window; heavy bodies are summed elsewhere). r^-3
// alone has to stay in FP32's range then: the callers take UNI for coordinates
// below kUniMax, where every r^-3 is a normal float, and repeat a chunk whose sums
// are not finite (a pair closer than about 2^-43) with G m in the product.
constexpr float kUniMax = 0x1p40f;  // r < 2^42, r^-3 > 2^-126
__device__ __forceinline__ bool uni_range(const float4 &p) {
    return fmaxf(fabsf(p.x), fmaxf(fabsf(p.y), fabsf(p.z))) < kUniMax;
}
// whether the sums of a thread's rows are finite: one component tells, as an infinite
// r^-3 makes all three infinite or NaN (also times a zero difference)
template <int N>
__device__ __forceinline__ bool finite_sums(const float2 (&x)[N]) {
    float2 m = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int k = 0; k < N; ++k) m = __ffma2_rn(x[k], make_float2(0.0f, 0.0f), m);
    return m.x + m.y == 0.0f;  // (0 times infinity is NaN)
}
template <int IPT, bool FLAG, bool DIAG, bool FORCE, bool UNI>
__device__ __forceinline__ void mixed_chunk(const JPairs &s, int p0, int p1, int jt,
                                            const int (&gi)[IPT],
                                            const float2 (&nxh)[IPT], const float2 (&nyh)[IPT],
                                            const float2 (&nzh)[IPT], const float2 (&nxl)[IPT],
                                            const float2 (&nyl)[IPT], const float2 (&nzl)[IPT],
                                            float2 (&fx)[IPT], float2 (&fy)[IPT],
                                            float2 (&fz)[IPT], float (&mind)[IPT]) {
#pragma unroll kPairUnroll
    for (int p = p0; p < p1; ++p) {
        const float4 A = s.a[p], B = s.b[p], C = s.c[p], D = s.d[p];
        const float2 xh = make_float2(A.x, A.y), yh = make_float2(A.z, A.w);
        const float2 zh = make_float2(B.x, B.y), gm = make_float2(B.z, B.w);
        const float2 xl = make_float2(C.x, C.y), yl = make_float2(C.z, C.w);
        const float2 zl = make_float2(D.x, D.y), nc = make_float2(D.z, D.w);
#pragma unroll
        for (int k = 0; k < IPT; ++k) {
            const float2 dx = __fadd2_rn(__fadd2_rn(xh, nxh[k]), __fadd2_rn(xl, nxl[k]));
            const float2 dy = __fadd2_rn(__fadd2_rn(yh, nyh[k]), __fadd2_rn(yl, nyl[k]));
            const float2 dz = __fadd2_rn(__fadd2_rn(zh, nzh[k]), __fadd2_rn(zl, nzl[k]));
            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
            if (FORCE) {
                const float2 ri = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
                float2 sm = __fmul2_rn(UNI ? ri : __fmul2_rn(gm, ri), __fmul2_rn(ri, ri));
                if (DIAG) {
                    sm.x = (r2.x > 0.0f) ? sm.x : 0.0f;
                    sm.y = (r2.y > 0.0f) ? sm.y : 0.0f;
                }
                fx[k] = __ffma2_rn(sm, dx, fx[k]);
                fy[k] = __ffma2_rn(sm, dy, fy[k]);
                fz[k] = __ffma2_rn(sm, dz, fz[k]);
            }
            if (FLAG) {
                float2 t = __fadd2_rn(r2, nc);
                if (DIAG) {  // a row is not its own partner
                    t.x = (jt + 2 * p == gi[k]) ? 3.0e38f : t.x;
                    t.y = (jt + 2 * p + 1 == gi[k]) ? 3.0e38f : t.y;
                }
                mind[k] = fmin3(mind[k], t.x, t.y);
            }
        }
    }
}

// The same for a tile far from every row of the warp (far_tile): the j rows
// are held as FP32 offsets o_j = Q_j - c from the tile's reference point c
// (two j per float4 pair: (ox0, ox1, oy0, oy1), (oz0, oz1, Gm0, Gm1)) and
// each row as d_i = c - Q_i, formed once per tile in double-single and
// rounded; the separation is one packed add o_j + d_i per coordinate instead
// of three. With every pair at least the tile's radius R apart, both offsets
// are at most about the separation, so its relative error stays a few
// 2^-24; the rest (r^2, rsqrt, m r^-3, force, search) is the near form's.
struct JFar {
    float4 *a, *b, *d;  // d: the near layout's fourth float4, for -c0, -c1
};

template <int IPT, bool FLAG, bool FORCE, bool UNI>
__device__ __forceinline__ void far_chunk(const JFar &s, int p0, int p1, const float2 (&dxi)[IPT],
                                          const float2 (&dyi)[IPT], const float2 (&dzi)[IPT],
                                          float2 (&fx)[IPT], float2 (&fy)[IPT], float2 (&fz)[IPT],
                                          float (&mind)[IPT]) {
#pragma unroll kPairUnroll
    for (int p = p0; p < p1; ++p) {
        const float4 A = s.a[p], B = s.b[p];
        const float2 ox = make_float2(A.x, A.y), oy = make_float2(A.z, A.w);
        const float2 oz = make_float2(B.x, B.y), gm = make_float2(B.z, B.w);
        float2 nc = make_float2(0.0f, 0.0f);
        if (FLAG) {
            const float4 D = s.d[p];
            nc = make_float2(D.z, D.w);
        }
#pragma unroll
        for (int k = 0; k < IPT; ++k) {
            const float2 dx = __fadd2_rn(ox, dxi[k]);
            const float2 dy = __fadd2_rn(oy, dyi[k]);
            const float2 dz = __fadd2_rn(oz, dzi[k]);
            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
            if (FORCE) {
                const float2 ri = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
                const float2 sm = __fmul2_rn(UNI ? ri : __fmul2_rn(gm, ri), __fmul2_rn(ri, ri));
                fx[k] = __ffma2_rn(sm, dx, fx[k]);
                fy[k] = __ffma2_rn(sm, dy, fy[k]);
                fz[k] = __ffma2_rn(sm, dz, fz[k]);
            }
            if (FLAG) {
                const float2 t = __fadd2_rn(r2, nc);
                mind[k] = fmin3(mind[k], t.x, t.y);
            }
        }
    }
}

// record that row i's crude minimum over the j rows [j0, j1) fell below c_i
// (divergent branch, warp-aggregated); k_flag_chunks re-tests them
__device__ __forceinline__ void push_flag(const KickArgs &a, int i, int j0, int j1) {
    unsigned mask = __activemask();
    int lane = threadIdx.x & 31;
    int leader = __ffs(mask) - 1;
    unsigned long long base = 0;
    if (lane == leader) base = atomicAdd(a.nfchunk, (unsigned long long)__popc(mask));
    base = __shfl_sync(mask, base, leader);
    unsigned long long idx = base + __popc(mask & ((1u << lane) - 1u));
    if (idx < (unsigned long long)a.max_fchunk)
        a.fchunk[idx] = make_int4(i, j0, j1, 0);
    else if (lane == leader)
        atomicOr(a.status, QYM_ST_CAND_OVERFLOW);
}

// FORCE = false: the crude search alone (no partial sums written)
template <int IPT, bool FLAG, bool FORCE>
__global__ void __launch_bounds__(256) k_kick_mixed(KickArgs a) {
    chain_wait();
    __shared__ float4 s_a[TILE / 2], s_b[TILE / 2], s_c[TILE / 2], s_d[TILE / 2];
    __shared__ float4 s_fa[TILE / 2], s_fb[TILE / 2];
    const JPairs sp{s_a, s_b, s_c, s_d};
    const JFar sf{s_fa, s_fb, s_d};
    int slot;
    const int4 it = kick_item(a, IPT * (int)blockDim.x, slot);
    float rho[IPT];
    float2 nxh[IPT], nyh[IPT], nzh[IPT], nxl[IPT], nyl[IPT], nzl[IPT];  // -Q_i, duplicated
    int gi[IPT];
    float ahx[IPT], ahy[IPT], ahz[IPT], alx[IPT], aly[IPT], alz[IPT];
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        int i = it.x + threadIdx.x + k * blockDim.x;
        gi[k] = i;
        // idle lane: parked far away so its arithmetic stays finite
        float4 p = make_float4(1e18f, 1e18f, 1e18f, 0.0f), l = make_float4(0.f, 0.f, 0.f, -1e30f);
        if (i < it.y) {
            p = a.pos[i];
            l = a.lo[i];
        }
        rho[k] = l.w;
        nxh[k] = make_float2(-p.x, -p.x); nyh[k] = make_float2(-p.y, -p.y);
        nzh[k] = make_float2(-p.z, -p.z); nxl[k] = make_float2(-l.x, -l.x);
        nyl[k] = make_float2(-l.y, -l.y); nzl[k] = make_float2(-l.z, -l.z);
        ahx[k] = ahy[k] = ahz[k] = alx[k] = aly[k] = alz[k] = 0.0f;
    }
    // whether this thread's rows let a window take the form without G m (one and two
    // rows a thread; four have no registers for both forms)
    constexpr bool HAS_UNI = FORCE && IPT <= 2;
    bool i_in = HAS_UNI && a.uniform;
#pragma unroll
    for (int k = 0; k < IPT; ++k) i_in = i_in && (gi[k] >= it.y || uni_range(make_float4(nxh[k].x, nyh[k].x, nzh[k].x, 0.0f)));
    const int i_lo = it.x, i_hi = it.x + (int)(IPT * blockDim.x);
    for (int jt = it.z, n = 0; jt < it.w; jt += n) {
        // windows of at most TILE positions; with far tiles never across the
        // end of a tile (positions 1 + TILE t ..), whose data a window uses
        n = min(TILE, it.w - jt);
        if (a.far_tiles) n = min(n, 1 + ((jt - 1) / TILE + 1) * TILE - jt);
        const int np = (n + 1) >> 1;
        const bool diag = (jt < i_hi) && (jt + n > i_lo);
        // Far tiles (a.far_tiles: the bodies in Morton order, tiles aligned
        // at position 1 + TILE t, their data from k_tile_prep): a warp whose
        // every row lies at least the tile's radius R outside its box takes
        // the one-add separation; every pair is then at least R apart,
        // |o_j| <= R <= r and |d_i| <= 2 r, so that with o_j and d_i each
        // rounded once the separation is within 4 2^-24 r (the row test's
        // own rounding is within its 2% margin).
        bool far = false;
        // quiet (searching kick, a window of another block's tile): no pair
        // of the window can be a candidate, as every row lies farther from
        // the tile's box than its reach and the tile's largest one allow
        // (r^2 >= c_i + c_max, with a 3% and an absolute margin for the FP32
        // box distance): the window takes the plain form, far or near, with
        // no search arithmetic
        bool quiet = false;
        float2 dxi[IPT], dyi[IPT], dzi[IPT];
        float4 m0 = make_float4(0.f, 0.f, 0.f, 0.f);
        bool j_in = true;
        if (a.far_tiles && !diag) {
            const float4 *tm = a.tile + 3 * ((jt - 1) / TILE);
            m0 = tm[0];
            const float4 m1 = tm[1], m2 = tm[2];
            const float R = m0.w;
            j_in = uni_range(m1) && uni_range(m2);
            bool mine = true, calm = true;
#pragma unroll
            for (int k = 0; k < IPT; ++k) {
                const float x = -nxh[k].x, y = -nyh[k].x, z = -nzh[k].x;
                const float ex = fmaxf(fmaxf(m1.x - x, x - m2.x), 0.0f);
                const float ey = fmaxf(fmaxf(m1.y - y, y - m2.y), 0.0f);
                const float ez = fmaxf(fmaxf(m1.z - z, z - m2.z), 0.0f);
                const float d2 = ex * ex + ey * ey + ez * ez;
                mine = mine && (d2 >= 1.02f * R * R);
                if (FLAG)
                    calm = calm && (d2 >= 1.03f * (rho[k] + m1.w) + 1e-9f * (x * x + y * y + z * z));
            }
            far = __all_sync(0xffffffffu, mine);
            if (FLAG) quiet = __all_sync(0xffffffffu, calm);
        }
        // which layouts this CTA's warps need
        const bool any_far = __syncthreads_or(far);
        const bool any_near = __syncthreads_or(!far);
        // one G m for the whole window (and not zero, so that the pad and a
        // massless body are never taken for it)
        const float gm0 = HAS_UNI ? a.pos[jt].w : 0.0f;
        bool same = i_in && j_in && gm0 > 0.0f;
        for (int t = threadIdx.x; t < np; t += blockDim.x) {
            const int j0 = jt + 2 * t;
            const bool two = 2 * t + 1 < n;
            if (any_near) {
                const float4 p0 = a.pos[j0], l0 = a.lo[j0];
                // an odd tail is padded with a massless row far from everything
                float4 p1 = make_float4(2e18f, 2e18f, 2e18f, 0.0f), l1 = make_float4(0.f, 0.f, 0.f, 0.f);
                if (two) {
                    p1 = a.pos[j0 + 1];
                    l1 = a.lo[j0 + 1];
                }
                s_a[t] = make_float4(p0.x, p1.x, p0.y, p1.y);
                same = same && p0.w == gm0 && uni_range(p0) && (!two || (p1.w == gm0 && uni_range(p1)));
                s_b[t] = make_float4(p0.z, p1.z, p0.w, p1.w);
                s_c[t] = make_float4(l0.x, l1.x, l0.y, l1.y);
                s_d[t] = make_float4(l0.z, l1.z, -l0.w, -l1.w);
            }
            if (any_far) {
                const float4 f0 = a.far[j0];
                float4 f1 = make_float4(2e18f, 2e18f, 2e18f, 0.0f);
                float c1 = 0.0f;
                if (two) {
                    f1 = a.far[j0 + 1];
                    c1 = a.lo[j0 + 1].w;
                }
                s_fa[t] = make_float4(f0.x, f1.x, f0.y, f1.y);
                same = same && f0.w == gm0 && (!two || f1.w == gm0);
                s_fb[t] = make_float4(f0.z, f1.z, f0.w, f1.w);
                if (FLAG && !any_near) s_d[t] = make_float4(0.f, 0.f, -a.lo[j0].w, -c1);
            }
        }
        const bool uni = HAS_UNI ? __syncthreads_and(same) : (__syncthreads(), false);
        if (far) {
            // d_i = c - Q_i = (c - x_hi) - x_lo rounded once, duplicated for
            // the packed form
#pragma unroll
            for (int k = 0; k < IPT; ++k) {
                const float dx = ds_add(m0.x, nxh[k].x, nxl[k].x);
                const float dy = ds_add(m0.y, nyh[k].x, nyl[k].x);
                const float dz = ds_add(m0.z, nzh[k].x, nzl[k].x);
                dxi[k] = make_float2(dx, dx);
                dyi[k] = make_float2(dy, dy);
                dzi[k] = make_float2(dz, dz);
            }
        }
        for (int c = 0; c < np; c += FOLD / 2) {
            const int ce = min(c + FOLD / 2, np);
            float2 fx[IPT], fy[IPT], fz[IPT];
            float mind[IPT];
            const auto run = [&](auto u) {
                constexpr bool U = decltype(u)::value;
                if (far && quiet)
                    far_chunk<IPT, false, FORCE, U>(sf, c, ce, dxi, dyi, dzi, fx, fy, fz, mind);
                else if (far)
                    far_chunk<IPT, FLAG, FORCE, U>(sf, c, ce, dxi, dyi, dzi, fx, fy, fz, mind);
                else if (quiet)
                    mixed_chunk<IPT, false, false, FORCE, U>(sp, c, ce, jt, gi, nxh, nyh, nzh, nxl,
                                                             nyl, nzl, fx, fy, fz, mind);
                else if (diag)
                    mixed_chunk<IPT, FLAG, true, FORCE, U>(sp, c, ce, jt, gi, nxh, nyh, nzh, nxl, nyl,
                                                           nzl, fx, fy, fz, mind);
                else
                    mixed_chunk<IPT, FLAG, false, FORCE, U>(sp, c, ce, jt, gi, nxh, nyh, nzh, nxl, nyl,
                                                            nzl, fx, fy, fz, mind);
            };
            float gw = uni ? gm0 : 1.0f;
            for (;;) {
#pragma unroll
                for (int k = 0; k < IPT; ++k) {
                    fx[k] = fy[k] = fz[k] = make_float2(0.0f, 0.0f);
                    mind[k] = 3.0e38f;
                }
                if (!HAS_UNI || gw == 1.0f) {
                    run(std::false_type{});
                    break;
                }
                run(std::integral_constant<bool, HAS_UNI>{});
                if (finite_sums(fx)) break;
                gw = 1.0f;
            }
#pragma unroll
            for (int k = 0; k < IPT; ++k) {
                if (FORCE) {
                    float s, e;
                    two_sum(ahx[k], gw * (fx[k].x + fx[k].y), s, e); ahx[k] = s; alx[k] += e;
                    two_sum(ahy[k], gw * (fy[k].x + fy[k].y), s, e); ahy[k] = s; aly[k] += e;
                    two_sum(ahz[k], gw * (fz[k].x + fz[k].y), s, e); ahz[k] = s; alz[k] += e;
                }
                // only partners j > i become candidates, so a chunk wholly at or
                // below the row needs no record
                const int j1 = jt + min(2 * ce, n);
                if (FLAG && mind[k] < rho[k] && j1 - 1 > gi[k]) push_flag(a, gi[k], jt + 2 * c, j1);
            }
        }
    }
    if (!FORCE) return;
    const int64_t rows = a.rows;
    double *out = a.apart + (int64_t)slot * 3 * rows;
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        if (gi[k] < it.y) {
            out[gi[k]] = (double)ahx[k] + (double)alx[k];
            out[rows + gi[k]] = (double)ahy[k] + (double)aly[k];
            out[2 * rows + gi[k]] = (double)ahz[k] + (double)alz[k];
        }
    }
    if (a.blk_cnt) sum_block_slots<IPT>(a, gi, it.x, it.y);
}

// ---------------------------------------------------------------- pairs once
// The mixed kick of one system in Morton order with each pair formed once: the
// separation, r^2, 1/r and r^-2 serve both bodies (Newton's third law), 14 FMA-pipe
// instructions a far pair of equal masses instead of 2 x 11 (17 instead of 2 x 12 of
// several masses), which is what bounds the kick.
//
// An i-block is 512 consecutive positions, four per thread, a warp's 128
// consecutive ones (compact along the Morton curve, so that more windows are far
// from all of them). Windows of 256 positions past the block stream through shared
// memory as in k_kick_mixed; the block's own two tiles take that kernel's
// one-sided form. For the j side each lane starts at a different j pair of a
// 64-body chunk and holds the pair's sums, which move on with the pair from lane
// to lane (six shuffles a step, against twelve passes of shared memory for a
// read-modify-write there), so after 32 steps lane l holds the sums of pair l over
// the warp's 128 rows: added per step as sums of four, 32 in a row, as the i side
// adds its own. The warps' sums are added as two floats (hi, lo) and converted once:
// added in FP64 they took 54 FP64 instructions per 64 x 512 pairs, a quarter of the
// FMA pipe's time for them (16384 bodies 0.0988 -> 0.0970 ms, 262144 20.15 -> 19.98;
// with the checks of r^-3's range 0.0972 and 20.16).
//
// Work unit: G consecutive i-blocks against a range of rh half tiles (the part
// past each block). Rows get one slot of partial sums per range from their own
// block, and one per group of earlier i-blocks from the j side, added up in the
// group's order by the unit that owns the slot. SymSlots (qym_internal.cuh)
// gives a row's valid slots.
constexpr int SYM_T = 128, SYM_R = 4, SYM_BLK = SYM_T * SYM_R, SYM_W = SYM_T / 32;
static_assert(SYM_BLK == kSymBlock, "i-block of the pair-symmetric kick");

struct SymShared {
    float4 a[TILE / 2], b[TILE / 2], c[TILE / 2], d[TILE / 2];  // near layout (JPairs)
    float4 fa[TILE / 2], fb[TILE / 2];                           // far layout (JFar)
    float4 ip[SYM_BLK], il[SYM_BLK];                             // the i-block's packs
    float acc[6][SYM_BLK];                                       // i sums, two-sum pairs (hi, lo)
    float4 jxy[SYM_W][TILE / 2];                                 // j sums of a warp (x0, x1, y0, y1)
    float2 jz[SYM_W][TILE / 2];
};

// One chunk of 32 j pairs from p0 against the four rows of a thread. FAR: (ix, iy,
// iz) are the rows' d_i = c - Q_i; else -Q_i (hi) with (lx, ly, lz) -Q_i (lo).
// UNI: one G m for the rows and one for the window, multiplied in by the caller.
// Leaves in (jx, jy, jz) the j sums of pair p0 + lane, sign flipped.
template <bool FLAG, bool FORCE, bool UNI, bool FAR>
__device__ __forceinline__ void sym_chunk(const SymShared &S, int p0, const float2 (&ix)[SYM_R],
                                          const float2 (&iy)[SYM_R], const float2 (&iz)[SYM_R],
                                          const float2 (&lx)[SYM_R], const float2 (&ly)[SYM_R],
                                          const float2 (&lz)[SYM_R], const float (&gi)[SYM_R],
                                          float2 (&fx)[SYM_R], float2 (&fy)[SYM_R], float2 (&fz)[SYM_R],
                                          float (&mind)[SYM_R], float2 &jx, float2 &jy, float2 &jz) {
    const int lane = threadIdx.x & 31, next = (lane + 1) & 31;
    jx = jy = jz = make_float2(0.0f, 0.0f);
#pragma unroll 2
    for (int s = 0; s < 32; ++s) {
        const int p = p0 + ((lane + s) & 31);
        float4 A, B, C, D;
        if (FAR) {
            A = S.fa[p];
            B = S.fb[p];
            if (FLAG) D = S.d[p];
        } else {
            A = S.a[p];
            B = S.b[p];
            C = S.c[p];
            D = S.d[p];
        }
        const float2 x = make_float2(A.x, A.y), y = make_float2(A.z, A.w);
        const float2 z = make_float2(B.x, B.y), gm = make_float2(B.z, B.w);
        float2 tx, ty, tz;
#pragma unroll
        for (int k = 0; k < SYM_R; ++k) {
            float2 dx = __fadd2_rn(x, ix[k]), dy = __fadd2_rn(y, iy[k]), dz = __fadd2_rn(z, iz[k]);
            if (!FAR) {
                dx = __fadd2_rn(dx, __fadd2_rn(make_float2(C.x, C.y), lx[k]));
                dy = __fadd2_rn(dy, __fadd2_rn(make_float2(C.z, C.w), ly[k]));
                dz = __fadd2_rn(dz, __fadd2_rn(make_float2(D.x, D.y), lz[k]));
            }
            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
            if (FORCE) {
                const float2 ri = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
                const float2 w = __fmul2_rn(ri, ri);
                const float2 si = __fmul2_rn(UNI ? ri : __fmul2_rn(gm, ri), w);
                const float2 sj = UNI ? si : __fmul2_rn(__fmul2_rn(make_float2(gi[k], gi[k]), ri), w);
                fx[k] = __ffma2_rn(si, dx, fx[k]);
                fy[k] = __ffma2_rn(si, dy, fy[k]);
                fz[k] = __ffma2_rn(si, dz, fz[k]);
                tx = k ? __ffma2_rn(sj, dx, tx) : __fmul2_rn(sj, dx);
                ty = k ? __ffma2_rn(sj, dy, ty) : __fmul2_rn(sj, dy);
                tz = k ? __ffma2_rn(sj, dz, tz) : __fmul2_rn(sj, dz);
            }
            if (FLAG) {
                const float2 t = __fadd2_rn(r2, make_float2(D.z, D.w));
                mind[k] = fmin3(mind[k], t.x, t.y);
            }
        }
        if (FORCE) {
            jx = __fadd2_rn(jx, tx);
            jy = __fadd2_rn(jy, ty);
            jz = __fadd2_rn(jz, tz);
            // the next step takes the pair the lane above has just had
            jx.x = __shfl_sync(0xffffffffu, jx.x, next);
            jx.y = __shfl_sync(0xffffffffu, jx.y, next);
            jy.x = __shfl_sync(0xffffffffu, jy.x, next);
            jy.y = __shfl_sync(0xffffffffu, jy.y, next);
            jz.x = __shfl_sync(0xffffffffu, jz.x, next);
            jz.y = __shfl_sync(0xffffffffu, jz.y, next);
        }
    }
}

template <bool FLAG, bool FORCE>
__global__ void __launch_bounds__(SYM_T, 4) k_kick_sym(KickArgs a) {
    chain_wait();
    extern __shared__ __align__(16) unsigned char g_symsmem[];
    SymShared &S = *reinterpret_cast<SymShared *>(g_symsmem);
    const JPairs sp{S.a, S.b, S.c, S.d};
    const int4 u = a.items[blockIdx.x];  // i-blocks [x, y), half tiles [z, w)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int npos = (int)a.rows;
    const int64_t rows = a.rows;
    const int i_of = warp * 32 * SYM_R + lane;  // row k of this thread: block start + i_of + 32 k
    for (int blk = u.x; blk < u.y; ++blk) {
        const int i_lo = 1 + blk * SYM_BLK, i_hi = i_lo + SYM_BLK;
        const int h0 = max(u.z, 4 * blk);  // from the block's own half tiles on
        if (h0 >= u.w) continue;
        int gi[SYM_R];
        float rho[SYM_R], gmi[SYM_R];
        bool i_same = true;
        const float gi0 = a.pos[i_lo].w;
        __syncthreads();  // the packs of the block before are no longer read
#pragma unroll
        for (int k = 0; k < SYM_R; ++k) {
            const int o = i_of + 32 * k, i = i_lo + o;
            gi[k] = i;
            // idle row: parked far away so its arithmetic stays finite
            float4 p = make_float4(1e18f, 1e18f, 1e18f, 0.0f), l = make_float4(0.f, 0.f, 0.f, -1e30f);
            if (i < npos) {
                p = a.pos[i];
                l = a.lo[i];
            }
            i_same = i_same && p.w == gi0 && uni_range(p);
            rho[k] = l.w;
            gmi[k] = p.w;
            S.ip[o] = p;
            S.il[o] = l;
#pragma unroll
            for (int c = 0; c < 6; ++c) S.acc[c][o] = 0.0f;
        }
        const bool i_uni = __syncthreads_and(i_same) && gi0 > 0.0f;
        for (int jt = 1 + h0 * (TILE / 2), n = 0; jt < npos && jt < 1 + u.w * (TILE / 2); jt += n) {
            // windows to the end of the tile, the range or the system
            n = min(min(1 + ((jt - 1) / TILE + 1) * TILE, 1 + u.w * (TILE / 2)), npos) - jt;
            const int np = (n + 1) >> 1;
            const bool diag = jt < i_hi;
            bool far = false, quiet = false, j_in = true;
            float4 m0 = make_float4(0.f, 0.f, 0.f, 0.f);
            if (!diag) {
                const float4 *tm = a.tile + 3 * ((jt - 1) / TILE);
                m0 = tm[0];
                const float4 m1 = tm[1], m2 = tm[2];
                j_in = uni_range(m1) && uni_range(m2);
                bool mine = true, calm = true;
#pragma unroll
                for (int k = 0; k < SYM_R; ++k) {
                    const float4 P = S.ip[i_of + 32 * k];
                    const float ex = fmaxf(fmaxf(m1.x - P.x, P.x - m2.x), 0.0f);
                    const float ey = fmaxf(fmaxf(m1.y - P.y, P.y - m2.y), 0.0f);
                    const float ez = fmaxf(fmaxf(m1.z - P.z, P.z - m2.z), 0.0f);
                    const float d2 = ex * ex + ey * ey + ez * ez;
                    mine = mine && (d2 >= 1.02f * m0.w * m0.w);
                    if (FLAG)
                        calm = calm && (d2 >= 1.03f * (rho[k] + m1.w) +
                                                  1e-9f * (P.x * P.x + P.y * P.y + P.z * P.z));
                }
                far = __all_sync(0xffffffffu, mine);
                if (FLAG) quiet = __all_sync(0xffffffffu, calm);
            }
            const bool any_far = __syncthreads_or(far);
            const bool any_near = __syncthreads_or(!far);
            const float gm0 = FORCE ? a.pos[jt].w : 0.0f;
            bool same = j_in && gm0 > 0.0f;
            // (padded to whole chunks of 32 pairs with massless bodies far from everything)
            for (int t = tid; t < ((np + 31) & ~31); t += SYM_T) {
                const int j0 = jt + 2 * t;
                const bool one = 2 * t < n, two = 2 * t + 1 < n;
                const float4 pad = make_float4(2e18f, 2e18f, 2e18f, 0.0f);
                const float4 pad_l = make_float4(0.f, 0.f, 0.f, -1e30f);
                const float4 l0 = one && (any_near || FLAG) ? a.lo[j0] : pad_l;
                const float4 l1 = two && (any_near || FLAG) ? a.lo[j0 + 1] : pad_l;
                if (any_near) {
                    const float4 p0 = one ? a.pos[j0] : pad, p1 = two ? a.pos[j0 + 1] : pad;
                    same = same && (!one || p0.w == gm0) && (!two || p1.w == gm0);
                    S.a[t] = make_float4(p0.x, p1.x, p0.y, p1.y);
                    S.b[t] = make_float4(p0.z, p1.z, p0.w, p1.w);
                    S.c[t] = make_float4(l0.x, l1.x, l0.y, l1.y);
                }
                S.d[t] = make_float4(l0.z, l1.z, -l0.w, -l1.w);
                if (any_far) {
                    const float4 f0 = one ? a.far[j0] : pad, f1 = two ? a.far[j0 + 1] : pad;
                    same = same && (!one || f0.w == gm0) && (!two || f1.w == gm0);
                    S.fa[t] = make_float4(f0.x, f1.x, f0.y, f1.y);
                    S.fb[t] = make_float4(f0.z, f1.z, f0.w, f1.w);
                }
            }
            const bool j_uni = FORCE ? __syncthreads_and(same) : (__syncthreads(), false);
            const bool uni = j_uni && i_uni && !diag;
            float2 ix[SYM_R], iy[SYM_R], iz[SYM_R], lx[SYM_R], ly[SYM_R], lz[SYM_R];
#pragma unroll
            for (int k = 0; k < SYM_R; ++k) {
                const float4 P = S.ip[i_of + 32 * k], L = S.il[i_of + 32 * k];
                // far: d_i = c - Q_i = (c - x_hi) - x_lo rounded once
                const float x = far ? ds_add(m0.x, -P.x, -L.x) : -P.x;
                const float y = far ? ds_add(m0.y, -P.y, -L.y) : -P.y;
                const float z = far ? ds_add(m0.z, -P.z, -L.z) : -P.z;
                ix[k] = make_float2(x, x);
                iy[k] = make_float2(y, y);
                iz[k] = make_float2(z, z);
                lx[k] = make_float2(-L.x, -L.x);
                ly[k] = make_float2(-L.y, -L.y);
                lz[k] = make_float2(-L.z, -L.z);
            }
            for (int c = 0; c < np; c += 32) {
                float2 fx[SYM_R], fy[SYM_R], fz[SYM_R], jx, jy, jz;
                float mind[SYM_R];
                const auto run = [&](auto U, auto F, auto Q) {
                    sym_chunk<FLAG && decltype(Q)::value, FORCE, decltype(U)::value, decltype(F)::value>(
                        S, c, ix, iy, iz, lx, ly, lz, gmi, fx, fy, fz, mind, jx, jy, jz);
                };
                using T1 = std::true_type;
                using T0 = std::false_type;
                bool u = uni && (quiet || !FLAG);
                for (;;) {
#pragma unroll
                    for (int k = 0; k < SYM_R; ++k) {
                        fx[k] = fy[k] = fz[k] = make_float2(0.0f, 0.0f);
                        mind[k] = 3.0e38f;
                    }
                    if (diag) {
                        mixed_chunk<SYM_R, FLAG, true, FORCE, false>(sp, c, min(c + 32, np), jt, gi, ix, iy,
                                                                     iz, lx, ly, lz, fx, fy, fz, mind);
                    } else if (far && (quiet || !FLAG)) {
                        if (u) run(T1{}, T1{}, T0{}); else run(T0{}, T1{}, T0{});
                    } else if (far) {
                        run(T0{}, T1{}, T1{});
                    } else if (quiet || !FLAG) {
                        if (u) run(T1{}, T0{}, T0{}); else run(T0{}, T0{}, T0{});
                    } else {
                        run(T0{}, T0{}, T1{});
                    }
                    if (!FORCE || !u || __all_sync(0xffffffffu, finite_sums(fx))) break;
                    u = false;
                }
                if (FORCE && !diag) {
                    const float v = u ? -gi0 : -1.0f;
                    S.jxy[warp][c + lane] = make_float4(v * jx.x, v * jx.y, v * jy.x, v * jy.y);
                    S.jz[warp][c + lane] = make_float2(v * jz.x, v * jz.y);
                }
                const float g = u ? gm0 : 1.0f;
#pragma unroll
                for (int k = 0; k < SYM_R; ++k) {
                    const int o = i_of + 32 * k;
                    if (FORCE) {
                        float s, e;
                        two_sum(S.acc[0][o], g * (fx[k].x + fx[k].y), s, e); S.acc[0][o] = s; S.acc[3][o] += e;
                        two_sum(S.acc[1][o], g * (fy[k].x + fy[k].y), s, e); S.acc[1][o] = s; S.acc[4][o] += e;
                        two_sum(S.acc[2][o], g * (fz[k].x + fz[k].y), s, e); S.acc[2][o] = s; S.acc[5][o] += e;
                    }
                    // only partners j > i become candidates
                    const int j1 = jt + min(2 * c + 64, n);
                    if (FLAG && mind[k] < rho[k] && j1 - 1 > gi[k]) push_flag(a, gi[k], jt + 2 * c, j1);
                }
            }
            __syncthreads();  // the window is no longer read; every warp's j sums are there
            if (FORCE && !diag) {
                // slot of the group's j sums: the group's first block stores, the others add
                double *const out = a.apart + (int64_t)(a.sym.nc + blk / a.sym.G) * 3 * rows + jt;
                const bool first = blk == u.x;
                for (int t = tid; t < np; t += SYM_T) {
                    const bool two = 2 * t + 1 < n;
                    float h[6], l[6];
#pragma unroll
                    for (int w = 0; w < SYM_W; ++w) {
                        const float4 xy = S.jxy[w][t];
                        const float2 z = S.jz[w][t];
                        const float x[6] = {xy.x, xy.y, xy.z, xy.w, z.x, z.y};
#pragma unroll
                        for (int c = 0; c < 6; ++c) {
                            float e = 0.0f;
                            if (w) two_sum(h[c], x[c], h[c], e); else h[c] = x[c];
                            l[c] = w > 1 ? l[c] + e : e;
                        }
                    }
                    double v[6];
#pragma unroll
                    for (int c = 0; c < 6; ++c) v[c] = (double)h[c] + (double)l[c];
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        double *const o = out + c * rows + 2 * t;
                        o[0] = first ? v[2 * c] : o[0] + v[2 * c];
                        if (two) o[1] = first ? v[2 * c + 1] : o[1] + v[2 * c + 1];
                    }
                }
            }
        }
        if (FORCE) {
            double *const out = a.apart + (int64_t)(u.z / a.sym.rh) * 3 * rows;
#pragma unroll
            for (int k = 0; k < SYM_R; ++k) {
                const int o = i_of + 32 * k;
                if (gi[k] < npos) {
                    out[gi[k]] = (double)S.acc[0][o] + (double)S.acc[3][o];
                    out[rows + gi[k]] = (double)S.acc[1][o] + (double)S.acc[4][o];
                    out[2 * rows + gi[k]] = (double)S.acc[2][o] + (double)S.acc[5][o];
                }
            }
        }
    }
}

// Units of the pair-symmetric kick of nb bodies with at most max_slots slots a
// row: about 2000 (four CTAs on each SM, several waves), ranges and groups of the
// same length where the slots allow; no shape (G = 0, no slots) where they do not.
SymShape sym_shape(int64_t nb, int64_t max_slots) {
    SymShape y;
    const int64_t nblk = (nb + SYM_BLK - 1) / SYM_BLK, nhalf = (nb + TILE / 2 - 1) / (TILE / 2);
    y.G = (int32_t)std::max<int64_t>(1, (nblk + 63) / 64);
    const int64_t ng = (nblk + y.G - 1) / y.G;
    const int64_t want = std::min<int64_t>(128, std::max<int64_t>(64, 4096 / ng));
    y.rh = (int32_t)std::max<int64_t>(1, (nhalf + want - 1) / want);
    y.nc = (int32_t)((nhalf + y.rh - 1) / y.rh);
    y.splits = (int32_t)(y.nc + ng);
    return y.splits <= max_slots ? y : SymShape();
}

void sym_items_host(int64_t nb, const SymShape &y, std::vector<int4> &items) {
    const int64_t nblk = (nb + SYM_BLK - 1) / SYM_BLK;
    items.clear();
    for (int64_t b = 0; b < nblk; b += y.G)
        for (int64_t c = 4 * b / y.rh; c < y.nc; ++c)
            items.push_back(make_int4((int)b, (int)std::min<int64_t>(b + y.G, nblk), (int)(c * y.rh),
                                      (int)((c + 1) * y.rh)));
}

template <bool FLAG, bool FORCE>
static cudaError_t launch_sym(const KickArgs &a, int nitems, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_kick_sym<FLAG, FORCE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(SymShared));
    if (e != cudaSuccess) return e;
    return launch_chain(k_kick_sym<FLAG, FORCE>, nitems, SYM_T, sizeof(SymShared), st, a);
}

// Exact test of the flagged chunks, one warp per entry, lane l on the j rows
// j0 + l and j0 + 32 + l: candidates (i, j), i < j, with r^2 < c_i + c_j, the
// separation formed from the same split positions in the same order as the
// kick forms it, so the candidate set is the kick's own. Entries hold
// positions of the packs' order (each pair once: from the smaller position);
// candidates are rows. The last CTA to finish resets the entry counter for
// the next search kick.
__global__ void __launch_bounds__(256) k_flag_chunks(KickArgs a, unsigned long long *done) {
    chain_wait();
    unsigned long long n = *(volatile unsigned long long *)a.nfchunk;
    if (n > (unsigned long long)a.max_fchunk) n = a.max_fchunk;
    const int lane = threadIdx.x & 31;
    const unsigned long long warps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    for (unsigned long long e = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
         e < n; e += warps) {
        const int4 f = a.fchunk[e];
        const float4 pi = a.pos[f.x], li = a.lo[f.x];
        for (int j = f.y + lane; j < f.z; j += 32) {
            if (j <= f.x) continue;
            const float4 pj = a.pos[j], lj = a.lo[j];
            const float dx = (pi.x - pj.x) + (li.x - lj.x);
            const float dy = (pi.y - pj.y) + (li.y - lj.y);
            const float dz = (pi.z - pj.z) + (li.z - lj.z);
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            if (r2 < li.w + lj.w) {
                // positions of the kick's order -> rows, smaller row first
                int ri = f.x, rj = j;
                if (a.perm) {
                    ri = a.perm[ri];
                    rj = a.perm[rj];
                }
                push_candidate(a, min(ri, rj), max(ri, rj));
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(done, 1ull) == gridDim.x - 1) {
            *a.nfchunk = 0;
            *done = 0;
        }
    }
}

// ---------------------------------------------------------------- FP64 form
// G m_j / r^3 of a pair in FP64, where the float form does not hold
__device__ __noinline__ double weight_fp64(double dx, double dy, double dz, double gm) {
    const long long ux = __double_as_longlong(dx), uy = __double_as_longlong(dy);
    const long long uz = __double_as_longlong(dz);
    // a body and itself, or a massless partner: no FP64 instruction
    if (((ux | uy | uz) << 1) == 0 || (__double_as_longlong(gm) << 1) == 0) return 0.0;
    const double r2 = dx * dx + dy * dy + dz * dz;
    const double ri = rsqrt(r2);
    const double s = gm * (ri * ri) * ri;
    return (r2 > 0.0) ? s : 0.0;
}

// The FP64 kick. The separations, r^2 and G m / r^3 of a pair are formed to FP64
// accuracy on the FP32 pipes (pair64.cuh, about 400 issue slots); beside them the
// FP64 pipe, one warp instruction per ~19 cycles and SM, forms the separation
// again and sums the pair's acceleration, six instructions where the plain form
// has 22: 10240 bodies take 1.20 ms, 107 cycles of an SM per warp of pairs, both
// pipes full (4.08 ms before; assembling the separation's doubles from the floats
// instead of three FP64 subtractions, 1.34 ms). Rows and partners are split into
// three floats once per CTA and tile, scaled by powers of two; pairs outside the
// float range take plain FP64.
template <int IPT, bool FLAG, bool FORCE>
__global__ void __launch_bounds__(256) k_kick_fp64(KickArgs a) {
    chain_wait();
    __shared__ D4 s_q[TILE];
    __shared__ float4 s_h[TILE], s_m[TILE], s_l[TILE];  // (x, y, z, G m) in three parts
    __shared__ float s_rho[TILE];
    __shared__ int s_hi[2][8];
    int slot;
    const int4 it = kick_item(a, IPT * (int)blockDim.x, slot);
    const int64_t rows = a.rows;
    const double G = a.G;
    double xi[IPT], yi[IPT], zi[IPT], ax[IPT], ay[IPT], az[IPT];
    float rho[IPT];
    int gi[IPT];
    int hl = 0, hw = 0;
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        const int i = it.x + threadIdx.x + k * blockDim.x;
        gi[k] = i;
        const int r = min(i, it.y - 1);  // an idle lane repeats the last row
        xi[k] = a.q[r]; yi[k] = a.q[rows + r]; zi[k] = a.q[2 * rows + r];
        rho[k] = FLAG && i < it.y ? a.lo[i].w : -1e30f;
        hl = max(hl, max(p64::hi_abs(xi[k]), max(p64::hi_abs(yi[k]), p64::hi_abs(zi[k]))));
        ax[k] = ay[k] = az[k] = 0.0;
    }
    if (it.z + (int)threadIdx.x < it.w) hw = p64::hi_abs(G * a.m[it.z + threadIdx.x]);
    hl = __reduce_max_sync(0xffffffffu, hl);
    hw = __reduce_max_sync(0xffffffffu, hw);
    if ((threadIdx.x & 31) == 0) {
        s_hi[0][threadIdx.x >> 5] = hl;
        s_hi[1][threadIdx.x >> 5] = hw;
    }
    __syncthreads();
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        hl = max(hl, s_hi[0][w]);
        hw = max(hw, s_hi[1][w]);
    }
    const p64::Scale sc(hl, hw);
    const uint64_t bias = sc.bias(3);
    // r^2 back to the caller's units for the encounter search
    const bool r2_ok = sc.kb >= -60 && sc.kb <= 60;
    const float r2u = r2_ok ? __int_as_float((127 + 2 * sc.kb) << 23) : 1.0f;
    p64::F3 px[IPT], py[IPT], pz[IPT];
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        px[k] = p64::split3(xi[k] * sc.len);
        py[k] = p64::split3(yi[k] * sc.len);
        pz[k] = p64::split3(zi[k] * sc.len);
    }
    for (int jt = it.z; jt < it.w; jt += TILE) {
        const int n = min(TILE, it.w - jt);
        __syncthreads();
        for (int t = threadIdx.x; t < n; t += blockDim.x) {
            const int j = jt + t;
            const D4 p{a.q[j], a.q[rows + j], a.q[2 * rows + j], G * a.m[j]};
            const p64::F3 x = p64::split3(p.x * sc.len), y = p64::split3(p.y * sc.len);
            const p64::F3 z = p64::split3(p.z * sc.len), g = p64::split3(p.w * sc.wt);
            s_q[t] = p;
            s_h[t] = make_float4(x.h, y.h, z.h, g.h);
            s_m[t] = make_float4(x.m, y.m, z.m, g.m);
            s_l[t] = make_float4(x.l, y.l, z.l, g.l);
            if (FLAG) s_rho[t] = a.lo[j].w;
        }
        __syncthreads();
#pragma unroll 1
        for (int j = 0; j < n; ++j) {
            const D4 p = s_q[j];
            const float4 H = s_h[j], M = s_m[j], L = s_l[j];
            const bool g_ok = p64::g_fits(H.w);
#pragma unroll
            for (int k = 0; k < IPT; ++k) {
                const p64::F3 r2 = p64::norm2(p64::diff(px[k], p64::F3{H.x, M.x, L.x}),
                                              p64::diff(py[k], p64::F3{H.y, M.y, L.y}),
                                              p64::diff(pz[k], p64::F3{H.z, M.z, L.z}));
                const bool fits = sc.ok && p64::r2_fits(r2.h);
                const double dx = xi[k] - p.x, dy = yi[k] - p.y, dz = zi[k] - p.z;
                if (FORCE) {
                    double s;
                    if (!(p64::g_over_r3(p64::F3{H.w, M.w, L.w}, r2, rsqrt_ftz(r2.h), bias, s) &&
                          fits && g_ok))
                        s = weight_fp64(dx, dy, dz, p.w);
                    ax[k] -= s * dx;
                    ay[k] -= s * dy;
                    az[k] -= s * dz;
                }
                if (FLAG) {
                    float r2f = __fadd_rn(r2.h, r2.m) * r2u;
                    if (!(fits && r2_ok)) r2f = (float)(dx * dx + dy * dy + dz * dz);
                    if (r2f < rho[k] + s_rho[j]) {
                        int gj = jt + j;
                        if (gi[k] < gj) push_candidate(a, gi[k], gj);
                    }
                }
            }
        }
    }
    if (!FORCE) return;
    double *out = a.apart + (int64_t)slot * 3 * rows;
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        if (gi[k] < it.y) {
            out[gi[k]] = ax[k];
            out[rows + gi[k]] = ay[k];
            out[2 * rows + gi[k]] = az[k];
        }
    }
    if (a.blk_cnt) sum_block_slots<IPT>(a, gi, it.x, it.y);
}

// ---------------------------------------------------------------- items
// Items for a batch: for each system (bodies are rows lo+1 .. hi-1), i-blocks
// of threads*ipt rows times `splits` contiguous j-ranges. Every (i-block,
// split) pair gets an item, even when its j-range is empty, so every slot of
// every row is written. Only rows in [i_lo, i_hi) get i-blocks (a rank's own
// rows when a system's step is split over several GPUs); the j-ranges always
// cover the whole system, so a row's partial sums do not depend on the range.
static int64_t items_i_begin(int64_t b0, int64_t i_lo) { return b0 > i_lo ? b0 : i_lo; }
static int64_t items_i_end(int64_t b1, int64_t i_hi) { return b1 < i_hi ? b1 : i_hi; }

int32_t kick_items_count(const int64_t *offsets, int32_t nsys, const KickTune &t, int64_t i_lo,
                         int64_t i_hi) {
    int64_t tot = 0;
    const int64_t ti = (int64_t)t.threads * t.ipt;
    for (int32_t s = 0; s < nsys; ++s) {
        const int64_t a = items_i_begin(offsets[s] + 1, i_lo), b = items_i_end(offsets[s + 1], i_hi);
        const int64_t nb = b - a;
        if (nb > 0) tot += ((nb + ti - 1) / ti) * t.splits;
    }
    return (int32_t)tot;
}

void kick_items_host(const int64_t *offsets, int32_t nsys, const KickTune &t, int4 *items,
                     int32_t *slots, int32_t *nitems, int32_t *splits_used, int32_t max_items,
                     int64_t i_lo, int64_t i_hi, int32_t align) {
    const int64_t ti = (int64_t)t.threads * t.ipt;
    int32_t n = 0;
    for (int32_t s = 0; s < nsys; ++s) {
        int64_t b0 = offsets[s] + 1, b1 = offsets[s + 1];
        int64_t nb = b1 - b0;
        int64_t chunk = (nb + t.splits - 1) / t.splits;
        chunk = (chunk + align - 1) / align * align;  // j-ranges start on half tiles (one inside a tile takes that tile's far data)
        const int64_t ia = items_i_begin(b0, i_lo), ib = items_i_end(b1, i_hi);
        for (int64_t i0 = ia; i0 < ib; i0 += ti) {
            int64_t i1 = i0 + ti < ib ? i0 + ti : ib;
            for (int32_t sp = 0; sp < t.splits; ++sp) {
                int64_t j0 = b0 + sp * chunk, j1 = j0 + chunk;
                if (j0 > b1) j0 = b1;
                if (j1 > b1) j1 = b1;
                if (n < max_items) {
                    items[n] = make_int4((int)i0, (int)i1, (int)j0, (int)j1);
                    slots[n] = sp;
                }
                ++n;
            }
        }
    }
    *nitems = n;
    *splits_used = t.splits;
}

// Default launch shape for i-blocks of nb bodies in all (nbmax in the largest
// system), at most max_splits ranges per i-block.
// Mixed: one or two rows per thread and j-ranges of one tile (one row, half a
// tile and less for small systems, where a CTA's walk is the launch's length),
// as long as the partial slots stay few: 64 a row, and about 12288 CTAs. Many
// short CTAs even out the near and far tiles and the last wave: 16384 bodies
// take 0.134 ms in 64 ranges, 0.150 in 16, 0.188 in 10 (four CTAs per SM);
// 262144 bodies 26.9 ms in 12, 29.6 in one; 4096 bodies 20.5 us in 32, 1024
// bodies 6.2 us in 32 (14.4 in 4); each a twelfth less since windows of one G m
// leave its multiplication to the fold.
// FP64: as many CTAs as fit the GPU at once (eight of 128 threads per SM),
// since a pair takes some 300 issue slots: 10240 bodies on 80 i-blocks fill
// the chip with 15 splits; small systems take splits of at least 8 rows, of 4
// while that makes at most 256 CTAs (a 260-body kick is one warp's walk over its
// j-range: 185 us in one range in plain FP64, 14 us in ranges of 16, 6.8 in ranges
// of 8, 5.2 in ranges of 4; 600 bodies 9.5 us in 75 ranges, 12.6 in 128).
KickTune default_kick_tune(int64_t iblocks_nb, int64_t nbmax, int prec, int64_t max_splits) {
    KickTune t;
    const bool mixed = prec == QYM_KICK_MIXED;
    t.threads = 128;
    t.ipt = mixed && iblocks_nb > 6144 ? 2 : 1;
    const int64_t ib = std::max<int64_t>(1, (iblocks_nb + t.threads * t.ipt - 1) / (t.threads * t.ipt));
    int64_t sp;
    if (mixed) {
        const int64_t range = nbmax > 6144 ? 256 : (nbmax > 2048 ? 128 : 32);
        sp = std::min<int64_t>({(nbmax + range - 1) / range, 12288 / ib, 64});
    } else {
        sp = std::min<int64_t>({8 * 152 / ib, std::max(nbmax / 8, std::min(nbmax / 4, 256 / ib)), 128});
    }
    t.splits = (int32_t)std::max<int64_t>(1, std::min(sp, max_splits));
    return t;
}

// One-sided kicks: chained where a CTA's walk is short (the launch counts), a plain
// launch from 2^18 pairs a CTA (some 20 us): chained CTAs settle on the SMs beside the
// kernel before, two and three to some of them, and with few long CTAs that stays the
// kick's length. 16384 bodies: 128 threads x 4 rows in 4 ranges 0.254 ms, chained
// 0.363; 256 x 2 in 4 0.199 and 0.326; 3000 bodies, 128 x 2 in 8: 18.9 and 16.5 us.
constexpr int64_t kPlainPairs = 1 << 18;
template <class... P>
static cudaError_t launch_kick(void (*kernel)(P...), int nitems, int threads, int ipt, int64_t nj,
                               cudaStream_t st, const KickArgs &a) {
    if (nj * threads * ipt < kPlainPairs) return launch_chain(kernel, nitems, threads, 0, st, a);
    kernel<<<nitems, threads, 0, st>>>(a);
    return cudaGetLastError();
}

template <bool FLAG, bool FORCE>
static cudaError_t launch_mixed(const KickArgs &a, int nitems, int threads, int ipt, int64_t nj,
                                cudaStream_t st) {
    switch (ipt) {
    case 1: return launch_kick(k_kick_mixed<1, FLAG, FORCE>, nitems, threads, ipt, nj, st, a);
    case 2: return launch_kick(k_kick_mixed<2, FLAG, FORCE>, nitems, threads, ipt, nj, st, a);
    case 4: return launch_kick(k_kick_mixed<4, FLAG, FORCE>, nitems, threads, ipt, nj, st, a);
    default: return cudaErrorInvalidValue;
    }
}

template <bool FLAG, bool FORCE>
static cudaError_t launch_f64(const KickArgs &a, int nitems, int threads, int ipt, int64_t nj,
                              cudaStream_t st) {
    return ipt == 1 ? launch_kick(k_kick_fp64<1, FLAG, FORCE>, nitems, threads, ipt, nj, st, a)
                    : launch_kick(k_kick_fp64<2, FLAG, FORCE>, nitems, threads, ipt, nj, st, a);
}

// Per tile of TILE consecutive positions (from position 1; the bodies in
// Morton order): the bounding box of the hi parts, a reference point c at its
// middle, a radius R >= max |Q_j - c| (rounded up, with room for the lo parts
// and the rounding of c), the largest crude-search reach c_j of its bodies
// (tile[1].w), and each body's offset o_j = Q_j - c, rounded once (two-sum of
// x_hi - c, then x_lo added), beside its G m. One CTA of TILE threads per tile;
// (P, L): the packs of position p of this thread.
__device__ __forceinline__ void tile_prep(bool act, int64_t p, const float4 &P, const float4 &L,
                                          float4 *far, float4 *tile) {
    __shared__ float s_m[TILE / 32][7];
    __shared__ float s_c[3];
    // (m[6]: minus the largest search reach c of the tile's bodies)
    float m[7] = {act ? P.x : 3e38f, act ? P.y : 3e38f, act ? P.z : 3e38f,
                  act ? -P.x : 3e38f, act ? -P.y : 3e38f, act ? -P.z : 3e38f,
                  act ? -L.w : 3e38f};
#pragma unroll
    for (int q = 0; q < 7; ++q) m[q] = warp_min(m[q]);
    if ((threadIdx.x & 31) == 0)
        for (int q = 0; q < 7; ++q) s_m[threadIdx.x >> 5][q] = m[q];
    __syncthreads();
    if (threadIdx.x == 0) {
        float b[7];
        for (int q = 0; q < 7; ++q) {
            b[q] = s_m[0][q];
            for (int w = 1; w < TILE / 32; ++w) b[q] = fminf(b[q], s_m[w][q]);
        }
        float hr2 = 0.0f, big = 0.0f, c[3];
        for (int q = 0; q < 3; ++q) {
            const float l = b[q], h = -b[q + 3];
            c[q] = 0.5f * (l + h);
            const float e = fmaxf(__fsub_ru(h, c[q]), __fsub_ru(c[q], l));
            hr2 = __fmaf_ru(e, e, hr2);
            big = fmaxf(big, fmaxf(fabsf(l), fabsf(h)));
            s_c[q] = c[q];
        }
        const float R = __fadd_ru(__fsqrt_ru(hr2), 4.0f * 1.1920929e-7f * big);
        float4 *t = tile + 3 * blockIdx.x;
        t[0] = make_float4(c[0], c[1], c[2], R);
        t[1] = make_float4(b[0], b[1], b[2], fmaxf(-b[6], 0.0f));
        t[2] = make_float4(-b[3], -b[4], -b[5], 0.0f);
    }
    __syncthreads();
    if (act)
        far[p] = make_float4(ds_add(P.x, -s_c[0], L.x), ds_add(P.y, -s_c[1], L.y),
                             ds_add(P.z, -s_c[2], L.z), P.w);
}

__global__ void __launch_bounds__(TILE) k_tile_prep(int64_t npos, const float4 *pos,
                                                    const float4 *lo, float4 *far, float4 *tile) {
    chain_wait();
    const int64_t p = 1 + (int64_t)blockIdx.x * TILE + threadIdx.x;
    const bool act = p < npos;
    float4 P = make_float4(0.f, 0.f, 0.f, 0.f), L = P;
    if (act) {
        P = pos[p];
        L = lo[p];
    }
    tile_prep(act, p, P, L, far, tile);
}

cudaError_t launch_kick_tiles(const Dev &d, int prec, int flag, double G, int threads, int ipt,
                              cudaStream_t st) {
    if (d.nitems <= 0) return cudaSuccess;
    KickArgs a;
    a.items = d.items;
    a.slots = d.item_slot;
    a.pos = d.pk_pos;
    a.lo = d.pk_lo;
    a.q = d.q;
    a.m = d.m;
    a.G = G;
    a.apart = d.apart;
    a.rows = d.rows;
    a.cand = d.cand;
    a.max_cand = d.max_cand;
    a.ncand = d.ctr + C_NCAND;
    a.fchunk = d.fchunk;
    a.max_fchunk = d.max_fchunk;
    a.nfchunk = d.ctr + C_NFCHUNK;
    a.status = d.status;
    a.far_tiles = (d.perm && d.far && prec == QYM_KICK_MIXED) ? 1 : 0;
    a.perm = d.perm;
    a.far = d.far;
    a.tile = d.tile;
    a.blk_cnt = d.kick_cnt;
    a.splits = d.splits;
    a.chunk = d.item_chunk;
    a.parts = d.item_parts;
    a.uniform = !d.batch;
    if (a.far_tiles && !d.tiles_ready) {
        const int64_t ntiles = (d.rows - 1 + TILE - 1) / TILE;
        launch_chain(k_tile_prep, (unsigned)ntiles, TILE, 0, st, d.rows, d.pk_pos, d.pk_lo, d.far, d.tile);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (flag != KICK_FORCE && flag != KICK_SEARCH && flag != KICK_SEARCH_ONLY)
        return cudaErrorInvalidValue;
    const int64_t nj = d.rows / std::max(1, d.nsys) / d.splits;  // j rows of a CTA, about
    if (prec == QYM_KICK_MIXED) {
        const bool sym = d.sym.G > 0;
        if (sym) {
            a.items = d.sym_items;
            a.sym = d.sym;
        }
        if (flag == KICK_FORCE)
            return sym ? launch_sym<false, true>(a, d.sym_nitems, st)
                       : launch_mixed<false, true>(a, d.nitems, threads, ipt, nj, st);
        cudaError_t e = flag == KICK_SEARCH
                            ? (sym ? launch_sym<true, true>(a, d.sym_nitems, st)
                                   : launch_mixed<true, true>(a, d.nitems, threads, ipt, nj, st))
                            : (sym ? launch_sym<true, false>(a, d.sym_nitems, st)
                                   : launch_mixed<true, false>(a, d.nitems, threads, ipt, nj, st));
        if (e) return e;
        // about one entry per row (its own chunk) plus the close pairs
        int64_t blocks = (d.rows + 63) / 64;
        if (blocks > 4 * 152) blocks = 4 * 152;
        if (blocks < 1) blocks = 1;
        launch_chain(k_flag_chunks, (int)blocks, 256, 0, st, a, d.ctr + C_FCDONE);
        return cudaGetLastError();
    }
    if (flag == KICK_FORCE) return launch_f64<false, true>(a, d.nitems, threads, ipt, nj, st);
    return flag == KICK_SEARCH ? launch_f64<true, true>(a, d.nitems, threads, ipt, nj, st)
                               : launch_f64<true, false>(a, d.nitems, threads, ipt, nj, st);
}

// ---------------------------------------------------------------- single system
// Workspace for qym_accel_dev: packs + items + partials for one system.
struct SingleLayout {
    size_t off_pos, off_lo, off_apart, off_heavy, total;
    int32_t nitems, chunk, parts;
    KickTune tune;
    bool sorted;   // bodies held in Morton order (mixed kick, >= kSortMinBodies bodies)
    size_t off_perm, off_inv, off_box, off_k0, off_k1, off_v0, off_v1, off_hist, off_far, off_tile;
};

// bodies from which a system's mixed kick holds them in Morton order (sort.cu)
constexpr int64_t kSingleSortMin = 2048;

// An acceleration is dominated by its closest pair, so how a pair's pull is rounded and
// which 64 bodies share an FP32 sum are part of a mixed call's result (1e-8 of it where
// a close pair stands out). Pulls carry G m in each product (as a batch's do; windows of
// one mass would give 16384 bodies 176 us instead of 184, 260 bodies 12.6 instead of
// 13.5), and the ranges end where sums of FOLD bodies end: on tiles or their halves in
// Morton order (4500 bodies 50.6 us in halves, 52.5 in tiles), else the system in equal
// chunks of at most a tile, each in parts of FOLD rows (2040 bodies 18.3 us). Two rows a
// thread in Morton order: a tile is near or far to a warp by all of its 64 rows.
static SingleLayout single_layout(int64_t rows, int prec) {
    SingleLayout L;
    int64_t nb = rows - 1;
    // slots that fit the fixed scratch of qym_accel_dev_static beside 60 bytes a
    // row of packs, order and tiles; beyond its sizes, 16
    L.tune = default_kick_tune(nb, nb, prec, rows <= QYM_STATIC_MAX_ROWS ? (((8 << 20) - (1 << 17)) / rows - 60) / 24 : 16);
    KickTune &t = L.tune;
    L.sorted = prec == QYM_KICK_MIXED && nb >= kSingleSortMin;
    L.parts = 1;
    if (L.sorted) t.ipt = 2;
    int64_t ti = (int64_t)t.threads * t.ipt;
    const int64_t align = L.sorted ? (nb > 6144 ? TILE : TILE / 2) : 1;
    if (prec == QYM_KICK_MIXED && !L.sorted) t.splits = (int32_t)((nb + TILE - 1) / TILE);
    int64_t chunk = (nb + t.splits - 1) / t.splits;
    chunk = (chunk + align - 1) / align * align;
    t.splits = (int32_t)((nb + chunk - 1) / chunk);
    L.chunk = (int32_t)chunk;
    if (prec == QYM_KICK_MIXED && !L.sorted) {
        L.parts = (int32_t)((chunk + FOLD - 1) / FOLD);
        t.splits *= L.parts;
    }
    L.nitems = (int32_t)((nb + ti - 1) / ti * t.splits);
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    size_t o = 0;
    const int64_t packs = prec == QYM_KICK_MIXED ? rows : 0;
    L.off_pos = o; o = al(o + sizeof(float4) * packs);
    L.off_lo = o; o = al(o + sizeof(float4) * packs);
    L.off_heavy = o; o = al(o + sizeof(int32_t) * (QYM_HEAVY_CAP + 1));
    L.off_perm = L.off_inv = L.off_box = L.off_k0 = L.off_k1 = L.off_v0 = L.off_v1 = L.off_hist = 0;
    L.off_far = L.off_tile = 0;
    if (L.sorted) {
        L.off_perm = o; o = al(o + sizeof(int32_t) * rows);
        L.off_inv = o; o = al(o + sizeof(int32_t) * rows);
        L.off_far = o; o = al(o + sizeof(float4) * rows);
        L.off_tile = o; o = al(o + sizeof(float4) * 3 * (size_t)((rows - 1 + TILE - 1) / TILE));
    }
    // the partial slots, over the sort's scratch (dead by then)
    L.off_apart = o;
    size_t end = al(o + sizeof(double) * 3 * rows * t.splits);
    if (L.sorted) {
        L.off_box = o; o = al(o + sizeof(int) * 8);
        L.off_k0 = o; o = al(o + sizeof(uint32_t) * rows);
        L.off_k1 = o; o = al(o + sizeof(uint32_t) * rows);
        L.off_v0 = o; o = al(o + sizeof(int32_t) * rows);
        L.off_v1 = o; o = al(o + sizeof(int32_t) * rows);
        L.off_hist = o; o = al(o + sizeof(uint32_t) * 256 * (size_t)sort_blocks(rows));
    }
    o = std::max(o, end);
    L.total = o;
    return L;
}

size_t accel_single_workspace(int64_t rows, int prec) {
    if (rows < 2) return 0;
    return single_layout(rows, prec).total;
}

// the packs of row r: its position as hi + lo floats and its G m (zero for a
// heavy body in the list; the list is ascending, so bodies past a full one are
// those beyond its last row)
__device__ __forceinline__ void pack_row(int64_t rows, int64_t r, const double *m, const double *q,
                                         double G, const int32_t *hl, double thr, float4 &P, float4 &L) {
    const p64::F3 x = p64::split3(q[r]), y = p64::split3(q[rows + r]), z = p64::split3(q[2 * rows + r]);
    const double mr = m[r];
    float gm = (float)(G * mr);
    if (hl && mass_reaches(mr, thr) && (hl[QYM_HEAVY_CAP] < QYM_HEAVY_CAP || r <= hl[QYM_HEAVY_CAP - 1])) gm = 0.0f;
    P = make_float4(x.h, y.h, z.h, gm);
    L = make_float4(x.m + x.l, y.m + y.l, z.m + z.l, 0.0f);
}

// packs and tile data of a sorted system, by position: one CTA per tile
__global__ void __launch_bounds__(TILE) k_pack_tiles(int64_t rows, const double *m, const double *q,
                                                     double G, double heavy_mass, const int32_t *hl,
                                                     const int32_t *perm, float4 *pos, float4 *lo,
                                                     float4 *far, float4 *tile) {
    chain_wait();
    const int64_t p = 1 + (int64_t)blockIdx.x * TILE + threadIdx.x;
    const bool act = p < rows;
    float4 P = make_float4(0.f, 0.f, 0.f, 0.f), L = P;
    if (act) {
        pack_row(rows, perm[p], m, q, G, hl, heavy_mass * m[0], P, L);
        pos[p] = P;
        lo[p] = L;
    }
    tile_prep(act, p, P, L, far, tile);
}

// heavy list and packs of a small system in row order, one CTA
__global__ void __launch_bounds__(1024) k_pack_small(int64_t rows, const double *m, const double *q,
                                                     double G, double heavy_mass, int32_t *hl,
                                                     float4 *pos, float4 *lo) {
    chain_wait();
    __shared__ int s[33];
    if (hl) {
        heavy_list(rows, m, heavy_mass, hl, s);
        __syncthreads();  // (the list is read back below by the CTA that wrote it)
    }
    for (int64_t r = threadIdx.x; r < rows; r += blockDim.x)
        pack_row(rows, r, m, q, G, hl, heavy_mass * m[0], pos[r], lo[r]);
}

// per row the sum of its slots and the heavy bodies' pull, SL threads a row
// (thread group q of the CTA the slots and heavies q, q + SL, ...), the parts
// added in a fixed tree
constexpr int SL = 8;
__global__ void __launch_bounds__(256) k_sum_partials(int64_t rows, int32_t splits, const double *apart,
                                                      const int32_t *hl, const double *m, const double *q,
                                                      double G, double *a, const int32_t *inv) {
    chain_wait();
    constexpr int RB = 256 / SL;
    __shared__ double sh[SL][3][RB];
    const int t = threadIdx.x % RB, g = threadIdx.x / RB;
    const int64_t i = (int64_t)blockIdx.x * RB + t;
    double s[3] = {0.0, 0.0, 0.0};
    if (i > 0 && i < rows) {
        const int64_t pi = inv ? inv[i] : i;  // the kick's order
        for (int sp = g; sp < splits; sp += SL)
            for (int c = 0; c < 3; ++c) s[c] += apart[((int64_t)sp * 3 + c) * rows + pi];
        if (hl)
            heavy_pull(hl, g, SL, hl[QYM_HEAVY_CAP], i, q[i], q[rows + i], q[2 * rows + i], q, m, rows,
                       G, s[0], s[1], s[2]);
    }
    for (int c = 0; c < 3; ++c) sh[g][c][t] = s[c];
    __syncthreads();
    if (g >= 3 || i >= rows) return;
    a[g * rows + i] = ((sh[0][g][t] + sh[1][g][t]) + (sh[2][g][t] + sh[3][g][t])) +
                      ((sh[4][g][t] + sh[5][g][t]) + (sh[6][g][t] + sh[7][g][t]));
}

cudaError_t launch_accel_single(int64_t rows, const double *m, const double *q, double *a,
                                double G, int prec, double heavy_mass, void *work,
                                size_t work_bytes, cudaStream_t st) {
    SingleLayout L = single_layout(rows, prec);
    if (work_bytes < L.total) return cudaErrorInvalidValue;
    char *w = (char *)work;
    Dev d;
    d.rows = rows;
    d.m = m ? const_cast<double *>(m) : nullptr;
    d.q = const_cast<double *>(q);
    d.pk_pos = (float4 *)(w + L.off_pos);
    d.pk_lo = (float4 *)(w + L.off_lo);
    d.apart = (double *)(w + L.off_apart);
    d.nitems = L.nitems;
    d.splits = L.tune.splits;
    d.item_chunk = L.chunk;
    d.item_parts = L.parts;
    d.batch = 1;
    // heavy split (mixed kick only): threshold relative to the star mass m[0],
    // read on the device
    int32_t *hl = prec == QYM_KICK_MIXED && heavy_mass > 0.0 ? (int32_t *)(w + L.off_heavy) : nullptr;
    cudaError_t e;
    if (prec == QYM_KICK_MIXED) {
        if (L.sorted) {
            // the bodies in Morton order, as the step's kick holds them
            d.perm = (int32_t *)(w + L.off_perm);
            d.inv = (int32_t *)(w + L.off_inv);
            d.far = (float4 *)(w + L.off_far);
            d.tile = (float4 *)(w + L.off_tile);
            d.tiles_ready = 1;
            SortScratch ss;
            ss.box = (int *)(w + L.off_box);
            ss.k0 = (uint32_t *)(w + L.off_k0);
            ss.k1 = (uint32_t *)(w + L.off_k1);
            ss.v0 = (int32_t *)(w + L.off_v0);
            ss.v1 = (int32_t *)(w + L.off_v1);
            ss.hist = (uint32_t *)(w + L.off_hist);
            if ((e = launch_sort_rows(rows, q, ss, d.perm, d.inv, st, m, heavy_mass, hl)) != cudaSuccess)
                return e;
            launch_chain(k_pack_tiles, (unsigned)((rows - 1 + TILE - 1) / TILE), TILE, 0, st, rows, m, q,
                         G, heavy_mass, hl, d.perm, d.pk_pos, d.pk_lo, d.far, d.tile);
        } else {
            launch_chain(k_pack_small, 1, 1024, 0, st, rows, m, q, G, heavy_mass, hl, d.pk_pos, d.pk_lo);
        }
        e = launch_kick_tiles(d, prec, 0, G, L.tune.threads, L.tune.ipt, st);
    } else {
        KickArgs ka{};
        ka.q = q; ka.m = m; ka.G = G; ka.apart = d.apart; ka.rows = rows;
        ka.splits = d.splits; ka.chunk = d.item_chunk;
        e = launch_f64<false, true>(ka, L.nitems, L.tune.threads, L.tune.ipt, L.chunk, st);
    }
    if (e != cudaSuccess) return e;
    launch_chain(k_sum_partials, (unsigned)((rows + 256 / SL - 1) / (256 / SL)), 256, 0, st, rows, d.splits, d.apart, hl, m,
                                                                     q, G, a, d.inv);
    return cudaGetLastError();
}

}  // namespace qym
