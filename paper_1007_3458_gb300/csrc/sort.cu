// sort.cu -- the order in which the mixed kick holds a system's bodies: along
// a Morton (Z-order) curve of their positions, so that each tile of 256
// consecutive bodies is compact in space and the kick can treat tiles far
// from a warp's rows with its one-add separation (kick.cu). Only the layout of
// the kick's operand packs follows this order; the state stays in row order,
// and results depend on it only through the grouping of the FP32 tile sums.
//
// Keys: 10 bits per axis of the position scaled into the cube over the
// system's bounding box, interleaved into 30 bits; bodies ordered by (key,
// row). Sort: stable least-significant-digit radix sort of (key, row),
// deterministic (digit counts, scans, and ranks within a warp from match masks).
// Up to 65536 bodies one cluster of eight CTAs does it all in shared memory
// (k_sort_cluster); above, 16 launches over the GPU. (A bitonic sort of the
// 64-bit words (key, row) in one CTA's shared memory took 0.16 ms for 16384
// bodies: each of its 105 stages moves every word through shared memory.)
#include <algorithm>
#include <utility>

#include <cooperative_groups.h>

#include "qym_internal.cuh"

namespace qym {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;                       // keys per thread per pass
constexpr int kSortTile = kSortThreads * kSortItems;  // keys per block

int64_t sort_blocks(int64_t n) { return (n + kSortTile - 1) / kSortTile; }

// bounding box of the bodies (rows 1 .. rows-1) as order-preserving integer
// images of their float coordinates (min and -max), reduced with atomics
__device__ __forceinline__ int fkey(float f) {
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float kfloat(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

__global__ void k_sort_box_init(int *box) {
    chain_wait();
    if (threadIdx.x < 6) box[threadIdx.x] = 0x7fffffff;
}

__global__ void __launch_bounds__(256) k_sort_box(int64_t rows, const double *q, int *box) {
    chain_wait();
    float m[6] = {3e38f, 3e38f, 3e38f, 3e38f, 3e38f, 3e38f};
    for (int64_t r = 1 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows;
         r += (int64_t)gridDim.x * blockDim.x) {
        for (int c = 0; c < 3; ++c) {
            const float x = (float)q[c * rows + r];
            m[c] = fminf(m[c], x);
            m[c + 3] = fminf(m[c + 3], -x);
        }
    }
    for (int c = 0; c < 6; ++c) {
        const float v = warp_min(m[c]);
        if ((threadIdx.x & 31) == 0) atomicMin(box + c, fkey(v));
    }
}

__device__ __forceinline__ uint32_t spread10(uint32_t x) {
    // 10 bits -> every third bit of 30
    x &= 0x3ff;
    x = (x | (x << 16)) & 0x030000ff;
    x = (x | (x << 8)) & 0x0300f00f;
    x = (x | (x << 4)) & 0x030c30c3;
    x = (x | (x << 2)) & 0x09249249;
    return x;
}

// Morton code of a position from the box (min, -max per axis, as fkey images)
__device__ __forceinline__ uint32_t morton_code(const float (&x)[3], const int *box) {
    // one scale for the three axes (cubic cells): a thin disk then orders by
    // its plane first instead of splitting its few bodies' heights at the top
    float span = 0.0f;
    for (int c = 0; c < 3; ++c) span = fmaxf(span, -kfloat(box[c + 3]) - kfloat(box[c]));
    uint32_t code = 0;
    for (int c = 0; c < 3; ++c) {
        const float lo = kfloat(box[c]);
        float u = span > 0.0f ? (x[c] - lo) / span : 0.0f;
        u = fminf(fmaxf(u, 0.0f), 1.0f);
        const uint32_t b = min((uint32_t)(u * 1024.0f), 1023u);
        code |= spread10(b) << c;
    }
    return code;
}
__global__ void __launch_bounds__(256) k_sort_keys(int64_t rows, const double *q, const int *box,
                                                    uint32_t *keys, int32_t *vals) {
    chain_wait();
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // body k = row k + 1
    if (k >= rows - 1) return;
    const int64_t r = k + 1;
    const float x[3] = {(float)q[r], (float)q[rows + r], (float)q[2 * rows + r]};
    keys[k] = morton_code(x, box);
    vals[k] = (int32_t)r;
}

// digit counts of each block: hist[digit * nblk + block]
__global__ void __launch_bounds__(kSortThreads) k_sort_hist(int64_t n, const uint32_t *keys,
                                                            int shift, uint32_t *hist, int nblk) {
    chain_wait();
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    for (int it = 0; it < kSortItems; ++it) {
        const int64_t k = base + it * kSortThreads + threadIdx.x;
        if (k < n) atomicAdd(&h[(keys[k] >> shift) & 255], 1u);
    }
    __syncthreads();
    hist[threadIdx.x * nblk + blockIdx.x] = h[threadIdx.x];
}

// exclusive scan of the m = 256 * nblk counts (one CTA)
__global__ void __launch_bounds__(1024) k_sort_scan(uint32_t *hist, int m) {
    chain_wait();
    __shared__ uint32_t part[1024];
    const int per = (m + 1023) / 1024;
    const int b0 = threadIdx.x * per;
    uint32_t s = 0;
    for (int b = b0; b < b0 + per && b < m; ++b) s += hist[b];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        const uint32_t t = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
        __syncthreads();
        part[threadIdx.x] += t;
        __syncthreads();
    }
    uint32_t run = threadIdx.x ? part[threadIdx.x - 1] : 0;
    for (int b = b0; b < b0 + per && b < m; ++b) {
        const uint32_t c = hist[b];
        hist[b] = run;
        run += c;
    }
}

// stable scatter: each block's keys in rounds of 256 (thread order), a key's
// place = the block's offset for its digit + the keys with that digit in
// earlier rounds + those in earlier warps of this round + earlier lanes
__global__ void __launch_bounds__(kSortThreads) k_sort_scatter(int64_t n, const uint32_t *kin,
                                                               const int32_t *vin, uint32_t *kout,
                                                               int32_t *vout, int shift,
                                                               const uint32_t *hist, int nblk) {
    chain_wait();
    constexpr int NW = kSortThreads / 32;
    __shared__ uint32_t run[256];
    __shared__ uint32_t wc[NW][256];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    run[tid] = hist[tid * nblk + blockIdx.x];
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    for (int it = 0; it < kSortItems; ++it) {
        for (int q = 0; q < NW; ++q) wc[q][tid] = 0;
        __syncthreads();
        const int64_t k = base + it * kSortThreads + tid;
        const bool act = k < n;
        const uint32_t key = act ? kin[k] : 0u;
        const int dig = act ? (int)((key >> shift) & 255) : 256 + lane;  // idle lanes apart
        const unsigned peers = __match_any_sync(0xffffffffu, dig);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        if (act && rank == 0) wc[w][dig] = (uint32_t)__popc(peers);
        __syncthreads();
        if (act) {
            uint32_t before = run[dig];
            for (int q = 0; q < w; ++q) before += wc[q][dig];
            const uint32_t pos = before + (uint32_t)rank;
            kout[pos] = key;
            vout[pos] = vin[k];
        }
        __syncthreads();
        uint32_t tot = 0;
        for (int q = 0; q < NW; ++q) tot += wc[q][tid];
        run[tid] += tot;
        __syncthreads();
    }
}

// position p (1 .. rows-1) holds row perm[p]; inv[perm[p]] = p; row 0 stays
__global__ void __launch_bounds__(256) k_sort_perm(int64_t rows, const int32_t *vals,
                                                    int32_t *perm, int32_t *inv) {
    chain_wait();
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k == 0) {
        perm[0] = 0;
        inv[0] = 0;
    }
    if (k >= rows - 1) return;
    const int32_t r = vals[k];
    perm[k + 1] = r;
    inv[r] = (int32_t)(k + 1);
}

// ---------------------------------------------------------------- one cluster
// The whole sort of up to 65536 bodies in one launch: eight CTAs of 1024 threads
// hold the (row, key) words of consecutive positions in shared memory and pass
// them on through distributed shared memory, three passes of 10-bit digits (one
// thread per digit in the scans). A pass: each warp counts the digits of its
// words in order (a word's rank among its warp's equal digits comes with the
// count), a digit's counts are summed over the CTA's warps and the cluster's
// CTAs, and every word is stored into the CTA that holds its new position. The
// sort is latency: the 16 launches of the general path take 100 us for 16384
// bodies, four passes of three kernels among them.
namespace cg = cooperative_groups;
constexpr int CS_CTAS = 8, CS_T = 1024, CS_W = CS_T / 32, CS_ITEMS = 8;
constexpr int64_t kClusterSortMax = (int64_t)CS_CTAS * CS_T * CS_ITEMS;
struct ClusterSortShared {
    uint16_t wc[CS_W][1024];  // a warp's words per digit, then the words before it
    uint32_t hist[1024];      // the CTA's words per digit
    uint32_t base[1024];      // position of the CTA's first word with the digit
    uint32_t wsum[CS_W];
    int box[6];
};

template <int IT>
__global__ void __cluster_dims__(CS_CTAS, 1, 1) __launch_bounds__(CS_T)
    k_sort_cluster(int64_t rows, const double *q, int32_t *perm, int32_t *inv, const double *m,
                   double heavy_mass, int32_t *hl) {
    chain_wait();
    extern __shared__ __align__(16) unsigned char sm[];
    if (blockIdx.x >= CS_CTAS) {  // a second cluster: the list of heavy bodies (hl != NULL)
        if (blockIdx.x == CS_CTAS) heavy_list(rows, m, heavy_mass, hl, reinterpret_cast<int *>(sm));
        return;
    }
    constexpr int CHUNK = CS_T * IT;
    ClusterSortShared &S = *reinterpret_cast<ClusterSortShared *>(sm);
    uint2 *const buf = reinterpret_cast<uint2 *>(sm + sizeof(ClusterSortShared));  // [2][CHUNK] (row, key)
    cg::cluster_group cl = cg::this_cluster();
    const int cta = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int64_t n = rows - 1;
    const int i0 = w * 32 * IT + lane;  // word it of this thread: i0 + 32 it
    // bounding box
    float x[IT][3];
    if (tid < 6) S.box[tid] = 0x7fffffff;
    __syncthreads();
    float mn[6] = {3e38f, 3e38f, 3e38f, 3e38f, 3e38f, 3e38f};
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int64_t k = (int64_t)cta * CHUNK + i0 + 32 * it;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x[it][c] = k < n ? p64::to_float(q[c * rows + k + 1]) : 0.0f;
            if (k < n) {
                mn[c] = fminf(mn[c], x[it][c]);
                mn[c + 3] = fminf(mn[c + 3], -x[it][c]);
            }
        }
    }
    for (int c = 0; c < 6; ++c) {
        const int v = __reduce_min_sync(0xffffffffu, fkey(mn[c]));
        if (lane == 0) atomicMin(&S.box[c], v);
    }
    cl.sync();
    int box[6];
    for (int c = 0; c < 6; ++c) {
        box[c] = 0x7fffffff;
        for (int r = 0; r < CS_CTAS; ++r) box[c] = min(box[c], cl.map_shared_rank(S.box, r)[c]);
    }
#pragma unroll
    for (int it = 0; it < IT; ++it)
        buf[i0 + 32 * it] = make_uint2((uint32_t)(cta * CHUNK + i0 + 32 * it + 1), morton_code(x[it], box));
    for (int pass = 0; pass < 3; ++pass) {
        const uint2 *src = buf + (pass & 1) * CHUNK;
        uint2 *dst = buf + ((pass & 1) ^ 1) * CHUNK;
        const int shift = 10 * pass;
        uint32_t *z = reinterpret_cast<uint32_t *>(S.wc);
        for (int k = tid; k < CS_W * 1024 / 2; k += CS_T) z[k] = 0;
        __syncthreads();
        uint2 word[IT];
        int dig[IT];
        uint32_t ahead[IT];  // words of this warp with the digit before this one
#pragma unroll
        for (int it = 0; it < IT; ++it) {
            const bool act = (int64_t)cta * CHUNK + i0 + 32 * it < n;
            word[it] = src[i0 + 32 * it];
            dig[it] = act ? (int)((word[it].y >> shift) & 1023) : 1024 + lane;
            const unsigned peers = __match_any_sync(0xffffffffu, dig[it]);
            const int rank = __popc(peers & ((1u << lane) - 1u));
            const uint32_t c = act ? S.wc[w][dig[it]] : 0u;
            __syncwarp();
            if (act && rank == 0) S.wc[w][dig[it]] = (uint16_t)(c + __popc(peers));
            __syncwarp();
            ahead[it] = c + rank;
        }
        __syncthreads();
        uint32_t run = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint16_t c[CS_W / 2];
#pragma unroll
            for (int k = 0; k < CS_W / 2; ++k) c[k] = S.wc[h * (CS_W / 2) + k][tid];
#pragma unroll
            for (int k = 0; k < CS_W / 2; ++k) {
                S.wc[h * (CS_W / 2) + k][tid] = (uint16_t)run;
                run += c[k];
            }
        }
        S.hist[tid] = run;
        cl.sync();
        uint32_t tot = 0, before = 0;
#pragma unroll
        for (int r = 0; r < CS_CTAS; ++r) {
            const uint32_t c = cl.map_shared_rank(S.hist, r)[tid];
            tot += c;
            if (r < cta) before += c;
        }
        uint32_t inc = tot;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) S.wsum[w] = inc;
        __syncthreads();
        const uint32_t off = __reduce_add_sync(0xffffffffu, lane < w ? S.wsum[lane] : 0u);
        S.base[tid] = off + inc - tot + before;
        __syncthreads();
#pragma unroll
        for (int it = 0; it < IT; ++it) {
            if (dig[it] >= 1024) continue;
            const uint32_t pos = S.base[dig[it]] + S.wc[w][dig[it]] + ahead[it];
            cl.map_shared_rank(dst, (int)(pos / CHUNK))[pos % CHUNK] = word[it];
        }
        cl.sync();
    }
    const uint2 *out = buf + CHUNK;  // three passes end in the second buffer
    if (cta == 0 && tid == 0) perm[0] = inv[0] = 0;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int64_t p = (int64_t)cta * CHUNK + tid + CS_T * it;
        if (p < n) {
            const int32_t r = (int32_t)out[tid + CS_T * it].x;
            perm[p + 1] = r;
            inv[r] = (int32_t)(p + 1);
        }
    }
}

template <int IT>
static cudaError_t sort_cluster(int64_t rows, const double *q, int32_t *perm, int32_t *inv,
                                const double *m, double heavy_mass, int32_t *hl, cudaStream_t st) {
    const size_t smem = sizeof(ClusterSortShared) + 2 * sizeof(uint2) * CS_T * IT;
    cudaError_t e = cudaFuncSetAttribute(k_sort_cluster<IT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chain(k_sort_cluster<IT>, (hl ? 2 : 1) * CS_CTAS, CS_T, smem, st, rows, q, perm, inv,
                        m, heavy_mass, hl);
}

int sort_launches(int64_t rows) { return rows - 1 <= kClusterSortMax ? 1 : 16; }

__global__ void __launch_bounds__(1024) k_heavy_list(int64_t rows, const double *m, double heavy_mass,
                                                     int32_t *hl) {
    chain_wait();
    __shared__ int s[33];
    heavy_list(rows, m, heavy_mass, hl, s);
}
cudaError_t launch_heavy_list(int64_t rows, const double *m, double heavy_mass, int32_t *hl,
                              cudaStream_t st) {
    return launch_chain(k_heavy_list, 1, 1024, 0, st, rows, m, heavy_mass, hl);
}

cudaError_t launch_sort_rows(int64_t rows, const double *q, const SortScratch &s, int32_t *perm,
                             int32_t *inv, cudaStream_t st, const double *m, double heavy_mass,
                             int32_t *hl) {
    const int64_t n = rows - 1;
    if (n < 1) return cudaSuccess;
    if (n <= kClusterSortMax) {
        const int it = (int)((n + CS_CTAS * CS_T - 1) / (CS_CTAS * CS_T));
        return it <= 1   ? sort_cluster<1>(rows, q, perm, inv, m, heavy_mass, hl, st)
               : it <= 2 ? sort_cluster<2>(rows, q, perm, inv, m, heavy_mass, hl, st)
               : it <= 4 ? sort_cluster<4>(rows, q, perm, inv, m, heavy_mass, hl, st)
                         : sort_cluster<8>(rows, q, perm, inv, m, heavy_mass, hl, st);
    }
    if (hl) launch_heavy_list(rows, m, heavy_mass, hl, st);
    const int nblk = (int)sort_blocks(n);
    const unsigned g = (unsigned)((n + 255) / 256);
    launch_chain(k_sort_box_init, 1, 32, 0, st, s.box);
    launch_chain(k_sort_box, (unsigned)std::min<int64_t>(g, 4 * 152), 256, 0, st, rows, q, s.box);
    launch_chain(k_sort_keys, g, 256, 0, st, rows, q, s.box, s.k0, s.v0);
    uint32_t *ka = s.k0, *kb = s.k1;
    int32_t *va = s.v0, *vb = s.v1;
    for (int shift = 0; shift < 32; shift += 8) {
        launch_chain(k_sort_hist, nblk, kSortThreads, 0, st, n, ka, shift, s.hist, nblk);
        launch_chain(k_sort_scan, 1, 1024, 0, st, s.hist, 256 * nblk);
        launch_chain(k_sort_scatter, nblk, kSortThreads, 0, st, n, ka, va, kb, vb, shift, s.hist, nblk);
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    launch_chain(k_sort_perm, g, 256, 0, st, rows, va, perm, inv);
    return cudaGetLastError();
}

}  // namespace qym
