// mlp.cu -- inference and training kernels of the learned Kepler starting
// guess (network and layouts in mlp.cuh).
//
// Training minimises the mean squared error of the network output y against
// yt = (t - om) / osd over rows (u1, u2, u3, u4, t) with Adam. One step is two
// launches:
//   k_mlp_grad    forward and backward of a minibatch; each CTA takes rounds
//                 of 64 rows (16 per warp), keeps the 64 x 64 weight gradient
//                 of its rows in tensor-core accumulators and writes one
//                 partial gradient vector;
//   k_mlp_reduce  sums the partials in a fixed order (deterministic) and
//                 applies the Adam update to the float32 master weights.
// The operands the tensor cores take are bf16: h1 and W2 in the forward
// product, dp2 = dL/dp2 with W2 (for dL/dh1) and with h1 (for dL/dW2) in the
// backward ones. The other sums (dL/dW1, the biases, dL/dW3) stay in FP32.
#include <cmath>

#include "mlp.cuh"

namespace qym {
using namespace mlp;

namespace {
constexpr int GT = 256;      // threads of a gradient CTA
constexpr int GWARPS = GT / 32;
constexpr int LDT = 72;      // bf16 row stride of the shared tiles: 16-byte rows of eight lanes
                             // fall on distinct banks (ldmatrix)
constexpr int MAXBLK = 256;  // CTAs of a gradient launch the workspace holds
constexpr int GRID = 152;    // one CTA per SM
constexpr int NRED = 448;    // column sums: W1 (4 x 64), b1, b2, W3
}  // namespace

__global__ void __launch_bounds__(256) k_mlp_forward(int64_t n, const float *__restrict__ w,
                                                     const float *__restrict__ u,
                                                     float *__restrict__ y) {
    chain_wait();
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float uu[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (k < n) {
        const float4 r = *reinterpret_cast<const float4 *>(u + 4 * k);
        uu[0] = r.x; uu[1] = r.y; uu[2] = r.z; uu[3] = r.w;
    }
    float fn[4];
    normalise(w, uu, fn);
    const float out = warp_forward(w, fn);
    if (k < n) y[k] = out;
}

// ldmatrix (PTX ISA): four (two) 8 x 8 matrices of b16, one row of 16 bytes
// per lane address; .trans hands each lane the transposed element pair
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t &r0, uint32_t &r1, uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(r0), "=r"(r1) : "r"(a) : "memory");
}

// Sum of c[16] (entry 2 nt + e: column 8 nt + 2 t + e) over the eight lanes g
// of a quad column, scattered: lane (g, t) adds the sums of columns
// 8 g + 2 t + e to s[e]. Halves are exchanged, 8 + 4 + 2 shuffles instead of
// three per column.
__device__ __forceinline__ void scatter_sum(float (&c)[16], int lane, float (&s)[2]) {
#pragma unroll
    for (int h = 8; h >= 2; h >>= 1) {
        const int bit = 2 * h;  // lanes 16, 8, 4 apart
        const bool up = lane & bit;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float keep = up ? c[h + i] : c[i], give = up ? c[i] : c[h + i];
            c[i] = keep + __shfl_xor_sync(0xffffffffu, give, bit);
        }
    }
    s[0] += c[0];
    s[1] += c[1];
}

// Forward and backward of a minibatch. A warp takes 16-row tiles (tile =
// warp * grid + CTA, so any batch spreads over every SM before a warp gets a
// second one); the batch is latency here, not arithmetic (16384 rows are 0.6
// GFLOP), so the kernel is built for few dependent round trips: the weights
// staged once per CTA with all loads in flight, one copy of W2 serving both
// its products through ldmatrix (plain and transposed), the tiles' bf16 h1 and
// dL/dp2 left row by row and read transposed for dL/dW2 (warp w owns its
// columns 8w ..), the column sums by a halving exchange in registers. With
// 64-row CTAs of 128 threads, 16-bit transposing stores and a serial walk of
// 64 rows for the column sums a 16384-row minibatch took 20 us.
__global__ void __launch_bounds__(GT, 1) k_mlp_grad(const float *__restrict__ w,
                                                    const float *__restrict__ rows, int64_t n,
                                                    float inv_n, float *__restrict__ part,
                                                    float *__restrict__ lpart) {
    chain_wait();
    __shared__ __align__(16) __nv_bfloat16 s_w2[64 * LDT];             // bf16 W2[j][k]
    __shared__ __align__(16) uint32_t s_t[2][16 * GWARPS * LDT / 2];   // h1, dL/dp2 [row][col]
    __shared__ __align__(16) float s_w1[256];                          // bf16-rounded W1
    __shared__ float s_b1[64], s_b2[64], s_w3[64];
    __shared__ float s_red[2][GWARPS];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    {
        const float4 *w2 = reinterpret_cast<const float4 *>(w + W2);
        float4 x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = w2[tid + i * GT];
        const float y = w[W1 + tid];
        if (tid < 64) {
            s_b1[tid] = w[B1 + tid];
            s_b2[tid] = w[B2 + tid];
            s_w3[tid] = bf(w[W3 + tid]);
        }
        s_w1[tid] = bf(y);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = 4 * (tid + i * GT);
            *reinterpret_cast<uint2 *>(s_w2 + (e >> 6) * LDT + (e & 63)) =
                make_uint2(pack2(x[i].x, x[i].y), pack2(x[i].z, x[i].w));
        }
    }
    const float om = w[OM], osd = w[OSD], b3 = w[B3];
    // lane addresses of the ldmatrix loads
    const uint32_t w2s = smem_u32(s_w2);
    const uint32_t aF = w2s + 2 * ((lane & 7) * LDT + 8 * (lane >> 3));
    const uint32_t aB = w2s + 2 * (((lane & 7) + 8 * ((lane >> 3) & 1)) * LDT + 8 * (lane >> 4));
    const uint32_t aD = smem_u32(s_t[1]) + 2 * (((lane & 7) + 8 * (lane >> 4)) * LDT + 8 * ((lane >> 3) & 1));
    const uint32_t aH = smem_u32(s_t[0]) + 2 * ((lane & 15) * LDT + 8 * warp);
    float gw2[4][4];  // dL/dW2 rows 16 mt + g (+ 8), columns 8 warp + 2 t (+ 1)
#pragma unroll
    for (int mt = 0; mt < 4; ++mt)
#pragma unroll
        for (int e = 0; e < 4; ++e) gw2[mt][e] = 0.0f;
    float cs[7][2];  // columns 8 g + 2 t + e: dL/dW1 (4), dL/db1, dL/db2, dL/dW3
#pragma unroll
    for (int i = 0; i < 7; ++i) cs[i][0] = cs[i][1] = 0.0f;
    float gb3 = 0.0f, lsum = 0.0f;
    __syncthreads();

    const int64_t ntile = (n + 15) / 16;
    for (int64_t t0 = blockIdx.x; t0 < ntile; t0 += (int64_t)GWARPS * gridDim.x) {
        // warps 0 .. nw - 1 have a tile in this round
        const int64_t left = (ntile - t0 + gridDim.x - 1) / gridDim.x;
        const int nw = left < GWARPS ? (int)left : GWARPS;
        if (warp < nw) {
            const int64_t tile = t0 + (int64_t)warp * gridDim.x;
            const int64_t sa = tile * 16 + g, sb = sa + 8;
            const bool va = sa < n, vb = sb < n;
            float ua[4] = {0.0f, 0.0f, 0.0f, 0.0f}, ub[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            float ta = 0.0f, tb = 0.0f;
            if (va) {
#pragma unroll
                for (int i = 0; i < 4; ++i) ua[i] = rows[5 * sa + i];
                ta = rows[5 * sa + 4];
            }
            if (vb) {
#pragma unroll
                for (int i = 0; i < 4; ++i) ub[i] = rows[5 * sb + i];
                tb = rows[5 * sb + 4];
            }
            float fa[4], fb[4];
            normalise(w, ua, fa);
            normalise(w, ub, fb);
            // layer 1: h1 as the A fragments of layer 2, d1 = gelu'(p1)
            uint32_t A[4][4];
            float d1[8][4];
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                float h[4];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int c = 8 * nt + 2 * t + e;
                    const float4 wr = *reinterpret_cast<const float4 *>(s_w1 + 4 * c);
                    const float bb = s_b1[c];
                    const float pa = fmaf(wr.w, fa[3], fmaf(wr.z, fa[2], fmaf(wr.y, fa[1], fmaf(wr.x, fa[0], bb))));
                    const float pb = fmaf(wr.w, fb[3], fmaf(wr.z, fb[2], fmaf(wr.y, fb[1], fmaf(wr.x, fb[0], bb))));
                    h[e] = gelu(pa, d1[nt][e]);
                    h[2 + e] = gelu(pb, d1[nt][2 + e]);
                }
                A[nt >> 1][2 * (nt & 1)] = pack2(h[0], h[1]);      // row g
                A[nt >> 1][2 * (nt & 1) + 1] = pack2(h[2], h[3]);  // row g + 8
            }
            // p2[s][j] = sum_k h1[s][k] W2[j][k] + b2
            float acc[8][4];
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                acc[nt][0] = acc[nt][2] = s_b2[8 * nt + 2 * t];
                acc[nt][1] = acc[nt][3] = s_b2[8 * nt + 2 * t + 1];
            }
#pragma unroll
            for (int kp = 0; kp < 2; ++kp)
#pragma unroll
                for (int nt = 0; nt < 8; ++nt) {
                    uint32_t b[4];
                    ldsm4(b, aF + 2 * (8 * nt * LDT + 32 * kp));
                    mma_bf16(acc[nt], A[2 * kp], b[0], b[1]);
                    mma_bf16(acc[nt], A[2 * kp + 1], b[2], b[3]);
                }
            uint32_t *const h1s = s_t[0] + (16 * warp + g) * (LDT / 2) + t;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                h1s[4 * nt] = A[nt >> 1][2 * (nt & 1)];
                h1s[8 * (LDT / 2) + 4 * nt] = A[nt >> 1][2 * (nt & 1) + 1];
            }
            // output layer: h2, acc <- gelu'(p2)
            float h2[8][4], sya = 0.0f, syb = 0.0f;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float w3 = s_w3[8 * nt + 2 * t + e];
                    float da, db;
                    h2[nt][e] = gelu(acc[nt][e], da);
                    h2[nt][2 + e] = gelu(acc[nt][2 + e], db);
                    sya = fmaf(w3, h2[nt][e], sya);
                    syb = fmaf(w3, h2[nt][2 + e], syb);
                    acc[nt][e] = da;
                    acc[nt][2 + e] = db;
                }
            sya += __shfl_xor_sync(0xffffffffu, sya, 1);
            syb += __shfl_xor_sync(0xffffffffu, syb, 1);
            sya += __shfl_xor_sync(0xffffffffu, sya, 2);
            syb += __shfl_xor_sync(0xffffffffu, syb, 2);
            const float rra = va ? (sya + b3) - (ta - om) / osd : 0.0f;
            const float rrb = vb ? (syb + b3) - (tb - om) / osd : 0.0f;
            const float dya = 2.0f * rra * inv_n, dyb = 2.0f * rrb * inv_n;
            if (t == 0) {
                lsum = fmaf(rra, rra, fmaf(rrb, rrb, lsum));
                gb3 += dya + dyb;
            }
            float c[16];
#pragma unroll
            for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                for (int e = 0; e < 2; ++e) c[2 * nt + e] = fmaf(h2[nt][e], dya, h2[nt][2 + e] * dyb);
            scatter_sum(c, lane, cs[6]);
            // dp2 = dy W3 gelu'(p2): FP32 for the bias gradient, bf16 in the
            // two tensor-core products
            uint32_t dA[4][4];
            uint32_t *const d2s = s_t[1] + (16 * warp + g) * (LDT / 2) + t;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                float p[4];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float w3 = s_w3[8 * nt + 2 * t + e];
                    p[e] = dya * w3 * acc[nt][e];
                    p[2 + e] = dyb * w3 * acc[nt][2 + e];
                    c[2 * nt + e] = p[e] + p[2 + e];
                }
                const uint32_t xa = pack2(p[0], p[1]), xb = pack2(p[2], p[3]);
                dA[nt >> 1][2 * (nt & 1)] = xa;
                dA[nt >> 1][2 * (nt & 1) + 1] = xb;
                d2s[4 * nt] = xa;
                d2s[8 * (LDT / 2) + 4 * nt] = xb;
            }
            scatter_sum(c, lane, cs[5]);
            // dh1[s][k] = sum_j dp2[s][j] W2[j][k]
            float dh[8][4];
#pragma unroll
            for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) dh[nt][e] = 0.0f;
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
#pragma unroll
                for (int np = 0; np < 4; ++np) {
                    uint32_t b[4];
                    ldsm4t(b, aB + 2 * (16 * ks * LDT + 16 * np));
                    mma_bf16(dh[2 * np], dA[ks], b[0], b[1]);
                    mma_bf16(dh[2 * np + 1], dA[ks], b[2], b[3]);
                }
            // dp1 = dh1 gelu'(p1), its column sums and those with the features
#pragma unroll
            for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) d1[nt][e] *= dh[nt][e];
#pragma unroll
            for (int i = 0; i < 5; ++i) {
#pragma unroll
                for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        c[2 * nt + e] = i < 4 ? fmaf(d1[nt][e], fa[i & 3], d1[nt][2 + e] * fb[i & 3])
                                              : d1[nt][e] + d1[nt][2 + e];
                scatter_sum(c, lane, cs[i]);
            }
        }
        __syncthreads();
        // dL/dW2[j][k] = sum_s dp2[s][j] h1[s][k] over the round's rows
        for (int st = 0; st < nw; ++st) {
            uint32_t b0, b1;
            ldsm2t(b0, b1, aH + 2 * 16 * st * LDT);
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) {
                uint32_t a[4];
                ldsm4t(a, aD + 2 * (16 * st * LDT + 16 * mt));
                mma_bf16(gw2[mt], a, b0, b1);
            }
        }
        __syncthreads();
    }
    // one partial gradient per CTA
    float *P = part + (size_t)blockIdx.x * NW;
#pragma unroll
    for (int mt = 0; mt < 4; ++mt) {
        float *o = P + W2 + 64 * (16 * mt + g) + 8 * warp + 2 * t;
        o[0] = gw2[mt][0];
        o[1] = gw2[mt][1];
        o[8 * 64] = gw2[mt][2];
        o[8 * 64 + 1] = gw2[mt][3];
    }
    // column sums over the warps, in warp order (in the tiles' storage)
    float(*red)[NRED] = reinterpret_cast<float(*)[NRED]>(s_t);
    static_assert(sizeof(float) * GWARPS * NRED <= sizeof(s_t), "column sums overlay the tiles");
    const int c0 = 8 * g + 2 * t;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
#pragma unroll
        for (int i = 0; i < 4; ++i) red[warp][4 * (c0 + e) + i] = cs[i][e];
#pragma unroll
        for (int i = 4; i < 7; ++i) red[warp][64 * i + c0 + e] = cs[i][e];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
        lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    }
    if (lane == 0) {
        s_red[0][warp] = gb3;
        s_red[1][warp] = lsum;
    }
    __syncthreads();
    for (int i = tid; i < NRED; i += GT) {
        float x = 0.0f;
#pragma unroll
        for (int k = 0; k < GWARPS; ++k) x += red[k][i];
        // W1, b1 | b2, W3 of the weight vector
        P[i < 320 ? i : i - 320 + B2 + (i >= 384 ? W3 - B2 - 64 : 0)] = x;
    }
    if (tid == 0) {
        float a = 0.0f, b = 0.0f;
        for (int i = 0; i < GWARPS; ++i) {
            a += s_red[0][i];
            b += s_red[1][i];
        }
        P[B3] = a;
        lpart[blockIdx.x] = b;
    }
    if (tid < NFROZEN) P[NW - NFROZEN + tid] = 0.0f;
}

// Sum of nblk partial gradients (fixed order), optional copy to grad, and
// with adam != 0 the Adam update of w, m, v (normalisation entries kept).
// A CTA takes 32 weights, its warps every eighth partial each with all their
// loads in flight; sums are compensated pairs of floats (two-sum, about 2^-48:
// rounded to float it is the FP64 sum's value but for ties), since an FP64 add
// holds a warp 64 cycles here: one thread per weight adding 256 partials in
// FP64 took 63 us, three times the gradient itself. The last CTA also
// reduces the loss partials into *loss (mean over inv_n).
constexpr int RT = 256;
__global__ void __launch_bounds__(RT) k_mlp_reduce(const float *__restrict__ part, int nblk,
                                                   const float *__restrict__ lpart, float inv_n,
                                                   float *__restrict__ grad, float *__restrict__ loss,
                                                   float *__restrict__ w, float *__restrict__ m,
                                                   float *__restrict__ v, int adam, float lr,
                                                   float beta1, float beta2, float eps, float bc1,
                                                   float bc2) {
    chain_wait();
    constexpr int SL = RT / 32;
    __shared__ float s_hi[SL][32], s_lo[SL][32];
    const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    float hi = 0.0f, lo = 0.0f;
    if (i < NW) {
        const float *p = part + i;
#pragma unroll 8
        for (int b = sl; b < nblk; b += SL) {
            float s, e;
            two_sum(hi, p[(size_t)b * NW], s, e);
            hi = s;
            lo += e;
        }
    }
    s_hi[sl][lane] = hi;
    s_lo[sl][lane] = lo;
    __syncthreads();
    if (loss && lpart && blockIdx.x == gridDim.x - 1 && sl == 1) {
        double s = 0.0;
        for (int b = lane; b < nblk; b += 32) s += lpart[b];
        s = warp_sum(s);
        if (lane == 0) *loss = (float)(s * inv_n);
    }
    if (sl != 0 || i >= NW) return;
#pragma unroll
    for (int k = 1; k < SL; ++k) {
        float s, e;
        two_sum(hi, s_hi[k][lane], s, e);
        hi = s;
        lo += e + s_lo[k][lane];
    }
    const float gi = hi + lo;
    if (grad) grad[i] = gi;
    if (adam && i < NW - NFROZEN) {
        const float mm = fmaf(beta1, m[i], (1.0f - beta1) * gi);
        const float vv = fmaf(beta2, v[i], (1.0f - beta2) * gi * gi);
        m[i] = mm;
        v[i] = vv;
        w[i] -= lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
    }
}

// ------------------------------------------------------------------ host side
size_t mlp_workspace_bytes() { return (size_t)MAXBLK * NW * sizeof(float) + MAXBLK * sizeof(float); }

cudaError_t launch_mlp_forward(int64_t n, const float *w, const float *u, float *y, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const int64_t blocks = (n + 255) / 256;
    launch_chain(k_mlp_forward, (unsigned)blocks, 256, 0, st, n, w, u, y);
    return cudaGetLastError();
}

static cudaError_t grad_partials(int64_t n, const float *w, const float *rows, void *work, int &nblk,
                                 cudaStream_t st) {
    const int64_t tiles = (n + 15) / 16;
    nblk = (int)(tiles < GRID ? tiles : GRID);
    float *part = static_cast<float *>(work);
    float *lpart = part + (size_t)MAXBLK * NW;
    launch_chain(k_mlp_grad, nblk, GT, 0, st, w, rows, n, 1.0f / (float)n, part, lpart);
    return cudaGetLastError();
}

cudaError_t launch_mlp_grad(int64_t n, const float *w, const float *rows, float *grad, float *loss,
                            void *work, cudaStream_t st) {
    int nblk = 0;
    cudaError_t e = grad_partials(n, w, rows, work, nblk, st);
    if (e != cudaSuccess) return e;
    float *part = static_cast<float *>(work);
    float *lpart = part + (size_t)MAXBLK * NW;
    launch_chain(k_mlp_reduce, (NW + 31) / 32, RT, 0, st, part, nblk, lpart, 1.0f / (float)n, grad, loss,
                                                   nullptr, nullptr, nullptr, 0, 0.f, 0.f, 0.f, 0.f,
                                                   1.f, 1.f);
    return cudaGetLastError();
}

static void bias_corr(int64_t t, float beta1, float beta2, float &bc1, float &bc2) {
    bc1 = (float)(1.0 - std::pow((double)beta1, (double)t));
    bc2 = (float)(1.0 - std::pow((double)beta2, (double)t));
}

cudaError_t launch_mlp_adam(float *w, float *m, float *v, const float *grad, int64_t t, float lr,
                            float beta1, float beta2, float eps, cudaStream_t st) {
    float bc1, bc2;
    bias_corr(t, beta1, beta2, bc1, bc2);
    launch_chain(k_mlp_reduce, (NW + 31) / 32, RT, 0, st, grad, 1, nullptr, 0.f, nullptr, nullptr, w, m, v,
                                                   1, lr, beta1, beta2, eps, bc1, bc2);
    return cudaGetLastError();
}

cudaError_t launch_mlp_train(float *w, float *m, float *v, int64_t t0, const float *rows, int64_t n,
                             int64_t batch, int32_t epochs, float lr, float lr_final, float *losses,
                             void *work, cudaStream_t st) {
    const int64_t nb = (n + batch - 1) / batch;
    const int64_t S = nb * (int64_t)epochs;
    float *part = static_cast<float *>(work);
    float *lpart = part + (size_t)MAXBLK * NW;
    const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
    for (int64_t s = 0; s < S; ++s) {
        const int64_t b = s % nb, off = b * batch;
        const int64_t len = (n - off) < batch ? (n - off) : batch;
        int nblk = 0;
        cudaError_t e = grad_partials(len, w, rows + 5 * off, work, nblk, st);
        if (e != cudaSuccess) return e;
        // cosine schedule from lr (s = 0) towards lr_final
        const double lrs = (double)lr_final +
                           0.5 * ((double)lr - (double)lr_final) * (1.0 + std::cos(kPi * (double)s / (double)S));
        float bc1, bc2;
        bias_corr(t0 + s + 1, beta1, beta2, bc1, bc2);
        launch_chain(k_mlp_reduce, (NW + 31) / 32, RT, 0, st, part, nblk, lpart, 1.0f / (float)len, nullptr,
                                                       losses ? losses + s : nullptr, w, m, v, 1,
                                                       (float)lrs, beta1, beta2, eps, bc1, bc2);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace qym
