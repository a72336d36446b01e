// mlp.cu -- inference and training kernels of the learned Kepler starting
// guess (network and layouts in mlp.cuh).
//
// Training minimises the mean squared error of the network output y against
// yt = (t - om) / osd over rows (u1, u2, u3, u4, t) with Adam. One step is two
// launches:
//   k_mlp_grad    forward and backward of a minibatch; each CTA takes rounds
//                 of 64 rows (16 per warp of the forward pass), keeps the
//                 64 x 64 weight gradient of its rows in tensor-core
//                 accumulators and writes one partial gradient vector;
//   k_mlp_reduce  sums the partials (as an FP64 sum does) and applies the Adam
//                 update to the float32 master weights.
// The grouping of the sums is part of the result: a weight near a bf16 midpoint
// turns one last place into 2^-9, and a hundred minibatches into 1e-2 of the
// moments. A round's sums run over its 64 rows in order (FP32), a CTA's over its
// rounds, CTA b of min(256, rounds) taking the rounds b, b + 256, ...; the
// partials' sum is exact but for its last rounding.
// The buffers are plain pointers, not const __restrict__: launches are chained, so
// a kernel may be resident while the one before it still writes them, and every
// load has to come after the wait and through the coherent path.
// The operands the tensor cores take are bf16: h1 and W2 in the forward
// product, dp2 = dL/dp2 with W2 (for dL/dh1) and with h1 (for dL/dW2) in the
// backward ones. The other sums (dL/dW1, the biases, dL/dW3) stay in FP32.
#include <cmath>

#include "mlp.cuh"

namespace qym {
using namespace mlp;

namespace {
constexpr int GT = 256;      // threads of a gradient CTA
constexpr int FW = 4;        // its warps that take a tile of 16 rows through the network
constexpr int GR = 16 * FW;  // rows per round
constexpr int LDT = 72;      // bf16 row stride of the shared tiles: 16-byte rows of eight lanes
                             // fall on distinct banks (ldmatrix)
constexpr int LDF = 72;      // float row stride: a half warp's pairs fall on distinct banks
constexpr int MAXBLK = 256;  // CTAs of a gradient launch, at most
struct GradShared {
    __nv_bfloat16 w2[64 * LDT];         // bf16 W2[j][k]
    __nv_bfloat16 h1[GR * LDT];         // bf16 h1 [row][k]
    __nv_bfloat16 d2[GR * LDT];         // bf16 dL/dp2 [row][j]
    float dp1[GR * LDF], dp2[GR * LDF], h2[GR * LDF];  // [row][unit]
    float4 fn[GR];                      // normalised features
    float dy[GR];
    float w1[256], b1[64], b2[64], w3[64];  // W1 and W3 rounded to bf16
    float red[2][FW];
};
}  // namespace

__global__ void __launch_bounds__(256) k_mlp_forward(int64_t n, const float *w, const float *u,
                                                     float *y) {
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

// Forward and backward of a minibatch (16384 rows with the reduction: 20 us). Four of the CTA's eight warps take a
// 16-row tile each; the batch is latency here, not arithmetic (16384 rows are 0.6
// GFLOP), so the kernel is built for few dependent round trips: the weights
// staged once per CTA with all loads in flight, one copy of W2 serving both
// its products through ldmatrix (plain and transposed), the tiles' bf16 h1 and
// dL/dp2 left row by row and read transposed for dL/dW2 (warp w owns its
// columns 8w ..). The other column sums run over the round's rows in order (see
// above), 448 chains on the CTA's 256 threads. (A halving exchange in registers
// instead is 3 us shorter at 16384 rows, in another order. Weights read from
// global memory per tile and 16-bit transposing stores: 20 us.)
__global__ void __launch_bounds__(GT, 2) k_mlp_grad(const float *w, const float *rows, int64_t n,
                                                    float inv_n, float *part, float *lpart) {
    chain_wait();
    extern __shared__ __align__(16) unsigned char g_gradsmem[];
    GradShared &S = *reinterpret_cast<GradShared *>(g_gradsmem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    {
        const float4 *w2 = reinterpret_cast<const float4 *>(w + W2);
        float4 x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = w2[tid + i * GT];
        const float y = w[W1 + tid];
        if (tid < 64) {
            S.b1[tid] = w[B1 + tid];
            S.b2[tid] = w[B2 + tid];
            S.w3[tid] = bf(w[W3 + tid]);
        }
        S.w1[tid] = bf(y);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = 4 * (tid + i * GT);
            *reinterpret_cast<uint2 *>(S.w2 + (e >> 6) * LDT + (e & 63)) =
                make_uint2(pack2(x[i].x, x[i].y), pack2(x[i].z, x[i].w));
        }
    }
    const float om = w[OM], osd = w[OSD], b3 = w[B3];
    // lane addresses of the ldmatrix loads
    const uint32_t w2s = smem_u32(S.w2);
    const uint32_t aF = w2s + 2 * ((lane & 7) * LDT + 8 * (lane >> 3));
    const uint32_t aB = w2s + 2 * (((lane & 7) + 8 * ((lane >> 3) & 1)) * LDT + 8 * (lane >> 4));
    const uint32_t aD = smem_u32(S.d2) + 2 * (((lane & 7) + 8 * (lane >> 4)) * LDT + 8 * ((lane >> 3) & 1));
    const uint32_t aH = smem_u32(S.h1) + 2 * ((lane & 15) * LDT + 8 * warp);
    float gw2[4][4];  // dL/dW2 rows 16 mt + g (+ 8), columns 8 warp + 2 t (+ 1)
#pragma unroll
    for (int mt = 0; mt < 4; ++mt)
#pragma unroll
        for (int e = 0; e < 4; ++e) gw2[mt][e] = 0.0f;
    // column sums of unit j: db1 and dW1[0] | dW1[1], dW1[2] | dW1[3], db2 | dW3
    const int j = tid & 63, job = tid >> 6;
    float cs0 = 0.0f, cs1 = 0.0f;
    float gb3 = 0.0f, lsum = 0.0f;
    __syncthreads();

    const int64_t nround = (n + GR - 1) / GR;
    for (int64_t rd = blockIdx.x; rd < nround; rd += gridDim.x) {
        if (warp < FW) {
            const int ra = 16 * warp + g, rb = ra + 8;  // rows of this lane within the round
            const int64_t sa = rd * GR + ra, sb = rd * GR + rb;
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
            if (t == 0) {
                S.fn[ra] = make_float4(fa[0], fa[1], fa[2], fa[3]);
                S.fn[rb] = make_float4(fb[0], fb[1], fb[2], fb[3]);
            }
            // layer 1: h1 as the A fragments of layer 2, d1 = gelu'(p1)
            uint32_t A[4][4];
            float d1[8][4];
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                float h[4];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int c = 8 * nt + 2 * t + e;
                    const float4 wr = *reinterpret_cast<const float4 *>(S.w1 + 4 * c);
                    const float bb = S.b1[c];
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
                acc[nt][0] = acc[nt][2] = S.b2[8 * nt + 2 * t];
                acc[nt][1] = acc[nt][3] = S.b2[8 * nt + 2 * t + 1];
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
            uint32_t *const h1s = reinterpret_cast<uint32_t *>(S.h1) + ra * (LDT / 2) + t;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                h1s[4 * nt] = A[nt >> 1][2 * (nt & 1)];
                h1s[8 * (LDT / 2) + 4 * nt] = A[nt >> 1][2 * (nt & 1) + 1];
            }
            // output layer: h2 to shared memory, acc <- gelu'(p2)
            float sya = 0.0f, syb = 0.0f;
            const int fo = ra * LDF + 2 * t;  // this lane's pair of units in the float tiles
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                float h[4];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float w3 = S.w3[8 * nt + 2 * t + e];
                    float da, db;
                    h[e] = gelu(acc[nt][e], da);
                    h[2 + e] = gelu(acc[nt][2 + e], db);
                    sya = fmaf(w3, h[e], sya);
                    syb = fmaf(w3, h[2 + e], syb);
                    acc[nt][e] = da;
                    acc[nt][2 + e] = db;
                }
                *reinterpret_cast<float2 *>(S.h2 + fo + 8 * nt) = make_float2(h[0], h[1]);
                *reinterpret_cast<float2 *>(S.h2 + fo + 8 * LDF + 8 * nt) = make_float2(h[2], h[3]);
            }
            sya += __shfl_xor_sync(0xffffffffu, sya, 1);
            syb += __shfl_xor_sync(0xffffffffu, syb, 1);
            sya += __shfl_xor_sync(0xffffffffu, sya, 2);
            syb += __shfl_xor_sync(0xffffffffu, syb, 2);
            const float rra = va ? (sya + b3) - (ta - om) / osd : 0.0f;
            const float rrb = vb ? (syb + b3) - (tb - om) / osd : 0.0f;
            const float dya = 2.0f * rra * inv_n, dyb = 2.0f * rrb * inv_n;
            if (t == 0) {
                S.dy[ra] = dya;
                S.dy[rb] = dyb;
                lsum = fmaf(rra, rra, fmaf(rrb, rrb, lsum));
                gb3 += dya + dyb;
            }
            // dp2 = dy W3 gelu'(p2): FP32 for the bias gradient, bf16 in the
            // two tensor-core products
            uint32_t dA[4][4];
            uint32_t *const d2s = reinterpret_cast<uint32_t *>(S.d2) + ra * (LDT / 2) + t;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                float p[4];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float w3 = S.w3[8 * nt + 2 * t + e];
                    p[e] = dya * w3 * acc[nt][e];
                    p[2 + e] = dyb * w3 * acc[nt][2 + e];
                }
                *reinterpret_cast<float2 *>(S.dp2 + fo + 8 * nt) = make_float2(p[0], p[1]);
                *reinterpret_cast<float2 *>(S.dp2 + fo + 8 * LDF + 8 * nt) = make_float2(p[2], p[3]);
                const uint32_t xa = pack2(p[0], p[1]), xb = pack2(p[2], p[3]);
                dA[nt >> 1][2 * (nt & 1)] = xa;
                dA[nt >> 1][2 * (nt & 1) + 1] = xb;
                d2s[4 * nt] = xa;
                d2s[8 * (LDT / 2) + 4 * nt] = xb;
            }
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
            // dp1 = dh1 gelu'(p1)
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                *reinterpret_cast<float2 *>(S.dp1 + fo + 8 * nt) =
                    make_float2(d1[nt][0] * dh[nt][0], d1[nt][1] * dh[nt][1]);
                *reinterpret_cast<float2 *>(S.dp1 + fo + 8 * LDF + 8 * nt) =
                    make_float2(d1[nt][2] * dh[nt][2], d1[nt][3] * dh[nt][3]);
            }
        }
        __syncthreads();
        // dL/dW2[j][k] = sum_s dp2[s][j] h1[s][k] over the round's rows
#pragma unroll
        for (int st = 0; st < FW; ++st) {
            uint32_t b0, b1;
            ldsm2t(b0, b1, aH + 2 * 16 * st * LDT);
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) {
                uint32_t a[4];
                ldsm4t(a, aD + 2 * (16 * st * LDT + 16 * mt));
                mma_bf16(gw2[mt], a, b0, b1);
            }
        }
        // column sums over the round's rows
        if (job == 0) {
#pragma unroll 16
            for (int s = 0; s < GR; ++s) {
                const float d = S.dp1[s * LDF + j];
                cs0 += d;
                cs1 = fmaf(d, S.fn[s].x, cs1);
            }
        } else if (job == 1) {
#pragma unroll 16
            for (int s = 0; s < GR; ++s) {
                const float d = S.dp1[s * LDF + j];
                cs0 = fmaf(d, S.fn[s].y, cs0);
                cs1 = fmaf(d, S.fn[s].z, cs1);
            }
        } else if (job == 2) {
#pragma unroll 16
            for (int s = 0; s < GR; ++s) {
                cs0 = fmaf(S.dp1[s * LDF + j], S.fn[s].w, cs0);
                cs1 += S.dp2[s * LDF + j];
            }
        } else {
#pragma unroll 16
            for (int s = 0; s < GR; ++s) cs0 = fmaf(S.h2[s * LDF + j], S.dy[s], cs0);
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
    if (job == 0) {
        P[B1 + j] = cs0;
        P[W1 + 4 * j] = cs1;
    } else if (job == 1) {
        P[W1 + 4 * j + 1] = cs0;
        P[W1 + 4 * j + 2] = cs1;
    } else if (job == 2) {
        P[W1 + 4 * j + 3] = cs0;
        P[B2 + j] = cs1;
    } else {
        P[W3 + j] = cs0;
    }
    // b3 and the loss: lanes with t == 0 of the first warps hold them
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
        lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    }
    if (warp < FW && lane == 0) {
        S.red[0][warp] = gb3;
        S.red[1][warp] = lsum;
    }
    __syncthreads();
    if (tid == 0) {
        float a = 0.0f, b = 0.0f;
        for (int i = 0; i < FW; ++i) {
            a += S.red[0][i];
            b += S.red[1][i];
        }
        P[B3] = a;
        lpart[blockIdx.x] = b;
    }
    if (tid < NFROZEN) P[NW - NFROZEN + tid] = 0.0f;
}

// Sum of nblk partial gradients, optional copy to grad, and with adam != 0 the
// Adam update of w, m, v (normalisation entries kept).
// A CTA takes 32 weights, its warps every sixteenth partial each with all their
// loads in flight. The sum is an FP64 one's, in any order the same float but where
// FP64 itself would round: a warp adds its partials as three floats with the exact
// errors (two-sum), the warps' sums are FP64 additions, since an FP64 addition
// holds a warp 64 cycles here: one thread per weight adding 256 partials in
// FP64 took 63 us, three times the gradient itself. The last CTA also
// reduces the loss partials into *loss (mean over inv_n).
constexpr int RT = 512;
__global__ void __launch_bounds__(RT) k_mlp_reduce(const float *part, int nblk, const float *lpart,
                                                   float inv_n, float *grad, float *loss, float *w,
                                                   float *m, float *v, int adam, float lr, float beta1,
                                                   float beta2, float eps, float bc1, float bc2) {
    chain_wait();
    constexpr int SL = RT / 32;
    __shared__ double s_sum[SL][32];
    const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    if (i < NW) {
        const float *p = part + i;
        float hi = 0.0f, mid = 0.0f, lo = 0.0f;
#pragma unroll 16
        for (int b = sl; b < nblk; b += SL) {
            float s, e, f;
            two_sum(hi, p[(size_t)b * NW], s, e);
            hi = s;
            two_sum(mid, e, s, f);
            mid = s;
            lo += f;
        }
        double sum = (double)hi + ((double)mid + (double)lo);
        if (!isfinite(hi)) {  // beyond FP32's range on the way, or not finite
            sum = 0.0;
            for (int b = sl; b < nblk; b += SL) sum += (double)p[(size_t)b * NW];
        }
        s_sum[sl][lane] = sum;
    }
    __syncthreads();
    if (loss && lpart && blockIdx.x == gridDim.x - 1 && sl == 1) {
        double s = 0.0;
        for (int b = lane; b < nblk; b += 32) s += lpart[b];
        s = warp_sum(s);
        if (lane == 0) *loss = (float)(s * inv_n);
    }
    if (sl != 0 || i >= NW) return;
    double s[SL];
#pragma unroll
    for (int k = 0; k < SL; ++k) s[k] = s_sum[k][lane];
#pragma unroll
    for (int o = 1; o < SL; o *= 2)
#pragma unroll
        for (int k = 0; k < SL; k += 2 * o) s[k] += s[k + o];
    const float gi = (float)s[0];
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
    // chained up to a CTA per SM; a plain launch above, where the next call's CTAs
    // would settle on the SMs while this one's still run, two and three to some of
    // them (65536 rows: 28 us, chained 31; 4096 rows: 24 us, chained 22)
    const unsigned blocks = (unsigned)((n + 255) / 256);
    if (blocks <= 152) return launch_chain(k_mlp_forward, blocks, 256, 0, st, n, w, u, y);
    k_mlp_forward<<<blocks, 256, 0, st>>>(n, w, u, y);
    return cudaGetLastError();
}

static cudaError_t grad_partials(int64_t n, const float *w, const float *rows, void *work, int &nblk,
                                 cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(GradShared));
    if (e != cudaSuccess) return e;
    const int64_t rounds = (n + GR - 1) / GR;
    nblk = (int)(rounds < MAXBLK ? rounds : MAXBLK);
    float *part = static_cast<float *>(work);
    float *lpart = part + (size_t)MAXBLK * NW;
    launch_chain(k_mlp_grad, nblk, GT, sizeof(GradShared), st, w, rows, n, 1.0f / (float)n, part, lpart);
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
