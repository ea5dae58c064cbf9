// gdi_mpnn.cu -- kernels of the learned warm start: a 3-layer message-passing network over a batch
// of graphs (disjoint union CSR), its training (loss, backward, Adam) and the rounding of its
// logits to an exactly balanced initial spin assignment for gdi_anneal.
//
// Layer l: H_l = ReLU(H_{l-1} Ws_l + (A_mean H_{l-1}) Wn_l + b_l), A_mean = D^-1 A (mean over
// neighbours).  Output z = H_3 wo + bo.  Weights are BF16 (round-to-nearest-even copies of FP32
// master weights); activations, accumulations and gradients are FP32.  The dense layers of the
// network (din = 16 and 64), forward and backward, run on the tensor cores (mma.sync m16n8k16,
// BF16 operands, FP32 accumulation) with the FP32 activations split into two BF16 parts; the
// neighbour aggregations are CSR gathers with one warp per vertex and lanes over channels.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gdi_device.cuh"
#include "gdi_mpnn.h"

using namespace gdi;

namespace {

constexpr int HID = GDI_MPNN_HIDDEN;   // 64
constexpr int FIN = GDI_MPNN_FEATURES; // 16
constexpr int NRAND = 8;               // random positional channels

inline bool aligned(const void *p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

__device__ __forceinline__ float bf16_to_f(uint16_t b)
{
    return __uint_as_float((uint32_t)b << 16);
}

__device__ __forceinline__ int64_t graph_of(const int64_t *graph_ptr, int G, int64_t i)
{
    int lo = 0, hi = G - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (graph_ptr[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------------------------------------
// Aggregation, one warp per destination vertex:
//   mode 0: Y_i = (1/deg_i) sum_{j in N(i)} X_j               (A_mean X)
//   mode 1: Y_j = sum_{i in N(j)} X_i / deg_i                 (A_mean^T X, graph symmetric)
//   mode 2: Y_i = 0.5 X_i + 0.5 sum_{j in N(i)} X_j / sqrt(deg_i deg_j)   (lazy normalised walk)
// accumulate: Y += result instead of Y = result.
__device__ __forceinline__ float edge_weight(int mode, const int64_t *row_ptr, int64_t j, float degi)
{
    if (mode == 0) return 1.f;
    const float dj = (float)(row_ptr[j + 1] - row_ptr[j]);
    return mode == 1 ? 1.f / dj : rsqrtf(degi * dj);
}

// Any width d <= 64, lanes over channels, neighbours one after the other: the widths and alignments
// that the vector kernel below does not take.
__global__ void aggregate_kernel(int64_t N, const int64_t *row_ptr, const int32_t *col, const float *X,
                                 int d, float *Y, int mode, int accumulate)
{
    const int lane = threadIdx.x & 31;
    const int64_t wglob = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = wglob; i < N; i += nw) {
        const int64_t e0 = row_ptr[i], e1 = row_ptr[i + 1];
        const float degi = (float)(e1 - e0);
        float a0 = 0.f, a1 = 0.f;
        for (int64_t e = e0; e < e1; ++e) {
            const int64_t j = col[e];
            float wgt = 1.f;
            if (mode == 1) {
                const float dj = (float)(row_ptr[j + 1] - row_ptr[j]);
                wgt = 1.f / dj;
            } else if (mode == 2) {
                const float dj = (float)(row_ptr[j + 1] - row_ptr[j]);
                wgt = rsqrtf(degi * dj);
            }
            if (lane < d) a0 += wgt * X[j * d + lane];
            if (lane + 32 < d) a1 += wgt * X[j * d + lane + 32];
        }
        if (mode == 0 && e1 > e0) { a0 /= degi; a1 /= degi; }
        if (mode == 2) {
            if (lane < d) a0 = 0.5f * X[i * d + lane] + 0.5f * a0;
            if (lane + 32 < d) a1 = 0.5f * X[i * d + lane + 32] + 0.5f * a1;
        }
        if (lane < d) Y[i * d + lane] = accumulate ? Y[i * d + lane] + a0 : a0;
        if (lane + 32 < d) Y[i * d + lane + 32] = accumulate ? Y[i * d + lane + 32] + a1 : a1;
    }
}

// Rows of D = 8, 16 or 64 floats on a 16-byte boundary: a row is D / 4 lanes of 16 bytes, so a warp
// reads 128 / D neighbours at once (2 of the 64-wide rows, 8 of the 16-wide).  The warp takes its
// columns 32 at a time, one coalesced load, and every lane forms the weight of one edge; a lane
// group then gets its neighbour and weight by shuffle, with four gathers in flight.  Bound by the
// L2 gathers (N = 46 thousand, 1.0 M edges, D = 64: 256 MB a launch; one neighbour at a time over 32
// lanes took 36 us, and 80 us with the transpose's weights formed once per channel group).
template <int D>
__global__ void __launch_bounds__(256) aggregate_vec_kernel(int64_t N, const int64_t *row_ptr, const int32_t *col,
                                                            const float *X, float *Y, int mode, int accumulate)
{
    constexpr int LPR = D / 4;              // lanes of a row
    constexpr int NB = 32 / LPR;            // neighbours at once
    const int lane = threadIdx.x & 31, sub = lane / LPR, c4 = lane % LPR;
    const int64_t wglob = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const float4 *X4 = reinterpret_cast<const float4 *>(X);
    for (int64_t i = wglob; i < N; i += nw) {
        const int64_t e0 = row_ptr[i], e1 = row_ptr[i + 1];
        const float degi = (float)(e1 - e0);
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int64_t eb = e0; eb < e1; eb += 32) {
            const int cnt = (int)min((int64_t)32, e1 - eb);
            int j = 0;
            float w = 0.f;
            if (lane < cnt) {
                j = col[eb + lane];
                w = edge_weight(mode, row_ptr, j, degi);
            }
#pragma unroll 4
            for (int k = 0; k < cnt; k += NB) {
                const int jj = __shfl_sync(0xFFFFFFFFu, j, (k + sub) & 31);
                const float ww = __shfl_sync(0xFFFFFFFFu, w, (k + sub) & 31);
                if (k + sub < cnt) {
                    const float4 v = X4[(int64_t)jj * LPR + c4];
                    a.x += ww * v.x; a.y += ww * v.y; a.z += ww * v.z; a.w += ww * v.w;
                }
            }
        }
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) {
            a.x += __shfl_xor_sync(0xFFFFFFFFu, a.x, o);
            a.y += __shfl_xor_sync(0xFFFFFFFFu, a.y, o);
            a.z += __shfl_xor_sync(0xFFFFFFFFu, a.z, o);
            a.w += __shfl_xor_sync(0xFFFFFFFFu, a.w, o);
        }
        if (sub == 0) {
            if (mode == 0 && e1 > e0) { a.x /= degi; a.y /= degi; a.z /= degi; a.w /= degi; }
            if (mode == 2) {
                const float4 x = X4[i * LPR + c4];
                a.x = 0.5f * x.x + 0.5f * a.x; a.y = 0.5f * x.y + 0.5f * a.y;
                a.z = 0.5f * x.z + 0.5f * a.z; a.w = 0.5f * x.w + 0.5f * a.w;
            }
            float4 *y = reinterpret_cast<float4 *>(Y) + i * LPR + c4;
            if (accumulate) {
                const float4 o = *y;
                a.x += o.x; a.y += o.y; a.z += o.z; a.w += o.w;
            }
            *y = a;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Dense forward: H = ReLU(X Ws + AGG Wn + b), X/AGG: N x din, Ws/Wn: din x 64 (BF16), H: N x 64.
__global__ void dense_fwd_kernel(int64_t N, const float *X, const float *AGG, int din, const uint16_t *Ws,
                                 const uint16_t *Wn, const float *b, float *H, int relu)
{
    extern __shared__ float sm[];
    float *ws = sm, *wn = sm + din * HID;
    for (int t = threadIdx.x; t < din * HID; t += blockDim.x) { ws[t] = bf16_to_f(Ws[t]); wn[t] = bf16_to_f(Wn[t]); }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t wglob = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = wglob; i < N; i += nw) {
        const float x0 = lane < din ? X[i * din + lane] : 0.f;
        const float x1 = lane + 32 < din ? X[i * din + lane + 32] : 0.f;
        const float g0 = lane < din ? AGG[i * din + lane] : 0.f;
        const float g1 = lane + 32 < din ? AGG[i * din + lane + 32] : 0.f;
        float o0 = b[lane], o1 = b[lane + 32];
        for (int k = 0; k < din; ++k) {
            const float xk = __shfl_sync(0xFFFFFFFFu, k < 32 ? x0 : x1, k & 31);
            const float gk = __shfl_sync(0xFFFFFFFFu, k < 32 ? g0 : g1, k & 31);
            o0 += xk * ws[k * HID + lane] + gk * wn[k * HID + lane];
            o1 += xk * ws[k * HID + lane + 32] + gk * wn[k * HID + lane + 32];
        }
        if (relu) { o0 = fmaxf(o0, 0.f); o1 = fmaxf(o1, 0.f); }
        H[i * HID + lane] = o0;
        H[i * HID + lane + 32] = o1;
    }
}

// Dense backward (data): dPRE = dH * [H > 0]; dXs = dPRE Ws^T; T = dPRE Wn^T  (N x din each).
__global__ void dense_bwd_kernel(int64_t N, int din, const uint16_t *Ws, const uint16_t *Wn, const float *H,
                                 const float *dH, float *dPRE, float *dXs, float *T)
{
    extern __shared__ float sm[];
    float *wsT = sm, *wnT = sm + din * HID;   // transposed: [c][k]
    for (int t = threadIdx.x; t < din * HID; t += blockDim.x) {
        const int k = t / HID, c = t % HID;
        wsT[c * din + k] = bf16_to_f(Ws[t]);
        wnT[c * din + k] = bf16_to_f(Wn[t]);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t wglob = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = wglob; i < N; i += nw) {
        const float p0 = H[i * HID + lane] > 0.f ? dH[i * HID + lane] : 0.f;
        const float p1 = H[i * HID + lane + 32] > 0.f ? dH[i * HID + lane + 32] : 0.f;
        dPRE[i * HID + lane] = p0;
        dPRE[i * HID + lane + 32] = p1;
        float s0 = 0.f, s1 = 0.f, t0 = 0.f, t1 = 0.f;   // outputs k = lane, lane + 32
        for (int c = 0; c < HID; ++c) {
            const float pc = __shfl_sync(0xFFFFFFFFu, c < 32 ? p0 : p1, c & 31);
            if (lane < din) { s0 += pc * wsT[c * din + lane]; t0 += pc * wnT[c * din + lane]; }
            if (lane + 32 < din) { s1 += pc * wsT[c * din + lane + 32]; t1 += pc * wnT[c * din + lane + 32]; }
        }
        if (lane < din) { dXs[i * din + lane] = s0; T[i * din + lane] = t0; }
        if (lane + 32 < din) { dXs[i * din + lane + 32] = s1; T[i * din + lane + 32] = t1; }
    }
}

// ---------------------------------------------------------------------------------------------
// Tensor-core dense layers (din = 16 or 64): mma.sync m16n8k16 with BF16 operands and FP32
// accumulation, one warp per tile of 16 vertices.  The weights are BF16 already; an FP32
// activation x is split into two BF16 parts hi = bf16(x), lo = bf16(x - hi), and hi W + lo W is
// accumulated in FP32: each product of BF16 values is exact in FP32, so the only rounding beyond
// the FP32 sums is the part of x below lo (about 2^-17 of |x|).
// Fragment layout of m16n8k16 (PTX ISA): g = lane / 4, q = lane % 4; A (16 x 16, row major) regs
// a0..a3 = rows g, g + 8, g, g + 8 at columns 2q, 2q + 1 (a0, a1) and 2q + 8, 2q + 9 (a2, a3);
// B (16 x 8, column major) regs b0, b1 = rows 2q, 2q + 1 and 2q + 8, 2q + 9 of column g;
// C/D (16 x 8) c0, c1 = row g, columns 2q, 2q + 1; c2, c3 = row g + 8, same columns.  The lower
// 16 bits of a register hold the element with the smaller index.
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
                 "{%8, %9}, {%0, %1, %2, %3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// two FP32 values (element k, k + 1) -> packed BF16 high parts and packed BF16 residuals
__device__ __forceinline__ void split_bf16x2(float x0, float x1, uint32_t &hi, uint32_t &lo)
{
    const __nv_bfloat16 h0 = __float2bfloat16_rn(x0), h1 = __float2bfloat16_rn(x1);
    const __nv_bfloat16 l0 = __float2bfloat16_rn(x0 - __bfloat162float(h0));
    const __nv_bfloat16 l1 = __float2bfloat16_rn(x1 - __bfloat162float(h1));
    hi = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
    lo = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
}

// H = ReLU([X | AGG] [Ws; Wn] + b): K = 2 DIN, 64 outputs = 8 column tiles.  Bound by reading X and
// AGG and writing H once.  The rows of X and of AGG that a warp's tile needs are all in flight before
// the first is multiplied (64 registers for DIN = 64: 8 KB a warp, 128 KB an SM with two blocks), and
// a block stays for several tiles (at most two blocks per SM), since laying the weights out as pairs
// costs as much as a tile (2,432 blocks that each laid them out for about one tile per warp: 161 us at
// N = 390 thousand, DIN = 64).
template <int DIN>
__global__ void __launch_bounds__(256, 2) dense_fwd_mma_kernel(int64_t N, const float *X, const float *AGG,
                                                               const uint16_t *Ws, const uint16_t *Wn,
                                                               const float *b, float *H)
{
    constexpr int K = 2 * DIN, KP = K / 2 + 4;           // pairs per output column (+4: banks)
    constexpr int KS = DIN / 16;                          // k-steps of X, and of AGG
    __shared__ uint32_t wt[HID * KP];                     // [n][k pair]: (k, k+1) of output n
    for (int t = threadIdx.x; t < HID * (K / 2); t += blockDim.x) {
        const int n = t % HID, kp = t / HID, k = 2 * kp;  // a warp reads 32 consecutive columns
        const uint16_t *W = k < DIN ? Ws + k * HID : Wn + (k - DIN) * HID;
        wt[n * KP + kp] = (uint32_t)W[n] | ((uint32_t)W[HID + n] << 16);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const int64_t wglob = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t tile = wglob; tile * 16 < N; tile += nw) {
        const int64_t r0 = tile * 16 + g, r1 = r0 + 8;
        float2 v[2][KS][4];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const float *src = m == 0 ? X : AGG;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks)
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const int64_t r = (h & 1) ? r1 : r0;
                    const int kk = ks * 16 + 2 * q + ((h & 2) ? 8 : 0);
                    v[m][ks][h] = r < N ? *reinterpret_cast<const float2 *>(src + r * DIN + kk) : make_float2(0.f, 0.f);
                }
        }
        float acc[8][4];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            acc[nt][0] = acc[nt][2] = __ldg(b + nt * 8 + 2 * q);
            acc[nt][1] = acc[nt][3] = __ldg(b + nt * 8 + 2 * q + 1);
        }
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                uint32_t ah[4], al[4];
#pragma unroll
                for (int h = 0; h < 4; ++h) split_bf16x2(v[m][ks][h].x, v[m][ks][h].y, ah[h], al[h]);
#pragma unroll
                for (int nt = 0; nt < 8; ++nt) {
                    const uint32_t *wr = wt + (nt * 8 + g) * KP + (m * KS + ks) * 8 + q;
                    const uint32_t b0 = wr[0], b1 = wr[4];
                    mma_bf16_16816(acc[nt], ah, b0, b1);
                    mma_bf16_16816(acc[nt], al, b0, b1);
                }
            }
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const int c = nt * 8 + 2 * q;
            if (r0 < N) *reinterpret_cast<float2 *>(H + r0 * HID + c) = make_float2(fmaxf(acc[nt][0], 0.f), fmaxf(acc[nt][1], 0.f));
            if (r1 < N) *reinterpret_cast<float2 *>(H + r1 * HID + c) = make_float2(fmaxf(acc[nt][2], 0.f), fmaxf(acc[nt][3], 0.f));
        }
    }
}

// Backward (data) of one layer: dPRE = dH * [H > 0] (written out), then dXs = dPRE Ws^T and
// T = dPRE Wn^T: K = 64, DIN outputs each, one pass per weight matrix.
template <int DIN>
__global__ void __launch_bounds__(256) dense_bwd_mma_kernel(int64_t N, const uint16_t *Ws, const uint16_t *Wn,
                                                            const float *H, const float *dH, float *dPRE,
                                                            float *dXs, float *T)
{
    constexpr int KP = HID / 2 + 4;
    __shared__ uint32_t wt[2][DIN * KP];                  // [m][j][c pair]: W_m[j][c], W_m[j][c+1]
    for (int t = threadIdx.x; t < DIN * (HID / 2); t += blockDim.x) {
        const int j = t / (HID / 2), cp = t % (HID / 2);
        wt[0][j * KP + cp] = reinterpret_cast<const uint32_t *>(Ws)[t];
        wt[1][j * KP + cp] = reinterpret_cast<const uint32_t *>(Wn)[t];
    }
    __syncthreads();
    constexpr int NT = DIN / 8;
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const int64_t wglob = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t tile = wglob; tile * 16 < N; tile += nw) {
        const int64_t r0 = tile * 16 + g, r1 = r0 + 8;
        // A fragments of dPRE for the 4 k-steps (c = 16 ks + ...), hi and lo parts
        uint32_t ah[4][4], al[4][4];
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int64_t r = (h & 1) ? r1 : r0;
                const int c = ks * 16 + 2 * q + ((h & 2) ? 8 : 0);
                float2 p = make_float2(0.f, 0.f);
                if (r < N) {
                    const float2 hv = *reinterpret_cast<const float2 *>(H + r * HID + c);
                    const float2 dv = *reinterpret_cast<const float2 *>(dH + r * HID + c);
                    p = make_float2(hv.x > 0.f ? dv.x : 0.f, hv.y > 0.f ? dv.y : 0.f);
                    *reinterpret_cast<float2 *>(dPRE + r * HID + c) = p;
                }
                split_bf16x2(p.x, p.y, ah[ks][h], al[ks][h]);
            }
        }
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            float *out = m == 0 ? dXs : T;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    const uint32_t *wr = wt[m] + (nt * 8 + g) * KP + ks * 8 + q;
                    const uint32_t b0 = wr[0], b1 = wr[4];
                    mma_bf16_16816(acc, ah[ks], b0, b1);
                    mma_bf16_16816(acc, al[ks], b0, b1);
                }
                const int j = nt * 8 + 2 * q;
                if (r0 < N) *reinterpret_cast<float2 *>(out + r0 * DIN + j) = make_float2(acc[0], acc[1]);
                if (r1 < N) *reinterpret_cast<float2 *>(out + r1 * DIN + j) = make_float2(acc[2], acc[3]);
            }
        }
    }
}

// out[din x dout] += A^T B over the rows of a chunk; A: N x din, B: N x dout (both at most 64 wide).
// Also colsum[dout] += sum of the rows of B when colsum != null.  One block of 512 threads per SM:
// tiles of 32 rows go through shared memory (the next tile's loads are in flight while this one is
// multiplied), a thread keeps a 4 x 4 block of the product in registers (two 16-byte shared loads
// for 16 multiply-adds), and the 512 / (4 DK) thread groups take different rows of a tile.  Each
// tile is summed on its own before it joins the running sum, so a sum is a tree of 16 (or 4), then
// tiles, then blocks.  Bound by the FP32 multiply-adds.  (One block per 1,024 rows with two shared
// loads per multiply-add took 480 us at N = 46 thousand, DK = 64, 45 blocks; with it a training batch
// of 16 graphs took 2.57 ms, with this kernel and the two above and below 0.38 ms.)  DK = 16 or 64
// is din rounded up; columns and rows beyond the matrices are zeros.
constexpr int WG_T = 512, WG_R = 32;

// tile rows [t0, t0 + 32) of M (N x d, d <= DP): this thread's share, as DP * 32 / 512 floats
template <int DP>
__device__ __forceinline__ void wg_load(const float *M, int d, int64_t t0, int64_t r1, bool vec, float (&v)[DP * WG_R / WG_T])
{
    constexpr int PER = DP * WG_R / WG_T;          // 1 (DP = 16) or 4 (DP = 64)
    if (PER == 4 && vec) {                         // d == DP, rows contiguous, 16-byte aligned
        const int o = threadIdx.x * 4;
        const float4 x = t0 + o / DP < r1 ? *reinterpret_cast<const float4 *>(M + t0 * DP + o) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[0] = x.x; v[1 % PER] = x.y; v[2 % PER] = x.z; v[3 % PER] = x.w;
    } else {
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int o = threadIdx.x * PER + u, rr = o / DP, k = o % DP;
            v[u] = k < d && t0 + rr < r1 ? M[(t0 + rr) * d + k] : 0.f;
        }
    }
}

template <int DP>
__device__ __forceinline__ void wg_store(float *s, const float (&v)[DP * WG_R / WG_T])
{
    constexpr int PER = DP * WG_R / WG_T;
    if (PER == 4) *reinterpret_cast<float4 *>(s + threadIdx.x * 4) = make_float4(v[0], v[1 % PER], v[2 % PER], v[3 % PER]);
    else s[threadIdx.x] = v[0];
}

template <int DK>
__global__ void __launch_bounds__(WG_T, 1) wgrad_kernel(int64_t N, const float *A, int din, const float *B, int dout,
                                                        float *out, float *colsum, int64_t chunk, int vec)
{
    constexpr int TG = DK * HID / 16;              // threads of a group: one 4 x 4 block of out each
    constexpr int NG = WG_T / TG, RG = WG_R / NG;  // groups, rows of a tile per group
    __shared__ __align__(16) float sa[2][WG_R * DK];
    __shared__ __align__(16) float sb[2][WG_R * HID];
    __shared__ __align__(16) float red[DK * HID];
    const int64_t r0 = (int64_t)blockIdx.x * chunk, r1 = min(N, r0 + chunk);
    const int grp = threadIdx.x / TG, ty = (threadIdx.x % TG) / 16, tx = threadIdx.x % 16;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    float cs = 0.f;
    float va[DK * WG_R / WG_T], vb[HID * WG_R / WG_T];
    wg_load<DK>(A, din, r0, r1, vec & 1, va);
    wg_load<HID>(B, dout, r0, r1, (vec >> 1) & 1, vb);
    int buf = 0;
    for (int64_t t0 = r0; t0 < r1; t0 += WG_R, buf ^= 1) {
        // two buffers: the barrier below also says that everyone is done with the tile before last
        wg_store<DK>(sa[buf], va);
        wg_store<HID>(sb[buf], vb);
        __syncthreads();
        if (t0 + WG_R < r1) {
            wg_load<DK>(A, din, t0 + WG_R, r1, vec & 1, va);
            wg_load<HID>(B, dout, t0 + WG_R, r1, (vec >> 1) & 1, vb);
        }
        float s[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) s[i][j] = 0.f;
#pragma unroll
        for (int rr = 0; rr < RG; ++rr) {
            const float4 x = *reinterpret_cast<const float4 *>(&sa[buf][(grp * RG + rr) * DK + 4 * ty]);
            const float4 y = *reinterpret_cast<const float4 *>(&sb[buf][(grp * RG + rr) * HID + 4 * tx]);
            const float xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) s[i][j] += xs[i] * ys[j];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] += s[i][j];
        if (colsum) {                              // thread: column t % 64, 4 rows of the tile
            float c = 0.f;
#pragma unroll
            for (int rr = 0; rr < WG_R * HID / WG_T; ++rr)
                c += sb[buf][(threadIdx.x / HID + rr * (WG_T / HID)) * HID + threadIdx.x % HID];
            cs += c;
        }
    }
    // the groups' products meet in shared memory, then one 16-byte atomic per four outputs
    for (int g = 0; g < NG; ++g) {
        __syncthreads();
        if (grp == g) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float4 *q = reinterpret_cast<float4 *>(&red[(4 * ty + i) * HID + 4 * tx]);
                float4 o = g ? *q : make_float4(0.f, 0.f, 0.f, 0.f);
                o.x += acc[i][0]; o.y += acc[i][1]; o.z += acc[i][2]; o.w += acc[i][3];
                *q = o;
            }
        }
    }
    __syncthreads();
    if (vec & 4) {                                 // dout == 64 and out 16-byte aligned
        for (int t = threadIdx.x; t < din * (HID / 4); t += WG_T)
            atomicAdd(reinterpret_cast<float4 *>(out) + t, *reinterpret_cast<const float4 *>(&red[4 * t]));
    } else {
        for (int t = threadIdx.x; t < din * dout; t += WG_T)
            atomicAdd(&out[t], red[(t / dout) * HID + t % dout]);
    }
    if (colsum) {
        __syncthreads();
        if (threadIdx.x < HID) red[threadIdx.x] = 0.f;
        __syncthreads();
        atomicAdd(&red[threadIdx.x % HID], cs);
        __syncthreads();
        if (threadIdx.x < dout) atomicAdd(&colsum[threadIdx.x], red[threadIdx.x]);
    }
}

// the same for one column B (dout == 1): out[k] += sum_i A[i][k] B[i].  Bound by reading A once:
// lanes over columns, the four thread groups take every fourth row.
__global__ void __launch_bounds__(256) wgrad1_kernel(int64_t N, const float *A, int din, const float *B, float *out,
                                                     float *colsum, int64_t chunk)
{
    __shared__ float red[4][HID + 1];
    const int64_t r0 = (int64_t)blockIdx.x * chunk, r1 = min(N, r0 + chunk);
    const int k = threadIdx.x % HID, grp = threadIdx.x / HID;
    float acc = 0.f, cs = 0.f;
    for (int64_t t0 = r0 + grp; t0 < r1; t0 += 4 * 8) {
        float s = 0.f, c = 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t r = t0 + 4 * u;
            const float bv = r < r1 ? B[r] : 0.f;
            if (k < din && r < r1) s += A[r * din + k] * bv;
            c += bv;
        }
        acc += s;
        cs += c;
    }
    red[grp][k] = acc;
    if (k == 0) red[grp][HID] = cs;
    __syncthreads();
    if (threadIdx.x < din) atomicAdd(&out[threadIdx.x], (red[0][k] + red[1][k]) + (red[2][k] + red[3][k]));
    if (colsum && threadIdx.x == 0) atomicAdd(colsum, (red[0][HID] + red[1][HID]) + (red[2][HID] + red[3][HID]));
}

// z = H wo + bo
__global__ void out_fwd_kernel(int64_t N, const float *H, const uint16_t *wo, const float *bo, float *z)
{
    const int lane = threadIdx.x & 31;
    const int64_t wglob = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const float w0 = bf16_to_f(wo[lane]), w1 = bf16_to_f(wo[lane + 32]);
    for (int64_t i = wglob; i < N; i += nw) {
        float s = H[i * HID + lane] * w0 + H[i * HID + lane + 32] * w1;
        s = warp_sum(s);
        if (lane == 0) z[i] = s + bo[0];
    }
}

// dH = dz wo^T
__global__ void out_bwd_kernel(int64_t N, const uint16_t *wo, const float *dz, float *dH)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < N * HID; t += (int64_t)gridDim.x * blockDim.x)
        dH[t] = dz[t / HID] * bf16_to_f(wo[t % HID]);
}

// Per graph (one block): L1 = mean softplus(-y z), L2 = mean softplus(y z), m = mean tanh z;
// loss_g = min(L1, L2) + lambda m^2; dz for the chosen sign; loss += loss_g / G.
__device__ __forceinline__ float softplus_f(float x) { return x > 20.f ? x : log1pf(expf(x)); }
__device__ __forceinline__ float sigmoid_f(float x) { return 1.f / (1.f + expf(-x)); }

__global__ void loss_kernel(int G, const int64_t *graph_ptr, const float *z, const int8_t *y, float lambda,
                            float *stats, float *dz, float *loss)
{
    const int g = blockIdx.x;
    const int64_t v0 = graph_ptr[g], v1 = graph_ptr[g + 1];
    const float n = (float)(v1 - v0);
    float l1 = 0.f, l2 = 0.f, th = 0.f;
    for (int64_t i = v0 + threadIdx.x; i < v1; i += blockDim.x) {
        const float yz = (float)y[i] * z[i];
        l1 += softplus_f(-yz);
        l2 += softplus_f(yz);
        th += tanhf(z[i]);
    }
    __shared__ float red[3][32];
    l1 = warp_sum(l1); l2 = warp_sum(l2); th = warp_sum(th);
    if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = l1; red[1][threadIdx.x >> 5] = l2; red[2][threadIdx.x >> 5] = th; }
    __syncthreads();
    if (threadIdx.x == 0) {
        float a = 0.f, b = 0.f, c = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { a += red[0][w]; b += red[1][w]; c += red[2][w]; }
        red[0][0] = a / n; red[1][0] = b / n; red[2][0] = c / n;
    }
    __syncthreads();
    const float L1 = red[0][0], L2 = red[1][0], m = red[2][0];
    const float sgn = L1 <= L2 ? 1.f : -1.f;   // target y (sgn = 1) or -y
    const float lg = fminf(L1, L2) + lambda * m * m;
    if (threadIdx.x == 0) {
        stats[g * 4 + 0] = L1; stats[g * 4 + 1] = L2; stats[g * 4 + 2] = m; stats[g * 4 + 3] = lg;
        atomicAdd(loss, lg / (float)G);
    }
    for (int64_t i = v0 + threadIdx.x; i < v1; i += blockDim.x) {
        const float t = sgn * (float)y[i];
        const float th_i = tanhf(z[i]);
        dz[i] = (-t * sigmoid_f(-t * z[i]) + lambda * 2.f * m * (1.f - th_i * th_i)) / (n * (float)G);
    }
}

__global__ void adam_kernel(int64_t P, float *p, const float *g, float *m, float *v, uint16_t *pb, float lr,
                            float b1, float b2, float eps, float c1, float c2)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < P; t += (int64_t)gridDim.x * blockDim.x) {
        const float gt = g[t];
        const float mt = b1 * m[t] + (1.f - b1) * gt;
        const float vt = b2 * v[t] + (1.f - b2) * gt * gt;
        m[t] = mt;
        v[t] = vt;
        const float pt = p[t] - lr * (mt / c1) / (sqrtf(vt / c2) + eps);
        p[t] = pt;
        pb[t] = __bfloat16_as_ushort(__float2bfloat16_rn(pt));
    }
}

__global__ void to_bf16_kernel(int64_t P, const float *p, uint16_t *pb)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < P; t += (int64_t)gridDim.x * blockDim.x)
        pb[t] = __bfloat16_as_ushort(__float2bfloat16_rn(p[t]));
}

// ---------------------------------------------------------------------------------------------
// Features: 8 channels of +-1 Philox noise, diffused by `steps` lazy normalised-walk steps, then
// centred and scaled to unit RMS per graph; channel 8 = log(1 + deg), channel 9 = deg / mean deg
// of the graph; channels 10..15 = 0.
__device__ __forceinline__ float noise_sign(uint32_t vertex, int c, uint32_t graph, uint32_t k0, uint32_t k1)
{
    const uint4 u = philox4x32_10(make_uint4(vertex, (uint32_t)c, graph, 0x4D504E4Eu), k0, k1);
    return (u.x >> 31) ? -1.f : 1.f;
}

__global__ void feat_init_kernel(int64_t N, int G, const int64_t *graph_ptr, const uint32_t *graph_id,
                                 uint32_t k0, uint32_t k1, float *R)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < N * NRAND; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / NRAND;
        const int c = (int)(t % NRAND);
        const int g = (int)graph_of(graph_ptr, G, i);
        R[t] = noise_sign((uint32_t)(i - graph_ptr[g]), c, graph_id[g], k0, k1);
    }
}

// The noise channels of graphs of up to a few thousand vertices, all walk steps in one launch: a cluster
// of eight blocks per graph, one channel each (the channels are independent).  A block keeps
// y = D^-1/2 x of its graph in shared memory, two buffers; in y a lazy walk step is
//     y_i <- y_i / 2 + (mean over the neighbours of y_j) / 2,
// with no edge weights, and x = D^1/2 y at the end (an isolated vertex: x <- x / 2).
//
// Columns.  One lane per row reading the CSR in place costs an L1 pass per lane; so the vertices are
// renumbered by falling degree (a counting sort in shared memory), cut into slices of 32, and entry k
// of the 32 rows of a slice laid out as one run of 32 16-bit numbers, short rows filled up with the
// number n, whose y is 0.  A warp then reads 64 consecutive bytes for 32 entries, and nothing in the
// inner loop is predicated.  The sort leaves next to no filling.  The cluster's blocks lay out every
// eighth slice each; the runs live in the caller's X and scratch, which hold 128 bytes per vertex and
// are free until the result is written (run r of a graph of n vertices: X for r < n, then the two
// halves of the scratch), so a graph whose runs exceed 2 n, or of more than `cap` vertices, is left
// to walk_rest_kernel.  The sums run in CSR order whatever the renumbering.  Only columns inside the graph have
// a rank: one that leads to another graph is laid out as the number n, and the batch is marked for
// walk_rest_kernel.
//
// Bound by the random shared-memory reads: 32 random words take 3.5 passes on average.  Inference on
// 128 graphs of 1,000 to 5,000 vertices (256 steps): 120 ms with one launch per step (470 us each), 18.6 ms
// with four lanes per CSR row, 12.4 ms so; one graph of 1,999 vertices 2.18 -> 1.74 -> 0.87 ms.
constexpr int DF_T = 1024, DF_CL = NRAND, DF_BINS = 256;

// shared memory of a block, n + 1 <= cap + 1 entries an array (the kernel carves, the host sizes)
struct DfLayout {
    uint32_t y[2], perm, deg, slice, total;
};
__host__ __device__ inline DfLayout df_layout(int cap)
{
    DfLayout L;
    const uint32_t c = (uint32_t)(cap + 32) & ~31u;
    uint32_t o = 0;
    L.y[0] = o; o += 4 * c + 4 * 32;
    L.y[1] = o; o += 4 * c + 4 * 32;
    L.perm = o; o += 2 * c;
    L.deg = o; o += 2 * c;
    L.slice = o; o += 4 * (c / 32 + 1);
    L.total = (o + 15) & ~15u;
    return L;
}

// runs of a graph: r < n in X, the next n / 2 in R0, the next n / 2 in R1
struct DfRuns {
    uint16_t *x, *r0, *r1;
    int n;
    __device__ __forceinline__ int limit() const { return n + 2 * (n / 2); }
    // address of run r and how many runs follow it contiguously (itself included)
    __device__ __forceinline__ uint16_t *at(int r, int &room) const
    {
        const int h = n / 2;
        if (r < n) { room = n - r; return x + (size_t)r * 32; }
        if (r < n + h) { room = n + h - r; return r0 + (size_t)(r - n) * 32; }
        room = n + 2 * h - r;
        return r1 + (size_t)(r - n - h) * 32;
    }
};

__global__ void __cluster_dims__(DF_CL, 1, 1) __launch_bounds__(DF_T, 2)
diffuse_kernel(const int64_t *graph_ptr, const uint32_t *graph_id, const int64_t *row_ptr, const int32_t *col,
               uint32_t k0, uint32_t k1, int steps, int cap, float *X, float *R0, float *R1)
{
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ int hist[DF_BINS];
    __shared__ int nruns;
    __shared__ int leaves;                                             // block 0's: a column leads out of the graph
    const int g = blockIdx.x / DF_CL, ch = blockIdx.x % DF_CL;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t v0 = graph_ptr[g];
    const int64_t n64 = graph_ptr[g + 1] - v0;
    const int64_t *rp = row_ptr + v0;
    const uint32_t id = graph_id[g];
    float *res = R0 + v0 * NRAND + ch;                                 // vertex i at element i * NRAND
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    bool fits = n64 <= cap;                                            // the same in all blocks of the cluster
    const int n = (int)n64, ns = (n + 31) / 32;
    const DfLayout L = df_layout(cap);
    float *ya = reinterpret_cast<float *>(sm_raw + L.y[0]), *yb = reinterpret_cast<float *>(sm_raw + L.y[1]);
    uint16_t *perm = reinterpret_cast<uint16_t *>(sm_raw + L.perm);    // vertex of rank r
    uint16_t *deg = reinterpret_cast<uint16_t *>(sm_raw + L.deg);      // degree of rank r
    uint32_t *slice = reinterpret_cast<uint32_t *>(sm_raw + L.slice);  // first run of slice s
    uint16_t *rank = reinterpret_cast<uint16_t *>(yb);                 // rank of vertex i, until the walk
    DfRuns runs;
    runs.x = reinterpret_cast<uint16_t *>(X + v0 * FIN);
    runs.r0 = reinterpret_cast<uint16_t *>(R0 + v0 * NRAND);
    runs.r1 = reinterpret_cast<uint16_t *>(R1 + v0 * NRAND);
    runs.n = n;
    if (threadIdx.x == 0) leaves = 0;
    if (fits && ch == 0) {
        // ranks by falling degree (degrees from DF_BINS - 1 on share a bin), by block 0 for the cluster:
        // the atomics rank equal degrees in any order
        for (int b = threadIdx.x; b < DF_BINS; b += DF_T) hist[b] = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += DF_T)
            atomicAdd(&hist[DF_BINS - 1 - (int)min((int64_t)(DF_BINS - 1), rp[i + 1] - rp[i])], 1);
        __syncthreads();
        if (warp == 0) {
            int run = 0;
            for (int b0 = 0; b0 < DF_BINS; b0 += 32) {
                const int h = hist[b0 + lane];
                int x = h;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xFFFFFFFFu, x, o);
                    if (lane >= o) x += t;
                }
                hist[b0 + lane] = run + x - h;
                run += __shfl_sync(0xFFFFFFFFu, x, 31);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += DF_T) {
            const int64_t d = rp[i + 1] - rp[i];
            const int r = atomicAdd(&hist[DF_BINS - 1 - (int)min((int64_t)(DF_BINS - 1), d)], 1);
            perm[r] = (uint16_t)i;
            deg[r] = (uint16_t)min(d, (int64_t)65535);                 // (65,535 runs exceed the limit)
            rank[i] = (uint16_t)r;
        }
        for (int r = n + threadIdx.x; r < ns * 32; r += DF_T) deg[r] = 0;
        __syncthreads();
        // the slices' first runs
        for (int s = warp; s < ns; s += DF_T / 32) {
            const uint32_t len = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)deg[32 * s + lane]);
            if (lane == 0) slice[s + 1] = len;
        }
        __syncthreads();
        if (warp == 0) {
            int run = 0;
            for (int s0 = 0; s0 < ns; s0 += 32) {
                int x = s0 + lane < ns ? (int)slice[s0 + lane + 1] : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xFFFFFFFFu, x, o);
                    if (lane >= o) x += t;
                }
                if (s0 + lane < ns) slice[s0 + lane + 1] = (uint32_t)(run + x);
                run += __shfl_sync(0xFFFFFFFFu, x, 31);
            }
            if (lane == 0) { slice[0] = 0; nruns = run; }
        }
    }
    if (fits) {
        cluster.sync();
        fits = *cluster.map_shared_rank(&nruns, 0) <= runs.limit();
        if (fits && ch != 0) {
            const uint16_t *p0 = cluster.map_shared_rank(perm, 0), *d0 = cluster.map_shared_rank(deg, 0);
            const uint32_t *s0 = cluster.map_shared_rank(slice, 0);
            for (int r = threadIdx.x; r < ns * 32; r += DF_T) {
                deg[r] = d0[r];
                if (r >= n) continue;
                const uint16_t v = p0[r];
                perm[r] = v;
                rank[v] = (uint16_t)r;
            }
            for (int s = threadIdx.x; s <= ns; s += DF_T) slice[s] = s0[s];
        }
        cluster.sync();
    }
    if (fits) {
        bool out = false;
        for (int s = warp * DF_CL + ch; s < ns; s += DF_CL * (DF_T / 32)) {
            const int r = 32 * s + lane;
            const int64_t e0 = r < n ? rp[perm[r]] : 0;
            const int d = deg[r], len = (int)(slice[s + 1] - slice[s]);
            for (int k0 = 0; k0 < len; k0 += 4) {      // four columns in flight
                uint32_t j[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) j[u] = k0 + u < d ? (uint32_t)col[e0 + k0 + u] - (uint32_t)v0 : 0xFFFFFFFFu;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool in = j[u] < (uint32_t)n;
                    out |= k0 + u < d && !in;
                    if (k0 + u >= len) break;
                    int room;
                    runs.at((int)slice[s] + k0 + u, room)[lane] = in ? rank[j[u]] : (uint16_t)n;
                }
            }
        }
        if (out) *cluster.map_shared_rank(&leaves, 0) = 1;
        // all runs written (and seen by the whole cluster) before the first step reads them
        __threadfence();
        cluster.sync();
        __threadfence();
        for (int r = threadIdx.x; r < n; r += DF_T) {
            const float d = (float)deg[r];
            ya[r] = (d > 0.f ? 1.f / sqrtf(d) : 1.f) * noise_sign(perm[r], ch, id, k0, k1);
        }
        if (threadIdx.x == 0) { ya[n] = 0.f; yb[n] = 0.f; }
        __syncthreads();
        for (int t = 0; t < steps; ++t) {
            for (int s = warp; s < ns; s += DF_T / 32) {
                int r0 = (int)slice[s];
                const int rend = (int)slice[s + 1];
                float a = 0.f;
                while (r0 < rend) {
                    int room;
                    const uint16_t *p = runs.at(r0, room) + lane;
                    const int cnt = min(room, rend - r0);
                    int k = 0;
                    for (; k + 4 <= cnt; k += 4) {
                        const int j0 = p[0], j1 = p[32], j2 = p[64], j3 = p[96];
                        a += ya[j0]; a += ya[j1]; a += ya[j2]; a += ya[j3];
                        p += 128;
                    }
                    for (; k < cnt; ++k, p += 32) a += ya[*p];
                    r0 += cnt;
                }
                const int r = 32 * s + lane;
                if (r < n) {
                    const float d = (float)deg[r], y = ya[r];
                    yb[r] = d > 0.f ? 0.5f * y + 0.5f * (a / d) : 0.5f * y;
                }
            }
            __syncthreads();
            float *tmp = ya; ya = yb; yb = tmp;
        }
        // every block of the cluster is done with the runs in R0 before the result goes there
        cluster.sync();
        for (int r = threadIdx.x; r < n; r += DF_T) {
            const float d = (float)deg[r];
            res[(int64_t)perm[r] * NRAND] = ya[r] * (d > 0.f ? sqrtf(d) : 1.f);
        }
    } else {
        for (int64_t i = threadIdx.x; i < n64; i += DF_T) res[i * NRAND] = noise_sign((uint32_t)i, ch, id, k0, k1);
    }
    // what walk_rest_kernel has to take (X is free again): 1 = this graph, 2 = the whole batch, since a column
    // leads from this graph to another (written above before the cluster's barriers)
    if (ch == 0 && threadIdx.x == 0 && n64 > 0) {
        X[v0 * FIN] = !fits ? 1.f : (leaves ? 2.f : 0.f);
        X[v0 * FIN + 1] = 0.f;                                         // walk_rest_kernel's own mark
    }
}

// The walk steps of the graphs that diffuse_kernel marked, whose noise it left in R0: one cooperative
// launch, a warp per row as in aggregate_vec_kernel<8>, a grid barrier per step.  Without marked
// graphs it returns at once.  (One launch per step over all vertices would cost every batch `steps`
// launches for the rare graph that does not fit.)  Bound by the chain of dependent L2 reads of a row (bounds,
// column, its bounds and value), so by rows in flight, and by the grid barrier: 32 registers leave 64 warps an SM, and
// blocks of 1,024 threads keep the barrier to two arrivals an SM.  (us a step, 256 steps: a graph of 10^6 vertices of
// degree 6 beside 400 of 1,000: one launch per step, one neighbour at a time, 720; four blocks of 256 and a search for
// the row's graph in each step 1,120, without the search 951; this 285.  One of 12,000 beside one of 1,000: 12.9, 14.6,
// 14.1, 7.8.  With the block size written as a constant the compiler spills differently and the first takes 500.)
// A batch in which a column leads from one graph to another
// walks as a whole, from the noise on: every vertex's value is then read at its own step.
constexpr int WR_T = 1024;
__global__ void __launch_bounds__(WR_T, 2) walk_rest_kernel(int64_t N, int G, const int64_t *graph_ptr, const uint32_t *graph_id,
                                                        const int64_t *row_ptr, const int32_t *col, uint32_t k0, uint32_t k1,
                                                        int steps, float *X, float *R0, float *R1)
{
    // a mark of any graph: word 0 (diffuse_kernel's) at least v, or word 1 (set below)
    auto marked = [&](float v) {
        int any = 0;
        for (int g = threadIdx.x; g < G; g += blockDim.x) {
            if (graph_ptr[g + 1] <= graph_ptr[g]) continue;
            const float *m = X + graph_ptr[g] * FIN;
            any |= m[0] >= v || m[1] != 0.f;
        }
        return __syncthreads_or(any) != 0;
    };
    if (!marked(1.f)) return;
    cooperative_groups::grid_group grid = cooperative_groups::this_grid();
    const int lane = threadIdx.x & 31, sub = lane >> 1, c4 = lane & 1;
    const int64_t wglob = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    float4 *in = reinterpret_cast<float4 *>(R0), *out = reinterpret_cast<float4 *>(R1);
    // every row takes its graph's mark; diffuse_kernel has looked at the columns of the graphs that fit it, here
    // the others'
    for (int64_t i = wglob; i < N; i += nw) {
        const int64_t g = graph_of(graph_ptr, G, i), v0 = graph_ptr[g], v1 = graph_ptr[g + 1];
        const float mark = X[v0 * FIN];
        if (i != v0 && lane == 0) X[i * FIN] = mark;
        if (mark != 1.f) continue;
        for (int64_t e = row_ptr[i] + lane; e < row_ptr[i + 1]; e += 32)
            if (col[e] < v0 || col[e] >= v1) X[v0 * FIN + 1] = 1.f;
    }
    grid.sync();
    const bool all = marked(2.f);
    if (all) {
        for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < N * NRAND; t += (int64_t)gridDim.x * blockDim.x) {
            const int64_t i = t / NRAND;
            const int g = (int)graph_of(graph_ptr, G, i);
            R0[t] = noise_sign((uint32_t)(i - graph_ptr[g]), (int)(t % NRAND), graph_id[g], k0, k1);
        }
        grid.sync();
    }
    // the last round copies the result back to R0 when it ended in R1
    for (int s = 0; s < steps + (steps & 1); ++s) {
        for (int64_t i = wglob; i < N; i += nw) {
            if (!all && X[i * FIN] == 0.f) continue;
            if (s == steps) {
                if (lane < 2) out[i * 2 + lane] = in[i * 2 + lane];
                continue;
            }
            const int64_t e0 = row_ptr[i], e1 = row_ptr[i + 1];
            const float degi = (float)(e1 - e0);
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
            for (int64_t e = e0 + sub; e < e1; e += 16) {
                const int64_t j = col[e];
                const float w = edge_weight(2, row_ptr, j, degi);
                const float4 v = in[j * 2 + c4];
                a.x += w * v.x; a.y += w * v.y; a.z += w * v.z; a.w += w * v.w;
            }
#pragma unroll
            for (int o = 2; o < 32; o <<= 1) {
                a.x += __shfl_xor_sync(0xFFFFFFFFu, a.x, o);
                a.y += __shfl_xor_sync(0xFFFFFFFFu, a.y, o);
                a.z += __shfl_xor_sync(0xFFFFFFFFu, a.z, o);
                a.w += __shfl_xor_sync(0xFFFFFFFFu, a.w, o);
            }
            if (lane < 2) {
                const float4 x = in[i * 2 + lane];
                out[i * 2 + lane] = make_float4(0.5f * x.x + 0.5f * a.x, 0.5f * x.y + 0.5f * a.y,
                                                0.5f * x.z + 0.5f * a.z, 0.5f * x.w + 0.5f * a.w);
            }
        }
        grid.sync();
        float4 *t = in; in = out; out = t;
    }
}

// per graph (one block): centre and scale channels of R, write X (N x 16) with degree features.
// flags & GDI_MPNN_ALIGN: channel c >= 1 is multiplied by the sign of its inner product with
// channel 0 (after centring), so that the channels' low-frequency components point the same way
// inside a graph; flags & GDI_MPNN_NO_NOISE: the noise channels are written as 0.
__global__ void feat_finish_kernel(int G, const int64_t *graph_ptr, const int64_t *row_ptr, const float *R,
                                   float *X, int flags)
{
    const int g = blockIdx.x;
    const int64_t v0 = graph_ptr[g], v1 = graph_ptr[g + 1];
    const float n = (float)(v1 - v0);
    __shared__ float red[NRAND + 1][32];
    __shared__ float mean[NRAND + 1], rms[NRAND], sgn[NRAND];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    float s[NRAND + 1];
#pragma unroll
    for (int c = 0; c <= NRAND; ++c) s[c] = 0.f;
    for (int64_t i = v0 + threadIdx.x; i < v1; i += blockDim.x) {
#pragma unroll
        for (int c = 0; c < NRAND; ++c) s[c] += R[i * NRAND + c];
        s[NRAND] += (float)(row_ptr[i + 1] - row_ptr[i]);
    }
#pragma unroll
    for (int c = 0; c <= NRAND; ++c) {
        const float a = warp_sum(s[c]);
        if (lane == 0) red[c][w] = a;
    }
    __syncthreads();
    if (threadIdx.x <= NRAND) {
        float a = 0.f;
        for (int q = 0; q < nwarp; ++q) a += red[threadIdx.x][q];
        mean[threadIdx.x] = a / n;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NRAND; ++c) s[c] = 0.f;
    for (int64_t i = v0 + threadIdx.x; i < v1; i += blockDim.x)
#pragma unroll
        for (int c = 0; c < NRAND; ++c) {
            const float x = R[i * NRAND + c] - mean[c];
            s[c] += x * x;
        }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NRAND; ++c) {
        const float a = warp_sum(s[c]);
        if (lane == 0) red[c][w] = a;
    }
    __syncthreads();
    if (threadIdx.x < NRAND) {
        float a = 0.f;
        for (int q = 0; q < nwarp; ++q) a += red[threadIdx.x][q];
        rms[threadIdx.x] = sqrtf(a / n) + 1e-12f;
    }
    __syncthreads();
    // inner products of the centred channels with channel 0
#pragma unroll
    for (int c = 0; c < NRAND; ++c) s[c] = 0.f;
    if (flags & GDI_MPNN_ALIGN)
        for (int64_t i = v0 + threadIdx.x; i < v1; i += blockDim.x) {
            const float x0 = R[i * NRAND] - mean[0];
#pragma unroll
            for (int c = 1; c < NRAND; ++c) s[c] += x0 * (R[i * NRAND + c] - mean[c]);
        }
    __syncthreads();
#pragma unroll
    for (int c = 1; c < NRAND; ++c) {
        const float a = warp_sum(s[c]);
        if (lane == 0) red[c][w] = a;
    }
    __syncthreads();
    if (threadIdx.x < NRAND) {
        float a = 0.f;
        if (threadIdx.x > 0 && (flags & GDI_MPNN_ALIGN))
            for (int q = 0; q < nwarp; ++q) a += red[threadIdx.x][q];
        sgn[threadIdx.x] = (flags & GDI_MPNN_NO_NOISE) ? 0.f : (a < 0.f ? -1.f : 1.f);
    }
    __syncthreads();
    for (int64_t i = v0 + threadIdx.x; i < v1; i += blockDim.x) {
        const float deg = (float)(row_ptr[i + 1] - row_ptr[i]);
#pragma unroll
        for (int c = 0; c < NRAND; ++c) X[i * FIN + c] = sgn[c] * ((R[i * NRAND + c] - mean[c]) / rms[c]);
        X[i * FIN + NRAND] = log1pf(deg);
        X[i * FIN + NRAND + 1] = mean[NRAND] > 0.f ? deg / mean[NRAND] : 0.f;
#pragma unroll
        for (int c = NRAND + 2; c < FIN; ++c) X[i * FIN + c] = 0.f;
    }
}

// ---------------------------------------------------------------------------------------------
// Rounding (one block per graph): the floor(n/2) largest logits (ties: smaller vertex id first)
// become +1, the rest -1.  Bitonic sort of 64-bit keys in shared memory (n <= 8192).
__device__ __forceinline__ uint32_t float_order_desc(float f)
{
    // map float to uint32 so that larger floats give smaller keys
    uint32_t u = __float_as_uint(f);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);   // ascending order of floats
    return ~u;                                          // descending
}

__global__ void round_kernel(const int64_t *graph_ptr, const float *z, int8_t *spins)
{
    extern __shared__ unsigned long long keys[];
    const int g = blockIdx.x;
    const int64_t v0 = graph_ptr[g];
    const int n = (int)(graph_ptr[g + 1] - v0);
    int P2 = 1;
    while (P2 < n) P2 <<= 1;
    for (int t = threadIdx.x; t < P2; t += blockDim.x)
        keys[t] = t < n ? (((unsigned long long)float_order_desc(z[v0 + t]) << 32) | (unsigned)t)
                        : ~0ull;
    __syncthreads();
    for (int k = 2; k <= P2; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = threadIdx.x; t < P2; t += blockDim.x) {
                const int p = t ^ j;
                if (p > t) {
                    const bool up = (t & k) == 0;
                    const unsigned long long a = keys[t], b = keys[p];
                    if ((a > b) == up) { keys[t] = b; keys[p] = a; }
                }
            }
            __syncthreads();
        }
    }
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        const int v = (int)(keys[t] & 0xFFFFFFFFu);
        spins[v0 + v] = t < n / 2 ? 1 : -1;
    }
}

int grid_for(int64_t work, int per_block)
{
    int64_t g = (work + per_block - 1) / per_block;
    if (g < 1) g = 1;
    if (g > 152 * 16) g = 152 * 16;
    return (int)g;
}

constexpr int DF_CAP = 8960;              // two blocks of 1,024 threads and this many vertices fit an SM

// The one-launch walk's two launches: diffuse_kernel in clusters of DF_CL blocks, then walk_rest_kernel with as many
// blocks as the device, or the part of it that this process has, holds at once (a cooperative
// launch of more is refused).  1: enqueued; 0: the device holds no such cluster, and nothing was
// enqueued; else a negative error.
int launch_walk(int64_t N, int32_t G, const int64_t *graph_ptr, const uint32_t *graph_id, const int64_t *row_ptr,
                const int32_t *col, uint32_t k0, uint32_t k1, int32_t steps, float *X, float *R0, float *R1, cudaStream_t st)
{
    int dev = 0, sms = 0, rest = 0, clusters = 0;
    const size_t smem = df_layout(DF_CAP).total;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = DF_CL;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)G * DF_CL);
    cfg.blockDim = dim3(DF_T);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&rest, (const void *)walk_rest_kernel, WR_T, 0) != cudaSuccess ||
        sms * rest < 1 ||
        cudaFuncSetAttribute(diffuse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, diffuse_kernel, &cfg) != cudaSuccess || clusters < 1) {
        cudaGetLastError();                   // (a refused query is no error of the call)
        return 0;
    }
    const int cap = DF_CAP;
    if (cudaLaunchKernelEx(&cfg, diffuse_kernel, graph_ptr, graph_id, row_ptr, col, k0, k1, (int)steps, cap, X, R0, R1) !=
        cudaSuccess)
        return GDI_ERR_CUDA;
    void *args[] = {&N, &G, &graph_ptr, &graph_id, &row_ptr, &col, &k0, &k1, &steps, &X, &R0, &R1};
    if (cudaLaunchCooperativeKernel((const void *)walk_rest_kernel, dim3(sms * rest), dim3(WR_T), args, 0,
                                    st) != cudaSuccess)
        return GDI_ERR_CUDA;
    return 1;
}

// Whether the one-launch walk saves more than it costs.  Few steps do not repay laying out the columns: a step in a
// launch of its own costs about 3.5 us + N / 3000, in the one launch 0.4 + n / 800 (mean degree 12, n = the mean graph),
// which costs 12 us + n / 200 + G / 4 more to begin with.  (us for 1 / 2 / 4 / 8 steps, one launch against one per step: one
// graph of 300 vertices 51 53 54 56 / 43 44 50 67, of 2,000 75 74 83 95 / 53 58 65 80, of 5,000 120 126 141 165 / 84
// 89 100 127; 64 of 2,000 115 123 143 178 / 95 134 211 367.)
bool one_launch_walk(int64_t N, int32_t G, int32_t steps)
{
    if (steps >= 32) return true;
    const double n = (double)N / G;
    return steps * (3.1 + (double)N / 3000 - n / 800) > 12.0 + n / 200 + G / 4.0;
}

// 8-, 16- and 64-wide rows (the network's) on a 16-byte boundary take the vector kernel, other widths
// and alignments the general one.
void launch_aggregate(int64_t N, const int64_t *row_ptr, const int32_t *col, const float *X, int d, float *Y,
                      int mode, int accumulate, cudaStream_t st)
{
    const int grid = grid_for(N * 32, 256);
    const bool vec = aligned(X, 16) && aligned(Y, 16);
    if (vec && d == 64) aggregate_vec_kernel<64><<<grid, 256, 0, st>>>(N, row_ptr, col, X, Y, mode, accumulate);
    else if (vec && d == 16) aggregate_vec_kernel<16><<<grid, 256, 0, st>>>(N, row_ptr, col, X, Y, mode, accumulate);
    else if (vec && d == 8) aggregate_vec_kernel<8><<<grid, 256, 0, st>>>(N, row_ptr, col, X, Y, mode, accumulate);
    else aggregate_kernel<<<grid, 256, 0, st>>>(N, row_ptr, col, X, d, Y, mode, accumulate);
}

}  // namespace

extern "C" {

int gdi_mpnn_features(int64_t N, int32_t G, const int64_t *graph_ptr, const uint32_t *graph_id,
                      const int64_t *row_ptr, const int32_t *col, uint64_t seed, int32_t steps,
                      int32_t flags, float *X, float *scratch, void *stream)
{
    if (N < 1 || G < 1 || steps < 0 || !graph_ptr || !graph_id || !row_ptr || !col || !X || !scratch ||
        (flags & ~(GDI_MPNN_ALIGN | GDI_MPNN_NO_NOISE)))
        return GDI_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    float *R0 = scratch, *R1 = scratch + N * NRAND;
    // all steps in one launch where the mean graph fits a block, and one for the graphs that do not; else,
    // for few steps, and on a device that holds no cluster, one launch per step over all vertices
    int walked = 0;
    if (one_launch_walk(N, G, steps) && N / G <= DF_CAP && aligned(scratch, 16)) {
        walked = launch_walk(N, G, graph_ptr, graph_id, row_ptr, col, (uint32_t)seed, (uint32_t)(seed >> 32), steps, X, R0,
                             R1, st);
        if (walked < 0) return walked;
    }
    if (!walked) {
        feat_init_kernel<<<grid_for(N * NRAND, 256), 256, 0, st>>>(N, G, graph_ptr, graph_id, (uint32_t)seed,
                                                                    (uint32_t)(seed >> 32), R0);
        for (int s = 0; s < steps; ++s) {
            launch_aggregate(N, row_ptr, col, R0, NRAND, R1, 2, 0, st);
            float *t = R0; R0 = R1; R1 = t;
        }
    }
    feat_finish_kernel<<<G, 1024, 0, st>>>(G, graph_ptr, row_ptr, R0, X, flags);
    return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
}

int gdi_mpnn_aggregate(int64_t N, const int64_t *row_ptr, const int32_t *col, const float *X, int32_t d,
                       float *Y, int32_t mode, int32_t accumulate, void *stream)
{
    if (N < 1 || d < 1 || d > 64 || mode < 0 || mode > 2) return GDI_ERR_INVALID_ARG;
    launch_aggregate(N, row_ptr, col, X, d, Y, mode, accumulate, (cudaStream_t)stream);
    return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
}

int gdi_mpnn_dense_fwd(int64_t N, const float *X, const float *AGG, int32_t din, const uint16_t *Ws,
                       const uint16_t *Wn, const float *b, float *H, void *stream)
{
    if (N < 1 || din < 1 || din > 64) return GDI_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int tb = (int)min(((N + 15) / 16 + 7) / 8, (int64_t)152 * 2);         // tiles of 16 rows, 8 warps a block
    // the tensor-core kernels move activations in pairs (8-byte accesses)
    const bool pairs = aligned(X, 8) && aligned(AGG, 8) && aligned(H, 8);
    if (din == 64 && pairs) {
        dense_fwd_mma_kernel<64><<<tb, 256, 0, st>>>(N, X, AGG, Ws, Wn, b, H);
    } else if (din == 16 && pairs) {
        dense_fwd_mma_kernel<16><<<tb, 256, 0, st>>>(N, X, AGG, Ws, Wn, b, H);
    } else {
        const size_t smem = 2 * (size_t)din * HID * sizeof(float);
        dense_fwd_kernel<<<grid_for(N * 32, 256), 256, smem, st>>>(N, X, AGG, din, Ws, Wn, b, H, 1);
    }
    return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
}

int gdi_mpnn_dense_bwd(int64_t N, int32_t din, const uint16_t *Ws, const uint16_t *Wn, const float *H,
                       const float *dH, float *dPRE, float *dXs, float *T, void *stream)
{
    if (N < 1 || din < 1 || din > 64) return GDI_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int tb = (int)min((N + 15) / 16 * 32 / 256 + 1, (int64_t)152 * 16);
    // pairs of activations (8-byte accesses) and pairs of BF16 weights (4-byte accesses)
    const bool pairs = aligned(H, 8) && aligned(dH, 8) && aligned(dPRE, 8) && aligned(dXs, 8) && aligned(T, 8) &&
                       aligned(Ws, 4) && aligned(Wn, 4);
    if (din == 64 && pairs) {
        dense_bwd_mma_kernel<64><<<tb, 256, 0, st>>>(N, Ws, Wn, H, dH, dPRE, dXs, T);
    } else if (din == 16 && pairs) {
        dense_bwd_mma_kernel<16><<<tb, 256, 0, st>>>(N, Ws, Wn, H, dH, dPRE, dXs, T);
    } else {
        const size_t smem = 2 * (size_t)din * HID * sizeof(float);
        dense_bwd_kernel<<<grid_for(N * 32, 256), 256, smem, st>>>(N, din, Ws, Wn, H, dH, dPRE, dXs, T);
    }
    return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
}

int gdi_mpnn_wgrad(int64_t N, const float *A, int32_t din, const float *B, int32_t dout, float *out,
                   float *colsum, void *stream)
{
    if (N < 1 || din < 1 || din > 64 || dout < 1 || dout > 64) return GDI_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if (dout == 1) {
        // two blocks per SM, at least 64 rows each
        const int64_t chunk = max((int64_t)64, (N + 303) / 304);
        wgrad1_kernel<<<(int)((N + chunk - 1) / chunk), 256, 0, st>>>(N, A, din, B, out, colsum, chunk);
        return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
    }
    // one block per SM, whole tiles of 32 rows
    const int64_t chunk = ((N + 151) / 152 + WG_R - 1) / WG_R * WG_R;
    const int grid = (int)((N + chunk - 1) / chunk);
    const int dk = din <= 16 ? 16 : 64;
    const int vec = (din == dk && aligned(A, 16) ? 1 : 0) | (dout == HID && aligned(B, 16) ? 2 : 0) |
                    (dout == HID && aligned(out, 16) ? 4 : 0);
    if (dk == 16) wgrad_kernel<16><<<grid, WG_T, 0, st>>>(N, A, din, B, dout, out, colsum, chunk, vec);
    else wgrad_kernel<64><<<grid, WG_T, 0, st>>>(N, A, din, B, dout, out, colsum, chunk, vec);
    return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
}

int gdi_mpnn_out_fwd(int64_t N, const float *H, const uint16_t *wo, const float *bo, float *z, void *stream)
{
    if (N < 1) return GDI_ERR_INVALID_ARG;
    out_fwd_kernel<<<grid_for(N * 32, 256), 256, 0, (cudaStream_t)stream>>>(N, H, wo, bo, z);
    return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
}

int gdi_mpnn_out_bwd(int64_t N, const uint16_t *wo, const float *dz, float *dH, void *stream)
{
    if (N < 1) return GDI_ERR_INVALID_ARG;
    out_bwd_kernel<<<grid_for(N * HID, 256), 256, 0, (cudaStream_t)stream>>>(N, wo, dz, dH);
    return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
}

int gdi_mpnn_loss(int32_t G, const int64_t *graph_ptr, const float *z, const int8_t *y, float lambda,
                  float *stats, float *dz, float *loss, void *stream)
{
    if (G < 1) return GDI_ERR_INVALID_ARG;
    loss_kernel<<<G, 1024, 0, (cudaStream_t)stream>>>(G, graph_ptr, z, y, lambda, stats, dz, loss);
    return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
}

int gdi_mpnn_adam(int64_t P, float *params, const float *grads, float *m, float *v, uint16_t *params_bf16,
                  float lr, float beta1, float beta2, float eps, int32_t step, void *stream)
{
    if (P < 1 || step < 1) return GDI_ERR_INVALID_ARG;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    adam_kernel<<<grid_for(P, 256), 256, 0, (cudaStream_t)stream>>>(P, params, grads, m, v, params_bf16, lr, beta1,
                                                                     beta2, eps, c1, c2);
    return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
}

int gdi_mpnn_to_bf16(int64_t P, const float *params, uint16_t *params_bf16, void *stream)
{
    if (P < 1) return GDI_ERR_INVALID_ARG;
    to_bf16_kernel<<<grid_for(P, 256), 256, 0, (cudaStream_t)stream>>>(P, params, params_bf16);
    return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
}

int gdi_mpnn_round(int32_t G, const int64_t *graph_ptr, int32_t max_n, const float *z, int8_t *spins,
                   void *stream)
{
    if (G < 1 || max_n < 1 || max_n > 8192) return GDI_ERR_INVALID_ARG;
    int P2 = 1;
    while (P2 < max_n) P2 <<= 1;
    const size_t smem = (size_t)P2 * sizeof(unsigned long long);
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(round_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    round_kernel<<<G, 512, smem, (cudaStream_t)stream>>>(graph_ptr, z, spins);
    return cudaGetLastError() == cudaSuccess ? GDI_OK : GDI_ERR_CUDA;
}

}  // extern "C"
