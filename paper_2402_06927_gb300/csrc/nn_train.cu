// Training pass of the learned proposal in BF16 (nn_backward with NN_BF16 and 64 channels):
// the loss and every gradient, on channels-first BF16 activations.
//
// The generic pass (nn_proposal.cu) runs every contraction through one GEMM whose operands
// come element by element through gather functors: FP32 loads with two integer divisions
// each, 64 x 64 tiles whatever the shape.  At the training batch (256 samples, n = 1024) it
// took 1.80 ms for 16 GFLOP.  Here the activations and the gradients of layers 1..4 are
// kept as the BF16 values that the contractions round them to, [b][c][position], and each
// contraction has a kernel that stages slabs of them in shared memory and forms
// mma.sync fragments from the slabs:
//   conv_cf_kernel   forward convolutions;
//   dx_cf_kernel     input gradients, with the ReLU mask and the bias gradient's FP32
//                    partial sums in the epilogue (no FP32 gradient is stored);
//   dw_cf_kernel     weight gradients, all columns of a k-chunk in one CTA;
//   gemm_cf_kernel   the head, its weight gradient and its input gradient;
//   modes_*          the Fourier-mode projection and its transpose.
// Every contraction runs over the generic pass's k-order (k = channel * 5 + tap; batch x
// position; the same split-K chunks) in the same steps of 16, so its values are the
// generic pass's bit for bit: rounding to BF16 between the layers turns any other order of
// summation into 1e-4 changes.  The loss's and the biases' plain sums are FP32 and FP64 as before.
//
// Measured at the training batch (B = 256, n = 1024, K = 16, Ns = 20; one GB300): the step, Adam
// included, 1.80 -> 0.28 ms.  By kernel (us, layers last to first): dw 12, 12, 21, 10; dx 16, 21,
// 32; forward convolutions 14, 18, 21, 16; the final sums 29 (36 MB of split-K slices); the head's
// products 10, 6, 6; the rest 5 to 9 each.  The convolution kernels are bound by the latency
// of their slabs' copies at one to seven tiles a CTA, not by the tensor cores (16 GFLOP).
#include "nn_internal.h"

namespace sch {

namespace {

constexpr int CF_C = 64;

__device__ __forceinline__ uint32_t pair16(const __nv_bfloat16* p, const __nv_bfloat16* q) {
    return (uint32_t)*reinterpret_cast<const uint16_t*>(p) | ((uint32_t)*reinterpret_cast<const uint16_t*>(q) << 16);
}
__device__ __forceinline__ uint32_t bf2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ bool bf_pos(uint32_t half) { return half != 0u && half < 0x8000u && half <= 0x7f80u; }

// a row length in elements, at least n, that is 24 mod 64: rows of 16-byte chunks whose
// 32-bit words start 12 banks apart
constexpr int row24(int n) { return ((n + 39) / 64) * 64 + 24; }

// A fragments (m16 x k16, row-major rows of `ld` elements) of four 16-row tiles
template <int MT>
__device__ __forceinline__ void load_a(uint32_t (&a)[MT][4], const __nv_bfloat16* s, int ld, int m0, int k0) {
    const int lane = threadIdx.x & 31;
    const int row = (lane & 7) + 8 * ((lane >> 3) & 1), col = 8 * (lane >> 4);
#pragma unroll
    for (int i = 0; i < MT; ++i) ldmatrix_x4(a[i], s + (size_t)(m0 + 16 * i + row) * ld + k0 + col);
}

// ---------------------------------------------------------------------------------------
// operands of the parameters as BF16: the convolutions' weights [l][co][k] (k = ci 5 + tap;
// layer 0 padded to 16) and transposed [l][ci][co 5 + tap], the head's Wh, and the mode table
// S(q, k) both ways; and the loss cleared
// ---------------------------------------------------------------------------------------
struct PackArgs {
    const float* params;
    size_t off_w[4], off_wh;
    int K, Kp, P, O, FF;
    __nv_bfloat16 *w0, *w, *wt, *wh, *sq, *sk;   // sq [P][Kp], sk [K][P]
    double* loss;
};

__device__ __forceinline__ float mode_value(int q, int k, int P) {
    const int j = k / 2 + 1;
    float s, c;
    sincospif(2.0f * (float)((j * q) % P) / (float)P, &s, &c);
    return ((k & 1) ? c : s) / (float)P;
}

__global__ void pack_cf_kernel(PackArgs a) {
    const int T = gridDim.x * blockDim.x, t0 = blockIdx.x * blockDim.x + threadIdx.x;
    if (t0 == 0) *a.loss = 0.0;
    for (int e = t0; e < CF_C * 16; e += T)
        a.w0[e] = __float2bfloat16_rn(e % 16 < 10 ? a.params[a.off_w[0] + (e / 16) * 10 + e % 16] : 0.f);
    constexpr int W = CF_C * CF_C * 5;
    for (int e = t0; e < 3 * W; e += T) {
        const int l = e / W, r = e % W;
        const float v = a.params[a.off_w[l + 1] + r];
        const int co = r / (CF_C * 5), ci = (r / 5) % CF_C, j = r % 5;
        a.w[e] = __float2bfloat16_rn(v);
        a.wt[l * W + (ci * CF_C + co) * 5 + j] = __float2bfloat16_rn(v);
    }
    for (int e = t0; e < a.O * a.FF; e += T) a.wh[e] = __float2bfloat16_rn(a.params[a.off_wh + e]);
    for (int e = t0; e < a.P * a.Kp; e += T) {
        const int q = e / a.Kp, k = e % a.Kp;
        const __nv_bfloat16 v = __float2bfloat16_rn(k < a.K ? mode_value(q, k, a.P) : 0.f);
        a.sq[e] = v;
        if (k < a.K) a.sk[k * a.P + q] = v;
    }
}

// ---------------------------------------------------------------------------------------
// Forward convolution: out[b][co][q] = relu(bias[co] + sum_k W[co][k] X[k][q]), X[ci 5 + j][q] =
// x[b][ci][(2q + j - 2) mod 2Lo].  A CTA of four warps takes TQ = 32 NT output positions of
// the flattened (b, q) (several samples where Lo < TQ), all 64 channels: warp w the 8 NT
// positions from 8 NT w.  The weights stay in shared memory over the CTA's tiles; the slab
// holds position p of segment s at s SEG + p - 2 q0 + 8, with the two positions left and the
// one right of the tile taken round the circle.  B fragments are 16-bit loads through a
// table of k's offset in the slab (lanes of one load fall in distinct banks).
// CIN = 2: the features (u, innovation) are formed here.
// ---------------------------------------------------------------------------------------
struct ConvArgs {
    int B, Lo;
    const __nv_bfloat16* x;      // [b][64][2 Lo], stride bs (CIN = 64)
    const float *u, *y;          // CIN = 2
    int n, M, ystride;
    float sigma;
    const __nv_bfloat16* w;      // [64][KP]
    const float* bias;
    __nv_bfloat16* out;          // [b][64][Lo], stride bs
    size_t bs;
};

template <int CIN, int NT>
struct ConvCfg {
    static constexpr int TQ = 32 * NT, KP = CIN == 2 ? 16 : 320, WROW = KP + 8;
    // the largest slab row: TQ / Lo segments of 2 Lo + 16 elements, Lo >= 8
    static int seg(int Lo) { return 2 * (Lo < TQ ? Lo : TQ) + 16; }
    static int row(int Lo) { return row24((Lo < TQ ? TQ / Lo : 1) * seg(Lo)); }
    static size_t smem(int Lo) { return ((size_t)CF_C * WROW + (size_t)CIN * row(Lo)) * 2 + KP * 2; }
};

template <int CIN, int NT>
__global__ void __launch_bounds__(128) conv_cf_kernel(ConvArgs g, int seg, int rs) {
    using Cfg = ConvCfg<CIN, NT>;
    constexpr int TQ = Cfg::TQ, KP = Cfg::KP, WROW = Cfg::WROW;
    extern __shared__ __align__(16) unsigned char raw[];
    __nv_bfloat16* Ws = reinterpret_cast<__nv_bfloat16*>(raw);
    __nv_bfloat16* Xs = Ws + CF_C * WROW;
    uint16_t* koff = reinterpret_cast<uint16_t*>(Xs + (size_t)CIN * rs);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int Lo = g.Lo, Lin = 2 * Lo, Lq = min(Lo, TQ), nseg = TQ / Lq;
    for (int e = tid; e < CF_C * (KP / 8); e += 128)
        cp_async16(Ws + (e / (KP / 8)) * WROW + 8 * (e % (KP / 8)), g.w + 8 * (size_t)e);
    for (int k = tid; k < KP; k += 128) koff[k] = k < CIN * 5 ? (uint16_t)((k / 5) * rs + k % 5 + 6) : (uint16_t)6;
    const int tot = g.B * Lo, ntiles = (tot + TQ - 1) / TQ;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int f0 = tile * TQ;
        __syncthreads();   // the slab of the previous tile is read; the tables are written
        for (int s = 0; s < nseg; ++s) {
            const int b = (f0 + s * Lq) / Lo, q0 = (f0 + s * Lq) % Lo;
            __nv_bfloat16* xs = Xs + s * seg + 8;
            if (CIN == 64) {
                if (b < g.B) {
                    const __nv_bfloat16* xb = g.x + (size_t)b * g.bs;
                    for (int e = tid; e < CF_C * (Lq / 4); e += 128) {
                        const int c = e / (Lq / 4), i = 8 * (e % (Lq / 4));
                        cp_async16(xs + (size_t)c * rs + i, xb + (size_t)c * Lin + 2 * q0 + i);
                    }
                    for (int e = tid; e < CF_C * 3; e += 128) {
                        const int c = e / 3, h = e % 3;                 // positions -2, -1 and 2 Lq
                        const int p = h < 2 ? h - 2 : 2 * Lq;
                        xs[(ptrdiff_t)c * rs + p] = xb[(size_t)c * Lin + (2 * q0 + p + Lin) % Lin];
                    }
                } else {
                    for (int e = tid; e < CF_C * (2 * Lq + 3); e += 128)
                        xs[(ptrdiff_t)(e / (2 * Lq + 3)) * rs + e % (2 * Lq + 3) - 2] = __float2bfloat16_rn(0.f);
                }
            } else {
                const int stride = g.n / g.M;
                for (int e = tid; e < 2 * Lq + 3; e += 128) {
                    float ub = 0.f, inn = 0.f;
                    if (b < g.B) {
                        const int i = (2 * q0 + e - 2 + Lin) % Lin;
                        ub = g.u[(size_t)b * g.n + i];
                        if (i % stride == 0) {
                            const float yj = g.y[(size_t)b * g.ystride + i / stride];
                            if (yj == yj) inn = (yj - ub) / g.sigma;   // NaN: not observed
                        }
                    }
                    xs[e - 2] = __float2bfloat16_rn(ub);
                    xs[rs + e - 2] = __float2bfloat16_rn(inn);
                }
            }
        }
        cp_async_commit();
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        int pb[NT];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const int q = warp * 8 * NT + 8 * nt + gq;
            pb[nt] = (q / Lq) * seg + 2 * (q % Lq);
        }
        float acc[4][NT][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[i][nt][e] = 0.f;
#pragma unroll 2
        for (int k0 = 0; k0 < KP; k0 += 16) {
            uint32_t a[4][4];
            load_a<4>(a, Ws, WROW, 0, k0);
            const uint32_t o0 = *reinterpret_cast<const uint32_t*>(koff + k0 + 2 * tq);
            const uint32_t o1 = *reinterpret_cast<const uint32_t*>(koff + k0 + 2 * tq + 8);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const __nv_bfloat16* xp = Xs + pb[nt];
                const uint32_t b2[2] = {pair16(xp + (o0 & 0xffffu), xp + (o0 >> 16)),
                                        // CIN = 2: k >= 10 is padding
                                        CIN == 2 && tq > 0 ? 0u : pair16(xp + (o1 & 0xffffu), xp + (o1 >> 16))};
#pragma unroll
                for (int i = 0; i < 4; ++i) mma_bf16_16816(acc[i][nt], a[i], b2);
            }
        }
        // fragment (i, nt): channels 16 i + gq (+ 8), positions 8 nt + 2 tq (+ 1)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const int f = f0 + warp * 8 * NT + 8 * nt + 2 * tq, b = f / Lo, q = f % Lo;
            if (b >= g.B) continue;
            __nv_bfloat16* ob = g.out + (size_t)b * g.bs + q;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int co = 16 * i + gq + 8 * h;
                    const float bb = g.bias[co];
                    const float v0 = acc[i][nt][2 * h] + bb, v1 = acc[i][nt][2 * h + 1] + bb;
                    *reinterpret_cast<uint32_t*>(ob + (size_t)co * Lo) = bf2(v0 > 0.f ? v0 : 0.f, v1 > 0.f ? v1 : 0.f);
                }
        }
    }
}

// ---------------------------------------------------------------------------------------
// Input gradient of layer l: dx[b][ci][i] = sum_k WT[ci][k] G[k][i], k = co 5 + j, G[k][i] =
// g[b][co][q] where 2q + j - 2 = i (mod 2Lo) and 0 where i - j is odd (k keeps its place in the
// steps of 16), masked by x > 0.  The n-tiles of a fragment are eight positions of one
// parity, i = 2r + par, so a tap reads consecutive q = r + (par - j + 2)/2 and the odd
// taps a slab row of zeros.  A CTA takes TR = 16 NT values of r (2 TR positions).  Epilogue:
// the tile in FP32 in shared memory, then mask, BF16 store and the FP32 sums over the
// tile's positions that the bias gradient of the layer below adds up.
// ---------------------------------------------------------------------------------------
struct DxArgs {
    int B, Lo;
    const __nv_bfloat16* g;      // [b][64][Lo], stride gs
    const __nv_bfloat16* wt;     // [64][320]
    const __nv_bfloat16* x;      // [b][64][2 Lo], stride gs
    __nv_bfloat16* dx;           // [b][64][2 Lo], stride gs
    size_t gs;
    float* bpart;                // [tile][64]
};

template <int NT>
struct DxCfg {
    static constexpr int TR = 16 * NT, KP = 320, WROW = KP + 8, OROW = 2 * TR + 4, MROW = 2 * TR + 8;
    static int seg(int Lo) { return (Lo < TR ? Lo : TR) + 16; }
    static int row(int Lo) { return row24((Lo < TR ? TR / Lo : 1) * seg(Lo)); }
    static size_t smem(int Lo) {
        // weights, slab and the row of zeros, x's tile, the FP32 tile, the offset tables
        return ((size_t)CF_C * (WROW + MROW) + (size_t)(CF_C + 1) * row(Lo)) * 2 + (size_t)CF_C * OROW * 4 + 2 * KP * 2;
    }
};

template <int NT>
__global__ void __launch_bounds__(128) dx_cf_kernel(DxArgs g, int seg, int rs) {
    using Cfg = DxCfg<NT>;
    constexpr int TR = Cfg::TR, KP = Cfg::KP, WROW = Cfg::WROW, OROW = Cfg::OROW, MROW = Cfg::MROW;
    extern __shared__ __align__(16) unsigned char raw[];
    __nv_bfloat16* Ws = reinterpret_cast<__nv_bfloat16*>(raw);
    float* Os = reinterpret_cast<float*>(Ws + CF_C * WROW);
    __nv_bfloat16* Xm = reinterpret_cast<__nv_bfloat16*>(Os + CF_C * OROW);        // x's tile [64][MROW]
    __nv_bfloat16* Gs = Xm + CF_C * MROW;
    uint16_t* koff = reinterpret_cast<uint16_t*>(Gs + (size_t)(CF_C + 1) * rs);   // [2][KP]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int Lo = g.Lo, Lin = 2 * Lo, Lr = min(Lo, TR), nseg = TR / Lr;
    for (int e = tid; e < CF_C * (KP / 8); e += 128)
        cp_async16(Ws + (e / (KP / 8)) * WROW + 8 * (e % (KP / 8)), g.wt + 8 * (size_t)e);
    for (int e = tid; e < 2 * KP; e += 128) {
        const int par = e / KP, k = e % KP, j = k % 5;
        koff[e] = ((par - j) & 1) ? (uint16_t)(CF_C * rs) : (uint16_t)((k / 5) * rs + 8 + (par - j + 2) / 2);
    }
    for (int e = tid; e < rs; e += 128) Gs[(size_t)CF_C * rs + e] = __float2bfloat16_rn(0.f);
    const int tot = g.B * Lo, ntiles = (tot + TR - 1) / TR;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int f0 = tile * TR;
        __syncthreads();
        for (int s = 0; s < nseg; ++s) {
            const int b = (f0 + s * Lr) / Lo, r0 = (f0 + s * Lr) % Lo;
            __nv_bfloat16* gsl = Gs + s * seg + 8;
            if (b < g.B) {
                const __nv_bfloat16* gb = g.g + (size_t)b * g.gs;
                for (int e = tid; e < CF_C * (Lr / 8); e += 128) {
                    const int c = e / (Lr / 8), i = 8 * (e % (Lr / 8));
                    cp_async16(gsl + (size_t)c * rs + i, gb + (size_t)c * Lo + r0 + i);
                }
                const __nv_bfloat16* xb = g.x + (size_t)b * g.gs + 2 * r0;
                for (int e = tid; e < CF_C * (Lr / 4); e += 128) {
                    const int c = e / (Lr / 4), i = 8 * (e % (Lr / 4));
                    cp_async16(Xm + c * MROW + 2 * s * Lr + i, xb + (size_t)c * Lin + i);
                }
                for (int e = tid; e < CF_C * 2; e += 128) {
                    const int c = e / 2, p = (e & 1) ? Lr : -1;
                    gsl[(ptrdiff_t)c * rs + p] = gb[(size_t)c * Lo + (r0 + p + Lo) % Lo];
                }
            } else {
                for (int e = tid; e < CF_C * (Lr + 2); e += 128)
                    gsl[(ptrdiff_t)(e / (Lr + 2)) * rs + e % (Lr + 2) - 1] = __float2bfloat16_rn(0.f);
            }
        }
        cp_async_commit();
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        // n-tile nt of warp w: parity nt & 1, the eight r from 8 (w NT / 2 + nt / 2)
        int pb[NT / 2];
#pragma unroll
        for (int h = 0; h < NT / 2; ++h) {
            const int r = 8 * (warp * (NT / 2) + h) + gq;
            pb[h] = (r / Lr) * seg + r % Lr;
        }
        float acc[4][NT][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[i][nt][e] = 0.f;
#pragma unroll 2
        for (int k0 = 0; k0 < KP; k0 += 16) {
            uint32_t a[4][4];
            load_a<4>(a, Ws, WROW, 0, k0);
#pragma unroll
            for (int par = 0; par < 2; ++par) {
                const uint32_t o0 = *reinterpret_cast<const uint32_t*>(koff + par * KP + k0 + 2 * tq);
                const uint32_t o1 = *reinterpret_cast<const uint32_t*>(koff + par * KP + k0 + 2 * tq + 8);
#pragma unroll
                for (int h = 0; h < NT / 2; ++h) {
                    const __nv_bfloat16* xp = Gs + pb[h];
                    const uint32_t b2[2] = {pair16(xp + (o0 & 0xffffu), xp + (o0 >> 16)),
                                            pair16(xp + (o1 & 0xffffu), xp + (o1 >> 16))};
#pragma unroll
                    for (int i = 0; i < 4; ++i) mma_bf16_16816(acc[i][2 * h + par], a[i], b2);
                }
            }
        }
        // fragment (i, nt): channels 16 i + gq (+ 8), r = 8 (..) + 2 tq (+ 1), position 2 r + par
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int r = 8 * (warp * (NT / 2) + nt / 2) + 2 * tq + (e & 1);
                    Os[(16 * i + gq + 8 * (e >> 1)) * OROW + 2 * r + (nt & 1)] = acc[i][nt][e];
                }
        __syncthreads();
        // four channels at a time, so that their loads and reductions overlap
        for (int c0 = warp * 16; c0 < warp * 16 + 16; c0 += 4) {
            float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 2 * lane; i < 2 * TR; i += 64) {
                const int f = 2 * f0 + i, b = f / Lin, p = f % Lin;
                if (b >= g.B) continue;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint32_t xv = *reinterpret_cast<const uint32_t*>(Xm + (c0 + c) * MROW + i);
                    const float2 v = *reinterpret_cast<const float2*>(Os + (c0 + c) * OROW + i);
                    const float v0 = bf_pos(xv & 0xffffu) ? v.x : 0.f, v1 = bf_pos(xv >> 16) ? v.y : 0.f;
                    *reinterpret_cast<uint32_t*>(g.dx + (size_t)b * g.gs + (size_t)(c0 + c) * Lin + p) = bf2(v0, v1);
                    sum[c] += v0 + v1;
                }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) sum[c] = warp_sum(sum[c]);
            if (lane == 0)
                *reinterpret_cast<float4*>(g.bpart + (size_t)tile * CF_C + c0) = make_float4(sum[0], sum[1], sum[2], sum[3]);
        }
    }
}

// ---------------------------------------------------------------------------------------
// Weight gradient: dw[co][kk] = sum_{(b, q)} g[b][co][q] X[(b, q)][kk], kk = ci 5 + j, over the
// k-chunk blockIdx.x of the flattened (b, q), in sub-blocks of 128 staged in shared memory:
// the gradient rows [co][k], and per input channel the pair of positions (2q, 2q + 1) of
// every k, with a pair more at each end of a run of consecutive q in a sample.  Runs start on
// a 16-byte boundary of the slab whatever the chunk's first k is, so x comes in 16-byte
// copies; the gradient rows do where the sub-block starts at a multiple of eight (4-byte
// copies at an even start).  Each warp takes NTT column tiles (CIN = 64: eight warps of 40
// columns, all 64 rows; CIN = 2: four warps of one 16-row tile, both column tiles).
// ---------------------------------------------------------------------------------------
struct DwArgs {
    int B, Lo, lg, kchunk;       // Lo = 1 << lg
    const __nv_bfloat16* g;      // [b][64][Lo], stride bs
    const __nv_bfloat16* x;      // [b][64][2 Lo], stride bs (CIN = 64)
    const float *u, *y;          // CIN = 2: the features
    int n, M, ystride;
    float sigma;
    size_t bs;
    float* part;                 // [chunk][64][5 CIN]
};

// 16 (4) bytes to shared memory, of which the first `bytes` come from gmem and the rest are zero
__device__ __forceinline__ void cp_async16_part(void* smem, const void* gmem, int bytes) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(gmem), "r"(bytes));
}
__device__ __forceinline__ void cp_async4_part(void* smem, const void* gmem, int bytes) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(sa), "l"(gmem), "r"(bytes));
}

constexpr int DW_KB = 128;
template <int CIN>
struct DwCfg {
    static constexpr int WARPS = CIN == 2 ? 4 : 8, MT = CIN == 2 ? 1 : 4, NTT = CIN == 2 ? 2 : 5;
    static constexpr int GROW = DW_KB + 8;
    // pairs per channel: a sub-block's own, four more per run, and three zero pairs
    static int row(int Lo) { return row24(2 * (DW_KB + 4 * (DW_KB / Lo + 2) + 12)); }
    static size_t smem(int Lo) { return ((size_t)CF_C * GROW + (size_t)CIN * row(Lo)) * 2 + DW_KB * 2; }
};

template <int CIN>
__global__ void __launch_bounds__(DwCfg<CIN>::WARPS * 32) dw_cf_kernel(DwArgs g, int rs) {
    using Cfg = DwCfg<CIN>;
    constexpr int T = Cfg::WARPS * 32, MT = Cfg::MT, NTT = Cfg::NTT, GROW = Cfg::GROW, N = 5 * CIN;
    extern __shared__ __align__(16) unsigned char raw[];
    __nv_bfloat16* Gs = reinterpret_cast<__nv_bfloat16*>(raw);
    __nv_bfloat16* Xs = Gs + CF_C * GROW;
    uint16_t* poff = reinterpret_cast<uint16_t*>(Xs + (size_t)CIN * rs);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int Lo = g.Lo, Lin = 2 * Lo, tot = g.B * Lo;
    const int kbeg = blockIdx.x * g.kchunk, kend = min(tot, kbeg + g.kchunk);
    const int m0 = CIN == 2 ? 16 * warp : 0, n0 = CIN == 2 ? 0 : 8 * NTT * warp;
    int coff[NTT];
#pragma unroll
    for (int t = 0; t < NTT; ++t) {
        const int kk = n0 + 8 * t + gq;
        coff[t] = kk < N ? (kk / 5) * rs + kk % 5 - 2 : -2;
    }
    float acc[MT][NTT][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int t = 0; t < NTT; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][t][e] = 0.f;
    // (features) the pairs of positions (2 q, 2 q + 1) of u and of the innovation
    auto features = [&](int b, int q, uint32_t* xr) {
        const int stride = g.n / g.M;
        float v[2][2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = 2 * q + h;
            const float ub = g.u[(size_t)b * g.n + i];
            float inn = 0.f;
            if (i % stride == 0) {
                const float yj = g.y[(size_t)b * g.ystride + i / stride];
                if (yj == yj) inn = (yj - ub) / g.sigma;   // NaN: not observed
            }
            v[0][h] = ub;
            v[1][h] = inn;
        }
        xr[0] = bf2(v[0][0], v[0][1]);
        xr[rs / 2] = bf2(v[1][0], v[1][1]);
    };
    const int zero = rs / 2 - 2;               // the middle of three zero pairs in every channel's row
    for (int e = tid; e < 3 * CIN; e += T) reinterpret_cast<uint32_t*>(Xs)[(e / 3) * (rs / 2) + zero - 1 + e % 3] = 0u;
    for (int kb = kbeg; kb < kend; kb += DW_KB) {
        const int nk = min(DW_KB, kend - kb), b0 = kb >> g.lg, b1 = (kb + nk - 1) >> g.lg;
        __syncthreads();
        if ((kb & 7) == 0) {
            for (int e = tid; e < CF_C * (DW_KB / 8); e += T) {
                const int co = e / (DW_KB / 8), kl = 8 * (e % (DW_KB / 8)), f = kb + kl, left = min(8, nk - kl);
                cp_async16_part(Gs + co * GROW + kl,
                                left > 0 ? g.g + (size_t)(f >> g.lg) * g.bs + (size_t)co * Lo + (f & (Lo - 1)) : g.g,
                                left > 0 ? 2 * left : 0);
            }
        } else if ((kb & 1) == 0) {
            for (int e = tid; e < CF_C * (DW_KB / 2); e += T) {
                const int co = e / (DW_KB / 2), kl = 2 * (e % (DW_KB / 2)), f = kb + kl, left = min(2, nk - kl);
                cp_async4_part(Gs + co * GROW + kl,
                               left > 0 ? g.g + (size_t)(f >> g.lg) * g.bs + (size_t)co * Lo + (f & (Lo - 1)) : g.g,
                               left > 0 ? 2 * left : 0);
            }
        } else {
#pragma unroll 8
            for (int e = tid; e < CF_C * DW_KB; e += T) {
                const int co = e / DW_KB, kl = e % DW_KB, f = kb + kl;
                Gs[co * GROW + kl] = kl < nk ? g.g[(size_t)(f >> g.lg) * g.bs + (size_t)co * Lo + (f & (Lo - 1))]
                                             : __float2bfloat16_rn(0.f);
            }
        }
        // slot of k: kl + (kb mod 4) + 4 + 4 (runs before), congruent to q mod 4
        const int sft = (kb & 3) + 4;
        for (int kl = tid; kl < DW_KB; kl += T)
            poff[kl] = (uint16_t)(2 * (kl < nk ? kl + sft + 4 * (((kb + kl) >> g.lg) - b0) : zero));
        for (int b = b0; b <= b1; ++b) {
            const int fa = max(kb, b << g.lg), fb = min(kb + nk, (b + 1) << g.lg);
            const int qa = fa & (Lo - 1), qn = fb - fa, s0 = fa - kb + sft + 4 * (b - b0);   // slot of qa
            if constexpr (CIN == 64) {
                const __nv_bfloat16* xb = g.x + (size_t)b * g.bs;
                const int ca = qa >> 2, cn = ((qa + qn + 3) >> 2) - ca;                     // 16-byte copies
                for (int e = tid; e < CF_C * cn; e += T) {
                    const int c = e / cn, i = e % cn;
                    cp_async16(Xs + (size_t)c * rs + 2 * (s0 - (qa & 3) + 4 * i), xb + (size_t)c * Lin + 8 * (ca + i));
                }
                const int ql = (qa + Lo - 1) & (Lo - 1), qr = (qa + qn) & (Lo - 1);
                for (int e = tid; e < 2 * CF_C; e += T) {
                    const int c = e >> 1;
                    if ((e & 1) == 0) {
                        if ((qa & 3) == 0) cp_async4_part(Xs + (size_t)c * rs + 2 * (s0 - 1), xb + (size_t)c * Lin + 2 * ql, 4);
                    } else if (((qa + qn) & 3) == 0) {
                        cp_async4_part(Xs + (size_t)c * rs + 2 * (s0 + qn), xb + (size_t)c * Lin + 2 * qr, 4);
                    }
                }
            } else {
                for (int i = tid - 1; i <= qn; i += T)
                    if (i >= -1) features(b, (qa + i + Lo) & (Lo - 1), reinterpret_cast<uint32_t*>(Xs) + s0 + i);
            }
        }
        cp_async_commit();
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
#pragma unroll 1
        for (int k0 = 0; k0 < nk; k0 += 16) {
            uint32_t a[MT][4];
            load_a<MT>(a, Gs, GROW, m0, k0);
            const uint32_t o0 = *reinterpret_cast<const uint32_t*>(poff + k0 + 2 * tq);
            const uint32_t o1 = *reinterpret_cast<const uint32_t*>(poff + k0 + 2 * tq + 8);
#pragma unroll
            for (int t = 0; t < NTT; ++t) {
                const __nv_bfloat16* xp = Xs + coff[t];
                const uint32_t b2[2] = {pair16(xp + (o0 & 0xffffu), xp + (o0 >> 16)),
                                        pair16(xp + (o1 & 0xffffu), xp + (o1 >> 16))};
#pragma unroll
                for (int i = 0; i < MT; ++i) mma_bf16_16816(acc[i][t], a[i], b2);
            }
        }
    }
    float* out = g.part + (size_t)blockIdx.x * CF_C * N;
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int t = 0; t < NTT; ++t)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int co = m0 + 16 * i + gq + 8 * h, kk = n0 + 8 * t + 2 * tq;
                if (kk < N)
                    *reinterpret_cast<float2*>(out + co * N + kk) = make_float2(acc[i][t][2 * h], acc[i][t][2 * h + 1]);
            }
}

// ---------------------------------------------------------------------------------------
// C[m][n] = sum_k A(m, k) B(k, n) (+ bias[n]) on BF16 operands in memory, over the k-chunk
// blockIdx.z: A stored [m][k] or (TA) [k][m], B stored [n][k] or (TB) [k][n], rows of lda,
// ldb elements (multiples of 8).  T x T tiles, four warps of (T/2) x (T/2), k-steps of 32 (64 at
// T = 32) in a ring of three cp.async buffers; what lies past M, N or the chunk is zero.
// ---------------------------------------------------------------------------------------
struct GemmArgs {
    int M, N, Kd, kchunk, lda, ldb, ldc;
    const __nv_bfloat16 *A, *Bm;
    const float* bias;
    float* C;                    // FP32 output, or
    __nv_bfloat16* Cb;           // BF16 output
    size_t cslice;               // elements between the chunks' outputs
};

constexpr int GM_ST = 3;

template <int T, bool TA, bool TB>
__global__ void __launch_bounds__(128) gemm_cf_kernel(GemmArgs g) {
    constexpr int GM_BK = T == 32 ? 64 : 32;
    constexpr int MT = T / 32, NP = T / 32;       // 16-row tiles and pairs of 8-column tiles a warp
    constexpr int AR = TA ? GM_BK : T, AC = TA ? T : GM_BK, BR = TB ? GM_BK : T, BC = TB ? T : GM_BK;
    __shared__ __align__(16) __nv_bfloat16 As[GM_ST][AR][AC + 8];
    __shared__ __align__(16) __nv_bfloat16 Bs[GM_ST][BR][BC + 8];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int m0 = blockIdx.y * T, n0 = blockIdx.x * T;
    const int kbeg = blockIdx.z * g.kchunk, kend = min(g.Kd, kbeg + g.kchunk);
    const int wm = (warp >> 1) * (T / 2), wn = (warp & 1) * (T / 2);
    // rows `r` x columns `c` from (r0, c0) of a matrix [R][C], zero past R and C
    auto fill = [&](__nv_bfloat16* s, int rows, int cols, const __nv_bfloat16* p, int ld, int r0, int c0, int R, int C) {
        for (int e = tid; e < rows * (cols / 8); e += 128) {
            const int r = e / (cols / 8), c = 8 * (e % (cols / 8));
            const int left = (r0 + r < R) ? min(8, C - (c0 + c)) : 0;
            cp_async16_part(s + r * (cols + 8) + c, left > 0 ? p + (size_t)(r0 + r) * ld + c0 + c : p, left > 0 ? 2 * left : 0);
        }
    };
    auto issue = [&](int st, int k0) {
        if (TA) fill(&As[st][0][0], AR, AC, g.A, g.lda, k0, m0, kend, g.M);
        else fill(&As[st][0][0], AR, AC, g.A, g.lda, m0, k0, g.M, kend);
        if (TB) fill(&Bs[st][0][0], BR, BC, g.Bm, g.ldb, k0, n0, kend, g.N);
        else fill(&Bs[st][0][0], BR, BC, g.Bm, g.ldb, n0, k0, g.N, kend);
    };
    float acc[MT][2 * NP][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int t = 0; t < 2 * NP; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][t][e] = 0.f;
    const int nk = (kend - kbeg + GM_BK - 1) / GM_BK;
#pragma unroll
    for (int s = 0; s < GM_ST - 1; ++s) {
        if (s < nk) issue(s, kbeg + s * GM_BK);
        cp_async_commit();
    }
    for (int kt = 0; kt < nk; ++kt) {
        asm volatile("cp.async.wait_group %0;" ::"n"(GM_ST - 2) : "memory");
        __syncthreads();   // step kt has arrived; the buffer of step kt - 1 is free
        if (kt + GM_ST - 1 < nk) issue((kt + GM_ST - 1) % GM_ST, kbeg + (kt + GM_ST - 1) * GM_BK);
        cp_async_commit();
        const int st = kt % GM_ST;
#pragma unroll
        for (int ks = 0; ks < GM_BK; ks += 16) {
            uint32_t a[MT][4], b[NP][4];
#pragma unroll
            for (int i = 0; i < MT; ++i) {
                // matrices (m 0-7, k 0-7), (m 8-15, k 0-7), (m 0-7, k 8-15), (m 8-15, k 8-15)
                const int m = wm + 16 * i + 8 * ((lane >> 3) & 1), k = ks + 8 * (lane >> 4);
                if (TA) ldmatrix_x4_trans(a[i], &As[st][k + (lane & 7)][m]);
                else ldmatrix_x4(a[i], &As[st][m + (lane & 7)][k]);
            }
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                // matrices (k 0-7, n 0-7), (k 8-15, n 0-7), (k 0-7, n 8-15), (k 8-15, n 8-15)
                const int n = wn + 16 * p + 8 * (lane >> 4), k = ks + 8 * ((lane >> 3) & 1);
                if (TB) ldmatrix_x4_trans(b[p], &Bs[st][k + (lane & 7)][n]);
                else ldmatrix_x4(b[p], &Bs[st][n + (lane & 7)][k]);
            }
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const uint32_t b0[2] = {b[p][0], b[p][1]}, b1[2] = {b[p][2], b[p][3]};
                    mma_bf16_16816(acc[i][2 * p], a[i], b0);
                    mma_bf16_16816(acc[i][2 * p + 1], a[i], b1);
                }
        }
    }
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int t = 0; t < 2 * NP; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int m = m0 + wm + 16 * i + gq + 8 * (e >> 1), n = n0 + wn + 8 * t + 2 * tq + (e & 1);
                if (m >= g.M || n >= g.N) continue;
                const float v = acc[i][t][e] + (g.bias ? g.bias[n] : 0.f);
                const size_t o = blockIdx.z * g.cslice + (size_t)m * g.ldc + n;
                if (g.C) g.C[o] = v;
                else g.Cb[o] = __float2bfloat16_rn(v);
            }
}

// ---------------------------------------------------------------------------------------
// Mode projection F[b][c][k] = sum_q h[b][c][q] S(q, k): a warp takes 16 channels of one
// sample, fragments straight from memory (q is contiguous in h and in sk [K][P]).
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) modes_fwd_kernel(int B, int K, int P, const __nv_bfloat16* h, size_t bs,
                                                        const __nv_bfloat16* sk, __nv_bfloat16* F) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gq = lane >> 2, tq = lane & 3;
    const int b = blockIdx.x, c0 = 16 * warp;
    const __nv_bfloat16* hr = h + (size_t)b * bs + (size_t)(c0 + gq) * P;
    for (int n0 = 0; n0 < K; n0 += 8) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        const int k = n0 + gq;
        for (int q0 = 0; q0 < P; q0 += 16) {
            const int qa = q0 + 2 * tq, qb = qa + 8;      // P is a multiple of 8
            const bool in = qb < P;
            const uint32_t a[4] = {*reinterpret_cast<const uint32_t*>(hr + qa),
                                   *reinterpret_cast<const uint32_t*>(hr + 8 * P + qa),
                                   in ? *reinterpret_cast<const uint32_t*>(hr + qb) : 0u,
                                   in ? *reinterpret_cast<const uint32_t*>(hr + 8 * P + qb) : 0u};
            const uint32_t b2[2] = {k < K ? *reinterpret_cast<const uint32_t*>(sk + (size_t)k * P + qa) : 0u,
                                    k < K && in ? *reinterpret_cast<const uint32_t*>(sk + (size_t)k * P + qb) : 0u};
            mma_bf16_16816(acc, a, b2);
        }
        const int ko = n0 + 2 * tq;
        if (ko < K) {
            __nv_bfloat16* o = F + (size_t)b * CF_C * K + (size_t)(c0 + gq) * K + ko;
            *reinterpret_cast<uint32_t*>(o) = bf2(acc[0], acc[1]);
            *reinterpret_cast<uint32_t*>(o + 8 * K) = bf2(acc[2], acc[3]);
        }
    }
}

// Its transpose: dh[b][c][q] = sum_k gF[b][c][k] S(q, k), masked by h > 0, BF16, with the FP32
// sums over q (the bias gradient of layer 3) to bpart[b][c].
__global__ void __launch_bounds__(128) modes_bwd_kernel(int B, int K, int Kp, int P, const __nv_bfloat16* gF,
                                                        const __nv_bfloat16* sq, const __nv_bfloat16* h,
                                                        __nv_bfloat16* dh, size_t bs, float* bpart) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gq = lane >> 2, tq = lane & 3;
    const int b = blockIdx.x, c0 = 16 * warp;
    const __nv_bfloat16* gr = gF + (size_t)b * CF_C * K + (size_t)(c0 + gq) * K;
    float s0 = 0.f, s1 = 0.f;
    for (int q0 = 0; q0 < P; q0 += 8) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int k0 = 0; k0 < Kp; k0 += 16) {
            const int ka = k0 + 2 * tq, kb = ka + 8;
            const uint32_t a[4] = {ka < K ? *reinterpret_cast<const uint32_t*>(gr + ka) : 0u,
                                   ka < K ? *reinterpret_cast<const uint32_t*>(gr + 8 * K + ka) : 0u,
                                   kb < K ? *reinterpret_cast<const uint32_t*>(gr + kb) : 0u,
                                   kb < K ? *reinterpret_cast<const uint32_t*>(gr + 8 * K + kb) : 0u};
            const __nv_bfloat16* sr = sq + (size_t)(q0 + gq) * Kp;
            const uint32_t b2[2] = {*reinterpret_cast<const uint32_t*>(sr + ka), *reinterpret_cast<const uint32_t*>(sr + kb)};
            mma_bf16_16816(acc, a, b2);
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const size_t o = (size_t)b * bs + (size_t)(c0 + gq + 8 * r) * P + q0 + 2 * tq;
            const uint32_t hv = *reinterpret_cast<const uint32_t*>(h + o);
            const float v0 = bf_pos(hv & 0xffffu) ? acc[2 * r] : 0.f, v1 = bf_pos(hv >> 16) ? acc[2 * r + 1] : 0.f;
            *reinterpret_cast<uint32_t*>(dh + o) = bf2(v0, v1);
            if (r == 0) s0 += v0 + v1;
            else s1 += v0 + v1;
        }
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        s0 += __shfl_xor_sync(FULL, s0, o);
        s1 += __shfl_xor_sync(FULL, s1, o);
    }
    if (tq == 0) {
        bpart[(size_t)b * CF_C + c0 + gq] = s0;
        bpart[(size_t)b * CF_C + c0 + gq + 8] = s1;
    }
}

// glam = (lam - target) / B in FP32 and in BF16 (rows of ldo, the columns past O zero), the loss in double
__global__ void loss_cf_kernel(int B, int O, int ldo, const float* lam, const float* target, float* glam,
                               __nv_bfloat16* glb, double* loss) {
    double acc = 0.0;
    const size_t tot = (size_t)B * ldo;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < tot; e += (size_t)gridDim.x * blockDim.x) {
        const size_t b = e / ldo, o = e % ldo;
        float gv = 0.f;
        if (o < (size_t)O) {
            const float d = lam[b * O + o] - target[b * O + o];
            gv = d / (float)B;
            glam[b * O + o] = gv;
            acc += 0.5 * (double)d * (double)d / B;
        }
        glb[e] = __float2bfloat16_rn(gv);
    }
    acc = warp_sum(acc);
    __shared__ double sh[8];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += sh[w];
        atomicAdd(loss, s);
    }
}

// ---------------------------------------------------------------------------------------
// The sums that end the pass, in one launch: the split-K slices of every weight gradient in
// slice order, and the bias gradients (the
// tiles' FP32 partials, or glam's rows: FP32 trees of 16 rows, added up in double; first, since
// they are the longest chains).
// ---------------------------------------------------------------------------------------
struct FinishArgs {
    struct W { const float* part; float* out; int count, nk, blocks; } w[5];
    struct Bs { const float* part; float* out; int rows, cols, blocks; } b[5];
};

__global__ void __launch_bounds__(256) finish_cf_kernel(FinishArgs a) {
    int blk = blockIdx.x;
#pragma unroll 1
    for (int l = 0; l < 5; ++l) {
        if (blk < a.b[l].blocks) {
            // a block sums 32 columns: eight warps over the rows, lanes over the columns
            __shared__ double sh[8][32];
            const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, col = blk * 32 + lane;
            double acc = 0.0;
            if (col < a.b[l].cols)
                for (int r = warp; r < a.b[l].rows; r += 128) {
                    float v[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        v[i] = r + 8 * i < a.b[l].rows ? a.b[l].part[(size_t)(r + 8 * i) * a.b[l].cols + col] : 0.f;
#pragma unroll
                    for (int h = 8; h >= 1; h >>= 1)
#pragma unroll
                        for (int i = 0; i < h; ++i) v[i] += v[i + h];
                    acc += (double)v[0];
                }
            sh[warp][lane] = acc;
            __syncthreads();
            if (warp == 0 && col < a.b[l].cols) {
                for (int w = 1; w < 8; ++w) acc += sh[w][lane];
                a.b[l].out[col] = (float)acc;
            }
            return;
        }
        blk -= a.b[l].blocks;
    }
#pragma unroll 1
    for (int l = 0; l < 5; ++l) {
        if (blk < a.w[l].blocks) {
            // 64 elements: 128 slices at a time into shared memory, then one thread an element
            __shared__ float tile[128][64];
            const int count = a.w[l].count, nk = a.w[l].nk, c = threadIdx.x & 63, e = blk * 64 + c;
            const float* p = a.w[l].part + e;
            float acc = 0.f;
            for (int s0 = 0; s0 < nk; s0 += 128) {
                const int ns = min(128, nk - s0);
                if (e < count)
#pragma unroll 16
                    for (int s = threadIdx.x >> 6; s < ns; s += 4) tile[s][c] = p[(size_t)(s0 + s) * count];
                __syncthreads();
                if (threadIdx.x < 64 && e < count)
#pragma unroll 8
                    for (int s = 0; s < ns; ++s) acc += tile[s][c];
                __syncthreads();
            }
            if (threadIdx.x < 64 && e < count) a.w[l].out[e] = acc;
            return;
        }
        blk -= a.w[l].blocks;
    }
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// the workspace's parts, as byte offsets from its first 256-byte boundary
struct Layout {
    size_t w0, w, wt, wh, sq, sk, act, grad, F, gF, lam, glam, glb, bpart[4], part[5], total;
    size_t bs;          // elements a sample of act and grad: layers 1..4
    size_t off[5];      // element offset of layer l (1..4) in a sample
    int Kp, ldo;
};

// rows of bias partials of layer l: tiles of the input-gradient kernel (l < 3), samples (l = 3)
int dx_tr(const NNDims& d, int B, int l) {
    // 64 values of r a CTA (128 positions), or 32 where that would leave SMs idle
    return (size_t)B * d.L[l + 1] >= (size_t)64 * 2 * device_sms() ? 64 : 32;
}
int bias_rows(const NNDims& d, int B, int l) {
    if (l == 3) return B;
    const int tr = dx_tr(d, B, l + 1);
    return (int)(((size_t)B * d.L[l + 2] + tr - 1) / tr);
}

Layout make_layout(const NNDims& d, int B) {
    Layout y{};
    const int O = d.K * d.Ns, FF = d.C * d.K, P = d.L[4];
    y.Kp = (d.K + 15) / 16 * 16;
    y.ldo = (O + 15) / 16 * 16;
    for (int l = 1; l <= 4; ++l) {
        y.off[l] = y.bs;
        y.bs += (size_t)CF_C * d.L[l];
    }
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += align256(bytes);
        return at;
    };
    y.w0 = take(CF_C * 16 * 2);
    y.w = take(3 * CF_C * CF_C * 5 * 2);
    y.wt = take(3 * CF_C * CF_C * 5 * 2);
    y.wh = take((size_t)O * FF * 2);
    y.sq = take((size_t)P * y.Kp * 2);
    y.sk = take((size_t)P * d.K * 2);
    y.act = take((size_t)B * y.bs * 2);
    y.grad = take((size_t)B * y.bs * 2);
    y.F = take((size_t)B * FF * 2);
    y.gF = take((size_t)B * FF * 2);
    y.lam = take((size_t)B * O * 4);
    y.glam = take((size_t)B * O * 4);
    y.glb = take((size_t)B * y.ldo * 2);
    for (int l = 0; l < 4; ++l) {
        y.bpart[l] = take((size_t)bias_rows(d, B, l) * CF_C * 4);
        const int KK = d.cin[l] * 5, Kd = B * d.L[l + 1];
        y.part[l] = take((size_t)splitk_chunks(Kd, splitk_for(d.C, KK, Kd)) * d.C * KK * 4);
    }
    y.part[4] = take((size_t)splitk_chunks(B, splitk_for(O, FF, B)) * O * FF * 4);
    y.total = o + 256;
    return y;
}

template <typename Kern>
int resident_ctas(Kern k, int threads, size_t sm) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, sm);
    return max(1, per_sm) * device_sms();
}

template <int CIN, int NT>
void launch_conv(const ConvArgs& g, cudaStream_t st) {
    using Cfg = ConvCfg<CIN, NT>;
    const size_t sm = Cfg::smem(g.Lo);
    const int ntiles = (int)(((size_t)g.B * g.Lo + Cfg::TQ - 1) / Cfg::TQ);
    const int res = resident_ctas(conv_cf_kernel<CIN, NT>, 128, sm);
    conv_cf_kernel<CIN, NT><<<min(ntiles, res), 128, sm, st>>>(g, Cfg::seg(g.Lo), Cfg::row(g.Lo));
}
// 128 output positions a CTA where that fills the SMs twice, else 64, else 32
template <int CIN>
void launch_conv_any(const ConvArgs& g, cudaStream_t st) {
    const size_t tot = (size_t)g.B * g.Lo, two = 2 * (size_t)device_sms();
    if (tot >= 128 * two) launch_conv<CIN, 4>(g, st);
    else if (tot >= 64 * two) launch_conv<CIN, 2>(g, st);
    else launch_conv<CIN, 1>(g, st);
}

template <int NT>
void launch_dx(const DxArgs& g, cudaStream_t st) {
    using Cfg = DxCfg<NT>;
    const size_t sm = Cfg::smem(g.Lo);
    const int ntiles = (int)(((size_t)g.B * g.Lo + Cfg::TR - 1) / Cfg::TR);
    const int res = resident_ctas(dx_cf_kernel<NT>, 128, sm);
    dx_cf_kernel<NT><<<min(ntiles, res), 128, sm, st>>>(g, Cfg::seg(g.Lo), Cfg::row(g.Lo));
}

template <int CIN>
void launch_dw(const DwArgs& g, int nk, cudaStream_t st) {
    using Cfg = DwCfg<CIN>;
    const size_t sm = Cfg::smem(g.Lo);
    cudaFuncSetAttribute(dw_cf_kernel<CIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    dw_cf_kernel<CIN><<<nk, Cfg::WARPS * 32, sm, st>>>(g, Cfg::row(g.Lo));
}

// 64 x 64 tiles where they fill the SMs twice, else 32 x 32
template <bool TA, bool TB>
void launch_gemm(const GemmArgs& g, int nk, cudaStream_t st) {
    const size_t big = (size_t)((g.N + 63) / 64) * ((g.M + 63) / 64) * nk;
    if (big >= 2 * (size_t)device_sms())
        gemm_cf_kernel<64, TA, TB><<<dim3((g.N + 63) / 64, (g.M + 63) / 64, nk), 128, 0, st>>>(g);
    else
        gemm_cf_kernel<32, TA, TB><<<dim3((g.N + 31) / 32, (g.M + 31) / 32, nk), 128, 0, st>>>(g);
}

int grid_for(size_t n) { return (int)max((size_t)1, min((n + 255) / 256, (size_t)device_sms() * 16)); }

}  // namespace

// 64 channels, and every layer a power of two of positions, at least eight at the last
bool cf_supported(const NNDims& d) {
    const int P = d.L[4];
    return d.prec == NN_BF16 && d.C == CF_C && P >= 8 && (P & (P - 1)) == 0 && d.n == 16 * P && d.K % 2 == 0 &&
           d.K <= 64 && head_count(d) <= HEAD_MAX;
}

size_t cf_workspace_bytes(const NNDims& d, int B) { return make_layout(d, B).total; }

int nn_backward_cf(const NNDims& d, int B, const float* params, const float* u, const float* y, int ystride,
                   const float* target, float* grads, double* loss, void* ws, cudaStream_t st) {
    const Layout L = make_layout(d, B);
    unsigned char* base = reinterpret_cast<unsigned char*>(align256(reinterpret_cast<size_t>(ws)));
    auto bf = [&](size_t o) { return reinterpret_cast<__nv_bfloat16*>(base + o); };
    auto fp = [&](size_t o) { return reinterpret_cast<float*>(base + o); };
    const int O = d.K * d.Ns, FF = d.C * d.K, P = d.L[4];
    __nv_bfloat16 *act = bf(L.act), *grad = bf(L.grad);
    constexpr int W = CF_C * CF_C * 5;

    PackArgs pk{params, {d.off_w[0], d.off_w[1], d.off_w[2], d.off_w[3]}, d.off_wh, d.K, L.Kp, P, O, FF, bf(L.w0),
                bf(L.w), bf(L.wt), bf(L.wh), bf(L.sq), bf(L.sk), loss};
    pack_cf_kernel<<<grid_for((size_t)O * FF), 256, 0, st>>>(pk);
    // forward
    for (int l = 0; l < 4; ++l) {
        ConvArgs c{B, d.L[l + 1], l ? act + L.off[l] : nullptr, u, y, d.n, d.M, ystride, d.sigma,
                   l ? bf(L.w) + (size_t)(l - 1) * W : bf(L.w0), params + d.off_b[l], act + L.off[l + 1], L.bs};
        if (l == 0) launch_conv_any<2>(c, st);
        else launch_conv_any<CF_C>(c, st);
    }
    modes_fwd_kernel<<<B, 128, 0, st>>>(B, d.K, P, act + L.off[4], L.bs, bf(L.sk), bf(L.F));
    launch_gemm<false, false>(GemmArgs{B, O, FF, FF, FF, FF, O, bf(L.F), bf(L.wh), params + d.off_bh, fp(L.lam),
                                       nullptr, 0}, 1, st);
    loss_cf_kernel<<<grid_for((size_t)B * L.ldo), 256, 0, st>>>(B, O, L.ldo, fp(L.lam), target, fp(L.glam), bf(L.glb),
                                                               loss);
    // the head: dWh, then gF = glam Wh
    FinishArgs fin{};
    const int ksk = splitk_for(O, FF, B), knk = splitk_chunks(B, ksk), kch = (B + ksk - 1) / ksk;
    launch_gemm<true, true>(GemmArgs{O, FF, B, kch, L.ldo, FF, FF, bf(L.glb), bf(L.F), nullptr,
                                     knk == 1 ? grads + d.off_wh : fp(L.part[4]), nullptr, (size_t)O * FF}, knk, st);
    launch_gemm<false, true>(GemmArgs{B, FF, O, O, L.ldo, FF, FF, bf(L.glb), bf(L.wh), nullptr, nullptr, bf(L.gF), 0}, 1,
                             st);
    modes_bwd_kernel<<<B, 128, 0, st>>>(B, d.K, L.Kp, P, bf(L.gF), bf(L.sq), act + L.off[4], grad + L.off[4], L.bs,
                                        fp(L.bpart[3]));
    // the convolutions, last to first
    for (int l = 3; l >= 0; --l) {
        const int KK = d.cin[l] * 5, Kd = B * d.L[l + 1], sk = splitk_for(d.C, KK, Kd), nk = splitk_chunks(Kd, sk);
        int lg = 0;
        while ((1 << lg) < d.L[l + 1]) ++lg;
        DwArgs w{B, d.L[l + 1], lg, (Kd + sk - 1) / sk, grad + L.off[l + 1], l ? act + L.off[l] : nullptr, u, y, d.n, d.M,
                 ystride, d.sigma, L.bs, fp(L.part[l])};
        if (l == 0) launch_dw<2>(w, nk, st);
        else launch_dw<CF_C>(w, nk, st);
        fin.w[l] = {fp(L.part[l]), grads + d.off_w[l], d.C * KK, nk, (d.C * KK + 63) / 64};
        fin.b[l] = {fp(L.bpart[l]), grads + d.off_b[l], bias_rows(d, B, l), CF_C, CF_C / 32};
        if (l > 0) {
            DxArgs x{B, d.L[l + 1], grad + L.off[l + 1], bf(L.wt) + (size_t)(l - 1) * W, act + L.off[l],
                     grad + L.off[l], L.bs, fp(L.bpart[l - 1])};
            if (dx_tr(d, B, l) == 64) launch_dx<4>(x, st);
            else launch_dx<2>(x, st);
        }
    }
    fin.w[4] = {fp(L.part[4]), grads + d.off_wh, O * FF, knk, knk == 1 ? 0 : (O * FF + 63) / 64};
    fin.b[4] = {fp(L.glam), grads + d.off_bh, B, O, (O + 31) / 32};
    int blocks = 0;
    for (int l = 0; l < 5; ++l) blocks += fin.w[l].blocks + fin.b[l].blocks;
    finish_cf_kernel<<<blocks, 256, 0, st>>>(fin);
    return cudaGetLastError() == cudaSuccess ? SCH_OK : SCH_ERR_CUDA;
}

}  // namespace sch
