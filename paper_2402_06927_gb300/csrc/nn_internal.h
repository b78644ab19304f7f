// Shared by the learned proposal's translation units: the network's dimensions and the
// tensor-core helpers.
#pragma once

#include <cuda_bf16.h>

#include "sch_internal.h"

namespace sch {

struct NNDims {
    int n, K, Ns, C, M, prec;
    float sigma;
    int L[5];     // positions at layers 0..4: n, n/2, n/4, n/8, n/16
    int cin[4];   // input channels of conv l
    size_t off_w[4], off_b[4], off_wh, off_bh, nparam;
    size_t act_off[5], off_F, off_lam, act_total;   // per-sample activation offsets (floats)
};

inline NNDims make_dims(const nn_shape* s) {
    NNDims d{};
    d.n = s->n; d.K = s->K; d.Ns = s->Ns; d.C = s->C; d.M = s->M; d.sigma = s->sigma; d.prec = s->precision;
    for (int l = 0; l <= 4; ++l) d.L[l] = s->n >> l;
    size_t o = 0;
    for (int l = 0; l < 4; ++l) {
        d.cin[l] = (l == 0) ? 2 : s->C;
        d.off_w[l] = o; o += (size_t)s->C * d.cin[l] * 5;
        d.off_b[l] = o; o += (size_t)s->C;
    }
    d.off_wh = o; o += (size_t)s->K * s->Ns * s->C * s->K;
    d.off_bh = o; o += (size_t)s->K * s->Ns;
    d.nparam = o;
    size_t a = 0;
    d.act_off[0] = a; a += 2 * (size_t)d.L[0];
    for (int l = 1; l <= 4; ++l) { d.act_off[l] = a; a += (size_t)s->C * d.L[l]; }
    d.off_F = a; a += (size_t)s->C * s->K;
    d.off_lam = a; a += (size_t)s->K * s->Ns;
    d.act_total = a;
    return d;
}

// entries of the head's matrix
inline size_t head_count(const NNDims& d) { return (size_t)d.K * d.Ns * d.C * d.K; }
// the BF16 passes of 64 channels count the head's entries in 32 bits; a larger head (from 4 GB of
// FP32 weights) takes the generic pass, which counts in 64
constexpr size_t HEAD_MAX = (size_t)1 << 30;

constexpr int TM = 64, TN = 64;   // output tile of the generic GEMMs (and of their split-K rule)

// k-splits for a reduction with few output tiles (weight gradients: the sum runs over
// batch x positions): about 8 CTAs per SM, chunks of at least 256 k-values
inline int splitk_for(int M, int N, int Kd) {
    const int tiles = ((M + TM - 1) / TM) * ((N + TN - 1) / TN);
    return max(1, min(Kd / 256, 8 * device_sms() / tiles));
}

// k-chunks that sgemm launches for a split of splitk
inline int splitk_chunks(int Kd, int splitk) {
    const int kchunk = (Kd + splitk - 1) / splitk;
    return (Kd + kchunk - 1) / kchunk;
}

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// 16-byte asynchronous copy global -> shared (cp.async, completion tracked by groups)
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;"); }

// four 8 x 8 BF16 matrices from shared memory (lane l gives the address of row l % 8 of
// matrix l / 8); register i receives matrix i in the mma fragment layout
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], const void* smem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(sa));
}

// the same, each matrix transposed
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], const void* smem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(sa));
}

// nn_forward with NN_BF16 on channels-last BF16 activations (nn_infer.cu)
bool cl_supported(const NNDims& d);
size_t cl_workspace_bytes(const NNDims& d, int B);
int nn_forward_cl(const NNDims& d, int B, const float* params, const float* u, const float* y, int ystride, void* ws,
                  float* lam_out, cudaStream_t st);

// nn_backward with NN_BF16 on channels-first BF16 activations (nn_train.cu): whether a shape
// takes it, its workspace bytes, and the pass itself (loss and every gradient)
bool cf_supported(const NNDims& d);
size_t cf_workspace_bytes(const NNDims& d, int B);
int nn_backward_cf(const NNDims& d, int B, const float* params, const float* u, const float* y, int ystride,
                   const float* target, float* grads, double* loss, void* ws, cudaStream_t st);

}  // namespace sch
