// Inference pass of the learned proposal in BF16 (nn_forward with NN_BF16, 64 channels and n a
// multiple of 1024), on channels-last BF16 activations [b][position][c].
//
// conv_tc5_kernel runs the convolutions of layers 1..3 on the fifth-generation tensor cores:
// a persistent CTA per SM keeps the layer's weights in shared memory and takes tiles of 128
// output positions (64 where a layer has no more) of one sample, all 64 output channels.
// Three kinds of warps work on different tiles at a time, through mbarriers:
//   producers fill one of four input slabs: eight warps of cp.async of the layer's input, or
//     (FIRST) layer 0 itself, computed from the features with mma.sync m16n8k16 by four
//     groups of four warps with a tile (and slab) each, so that its output (the network's
//     largest, 64 KB a sample at n = 1024) never goes to memory;
//   a relay warp puts the proxy fence between the two kinds of access to a slab;
//   one lane of the MMA warp issues the tile's 20 tcgen05.mma of 128 x 64 x 16 (five taps, 64
//     channels) into one of two TMEM accumulators;
//   two epilogue groups of four warps, an accumulator each, add the bias, apply the ReLU, round to
//     BF16 and store 128-byte rows in 32-byte pieces.
// With one group of each kind the chain of one tile's work (features, layer 0; TMEM load,
// conversion, stores) took three times the MMAs' 1100 cycles.
// A slab keeps the positions of each parity apart, channel octet by channel octet, rows 16
// bytes apart (the no-swizzle K-major operand layout with SBO = 128), so that tap j's operand
// is the parity's rows shifted by j / 2: a descriptor with another start address.
//
// The contraction order is that of a chain of mma.sync m16n8k16 over k = tap * 64 + channel; a
// chain of tcgen05.mma kind::f16 over the same steps of 16 gives the same bits on this part.
//
// Measured (8192 samples, n = 1024, K = 16, Ns = 20; one GB300): the whole pass 908 -> 384 us, same
// bits.  By kernel: layers 0 and 1 together 151 us (mma.sync and one launch each before: about
// 470), layer 2 98, layer 3 57, mode projection 30, head 31, packing 5.  Layer 1's kernel issues an
// instruction in 37% of the cycles and its shared-memory pipe is 49% busy (layer 0's stores, the
// output rows, the barriers' polls); layers 2 and 3 move 402 and 201 MB at 4.1 and 3.5 TB/s.
#include "nn_internal.h"

namespace sch {

namespace {

constexpr int CI = 64;                       // channels
constexpr int IK = 5 * CI;                   // reduction length, k = tap * 64 + channel
constexpr int TQ5 = 128;                     // MMA rows
constexpr int PROWS = 133;                   // slab rows of a parity (130 used): 2128 bytes an octet, conflict-free
constexpr int PLANE = PROWS * 16;
constexpr int SLAB = 2 * 8 * PLANE;          // both parities
constexpr int WBYTES = CI * IK * 2;
constexpr int XS_W = 592;                    // (u, innovation) words of a tile's features (528 used)
constexpr int ST5 = 4;                       // slabs in flight
constexpr int EPW = 8;                       // epilogue warps
template <bool FIRST>
constexpr int NPW = FIRST ? 16 : 8;          // producer warps
template <bool FIRST>
constexpr int T5 = 32 * (EPW + NPW<FIRST> + 2);
// tries of a wait before it gives up; a build with a low limit runs into it
#ifndef SCH_CONV_WAIT_LIMIT
#define SCH_CONV_WAIT_LIMIT 200000
#endif
constexpr int WAIT_LIMIT = SCH_CONV_WAIT_LIMIT;
constexpr int DRAIN_LIMIT = 200000;          // the same for the MMAs in flight at a CTA's end

__device__ __forceinline__ unsigned s2u(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint64_t* b, int n) {
    asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(s2u(b)), "r"(n));
}
__device__ __forceinline__ void bar_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared.b64 _, [%0];" ::"r"(s2u(b)) : "memory");
}
__device__ __forceinline__ bool bar_try(uint64_t* b, int parity) {
    unsigned done;
    asm volatile("{.reg .pred p; mbarrier.try_wait.parity.shared.b64 p, [%1], %2; selp.u32 %0, 1, 0, p;}"
                 : "=r"(done)
                 : "r"(s2u(b)), "r"(parity)
                 : "memory");
    return done;
}
// waits for the phase of this parity; false after WAIT_LIMIT tries, or once another wait gave up.
// Every lane polls, and a warp that goes on to an .aligned tcgen05 instruction takes its decision by
// a vote: with lane 0 polling for its warp and a shuffle of the answer the branch is no longer
// provably uniform, and a build of that form faulted.
__device__ __forceinline__ bool bar_wait(uint64_t* b, int parity, volatile int* gave_up) {
    for (int i = 0; i < WAIT_LIMIT; ++i) {
        if (bar_try(b, parity)) return true;
        if ((i & 1023) == 1023 && *gave_up) return false;
    }
    *gave_up = 1;
    return false;
}
// shared-memory operand descriptor: K-major, no swizzle, `lbo` bytes between channel octets, 128
// between groups of eight rows
__device__ __forceinline__ uint64_t op_desc(unsigned addr, unsigned lbo) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) | ((uint64_t)(128 >> 4) << 32) |
           (1ull << 46);
}

struct Conv5Args {
    int B, Lo, rows;             // rows: output positions a tile (128 or 64)
    const __nv_bfloat16* in;     // [b][2 Lo][64], stride in_bs (not FIRST)
    size_t in_bs;
    const __nv_bfloat16* w;      // [64][320]
    const float* bias;
    __nv_bfloat16* out;          // [b][Lo][64], stride out_bs
    size_t out_bs;
    // FIRST: layer 0 from the features
    const float *u, *y, *w0, *b0;
    int n, M, ystride;
    float sigma;
    int* failed;                 // set when a wait gave up
};

struct Conv5Smem {
    uint64_t full[ST5], ready[ST5], empty[ST5], tfull[2], tempty[2], drained;
    uint32_t tmem;
    int gave_up;
    alignas(16) float bias[CI];
};

template <bool FIRST>
constexpr size_t conv5_smem() {
    return 1024 + WBYTES + ST5 * (size_t)SLAB + (FIRST ? 2 * ST5 * XS_W * 4 : 0);
}

template <bool FIRST>
__global__ void __launch_bounds__(T5<FIRST>, 1) conv_tc5_kernel(Conv5Args g) {
    extern __shared__ __align__(128) unsigned char raw[];
    Conv5Smem* sh = reinterpret_cast<Conv5Smem*>(raw);
    static_assert(sizeof(Conv5Smem) <= 1024, "");
    unsigned char* Ws = raw + 1024;
    unsigned char* slab = Ws + WBYTES;
    uint32_t* Xs = reinterpret_cast<uint32_t*>(slab + ST5 * SLAB);
    constexpr int NP = NPW<FIRST>, NT = T5<FIRST>, PT = FIRST ? 128 : 32 * NP;   // PT: producers of a tile
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tpb = g.Lo / g.rows, ntiles = g.B * tpb, Lin = 2 * g.Lo;

    if (tid == 0) {
        for (int i = 0; i < ST5; ++i) {
            bar_init(&sh->full[i], PT);
            bar_init(&sh->ready[i], 32);
            bar_init(&sh->empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            bar_init(&sh->tfull[i], 1);
            bar_init(&sh->tempty[i], 128);
        }
        bar_init(&sh->drained, 1);
        sh->gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < CI) sh->bias[tid] = g.bias[tid];
    if (warp == EPW + NP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(s2u(&sh->tmem))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // the weights as 40 octets of k, 64 rows of 16 bytes each
    for (int e = tid; e < CI * (IK / 8); e += NT) cp_async16(Ws + 16 * e, g.w + (size_t)(e % CI) * IK + 8 * (e / CI));
    if (FIRST)
        for (int e = tid; e < 2 * ST5 * XS_W; e += NT) Xs[e] = 0u;
    cp_async_commit();
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = sh->tmem;
    volatile int* gave_up = &sh->gave_up;

    if (warp >= EPW && warp < EPW + NP) {
        // ------------------------------------------------------------------ producers
        const int pt = FIRST ? tid & 127 : tid - 32 * EPW;
        if constexpr (!FIRST) {
            // thread pt copies octet pt & 7 of the input positions 2 q0 - 2 + r, r = pt / 8 + 32 i: one parity
            const int c8 = pt & 7, r0 = pt >> 3, R = 2 * g.rows + 3;
            auto issue = [&](int t, int b) {
                const int s = t / tpb, q0 = (t - s * tpb) * g.rows;
                const __nv_bfloat16* src = g.in + (size_t)s * g.in_bs + 8 * c8;
                unsigned char* dst = slab + b * SLAB + (r0 & 1) * (8 * PLANE) + c8 * PLANE + (r0 >> 1) * 16;
                for (int r = r0; r < R; r += 32, dst += 256) {
                    int p = 2 * q0 - 2 + r;
                    p += p < 0 ? Lin : (p >= Lin ? -Lin : 0);
                    cp_async16(dst, src + (size_t)p * CI);
                }
            };
            // as far ahead as there are empty slabs: a thread's arrival follows its copies
            int it = 0;
            for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++it) {
                const int b = it % ST5;
                if (!bar_wait(&sh->empty[b], ((it / ST5) & 1) ^ 1, gave_up)) break;
                issue(t, b);
                asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];" ::"r"(s2u(&sh->full[b])) : "memory");
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
        } else {
            // layer 0: B fragments (its weights, k = 2 tap + channel, zero from k = 10) and biases
            const int gq = lane >> 2, tq = lane & 3;
            uint32_t bf[8][2];
            float bb[8][2];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int co = 8 * j + gq;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float v[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int k = 2 * tq + 8 * h + e;
                        v[e] = k < 10 ? g.w0[(co * 2 + (k & 1)) * 5 + (k >> 1)] : 0.f;
                    }
                    const __nv_bfloat162 pk = __floats2bfloat162_rn(v[0], v[1]);
                    bf[j][h] = *reinterpret_cast<const uint32_t*>(&pk);
                    bb[j][h] = g.b0[8 * j + 2 * tq + h];
                }
            }
            // the features of a tile: positions 4 q0 - 6 + i, i < 528, loaded a tile ahead
            const int stride = g.n / g.M;
            const float istride = 1.0f / (float)stride;
            constexpr int FPT = (528 + PT - 1) / PT;
            float ru[FPT], ry[FPT];
            auto load = [&](int t) {
                const int s = t / tpb, q0 = (t % tpb) * g.rows;
#pragma unroll
                for (int i = 0; i < FPT; ++i) {
                    const int e = pt + PT * i;
                    ru[i] = 0.f;
                    ry[i] = __int_as_float(0x7fffffff);
                    if (e < 528) {
                        int f = 4 * q0 - 6 + e;
                        f += f < 0 ? g.n : (f >= g.n ? -g.n : 0);
                        ru[i] = __ldg(g.u + (size_t)s * g.n + f);
                        const int j = (int)(((float)f + 0.5f) * istride);
                        if (j * stride == f) ry[i] = __ldg(g.y + (size_t)s * g.ystride + j);
                    }
                }
            };
            // group gr takes every fourth tile, in slab gr
            const int gr = (warp - EPW) >> 2, step = ST5 * gridDim.x;
            int t = blockIdx.x + gr * gridDim.x;
            if (t < ntiles) load(t);
            for (int k = 0; t < ntiles; t += step, ++k) {
                uint32_t* xs = Xs + (2 * gr + (k & 1)) * XS_W;
#pragma unroll
                for (int i = 0; i < FPT; ++i) {
                    const int e = pt + PT * i;
                    if (e < 528) {
                        const float inn = ry[i] == ry[i] ? (ry[i] - ru[i]) / g.sigma : 0.f;   // NaN: not observed
                        const __nv_bfloat162 pk = __floats2bfloat162_rn(ru[i], inn);
                        xs[e] = *reinterpret_cast<const uint32_t*>(&pk);
                    }
                }
                if (t + step < ntiles) load(t + step);
                // the slab is free; one decision for the group's producers, who also meet here over xs
                unsigned ok = bar_wait(&sh->empty[gr], (k & 1) ^ 1, gave_up);
                asm volatile(
                    "{.reg .pred p, q; setp.ne.u32 p, %0, 0; barrier.cta.red.and.pred q, %1, 128, p; "
                    "selp.u32 %0, 1, 0, q;}"
                    : "+r"(ok)
                    : "r"(1 + gr)
                    : "memory");
                if (!ok) break;
                unsigned char* sl = slab + gr * SLAB;
                // row idx of a parity is position 2 (q0 + idx - 1) + par, its features start at word
                // 4 idx + 2 par.  Sixteen rows of one parity at a time, then rows 128 on of both (the
                // fragment's upper half even, its lower half odd positions)
                for (int mt = warp & 3; mt < 17; mt += 4) {
                    const bool mixed = mt == 16;
                    const int par = mixed ? 0 : mt >> 3, i0 = mixed ? 128 : 16 * (mt & 7);
                    const uint32_t* x0 = xs + 4 * (i0 + gq) + 2 * par + tq;
                    const uint32_t* x1 = x0 + (mixed ? 2 : 32);
                    const uint32_t a[4] = {x0[0], x1[0], x0[4], x1[4]};
                    unsigned char* d0 = sl + par * (8 * PLANE) + (i0 + gq) * 16 + 4 * tq;
                    unsigned char* d1 = d0 + (mixed ? 8 * PLANE : 128);
                    const bool in = !mixed || gq < 2;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float acc[4] = {0.f, 0.f, 0.f, 0.f};
                        mma_bf16_16816(acc, a, bf[j]);
                        // (v > 0 ? v : 0; a NaN gives 0)
                        const __nv_bfloat162 p0 =
                            __floats2bfloat162_rn(fmaxf(acc[0] + bb[j][0], 0.f), fmaxf(acc[1] + bb[j][1], 0.f));
                        const __nv_bfloat162 p1 =
                            __floats2bfloat162_rn(fmaxf(acc[2] + bb[j][0], 0.f), fmaxf(acc[3] + bb[j][1], 0.f));
                        if (in) {
                            *reinterpret_cast<uint32_t*>(d0 + j * PLANE) = *reinterpret_cast<const uint32_t*>(&p0);
                            *reinterpret_cast<uint32_t*>(d1 + j * PLANE) = *reinterpret_cast<const uint32_t*>(&p1);
                        }
                    }
                }
                bar_arrive(&sh->full[gr]);
            }
        }
    } else if (warp == EPW + NP) {
        // ------------------------------------------------------------------ MMA issue
        // the whole warp runs the loop and one elected lane issues: with warp-uniform descriptors an
        // MMA is issued every 55 cycles, from a branch that one thread alone takes every 152
        unsigned one;
        asm volatile("{.reg .pred p; elect.sync _|p, 0xffffffff; selp.u32 %0, 1, 0, p;}" : "=r"(one));
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((CI >> 3) << 17) | ((TQ5 >> 4) << 24);
        const unsigned wa = s2u(Ws);
        int it = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++it) {
            const int b = it % ST5, a2 = it & 1;
            if (!__all_sync(FULL, bar_wait(&sh->ready[b], (it / ST5) & 1, gave_up))) break;
            if (!__all_sync(FULL, bar_wait(&sh->tempty[a2], ((it >> 1) & 1) ^ 1, gave_up))) break;
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const unsigned sa = s2u(slab) + b * SLAB;
            const uint32_t d = tmem + a2 * CI;
#pragma unroll
            for (int j = 0; j < 5; ++j)
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint64_t da = op_desc(sa + (j & 1) * (8 * PLANE) + 2 * kk * PLANE + (j >> 1) * 16, PLANE);
                    const uint64_t db = op_desc(wa + (8 * j + 2 * kk) * (CI * 16), CI * 16);
                    const uint32_t acc = (j | kk) != 0;
                    asm volatile(
                        "{.reg .pred p, e; setp.ne.u32 p, %4, 0; setp.ne.u32 e, %5, 0;"
                        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;}" ::"r"(d),
                        "l"(da), "l"(db), "r"(idesc), "r"(acc), "r"(one)
                        : "memory");
                }
            if (one) {
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 s2u(&sh->empty[b]))
                             : "memory");
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 s2u(&sh->tfull[a2]))
                             : "memory");
            }
            __syncwarp();
        }
        // The accumulators are freed and the shared memory given back only after every MMA issued,
        // also when a wait gave up and no epilogue waits for their commits any more.
        if (one)
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             s2u(&sh->drained))
                         : "memory");
        __syncwarp();
        bool ended = false;
        for (int i = 0; i < DRAIN_LIMIT && !ended; ++i) ended = bar_try(&sh->drained, 0);
        if (!__all_sync(FULL, ended)) *gave_up = 1;
    } else if (warp == EPW + NP + 1) {
        // ------------------------------------------------------------------ relay
        // orders the producers' writes, seen through `full`, before the MMAs' reads.  A warp of its
        // own: in the producers the proxy fence waits for their copies and loads of later tiles,
        // in the MMA warp it stands between two tiles' MMAs
        int it = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++it) {
            const int b = it % ST5;
            if (!bar_wait(&sh->full[b], (it / ST5) & 1, gave_up)) break;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            bar_arrive(&sh->ready[b]);
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        // group e (warps 4 e .. 4 e + 3) takes every second tile, in accumulator e
        const int e2 = warp >> 2, row = tid & 127;
        int k = 0;
        for (int t = blockIdx.x + e2 * gridDim.x; t < ntiles; t += 2 * gridDim.x, ++k) {
            if (!__all_sync(FULL, bar_wait(&sh->tfull[e2], k & 1, gave_up))) break;
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const bool mine = row < g.rows;      // whole warps
            const int s = t / tpb, q0 = (t - s * tpb) * g.rows;
            __nv_bfloat16* o = g.out + (size_t)s * g.out_bs + (size_t)(q0 + row) * CI;
            if (mine) {
#pragma unroll
                for (int c = 0; c < CI; c += 32) {
                    uint32_t v[32];
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                          "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]),
                          "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]),
                          "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                        : "r"(tmem + e2 * CI + ((uint32_t)(32 * (warp & 3)) << 16) + c));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    uint32_t pk[16];
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const float4 bb = *reinterpret_cast<const float4*>(&sh->bias[c + 2 * i]);
                        const __nv_bfloat162 p0 = __floats2bfloat162_rn(fmaxf(__uint_as_float(v[2 * i]) + bb.x, 0.f),
                                                                        fmaxf(__uint_as_float(v[2 * i + 1]) + bb.y, 0.f));
                        const __nv_bfloat162 p1 = __floats2bfloat162_rn(fmaxf(__uint_as_float(v[2 * i + 2]) + bb.z, 0.f),
                                                                        fmaxf(__uint_as_float(v[2 * i + 3]) + bb.w, 0.f));
                        pk[i] = *reinterpret_cast<const uint32_t*>(&p0);
                        pk[i + 1] = *reinterpret_cast<const uint32_t*>(&p1);
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(o + c + 16 * h),
                                     "r"(pk[8 * h]), "r"(pk[8 * h + 1]), "r"(pk[8 * h + 2]), "r"(pk[8 * h + 3]),
                                     "r"(pk[8 * h + 4]), "r"(pk[8 * h + 5]), "r"(pk[8 * h + 6]), "r"(pk[8 * h + 7])
                                     : "memory");
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            bar_arrive(&sh->tempty[e2]);
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == EPW + NP) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(tmem));
    if (tid == 0 && sh->gave_up) *g.failed = 1;
}

// operands of the parameters as BF16: the weights of layers 1..3 as [l][co][tap 64 + ci], the
// head's Wh, the mode table [k][q]; and the failure word cleared
__global__ void pack_infer_kernel(const float* params, size_t off1, size_t off2, size_t off3, size_t off_wh, int OF,
                                  int K, int P, __nv_bfloat16* w, __nv_bfloat16* wh, __nv_bfloat16* sk, int* failed) {
    const int T = gridDim.x * blockDim.x, t0 = blockIdx.x * blockDim.x + threadIdx.x;
    if (t0 == 0) *failed = 0;
    for (int e = t0; e < 3 * CI * IK; e += T) {
        const int l = e / (CI * IK), r = e % (CI * IK), co = r / IK, k = r % IK;
        const size_t off = (l == 0) ? off1 : (l == 1) ? off2 : off3;
        w[e] = __float2bfloat16_rn(params[off + ((size_t)co * CI + k % CI) * 5 + k / CI]);
    }
    for (int e = t0; e < OF; e += T) wh[e] = __float2bfloat16_rn(params[off_wh + e]);
    for (int e = t0; e < K * P; e += T) {
        const int k = e / P, q = e % P, j = k / 2 + 1;
        float s, c;
        sincospif(2.0f * (float)((j * q) % P) / (float)P, &s, &c);
        sk[e] = __float2bfloat16_rn(((k & 1) ? c : s) / (float)P);
    }
}

// Mode projection F[b][c][k] = sum_q h[b][q][c] S(q, k), channels-last h: a CTA takes one sample
// and 64 modes from 64 blockIdx.y, warp w 16 channels.  The rows of h come through shared memory 64 positions at a time, and the
// A fragments (q along k) by transposed ldmatrix.
__global__ void __launch_bounds__(128) modes_cl_kernel(int K, int P, const __nv_bfloat16* h, size_t bs,
                                                       const __nv_bfloat16* sk, __nv_bfloat16* F) {
    constexpr int MAXT = 8;                       // mode tiles of 8
    const int kb = 64 * blockIdx.y;
    __shared__ __align__(16) __nv_bfloat16 Hs[64][CI + 8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gq = lane >> 2, tq = lane & 3, c0 = 16 * warp;
    const __nv_bfloat16* hb = h + (size_t)blockIdx.x * bs;
    float acc[MAXT][4];
#pragma unroll
    for (int t = 0; t < MAXT; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[t][e] = 0.f;
    for (int q0 = 0; q0 < P; q0 += 64) {
        __syncthreads();
        for (int e = threadIdx.x; e < 64 * (CI / 8); e += 128)
            cp_async16(&Hs[e >> 3][8 * (e & 7)], hb + (size_t)(q0 + (e >> 3)) * CI + 8 * (e & 7));
        cp_async_commit();
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < 64; ks += 16) {
            // matrices (c 0-7, q 0-7), (c 8-15, q 0-7), (c 0-7, q 8-15), (c 8-15, q 8-15), stored [q][c]
            uint32_t a[4];
            ldmatrix_x4_trans(a, &Hs[ks + 8 * (lane >> 4) + (lane & 7)][c0 + 8 * ((lane >> 3) & 1)]);
#pragma unroll
            for (int t = 0; t < MAXT; ++t) {
                if (kb + 8 * t >= K) break;
                const int k = kb + 8 * t + gq;
                const __nv_bfloat16* sr = sk + (size_t)k * P + q0 + ks + 2 * tq;
                const uint32_t b2[2] = {k < K ? *reinterpret_cast<const uint32_t*>(sr) : 0u,
                                        k < K ? *reinterpret_cast<const uint32_t*>(sr + 8) : 0u};
                mma_bf16_16816(acc[t], a, b2);
            }
        }
    }
#pragma unroll
    for (int t = 0; t < MAXT; ++t) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = kb + 8 * t + 2 * tq + (e & 1);
            if (k < K)
                F[(size_t)blockIdx.x * CI * K + (size_t)(c0 + gq + 8 * (e >> 1)) * K + k] = __float2bfloat16_rn(acc[t][e]);
        }
    }
}

// The head: lambda[b][o] = sum_f F[b][f] Wh[o][f] + bh[o], both operands row-major BF16, Kd a
// multiple of 64.  T x T tiles, four warps of (T/2) x (T/2), k-steps of 64 in a ring of three
// cp.async buffers.  Not-a-number throughout when a wait of the convolutions gave up.
template <int T>
__global__ void __launch_bounds__(128) head_kernel(int M, int N, int Kd, const __nv_bfloat16* __restrict__ A,
                                                   const __nv_bfloat16* __restrict__ Bm,
                                                   const float* __restrict__ bias, const int* __restrict__ failed,
                                                   float* __restrict__ C) {
    constexpr int BK = 64, ST = 3, MT = T / 32, NP = T / 32;
    extern __shared__ __align__(128) unsigned char raw[];
    auto As = reinterpret_cast<__nv_bfloat16(*)[T][BK + 8]>(raw);
    auto Bs = As + ST;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int m0 = blockIdx.y * T, n0 = blockIdx.x * T, wm = (warp >> 1) * (T / 2), wn = (warp & 1) * (T / 2);
    auto issue = [&](int st, int k0) {
        for (int e = tid; e < T * (BK / 8); e += 128) {
            const int r = e / (BK / 8), c = 8 * (e % (BK / 8));   // rows past the end: any row
            cp_async16(&As[st][r][c], A + (size_t)min(m0 + r, M - 1) * Kd + k0 + c);
            cp_async16(&Bs[st][r][c], Bm + (size_t)min(n0 + r, N - 1) * Kd + k0 + c);
        }
    };
    float acc[MT][2 * NP][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int t = 0; t < 2 * NP; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][t][e] = 0.f;
    const int nk = Kd / BK;
#pragma unroll
    for (int s = 0; s < ST - 1; ++s) {
        if (s < nk) issue(s, s * BK);
        cp_async_commit();
    }
    for (int kt = 0; kt < nk; ++kt) {
        asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
        __syncthreads();
        if (kt + ST - 1 < nk) issue((kt + ST - 1) % ST, (kt + ST - 1) * BK);
        cp_async_commit();
        const int st = kt % ST;
#pragma unroll
        for (int ks = 0; ks < BK; ks += 16) {
            uint32_t a[MT][4], b[NP][4];
#pragma unroll
            for (int i = 0; i < MT; ++i)
                ldmatrix_x4(a[i], &As[st][wm + 16 * i + 8 * ((lane >> 3) & 1) + (lane & 7)][ks + 8 * (lane >> 4)]);
#pragma unroll
            for (int p = 0; p < NP; ++p)
                ldmatrix_x4(b[p], &Bs[st][wn + 16 * p + 8 * (lane >> 4) + (lane & 7)][ks + 8 * ((lane >> 3) & 1)]);
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
    const bool bad = *failed != 0;
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int t = 0; t < 2 * NP; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int m = m0 + wm + 16 * i + gq + 8 * (e >> 1), n = n0 + wn + 8 * t + 2 * tq + (e & 1);
                if (m < M && n < N) C[(size_t)m * N + n] = bad ? __int_as_float(0x7fffffff) : acc[i][t][e] + bias[n];
            }
}

template <int T>
void launch_head(int B, int O, int FF, const __nv_bfloat16* F, const __nv_bfloat16* wh, const float* bh,
                 const int* failed, float* lam, cudaStream_t st) {
    constexpr size_t sm = (size_t)2 * 3 * T * 72 * 2;
    cudaFuncSetAttribute(head_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    head_kernel<T><<<dim3((O + T - 1) / T, (B + T - 1) / T), 128, sm, st>>>(B, O, FF, F, wh, bh, failed, lam);
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

bool cl_supported(const NNDims& d) {
    // 64 channels; every layer's output a whole number of 64-position tiles
    return d.prec == NN_BF16 && d.C == CI && d.L[4] % 64 == 0 && d.n <= (1 << 21) && head_count(d) <= HEAD_MAX;
}

// layers 2..4 and the mode features of the batch, the packed parameters, the failure word
size_t cl_workspace_bytes(const NNDims& d, int B) {
    const size_t O = (size_t)d.K * d.Ns, FF = (size_t)d.C * d.K;
    return 512 + align256(3 * (size_t)CI * IK * 2) + align256(O * FF * 2) + align256((size_t)d.K * d.L[4] * 2) +
           align256((size_t)B * CI * (d.L[2] + d.L[3] + d.L[4]) * 2) + align256((size_t)B * FF * 2);
}

int nn_forward_cl(const NNDims& d, int B, const float* params, const float* u, const float* y, int ystride, void* ws,
                  float* lam_out, cudaStream_t st) {
    const int P = d.L[4], FF = d.C * d.K, O = d.K * d.Ns;
    unsigned char* at = reinterpret_cast<unsigned char*>(align256(reinterpret_cast<size_t>(ws)));
    auto take = [&](size_t bytes) {
        unsigned char* p = at;
        at += align256(bytes);
        return reinterpret_cast<__nv_bfloat16*>(p);
    };
    int* failed = reinterpret_cast<int*>(take(256));
    __nv_bfloat16* w = take(3 * (size_t)CI * IK * 2);
    __nv_bfloat16* wh = take((size_t)O * FF * 2);
    __nv_bfloat16* sk = take((size_t)d.K * P * 2);
    const size_t bs = (size_t)CI * (d.L[2] + d.L[3] + d.L[4]);
    __nv_bfloat16* act = take((size_t)B * bs * 2);
    __nv_bfloat16* F = take((size_t)B * FF * 2);
    const size_t off[5] = {0, 0, 0, (size_t)CI * d.L[2], (size_t)CI * (d.L[2] + d.L[3])};
    const int sms = device_sms();
    pack_infer_kernel<<<4 * sms, 256, 0, st>>>(params, d.off_w[1], d.off_w[2], d.off_w[3], d.off_wh, O * FF, d.K, P, w,
                                               wh, sk, failed);
    for (int l = 1; l < 4; ++l) {
        Conv5Args g{};
        g.B = B;
        g.Lo = d.L[l + 1];
        g.rows = g.Lo % TQ5 == 0 ? TQ5 : 64;
        g.in = act + off[l];
        g.in_bs = bs;
        g.w = w + (size_t)(l - 1) * CI * IK;
        g.bias = params + d.off_b[l];
        g.out = act + off[l + 1];
        g.out_bs = bs;
        g.u = u;
        g.y = y;
        g.w0 = params + d.off_w[0];
        g.b0 = params + d.off_b[0];
        g.n = d.n;
        g.M = d.M;
        g.ystride = ystride;
        g.sigma = d.sigma;
        g.failed = failed;
        const int tiles = B * (g.Lo / g.rows);
        if (l == 1) {
            cudaFuncSetAttribute(conv_tc5_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)conv5_smem<true>());
            conv_tc5_kernel<true><<<min(tiles, sms), T5<true>, conv5_smem<true>(), st>>>(g);
        } else {
            cudaFuncSetAttribute(conv_tc5_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)conv5_smem<false>());
            conv_tc5_kernel<false><<<min(tiles, sms), T5<false>, conv5_smem<false>(), st>>>(g);
        }
    }
    modes_cl_kernel<<<dim3(B, (d.K + 63) / 64), 128, 0, st>>>(d.K, P, act + off[4], bs, sk, F);
    if ((size_t)((O + 63) / 64) * ((B + 63) / 64) >= 2 * (size_t)sms)
        launch_head<64>(B, O, FF, F, wh, params + d.off_bh, failed, lam_out, st);
    else
        launch_head<32>(B, O, FF, F, wh, params + d.off_bh, failed, lam_out, st);
    return cudaGetLastError() == cudaSuccess ? SCH_OK : SCH_ERR_CUDA;
}

}  // namespace sch
