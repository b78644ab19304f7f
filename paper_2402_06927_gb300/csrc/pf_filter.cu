// Filter kernels on sm_103a: adaptive tempering by an ESS root search, systematic
// resampling on exact integers, and the row gather that copies resampled
// particles (Sec. 3.1.1 and 3.1.2 of the paper).  Weights and cumulative sums
// are FP64 / uint64 regardless of the field precision.
#include <cooperative_groups.h>

#include "sch_internal.h"

namespace sch {

constexpr int TEMPER_CTAS = 8;          // one thread-block cluster
constexpr int TEMPER_PER_THREAD = 8;    // N <= 8 * 256 * 8 = 16384
// threads per CTA: 128 up to N = 8 * 128 = 1024 (one particle per thread, every CTA
// busy), else 256: above N = 1024 the wider CTA shortens each thread's serial chain
// of exponentials.
constexpr int TEMPER_THREADS_SMALL = 128, TEMPER_THREADS_LARGE = 256;
constexpr int RESAMPLE_THREADS = 1024;

// Adaptive tempering on one cluster of TEMPER_CTAS CTAs: every CTA holds a slice of the
// particles, an evaluation reduces its sums over the cluster through distributed shared
// memory.  Every CTA sums the partials in the same order, so all CTAs take identical
// decisions.  Partials are double-buffered by evaluation parity, so one cluster barrier
// per evaluation suffices.
//
// What bounds it is the FP64 unit, on which a warp's instruction takes 64 cycles of its
// sub-partition: an FP64 evaluation costs about 25 of them a particle (the exponential),
// and any scalar that every warp computes for itself costs as much again.  So the root of
// ESS(d) = ess_min is located in float first (eight points an evaluation, the exponentials
// on the special-function unit), two or three Newton steps in FP64 finish it, and only
// warp 0 sums the partials and takes the decisions.  A searching call at N = 8001 takes 50 us
// (153 with an Illinois search of 12 to 15 FP64 evaluations summed by every warp), at N = 1024
// about 26 (62).
constexpr int TEMPER_POINTS = 8;
struct TemperShm {
    double dpart[2][8][2];                       // [parity][warp] S1, S2 of an FP64 evaluation
    float tpart[2][8][2];                        // ... and T1, T2
    float fwarp[8][2 * TEMPER_POINTS];           // a float evaluation: per-warp sums,
    float fpart[2][2 * TEMPER_POINTS];           // [parity] and the CTA's
    double minw[8], cmin;
    double c, s1, s2;                            // warp 0's decision: the next point, or the answer,
    int act;                                     // one of TemperAct,
    int keep;                                    // and whether the weights just formed are the answer's so far
};
enum TemperAct { TEMPER_EVAL = 0, TEMPER_LAST = 1, TEMPER_DONE = 2 };

template <int TPT>
__device__ __forceinline__ double cta_min(double v, TemperShm* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(FULL, v, o));
    if (lane == 0) sh->minw[warp] = v;
    __syncthreads();
    double m = sh->minw[0];
    for (int w = 1; w < TPT / 32; ++w) m = fmin(m, sh->minw[w]);
    __syncthreads();
    return m;
}

// The sums S1 = sum w_e and S2 = sum w_e^2 of the weights w_e = exp(-d phi_e - max),
// max = -d phi_min, over the cluster (ESS = S1^2 / S2, Eq. ess), and in float T1 = sum z_e
// w_e and T2 = sum z_e w_e^2, z_e = phi_e - phi_min, which give its slope: d log ESS / dd =
// -2 (T1 / S1 - T2 / S2).  The sums are warp 0's; the thread's weights are returned in w.
template <int TPT>
__device__ __forceinline__ void ess_sums(double d, const double (&phi)[TEMPER_PER_THREAD],
                                         const float (&z)[TEMPER_PER_THREAD], int cnt, double phimin, TemperShm* sh,
                                         int& parity, double& S1, double& S2, float& T1, float& T2,
                                         double (&w)[TEMPER_PER_THREAD]) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    constexpr int NW = TPT / 32;
    const double mx = -d * phimin;
    double s1 = 0.0, s2 = 0.0;
    float t1 = 0.f, t2 = 0.f;
#pragma unroll
    for (int e = 0; e < TEMPER_PER_THREAD; ++e) {
        w[e] = 0.0;
        if (e < cnt) {
            w[e] = exp(-d * phi[e] - mx);
            s1 += w[e];
            s2 += w[e] * w[e];
            const float wf = (float)w[e];
            if (wf > 0.f) {      // an infinite z has no weight
                t1 = fmaf(z[e], wf, t1);
                t2 = fmaf(z[e] * wf, wf, t2);
            }
        }
    }
    // the lower half of the warp sums s1, the upper s2: five FP64 additions for the two
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool up = lane & 16;
    const double sent = __shfl_xor_sync(FULL, up ? s1 : s2, 16);
    double s = (up ? s2 : s1) + sent;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        t1 += __shfl_xor_sync(FULL, t1, o);
        t2 += __shfl_xor_sync(FULL, t2, o);
    }
    if ((lane & 15) == 0) sh->dpart[parity][warp][lane >> 4] = s;
    if (lane == 0) {
        sh->tpart[parity][warp][0] = t1;
        sh->tpart[parity][warp][1] = t2;
    }
    cl.sync();
    if (warp == 0) {
        // one partial per (CTA, warp): lane l takes those of number l, l + 32, ...
        double a = 0.0, b = 0.0;
        t1 = 0.f;
        t2 = 0.f;
#pragma unroll
        for (int q = 0; q < TEMPER_CTAS * NW / 32; ++q) {
            const int k = lane + 32 * q;
            const TemperShm* o = cl.map_shared_rank(sh, k / NW);
            const double pa = o->dpart[parity][k % NW][0], pb = o->dpart[parity][k % NW][1];
            a = q ? a + pa : pa;
            b = q ? b + pb : pb;
            t1 += o->tpart[parity][k % NW][0];
            t2 += o->tpart[parity][k % NW][1];
        }
        const double got = __shfl_xor_sync(FULL, up ? a : b, 16);
        double v = (up ? b : a) + got;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
        S1 = __shfl_sync(FULL, v, 0);
        S2 = __shfl_sync(FULL, v, 16);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            t1 += __shfl_xor_sync(FULL, t1, o);
            t2 += __shfl_xor_sync(FULL, t2, o);
        }
        T1 = t1;
        T2 = t2;
    }
    parity ^= 1;
}

// One float evaluation at the TEMPER_POINTS points x_g = x0 + g dx (geo: x0 2^g): the number of
// points that pass before the first that does not, and g(x) = ESS - ess_min at the last that
// passes (gl) and at the next (gh); the same in every thread of the cluster.
template <int TPT>
__device__ __forceinline__ int ess_points(float x0, float dx, bool geo, const float (&z)[TEMPER_PER_THREAD], int cnt,
                                          float ess_min, TemperShm* sh, int& parity, float& gl, float& gh) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    constexpr int G = TEMPER_POINTS;
    float v[2 * G];
#pragma unroll
    for (int g = 0; g < 2 * G; ++g) v[g] = 0.f;
    for (int e = 0; e < cnt; ++e) {
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const float x = geo ? x0 * (float)(1 << g) : fmaf((float)g, dx, x0);
            float w;
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(w) : "f"(-1.44269504f * x * z[e]));
            v[g] += w;
            v[G + g] = fmaf(w, w, v[G + g]);
        }
    }
    // halving butterfly: after the exchanges over 16, 8, 4 and 2 a lane holds sum number lane / 2
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int h = G, o = 16; h >= 1; h >>= 1, o >>= 1)
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const bool up = lane & o;
            const float got = __shfl_xor_sync(FULL, up ? v[k] : v[k + h], o);
            v[k] = (up ? v[k + h] : v[k]) + got;
        }
    v[0] += __shfl_xor_sync(FULL, v[0], 1);
    if ((lane & 1) == 0) sh->fwarp[warp][lane >> 1] = v[0];
    __syncthreads();
    if (threadIdx.x < 2 * G) {
        float s = 0.f;
        for (int w = 0; w < TPT / 32; ++w) s += sh->fwarp[w][threadIdx.x];
        sh->fpart[parity][threadIdx.x] = s;
    }
    cl.sync();
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < TEMPER_CTAS; ++r) s += cl.map_shared_rank(sh, r)->fpart[parity][lane & (2 * G - 1)];
    parity ^= 1;
    const float s2 = __shfl_sync(FULL, s, (lane & (G - 1)) + G);
    const float g = s * s / s2 - ess_min;                     // lanes 0 .. G - 1
    const unsigned fail = __ballot_sync(FULL, !(g >= 0.f)) & ((1u << G) - 1);
    const int k = fail ? __ffs(fail) - 1 : G;
    gl = __shfl_sync(FULL, g, k > 0 ? k - 1 : 0);
    gh = __shfl_sync(FULL, g, k < G ? k : 0);
    return k;
}

template <int TPT>
__global__ void __cluster_dims__(TEMPER_CTAS, 1, 1) __launch_bounds__(TPT)
    temper_kernel(int N, const double* __restrict__ nll, const double* __restrict__ logG, double theta,
                  const double* __restrict__ theta_dev, double ess_min, int halving, double* __restrict__ wbar,
                  double* __restrict__ out) {
    namespace cg = cooperative_groups;
    __shared__ TemperShm shm;
    TemperShm* sh = &shm;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    // device-gated stage: the temperature comes from the previous stage's result; a
    // stage that starts at theta = 1 is inactive and only says so (out[4] = 0)
    if (theta_dev) {
        theta = *theta_dev;
        if (theta >= 1.0) {
            if (rank == 0 && threadIdx.x == 0) {
                out[0] = 0.0;
                out[1] = 0.0;
                out[2] = 1.0;
                out[3] = 0.0;
                out[4] = 0.0;
            }
            return;
        }
    }
    const int gt = rank * TPT + threadIdx.x;                  // global thread index in the cluster
    constexpr int STRIDE = TEMPER_CTAS * TPT;
    // thread gt owns particles gt, gt + STRIDE, ... (coalesced)
    double phi[TEMPER_PER_THREAD];
    int cnt = 0;
    double lmin = INFINITY;
#pragma unroll
    for (int e = 0; e < TEMPER_PER_THREAD; ++e) {
        const int i = gt + e * STRIDE;
        if (i < N) {
            phi[e] = logG ? nll[i] - logG[i] : nll[i];
            lmin = fmin(lmin, phi[e]);
            cnt = e + 1;
        } else {
            phi[e] = 0.0;
        }
    }
    // cluster-wide minimum of phi
    const double cmin = cta_min<TPT>(lmin, sh);
    if (threadIdx.x == 0) sh->cmin = cmin;
    cl.sync();
    double phimin = INFINITY;
    for (int r = 0; r < TEMPER_CTAS; ++r) phimin = fmin(phimin, cl.map_shared_rank(sh, r)->cmin);
    float z[TEMPER_PER_THREAD];
#pragma unroll
    for (int e = 0; e < TEMPER_PER_THREAD; ++e) z[e] = (e < cnt) ? (float)(phi[e] - phimin) : 0.f;
    int parity = 0;
    const double rest = 1.0 - theta;
    const bool lead = threadIdx.x < 32;
    // wk: this thread's weights at the answer so far, so that the normalised weights need no
    // further pass.  A point passes when S1^2 >= ess_min S2 (S2 > 0), without a division.
    double S1 = 0.0, S2 = 0.0, wk[TEMPER_PER_THREAD];
    float T1 = 0.f, T2 = 0.f;
    ess_sums<TPT>(rest, phi, z, cnt, phimin, sh, parity, S1, S2, T1, T2, wk);
    const double s1_rest = S1, s2_rest = S2;   // (warp 0)
    if (lead) {
        if (threadIdx.x == 0) {
            sh->s1 = S1;
            sh->s2 = S2;
            sh->c = rest;
            sh->act = (S1 * S1 >= ess_min * S2) ? TEMPER_DONE : TEMPER_EVAL;
        }
    }
    __syncthreads();
    if (sh->act != TEMPER_DONE && halving) {
        // the paper's search read literally: halve dtheta until the ESS passes, at most
        // 60 times (the last point tried is kept if none passes)
        for (int k = 1; k <= 60; ++k) {
            const double d = ldexp(rest, -k);
            ess_sums<TPT>(d, phi, z, cnt, phimin, sh, parity, S1, S2, T1, T2, wk);
            if (threadIdx.x == 0) {
                sh->s1 = S1;
                sh->s2 = S2;
                sh->c = d;
                sh->act = (S1 * S1 >= ess_min * S2) ? TEMPER_DONE : TEMPER_EVAL;
            }
            __syncthreads();
            if (sh->act == TEMPER_DONE) break;
        }
    } else if (sh->act != TEMPER_DONE) {
        // The largest dtheta with ESS >= ess_min.  ESS(d) falls monotonically in d (its
        // log-derivative is 2 (E_{w^2}[phi] - E_w[phi]) <= 0), so the root of g(d) = ESS(d) -
        // ess_min is bracketed by [0, rest] (g(0) = N - ess_min >= 0).
        // Float: the root's octave, then three ninths of the bracket and the secant point of
        // what is left (1/729 of an octave): the root to about 1e-6.
        float a = 0.f, b = (float)rest, ga = (float)N - (float)ess_min, gb = -1.f;
        const float ess_f = (float)ess_min;
        for (int r = 0; r < 8; ++r) {
            const float x0 = b * 0x1p-8f;
            float gl, gh;
            const int k = ess_points<TPT>(x0, 0.f, true, z, cnt, ess_f, sh, parity, gl, gh);
            if (k < TEMPER_POINTS) {
                b = x0 * (float)(1 << k);
                gb = gh;
            }
            if (k > 0) {
                a = x0 * (float)(1 << (k - 1));
                ga = gl;
                break;
            }
        }
        for (int r = 0; r < 3; ++r) {
            const float dx = (b - a) * (1.f / (TEMPER_POINTS + 1));
            float gl, gh;
            const int k = ess_points<TPT>(a + dx, dx, false, z, cnt, ess_f, sh, parity, gl, gh);
            const float a0 = a;
            if (k > 0) {
                a = fmaf((float)k, dx, a0);
                ga = gl;
            }
            if (k < TEMPER_POINTS) {
                b = fmaf((float)(k + 1), dx, a0);
                gb = gh;
            }
        }
        // FP64: Newton steps from the float root inside the bracket [lo, hi] (lo passes, hi does
        // not), the step itself in float; a midpoint where a step leaves the bracket and every
        // sixth time.  Near the root the point is put 2^-51 below the estimate, so that it
        // passes.  The search stops at a passing point whose distance to the root is at most
        // 2^-49 of it, or when the bracket is that narrow.  A root below rest 2^-60
        // (astronomically spread phi) gives rest 2^-60, the smallest point 60 bisection steps
        // would try.
        const double dmin = rest * 0x1.0p-60;
        double lo = 0.0, hi = rest, c = (double)(a + (b - a) * (ga / (ga - gb)));
        if (!(c > lo && c < hi)) c = 0.5 * hi;
        double ks1 = 0.0, ks2 = 0.0;                // the sums at lo (warp 0)
        for (int it = 1;; ++it) {
            double wc[TEMPER_PER_THREAD];
            ess_sums<TPT>(c, phi, z, cnt, phimin, sh, parity, S1, S2, T1, T2, wc);
            if (lead) {
                const double num = fma(S1, S1, -(ess_min * S2));
                const bool pass = num >= 0.0;
                // g / |g'| = (num / S2) / (ESS |dlog ESS|): the root is at c + dl
                const float s1f = (float)S1, s2f = (float)S2;
                const float m1 = T1 / s1f, slope = m1 - T2 / s2f;
                const float dl = (float)num / (2.f * s1f * s1f * slope);
                // On a plateau of the ESS the float slope is the difference of two nearly equal
                // means (each right to about 1e-6) and may even have the wrong sign: then dl says
                // nothing, and the search goes on by midpoints to the narrow bracket
                const bool steep = slope > 1e-5f * m1;
                const float cf = (float)c;
                int act = TEMPER_EVAL;
                if (pass) {
                    lo = c;
                    ks1 = S1;
                    ks2 = S2;
                    if (steep && dl <= cf * 0x1p-49f) act = TEMPER_DONE;
                } else {
                    hi = c;
                }
                double cn = lo;
                if (hi - lo <= hi * 0x1.0p-49 || hi < dmin || it >= 400) act = TEMPER_DONE;
                if (act == TEMPER_DONE) {
                    if (!(lo > 0.0)) {
                        act = TEMPER_LAST;
                        cn = fmax(hi, dmin);
                    }
                } else {
                    cn = c + (double)dl;
                    if (fabsf(dl) < cf * 0x1p-30f) cn = fma(c, -0x1.0p-51, cn);
                    if (!steep || !(cn > lo && cn < hi) || it % 6 == 0) cn = 0.5 * (lo + hi);
                }
                if (threadIdx.x == 0) {
                    sh->c = cn;
                    sh->s1 = ks1;
                    sh->s2 = ks2;
                    sh->act = act;
                    sh->keep = pass;
                }
            }
            __syncthreads();
            c = sh->c;
            if (sh->keep) {
#pragma unroll
                for (int e = 0; e < TEMPER_PER_THREAD; ++e) wk[e] = wc[e];
            }
            if (sh->act != TEMPER_EVAL) break;
        }
        if (sh->act == TEMPER_LAST) {
            ess_sums<TPT>(c, phi, z, cnt, phimin, sh, parity, S1, S2, T1, T2, wk);
            if (threadIdx.x == 0) {
                sh->s1 = S1;
                sh->s2 = S2;
            }
            __syncthreads();
        }
    }
    const double d = sh->c, s1 = sh->s1;
#pragma unroll
    for (int e = 0; e < TEMPER_PER_THREAD; ++e) {
        const int i = gt + e * STRIDE;
        if (i < N) wbar[i] = wk[e] / s1;
    }
    if (rank == 0 && threadIdx.x == 0) {
        out[0] = d;
        out[1] = s1 * s1 / sh->s2;
        out[2] = (d >= 1.0 - theta) ? 1.0 : theta + d;
        out[3] = s1_rest * s1_rest / s2_rest;
        if (theta_dev) out[4] = 1.0;
    }
    cl.sync();   // no CTA leaves while another may still read its shared memory
}

// floor(w 2^50) of a weight 0 <= w < 2, from its bits (anything else as the conversion gives it)
__device__ __forceinline__ unsigned long long weight_q50(double w) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(w);
    const int e = (int)(b >> 52);                         // sign and exponent
    if (e > 1023) return __double2ull_rd(w * 0x1.0p50);   // at least 2, negative, infinite or NaN
    const int sh = 1025 - e;
    return (e == 0 || sh > 63) ? 0ull : ((b & 0xfffffffffffffull) | 0x10000000000000ull) >> sh;
}

// Offspring indices of systematic resampling on integers:
// q_i = floor(wbar_i 2^50), C = inclusive scan, T = C_{N-1},
// slot i -> smallest j with C_j > t_i = (i T + floor(U T / 2^53)) / N
// (equal to floor((i 2^53 + U) T / (N 2^53)) since 2^53 divides i 2^53 T).
// One CTA, bound by latency and by what each thread does for its N / 1024 weights: q_i is
// cut out of the weight's bits (a product and a conversion hold the FP64 unit for 64 cycles a
// warp each), a thread's share is odd so that a warp's shared accesses fall into different
// banks, and t_i = i (T / N) + V / N + (i (T mod N) + V mod N) / N, V = floor(U T / 2^53),
// leaves a 32-bit division a slot.  N = 8001: 23 us before, 16 us so.
__global__ void __launch_bounds__(RESAMPLE_THREADS) resample_kernel(int N, const double* __restrict__ wbar,
                                                                    uint64_t seed, uint64_t stage_ctr,
                                                                    const double* __restrict__ gate,
                                                                    int32_t* __restrict__ idx) {
    extern __shared__ __align__(16) unsigned long long Cs[];   // N inclusive sums
    __shared__ unsigned long long wsum[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // an inactive device-gated stage keeps every particle in place
    if (gate && *gate == 0.0) {
        for (int i = t; i < N; i += blockDim.x) idx[i] = i;
        return;
    }
    const int per = (N + RESAMPLE_THREADS - 1) / RESAMPLE_THREADS | 1;
    const int beg = t * per;
    const int end = min(N, beg + per);
    unsigned long long loc = 0;
    for (int i = beg; i < end; ++i) {
        loc += weight_q50(wbar[i]);
        Cs[i] = loc;
    }
    // exclusive scan of per-thread totals
    unsigned long long v = loc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long n = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += n;
    }
    if (lane == 31) wsum[warp] = v;
    __syncthreads();
    if (warp == 0) {
        unsigned long long w = (lane < (int)(blockDim.x >> 5)) ? wsum[lane] : 0ull;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long n = __shfl_up_sync(FULL, w, o);
            if (lane >= o) w += n;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    const unsigned long long off = (v - loc) + (warp > 0 ? wsum[warp - 1] : 0ull);
    for (int i = beg; i < end; ++i) Cs[i] += off;
    __syncthreads();
    const unsigned long long T = Cs[N - 1];
    const U64x4 r = philox4x64(0, 0, 0, stage_ctr, seed, SCH_TAG_RESAMPLE);
    const unsigned long long U = r.v0 >> 11;
    const unsigned long long ut_hi = __umul64hi(U, T), ut_lo = U * T;
    const unsigned long long ut53 = (ut_hi << 11) | (ut_lo >> 53);
    const unsigned long long qT = T / (unsigned)N, qV = ut53 / (unsigned)N;
    const unsigned rT = (unsigned)(T - qT * (unsigned)N), rV = (unsigned)(ut53 - qV * (unsigned)N);
    for (int i = t; i < N; i += blockDim.x) {
        const unsigned long long thr = (unsigned)i * qT + qV + ((unsigned)i * rT + rV) / (unsigned)N;
        int lo = 0, hi = N - 1;   // smallest j with C_j > thr (C_{N-1} = T > thr)
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (Cs[mid] > thr) hi = mid; else lo = mid + 1;
        }
        idx[i] = lo;
    }
}

template <typename V>
__global__ void gather_kernel(int N, const int32_t* __restrict__ idx, const V* __restrict__ src,
                              V* __restrict__ dst, size_t rowv) {
    const size_t tot = (size_t)N * rowv;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < tot; q += (size_t)gridDim.x * blockDim.x) {
        const size_t row = q / rowv, col = q % rowv;
        dst[q] = src[(size_t)idx[row] * rowv + col];
    }
}

// Row gathers of several arrays in one launch: blockIdx.y picks the array, whose rows
// move in the widest vector (16, 8 or 4 bytes) that divides the row length.
struct GatherSet {
    const void* src[GATHER_MAX_ARRAYS];
    void* dst[GATHER_MAX_ARRAYS];
    size_t rowv[GATHER_MAX_ARRAYS];
    int vw[GATHER_MAX_ARRAYS];
};

template <typename V>
__device__ __forceinline__ void gather_rows(int N, const int32_t* __restrict__ idx, const V* __restrict__ src,
                                            V* __restrict__ dst, size_t rowv) {
    const size_t tot = (size_t)N * rowv;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < tot; q += (size_t)gridDim.x * blockDim.x) {
        const size_t row = q / rowv, col = q % rowv;
        dst[q] = src[(size_t)idx[row] * rowv + col];
    }
}

__global__ void gather_multi_kernel(int N, const int32_t* __restrict__ idx, GatherSet g) {
    const int a = blockIdx.y;
    if (g.vw[a] == 16) gather_rows<uint4>(N, idx, (const uint4*)g.src[a], (uint4*)g.dst[a], g.rowv[a]);
    else if (g.vw[a] == 8) gather_rows<uint2>(N, idx, (const uint2*)g.src[a], (uint2*)g.dst[a], g.rowv[a]);
    else gather_rows<unsigned>(N, idx, (const unsigned*)g.src[a], (unsigned*)g.dst[a], g.rowv[a]);
}

__global__ void copy_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst, size_t n16) {
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n16; q += (size_t)gridDim.x * blockDim.x)
        dst[q] = src[q];
}

int launch_temper(int N, const double* nll, const double* logG, double theta, const double* theta_dev,
                  double ess_min, int halving, double* wbar, double* out, cudaStream_t st) {
    if (N <= TEMPER_CTAS * TEMPER_THREADS_SMALL)
        temper_kernel<TEMPER_THREADS_SMALL><<<TEMPER_CTAS, TEMPER_THREADS_SMALL, 0, st>>>(
            N, nll, logG, theta, theta_dev, ess_min, halving, wbar, out);
    else
        temper_kernel<TEMPER_THREADS_LARGE><<<TEMPER_CTAS, TEMPER_THREADS_LARGE, 0, st>>>(
            N, nll, logG, theta, theta_dev, ess_min, halving, wbar, out);
    return cudaGetLastError() == cudaSuccess ? SCH_OK : SCH_ERR_CUDA;
}

int launch_resample_idx(int N, const double* wbar, uint64_t seed, uint64_t stage_ctr, const double* gate,
                        int32_t* idx, cudaStream_t st) {
    const size_t sm = (size_t)N * sizeof(unsigned long long);
    if (sm > 48 * 1024)
        cudaFuncSetAttribute(resample_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    resample_kernel<<<1, RESAMPLE_THREADS, sm, st>>>(N, wbar, seed, stage_ctr, gate, idx);
    return cudaGetLastError() == cudaSuccess ? SCH_OK : SCH_ERR_CUDA;
}

static int grid_for(size_t work) {
    size_t b = (work + 255) / 256;
    if (b > (size_t)device_sms() * 8) b = (size_t)device_sms() * 8;
    if (b < 1) b = 1;
    return (int)b;
}

int launch_gather(int N, const int32_t* idx, const void* src, void* dst, size_t row_bytes, cudaStream_t st) {
    if (row_bytes % 16 == 0) {
        const size_t rv = row_bytes / 16;
        gather_kernel<uint4><<<grid_for((size_t)N * rv), 256, 0, st>>>(N, idx, (const uint4*)src, (uint4*)dst, rv);
    } else if (row_bytes % 8 == 0) {
        const size_t rv = row_bytes / 8;
        gather_kernel<uint2><<<grid_for((size_t)N * rv), 256, 0, st>>>(N, idx, (const uint2*)src, (uint2*)dst, rv);
    } else {
        const size_t rv = row_bytes / 4;
        gather_kernel<unsigned><<<grid_for((size_t)N * rv), 256, 0, st>>>(N, idx, (const unsigned*)src,
                                                                         (unsigned*)dst, rv);
    }
    return cudaGetLastError() == cudaSuccess ? SCH_OK : SCH_ERR_CUDA;
}

int launch_gather_multi(int N, const int32_t* idx, int n, const void* const* src, void* const* dst,
                        const size_t* row_bytes, cudaStream_t st) {
    if (n < 1 || n > GATHER_MAX_ARRAYS) return SCH_ERR_ARG;
    GatherSet g{};
    size_t most = 0;
    for (int a = 0; a < n; ++a) {
        const int vw = row_bytes[a] % 16 == 0 ? 16 : (row_bytes[a] % 8 == 0 ? 8 : 4);
        g.src[a] = src[a];
        g.dst[a] = dst[a];
        g.vw[a] = vw;
        g.rowv[a] = row_bytes[a] / vw;
        most = most > (size_t)N * g.rowv[a] ? most : (size_t)N * g.rowv[a];
    }
    gather_multi_kernel<<<dim3(grid_for(most), n), 256, 0, st>>>(N, idx, g);
    return cudaGetLastError() == cudaSuccess ? SCH_OK : SCH_ERR_CUDA;
}

int launch_copy(const void* src, void* dst, size_t bytes, cudaStream_t st) {
    const size_t n16 = bytes / 16;
    copy_kernel<<<grid_for(n16), 256, 0, st>>>((const uint4*)src, (uint4*)dst, n16);
    return cudaGetLastError() == cudaSuccess ? SCH_OK : SCH_ERR_CUDA;
}

}  // namespace sch
