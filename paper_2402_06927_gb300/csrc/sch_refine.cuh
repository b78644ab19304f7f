// FP64 fields, linearly implicit Picard steps by defect correction: the step's two
// residuals are formed in double, the corrections are solved for in float.
//
// What bounds the FP64 kernels on this part is the FP64 unit: a warp-wide DFMA occupies
// a sub-partition for 64 cycles (an FFMA for one), and the one warp that solves a
// reduced interface system waits that long for every instruction of it.  The plain
// iteration (sch_step) runs about 55 FP64 instructions a node and iteration, a
// quarter of them in that one warp.  Here an iteration forms, in double,
//   r = (M - mu dt/2 K - 1/2 A_dv) m0 - (M + mu dt/2 K + 1/2 A_dv) m,
// solves the same variable matrix for the change of m in float, adds it in double, then
// forms r' = M m - H u and solves for the change of u in the same way: 20 FP64
// instructions a node and iteration (counted with ncu), none in the reduced solves.  The iterates
// are those of sch_step up to the float solve's relative error (about 1e-7) in each
// *change*, which the next residual sees and removes, so the sequence contracts as
// before, stops by the same test after the same number of iterations (a few more where
// alpha is far below a cell: 108 against 71 over five steps at alpha = h / 20, n = 2048) and ends
// at the fixed point of the double residuals.  A step whose corrected iteration does not
// converge, or leaves the float range, is run again from its start by sch_step: its result
// and its status are those of the plain FP64 iteration.  u, no longer solved for anew, is within
// 1e-13 of H^{-1} M m for alpha up to 1e4 cells (the plain iteration's 1e-9 there); beyond 2e4
// cells every step is the plain iteration.
//
// Measured (one GB300, before -> after): gradients of 256 particles, n = 1024, 20 steps 11.60
// -> 4.20 ms; a filter cycle with n = 256, N = 32 9.63 -> 3.61 ms, with the Matern noise at
// n = 128, N = 150 14.5 -> 7.6 ms.  Against 64-bit values the gradients' error went from
// 2.1e-13 to 1.2e-13; the iteration counts are those of the plain iteration.
//
// The adjoint solve is treated alike (adjoint_step_refined in sch_adjoint.cuh).
#pragma once

#include "sch_kernels.cuh"

namespace sch {

// double -> float by truncation and float -> double, on the integer pipe (the
// conversion instructions run on the narrow pipe).  sh: power-of-two scale of the float
// side as an exponent-field offset, float = 2^(sh / 2^20) double, -1023 <= sh / 2^20 <= 800.
// Below the float range: zero; above it, infinite or NaN: NaN.  (The scaled exponent field is
// unsigned: up to 2847 << 20, and a negative one wraps to 3073 << 20 or more.)
__device__ __forceinline__ float d2f_bits(double x, int sh = 0) {
    const unsigned hi = (unsigned)__double2hiint(x);
    const unsigned ah = (hi & 0x7fffffffu) + (unsigned)sh;
    const unsigned t = __funnelshift_l((unsigned)__double2loint(x), hi + (unsigned)sh, 3) + 0x40000000u;
    unsigned r = (t & 0x7fffffffu) | (hi & 0x80000000u);
    if (ah < (897u << 20) || ah >= (3073u << 20)) r = 0u;
    if ((ah >= (1151u << 20) && ah < (3073u << 20)) || (hi & 0x7ff00000u) == 0x7ff00000u) r = 0x7fffffffu;
    return __uint_as_float(r);
}
// (A float NaN or infinity gives a finite value: an iteration that meets one in a right-hand side
// or a change ends without its result.)
__device__ __forceinline__ double f2d_bits(float x, int sh = 0) {
    const unsigned b = __float_as_uint(x);
    const unsigned ab = b & 0x7fffffffu;
    const int hi = (int)((b & 0x80000000u) | ((ab >> 3) + (unsigned)((896 << 20) - sh)));
    return ab < 0x00800000u ? 0.0 : __hiloint2double(hi, (int)(b << 29));
}

// the float view of a shared array of doubles (same slot, so that an exchange has the
// hazards of the double solve it replaces)
__device__ __forceinline__ float* fview(double* p) { return reinterpret_cast<float*>(p); }

// max over a warp of non-negative floats (or NaN with the sign bit clear, which wins):
// such floats order as their bit patterns
__device__ __forceinline__ float warp_max_bits(float v) {
    return __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(v)));
}

// Reduced solve of a variable matrix in float, warp 0 (as warp_reduce_var)
template <int TP>
__device__ __forceinline__ void warp_reduce_var_f(Shm<double, TP>* sh) {
    const float *ae_ = fview(sh->ae), *ge_ = fview(sh->ge), *de_ = fview(sh->de);
    const float *pa_ = fview(sh->pa), *pc_ = fview(sh->pc), *pd_ = fview(sh->pd);
    float *E = fview(sh->E), *F = fview(sh->F);
    auto row = [=](int t, float& A, float& B, float& Cc, float& D) {
        const int tn = (t + 1) & (TP - 1);
        const float ae = ae_[t], ge = ge_[t];
        A = -ae * pa_[t];
        B = 1.0f - ae * pc_[t] - ge * pa_[tn];
        Cc = -ge * pc_[tn];
        D = de_[t] - ae * pd_[t] - ge * pd_[tn];
    };
    warp_cyclic_solve<float, TP>(row, E, fview(sh->sw));
    constexpr int RR = Shm<double, TP>::RR;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < RR; ++r) {
        const int t = lane * RR + r;
        F[t] = pd_[t] - pa_[t] * E[(t - 1) & (TP - 1)] - pc_[t] * E[t];
    }
}

// Chunk sweep of rows a_i x_{i-1} + b_i x_i + c_i x_{i+1} = d_i in float: the reduced rows
// to shared memory; de, al, ga hold the back-swept interior afterwards.
template <int C, int TP>
__device__ __forceinline__ void var_local_f(const float (&a)[C], const float (&b)[C], const float (&c)[C],
                                            const float (&d)[C], float (&de)[C], float (&al)[C], float (&ga)[C],
                                            Shm<double, TP>* sh) {
    const int t = threadIdx.x;
    al[0] = -1.0f;
    ga[0] = 0.0f;
    de[0] = 0.0f;
#pragma unroll
    for (int i = 1; i < C; ++i) {
        const float q = rcp(b[i] - a[i] * ga[i - 1]);
        ga[i] = c[i] * q;
        al[i] = -a[i] * al[i - 1] * q;
        de[i] = (d[i] - a[i] * de[i - 1]) * q;
    }
    fview(sh->ae)[t] = al[C - 1];
    fview(sh->ge)[t] = ga[C - 1];
    fview(sh->de)[t] = de[C - 1];
    float dp = 0.0f, ap = 0.0f, gp = -1.0f;
#pragma unroll
    for (int i = C - 2; i >= 1; --i) {
        dp = de[i] - ga[i] * dp;
        ap = al[i] - ga[i] * ap;
        gp = -ga[i] * gp;
        de[i] = dp;
        al[i] = ap;
        ga[i] = gp;
    }
    if constexpr (C == 2) {   // no interior: the first row couples the last directly
        const float qF = rcp(b[0]);
        fview(sh->pa)[t] = a[0] * qF;
        fview(sh->pc)[t] = c[0] * qF;
        fview(sh->pd)[t] = d[0] * qF;
    } else {
        const float qF = rcp(b[0] - c[0] * al[1]);
        fview(sh->pa)[t] = a[0] * qF;
        fview(sh->pc)[t] = -c[0] * ga[1] * qF;
        fview(sh->pd)[t] = (d[0] - c[0] * de[1]) * qF;
    }
}

// The constant matrix (6/h)(M + alpha^2 K) in float: chunk sweep, reduced rows to shared memory.
// True where a right-hand side is out of the float range (NaN, which the change of m or psi need not
// show and which makes a reduced row NaN): the barrier that follows takes it to the stop test.  (As a
// flag in shared memory it cost windows of n = 128 up to 4%, on the barrier nothing that shows.)
template <int C, int TP>
__device__ __forceinline__ bool helm_local_f(const CTab<float>& T, const float (&r)[C], float (&dp)[C],
                                             Shm<double, TP>* sh) {
    float de[C];
    de[0] = 0.0f;
#pragma unroll
    for (int i = 1; i < C; ++i) de[i] = (r[i] - T.a * de[i - 1]) * T.rden[i];
    dp[0] = 0.0f;
    dp[C - 1] = 0.0f;
#pragma unroll
    for (int i = C - 2; i >= 1; --i) dp[i] = de[i] - T.gam[i] * dp[i + 1];
    const float pd = (r[0] - T.a * dp[1]) * T.iBF;
    fview(sh->hpd)[threadIdx.x] = pd;
    fview(sh->hde)[threadIdx.x] = de[C - 1];
    return !(fabsf(pd) + fabsf(de[C - 1]) < INFINITY);
}

// Reduced solve of a variable matrix whose interface rows stay the same over several
// right-hand sides, in float, by warp 0: factor() eliminates the rows (lane l: rows
// l RR .. l RR + RR - 1, as warp_cyclic_solve) and tabulates the lane system's PCR
// multipliers; solve() runs pd, de through them.  sw: 5 RR 32 floats kept between the calls
// (the lanes' sweep coefficients al, ga, q, gf, A).
template <int TP>
struct VarReduced {
    static constexpr int RR = TP / 32;
    float aeL, geL, qa, qc, iBF, Cc0;
    float k1[4], k2[4], f1, f2;

    __device__ __forceinline__ void factor(const float* ae, const float* ge, const float* pa, const float* pc,
                                           float* sw) {
        const int lane = threadIdx.x & 31, t0 = lane * RR;
        float a[RR], b[RR], c[RR];
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            const int t = t0 + r, tn = (t + 1) & (TP - 1);
            a[r] = -ae[t] * pa[t];
            b[r] = 1.0f - ae[t] * pc[t] - ge[t] * pa[tn];
            c[r] = -ge[t] * pc[tn];
            sw[(4 * RR + r) * 32 + lane] = a[r];
        }
        float LA = a[0], LB = b[0], LC = c[0];
        if constexpr (RR > 1) {
            float al[RR], gf[RR];
            al[0] = -1.0f;
            gf[0] = 0.0f;
#pragma unroll
            for (int r = 1; r < RR; ++r) {
                const float q = rcp(b[r] - a[r] * gf[r - 1]);
                gf[r] = c[r] * q;
                al[r] = -a[r] * al[r - 1] * q;
                sw[(2 * RR + r) * 32 + lane] = q;
                sw[(3 * RR + r) * 32 + lane] = gf[r];
            }
            aeL = al[RR - 1];
            geL = gf[RR - 1];
            float ap = 0.0f, gp = -1.0f;
#pragma unroll
            for (int r = RR - 2; r >= 1; --r) {
                ap = al[r] - gf[r] * ap;
                gp = -gf[r] * gp;
                sw[r * 32 + lane] = ap;
                sw[(RR + r) * 32 + lane] = gp;
            }
            Cc0 = c[0];
            const float BF = (RR == 2) ? b[0] : b[0] - c[0] * ap, CF = (RR == 2) ? c[0] : -c[0] * gp;
            iBF = rcp(BF);
            qa = a[0] * iBF;
            qc = CF * iBF;
            const int nx = (lane + 1) & 31;
            const float nqa = __shfl_sync(FULL, qa, nx), nqc = __shfl_sync(FULL, qc, nx);
            LA = -aeL * qa;
            LB = 1.0f - aeL * qc - geL * nqa;
            LC = -geL * nqc;
        }
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const int s = 1 << l, lo = (lane - s) & 31, hi = (lane + s) & 31;
            const float rb = rcp(LB);
            const float Am = __shfl_sync(FULL, LA, lo), Cm = __shfl_sync(FULL, LC, lo), rm = __shfl_sync(FULL, rb, lo);
            const float Ap = __shfl_sync(FULL, LA, hi), Cp = __shfl_sync(FULL, LC, hi), rp = __shfl_sync(FULL, rb, hi);
            k1[l] = LA * rm;
            k2[l] = LC * rp;
            const float nB = LB - Cm * k1[l] - Ap * k2[l];
            LA = -Am * k1[l];
            LC = -Cp * k2[l];
            LB = nB;
        }
        const float e = LA + LC;
        const float ej = __shfl_sync(FULL, e, lane ^ 16), Bj = __shfl_sync(FULL, LB, lane ^ 16);
        const float rd = rcp(LB * Bj - e * ej);
        f1 = Bj * rd;
        f2 = -e * rd;
    }

    __device__ __forceinline__ void solve(const float* ae, const float* ge, const float* pa, const float* pc,
                                          const float* pd, const float* de, const float* sw, float* E,
                                          float* F) const {
        const int lane = threadIdx.x & 31, t0 = lane * RR;
        float p[RR], D[RR], x[RR];
#pragma unroll
        for (int r = 0; r < RR; ++r) p[r] = pd[t0 + r];
        const float pn = __shfl_sync(FULL, p[0], (lane + 1) & 31);
#pragma unroll
        for (int r = 0; r < RR; ++r)
            D[r] = de[t0 + r] - ae[t0 + r] * p[r] - ge[t0 + r] * ((r == RR - 1) ? pn : p[(r + 1) % RR]);
        float LD = D[0], qd = 0.0f, dl[RR];
        if constexpr (RR > 1) {
            dl[0] = 0.0f;
#pragma unroll
            for (int r = 1; r < RR; ++r) dl[r] = (D[r] - sw[(4 * RR + r) * 32 + lane] * dl[r - 1]) * sw[(2 * RR + r) * 32 + lane];
            const float deL = dl[RR - 1];
            float dp = 0.0f;
#pragma unroll
            for (int r = RR - 2; r >= 1; --r) {
                dp = dl[r] - sw[(3 * RR + r) * 32 + lane] * dp;
                dl[r] = dp;
            }
            qd = ((RR == 2) ? D[0] : D[0] - Cc0 * dp) * iBF;
            LD = deL - aeL * qd - geL * __shfl_sync(FULL, qd, (lane + 1) & 31);
        }
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const int s = 1 << l;
            const float Dm = __shfl_sync(FULL, LD, (lane - s) & 31), Dp = __shfl_sync(FULL, LD, (lane + s) & 31);
            LD = LD - k1[l] * Dm - k2[l] * Dp;
        }
        const float EL = f1 * LD + f2 * __shfl_sync(FULL, LD, lane ^ 16);
        const float Ep = __shfl_sync(FULL, EL, (lane + 31) & 31);
        x[RR - 1] = EL;
        if constexpr (RR > 1) {
            x[0] = qd - qa * Ep - qc * EL;
#pragma unroll
            for (int r = 1; r < RR - 1; ++r) x[r] = dl[r] - sw[r * 32 + lane] * x[0] - sw[(RR + r) * 32 + lane] * EL;
        }
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            E[t0 + r] = x[r];
            F[t0 + r] = p[r] - pa[t0 + r] * ((r == 0) ? Ep : x[(r + RR - 1) % RR]) - pc[t0 + r] * x[r];
        }
        __syncwarp();
    }
};

// SALT increment dU/4 at the nodes i0 - 1 .. i0 + C of a chunk of C = 4 or 2 nodes about its
// centre theta_c: at theta_c +- d harmonic j gives cos(jd) (a S + b C) +- sin(jd) (a C - b S),
// (S, C) = (sin, cos)(j theta_c), so a harmonic costs a four-node chunk 12 FP64 instructions
// (noise_nodes: 38).  (s0, c0): the angle of node i0 - 1.
template <int C>
__device__ __forceinline__ void noise_nodes_centred(const ModelArgs<double>& A, const double* wq, double s0, double c0,
                                                    double (&nq)[C + 2]) {
    static_assert(C == 2 || C == 4, "the centre tables hold three offsets");
    constexpr int H = C / 2 + 1;
    const double cd = A.nco[0][H - 1], sd = A.nsi[0][H - 1];
    const double s1 = s0 * cd + c0 * sd, c1 = c0 * cd - s0 * sd;
    const double twoc = 2.0 * c1;
    double sj = s1, cj = c1, sjm = 0.0, cjm = 1.0;
    double E[H], O[H];
#pragma unroll
    for (int k = 0; k < H; ++k) {
        E[k] = 0.0;
        O[k] = 0.0;
    }
    for (int j = 0; j < A.K2; ++j) {
        const double a = wq[2 * j], b = wq[2 * j + 1];
        const double v = a * sj + b * cj, q = a * cj - b * sj;
#pragma unroll
        for (int k = 0; k < H; ++k) {
            E[k] += v * A.nco[j][k];
            O[k] += q * A.nsi[j][k];
        }
        const double sn2 = twoc * sj - sjm, cn2 = twoc * cj - cjm;
        sjm = sj;
        cjm = cj;
        sj = sn2;
        cj = cn2;
    }
#pragma unroll
    for (int k = 0; k < H; ++k) {
        nq[H + k] = E[k] + O[k];
        nq[H - 1 - k] = E[k] - O[k];
    }
}

// the plain step from the start state, kept out of line: only a step that fails to converge comes here
template <int C, int TP, int NZ>
__device__ __noinline__ void sch_step_plain(const ModelArgs<double>& A, Shm<double, TP>* sh, Field<double, C>& f,
                                            const double* wq, double s0, double c0, int& iters, int& flags) {
    sch_step<double, C, TP, NZ>(A, sh, f, wq, s0, c0, iters, flags);
}

// One linearly implicit Picard step (Eq. fde1) by defect correction; arguments as sch_step.
template <int C, int TP, int NZ>
__device__ __forceinline__ void sch_step_refined(const ModelArgs<double>& A, Shm<double, TP>* sh,
                                                 Field<double, C>& f, const double* wq, double s0, double c0,
                                                 int& iters, int& flags) {
    const int t = threadIdx.x;
    double W0[C], W0p, W0n;
    {
        double nq[C + 2];
        if constexpr (NZ == SCH_NOISE_MATERN)
            matern_nodes<double, C, TP>(A, sh, wq, nq);
        else
            noise_nodes_centred<C>(A, wq, s0, c0, nq);
#pragma unroll
        for (int i = 0; i < C; ++i) W0[i] = A.dt8 * f.u[i] + nq[i + 1];
        W0p = A.dt8 * f.up + nq[0];
        W0n = A.dt8 * f.un + nq[C + 1];
    }
    // S_i = m0_i + m0_{i+1} (S[0]: i = -1), s_i = S_{i-1} + S_i and D0 = (M - mu dt/2 K) m0
    double S[C + 1], D0[C], q[C + 1];
    S[0] = f.mp + f.m[0];
#pragma unroll
    for (int i = 0; i < C; ++i) S[i + 1] = f.m[i] + ((i == C - 1) ? f.mn : f.m[i + 1]);
#pragma unroll
    for (int i = 0; i < C; ++i) D0[i] = A.c0p * (S[i] + S[i + 1]) + (A.b0p - 2.0 * A.c0p) * f.m[i];
    double m[C], u[C];
    double mp = f.mp, mn = f.mn, up = f.up, un = f.un;
#pragma unroll
    for (int i = 0; i < C; ++i) {
        m[i] = f.m[i];
        u[i] = f.u[i];
    }
#pragma unroll
    for (int i = 0; i <= C; ++i) q[i] = S[i];
    const double bq = A.b0 - 2.0 * A.c0;
    const double h2 = A.helg;                    // off-diagonal of (6/h)(M + alpha^2 K)
    const float c0f = A.c0f, b0f = A.b0f;
    int it = 1, bad = 0;
    for (;; ++it) {
        float al[C], ga[C], de[C];
        {
            // w = dv / 4; r_i = D0_i - c0 (m_{i-1} + m_{i+1}) - b0 m_i + w_{i-1} T_{i-1} - w_{i+1} T_i,
            // T_i = S_i + m_i + m_{i+1}
            double w[C + 2], T[C + 1];
            w[0] = W0p + A.dt8 * up;
#pragma unroll
            for (int i = 0; i < C; ++i) w[i + 1] = W0[i] + A.dt8 * u[i];
            w[C + 1] = W0n + A.dt8 * un;
#pragma unroll
            for (int i = 0; i <= C; ++i) T[i] = S[i] + q[i];
            float wf[C + 2], a[C], b[C], c[C], d[C];
#pragma unroll
            for (int i = 0; i < C + 2; ++i) wf[i] = d2f_bits(w[i]);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                double r = D0[i] - A.c0 * (q[i] + q[i + 1]);
                r -= bq * m[i];
                r += w[i] * T[i];
                r -= w[i + 2] * T[i + 1];
                d[i] = d2f_bits(r);
                a[i] = c0f - wf[i];
                c[i] = c0f + wf[i + 2];
                b[i] = b0f + (wf[i + 2] - wf[i]);
            }
            var_local_f<C, TP>(a, b, c, d, de, al, ga, sh);
        }
        __syncthreads();                                             // B1
        if (t < 32) warp_reduce_var_f<TP>(sh);
        __syncthreads();                                             // B2
        float dmax = 0.0f, mmax = 0.0f;
        {
            const float F = fview(sh->F)[t], E = fview(sh->E)[t];
            mp += f2d_bits(fview(sh->E)[(t - 1) & (TP - 1)]);
            mn += f2d_bits(fview(sh->F)[(t + 1) & (TP - 1)]);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const float dm = (i == 0) ? F : (i == C - 1) ? E : de[i] - al[i] * F - ga[i] * E;
                // NaN or infinite changes win the maximum (as bit patterns)
                dmax = __uint_as_float(max(__float_as_uint(dmax), __float_as_uint(dm) & 0x7fffffffu));
                m[i] += f2d_bits(dm);
                mmax = __uint_as_float(max(__float_as_uint(mmax), __float_as_uint(d2f_bits(m[i])) & 0x7fffffffu));
            }
        }
        dmax = warp_max_bits(dmax);
        mmax = warp_max_bits(mmax);
        if ((t & 31) == 0) {
            fview(sh->wred[0])[t >> 5] = dmax;
            fview(sh->wred[1])[t >> 5] = mmax;
        }
        // (6/h)(M m - H u): s_i + 2 m_i - 6 u_i - h2 (u_{i-1} - 2 u_i + u_{i+1}), the second
        // difference from the (nearly exact) first ones
        float dpH[C];
        bool out;
        {
            q[0] = mp + m[0];
#pragma unroll
            for (int i = 0; i < C; ++i) q[i + 1] = m[i] + ((i == C - 1) ? mn : m[i + 1]);
            float r[C];
            double dl = u[0] - up;
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const double dr = ((i == C - 1) ? un : u[i + 1]) - u[i];
                double e = (q[i] + q[i + 1]) + 2.0 * m[i];
                e -= 6.0 * u[i];
                e -= h2 * (dr - dl);
                r[i] = d2f_bits(e);
                dl = dr;
            }
            out = helm_local_f<C, TP>(A.helf, r, dpH, sh);
        }
        const int nan = __syncthreads_or(out);                       // B3
        if (t < 32) {
            CTab<float> const& T = A.helf;
            warp_solve_const<float, TP>(T, A.rhelf, fview(sh->hpd), fview(sh->hde), fview(sh->hE), fview(sh->hF));
            constexpr int NW = TP / 32;
            const float dm = warp_max_bits((t < NW) ? fview(sh->wred[0])[t] : 0.0f);
            const float mm = warp_max_bits((t < NW) ? fview(sh->wred[1])[t] : 0.0f);
            if (t == 0) {
                int fl = 0;
                if (!(dm < INFINITY) || !(mm < INFINITY) || nan) fl = FLAG_NONFINITE;
                else if (dm <= A.tolf * fmaxf(1.0f, mm)) fl = FLAG_CONVERGED;
                sh->flag = fl;
            }
        }
        __syncthreads();                                             // B4
        {
            const float hF = fview(sh->hF)[t], hE = fview(sh->hE)[t];
            up += f2d_bits(fview(sh->hE)[(t - 1) & (TP - 1)]);
            un += f2d_bits(fview(sh->hF)[(t + 1) & (TP - 1)]);
            u[0] += f2d_bits(hF);
            u[C - 1] += f2d_bits(hE);
#pragma unroll
            for (int i = 1; i < C - 1; ++i)
                u[i] += f2d_bits(dpH[i] - A.helf.alpp[i] * hF - A.helf.gamp[i] * hE);
        }
        const int fl = sh->flag;
        if (fl & FLAG_CONVERGED) break;
        if ((fl & FLAG_NONFINITE) || it == A.max_iter) {
            bad = 1;
            break;
        }
    }
    if (bad) {
        Field<double, C> g = f;
        int gi = 0, gf = 0;
        __syncthreads();   // every thread has read the flag and the interface values
        sch_step_plain<C, TP, NZ>(A, sh, g, wq, s0, c0, gi, gf);
        f = g;
        iters += gi;
        flags |= gf;
        return;
    }
    iters += it;
#pragma unroll
    for (int i = 0; i < C; ++i) {
        f.m[i] = m[i];
        f.u[i] = u[i];
    }
    f.mp = mp;
    f.mn = mn;
    f.up = up;
    f.un = un;
}

}  // namespace sch
