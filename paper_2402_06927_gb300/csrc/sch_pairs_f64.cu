// FP64 windows and jitters of small ensembles: chunks of two nodes per thread, n = 128 and 256
// (TP = n / 2), linearly implicit solver, either noise model.
//
// A warp's FP64 instruction holds its sub-partition's unit for 64 cycles, and an ensemble of
// N n / 128 warps on four-node chunks that does not fill the SMs' sub-partitions leaves units
// idle while each warp waits for its own.  Half the nodes a thread puts the same work on
// twice as many units; only the reduced solves (float, in warp 0) get longer.
// One GB300, five steps of one particle an SM, four-node against two-node chunks: n = 256 172 /
// 138 us, with the Matern noise 211 / 169; n = 128 171 / 128 and 193 / 140.  A filter cycle
// with n = 256, N = 32: 3.29 -> 2.53 ms.
#include "sch_matern.cuh"

namespace sch {

#define SCH_PAIRS(expr_tp, L, ...)                                \
    switch (expr_tp) {                                            \
        case 64: return L<double, 2, 64>::__VA_ARGS__;            \
        case 128: return L<double, 2, 128>::__VA_ARGS__;          \
        default: return SCH_ERR_UNSUPPORTED;                      \
    }

int launch_window_pairs(const ModelArgs<double>& A, int matern, const WindowIO<double>& io, int N, cudaStream_t st) {
    if (matern) SCH_PAIRS(A.n / 2, LaunchMatern, template window<SCH_SOLVER_LI>(A, io, N, st))
    SCH_PAIRS(A.n / 2, Launch, template window<SCH_SOLVER_LI>(A, io, N, st))
}
int launch_jitter_pairs(const ModelArgs<double>& A, int matern, const JitterIO<double>& io, int N, cudaStream_t st) {
    if (matern) SCH_PAIRS(A.n / 2, LaunchMatern, template jitter<SCH_SOLVER_LI>(A, io, N, st))
    SCH_PAIRS(A.n / 2, Launch, template jitter<SCH_SOLVER_LI>(A, io, N, st))
}
size_t pairs_smem(int n, int Ns, int K, int bufs) {
    switch (n / 2) {
        case 64: return Launch<double, 2, 64>::smem(Ns, K, bufs);
        case 128: return Launch<double, 2, 128>::smem(Ns, K, bufs);
        default: return (size_t)-1;
    }
}

}  // namespace sch
