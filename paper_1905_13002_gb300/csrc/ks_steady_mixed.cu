// The settled path (ks_steady.cuh) of a mixed-size batch (ks_mixed.cuh): one
// preparation over the sequences of all sizes, and the windows one size after
// another.  (One launch for all three gave every block nx = 6's 250 registers
// and 104 KB, two blocks per SM where nx = 4 and 2 fit three and four.)
#include "ks_mixed.cuh"
#include "ks_steady_kernels.cuh"

namespace ks {

extern template int launch_steady_kernel<6, 3>(const SteadyArgs<6, 3>&, cudaStream_t);   // ks_steady6.cu, ...
extern template int launch_steady_kernel<4, 2>(const SteadyArgs<4, 2>&, cudaStream_t);
extern template int launch_steady_kernel<2, 1>(const SteadyArgs<2, 1>&, cudaStream_t);

namespace {

template <int N, int M>
KS_DEV PlanArgs<N, M> plan_args(const MixedGroup<N, M>& g) {
    PlanArgs<N, M> a{g.F, g.u, g.Q, g.H, g.d, g.R, g.m0, g.P0, g.y, const_cast<ModelConst<N, M>*>(g.segs.mcg),
                     g.fs.status};
    a.zero = g.zero;
    a.nzero = g.nzero;
    a.off = g.segs.off;
    a.B = g.B;
    a.T = g.T;
    a.coef = const_cast<BlockCoef<N, M>*>(g.segs.coef);
    a.ch = g.ch;
    a.plan = g.plan;
    return a;
}

template <int N, int M>
SteadyArgs<N, M> steady_args(const MixedGroup<N, M>& g) {
    return SteadyArgs<N, M>{g.plan, g.segs.off, g.B, g.T, g.y, g.fmean, g.fcov, g.smean, g.scov, 1, g.fs.status};
}

// One block per sequence of all groups, nx = 6 first; block 0 also zeroes the
// scans' queue counters.
template <bool FOLD>
__global__ void __launch_bounds__(kPlanThreads) mixed_plan_kernel(MG6 g6, MG4 g4, MG2 g2, MixedQueue q) {
    extern __shared__ __align__(16) char prep_dsm[];
    pdl_trigger();
    int b = (int)blockIdx.x;
    if (b == 0 && threadIdx.x == 0) {
        *q.fcounter = 0u;
        *q.scounter = 0u;
    }
    if (b < g6.B) { plan_block<6, 3, FOLD>(prep_dsm, b, plan_args(g6)); return; }
    b -= g6.B;
    if (b < g4.B) { plan_block<4, 2, FOLD>(prep_dsm, b, plan_args(g4)); return; }
    b -= g4.B;
    if (b < g2.B) plan_block<2, 1, FOLD>(prep_dsm, b, plan_args(g2));
}

}  // namespace

int launch_mixed_plan(const MG6& g6, const MG4& g4, const MG2& g2, const MixedQueue& q, bool fold, cudaStream_t st) {
    constexpr int smem = (int)cmax(cmax(plan_dyn_smem<6, 3>(), plan_dyn_smem<4, 2>()), plan_dyn_smem<2, 1>());
    static_assert(smem <= 48 * 1024, "no opt-in needed");
    const int nseq = g6.B + g4.B + g2.B;
    if (fold)
        mixed_plan_kernel<true><<<nseq, kPlanThreads, smem, st>>>(g6, g4, g2, q);
    else
        mixed_plan_kernel<false><<<nseq, kPlanThreads, smem, st>>>(g6, g4, g2, q);
    return launch_status();
}

int launch_mixed_steady(const MG6& g6, const MG4& g4, const MG2& g2, cudaStream_t st) {
    int rc = KS_OK;
    if (g6.B && (rc = launch_steady_kernel(steady_args(g6), st))) return rc;
    if (g4.B && (rc = launch_steady_kernel(steady_args(g4), st))) return rc;
    if (g2.B) rc = launch_steady_kernel(steady_args(g2), st);
    return rc;
}

}  // namespace ks
