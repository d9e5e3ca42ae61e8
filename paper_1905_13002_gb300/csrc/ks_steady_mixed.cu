// The settled path (ks_steady.cuh) of a mixed-size batch (ks_mixed.cuh): one
// preparation and one window launch over the sequences of all sizes.
#include "ks_mixed.cuh"
#include "ks_steady_kernels.cuh"

namespace ks {

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
KS_DEV SteadyArgs<N, M> steady_args(const MixedGroup<N, M>& g) {
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

// The windows of all groups, nx = 6 first (n6, n4: its and nx = 4's slots).
__global__ void __launch_bounds__(kStNT, kSteadyMinBlocks<6>) mixed_steady_kernel(MG6 g6, MG4 g4, MG2 g2, int64_t n6,
                                                                                  int64_t n4) {
    extern __shared__ __align__(16) char dsm[];
    pdl_trigger();
    int64_t s = (int64_t)blockIdx.x;
    if (s < n6) { steady_block<6, 3>(dsm, steady_args(g6), s); return; }
    s -= n6;
    if (s < n4) { steady_block<4, 2>(dsm, steady_args(g4), s); return; }
    steady_block<2, 1>(dsm, steady_args(g2), s - n4);
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

int launch_mixed_steady(const MG6& g6, const MG4& g4, const MG2& g2, const MixedQueue&, cudaStream_t st) {
    constexpr int smem =
        (int)cmax(cmax(sizeof(SteadySmem<6, 3>), sizeof(SteadySmem<4, 2>)), sizeof(SteadySmem<2, 1>));
    static const bool ok = cudaFuncSetAttribute(mixed_steady_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                smem) == cudaSuccess;
    if (!ok) return KS_ECUDA;
    const int64_t n6 = g6.B ? steady_blocks(g6.T, g6.B) : 0, n4 = g4.B ? steady_blocks(g4.T, g4.B) : 0,
                  n2 = g2.B ? steady_blocks(g2.T, g2.B) : 0;
    return launch_pdl(mixed_steady_kernel, (int)(n6 + n4 + n2), kStNT, smem, st, g6, g4, g2, n6, n4);
}

}  // namespace ks
