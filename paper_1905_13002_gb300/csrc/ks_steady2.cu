// The settled path (ks_steady.cuh) at nx = 2, ny = 1.
#include "ks_steady_kernels.cuh"

namespace ks {
template int launch_plan_kernel<2, 1>(const PlanArgs<2, 1>&, cudaStream_t);
template int launch_steady_kernel<2, 1>(const SteadyArgs<2, 1>&, cudaStream_t);
}
