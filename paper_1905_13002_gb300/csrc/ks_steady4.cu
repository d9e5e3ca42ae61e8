// The settled path (ks_steady.cuh) at nx = 4, ny = 2.
#include "ks_steady_kernels.cuh"

namespace ks {
template int launch_plan_kernel<4, 2>(const PlanArgs<4, 2>&, cudaStream_t);
template int launch_steady_kernel<4, 2>(const SteadyArgs<4, 2>&, cudaStream_t);
}
