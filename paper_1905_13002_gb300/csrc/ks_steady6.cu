// The settled path (ks_steady.cuh) at nx = 6, ny = 3.
#include "ks_steady_kernels.cuh"

namespace ks {
template int launch_plan_kernel<6, 3>(const PlanArgs<6, 3>&, cudaStream_t);
template int launch_steady_kernel<6, 3>(const SteadyArgs<6, 3>&, cudaStream_t);
}
