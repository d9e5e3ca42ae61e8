// The settled path (ks_steady.cuh) at nx = 8, ny = 4.
#include "ks_steady_kernels.cuh"

namespace ks {
template int launch_plan_kernel<8, 4>(const PlanArgs<8, 4>&, cudaStream_t);
template int launch_steady_kernel<8, 4>(const SteadyArgs<8, 4>&, cudaStream_t);
}
