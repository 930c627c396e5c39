// Search kernels of SAILOR_OBJ_MAX_THROUGHPUT_PER_USD.
#include "sailor_plan_kernels.cuh"

namespace sailor {
template PlanKernel plan_kernel_of<SAILOR_OBJ_MAX_THROUGHPUT_PER_USD>(bool, bool, bool, bool);
}
