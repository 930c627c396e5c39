// Search kernels of SAILOR_OBJ_MAX_THROUGHPUT.
#include "sailor_plan_kernels.cuh"

namespace sailor {
template PlanKernel plan_kernel_of<SAILOR_OBJ_MAX_THROUGHPUT>(bool, bool, bool, bool);
}
