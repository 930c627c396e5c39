// Search kernels of SAILOR_OBJ_MIN_COST.
#include "sailor_plan_kernels.cuh"

namespace sailor {
template PlanKernel plan_kernel_of<SAILOR_OBJ_MIN_COST>(bool, bool, bool, bool);
}
