// schedule_walk_rb.cu -- the pipelined reduction, then broadcast, on large
// blocks (schedule_walk.cuh).
#include "schedule_walk.cuh"

namespace dpdr {

const void* walk_reduce_bcast_kernel(int dtype, bool vec) { return walk::kernel_for<true>(dtype, vec); }

}  // namespace dpdr
