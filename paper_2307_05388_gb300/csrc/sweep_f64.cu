// Complex128 dataflow sweeps (flow.cuh).
#include "flow.cuh"

namespace fdfd {
FDFD_FLOW_SHAPE(f64, kFlowThreads, 1, double2, 1)
}  // namespace fdfd
