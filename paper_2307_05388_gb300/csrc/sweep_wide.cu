// Complex64 dataflow sweeps of large problems (flow.cuh).
#include "flow.cuh"

namespace fdfd {
FDFD_FLOW_SHAPE(wide1, kFlowThreads, kFlowWideCtas, float2, 1)
FDFD_FLOW_SHAPE(wide2, kFlowThreads, kFlowWideCtas, float2, 2)
}  // namespace fdfd
