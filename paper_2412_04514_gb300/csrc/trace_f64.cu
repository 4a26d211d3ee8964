// trace_f64.cu -- cells by edge tracing, FP64 form.
#include "trace_impl.cuh"

namespace vt {

cudaError_t launch_trace_f64(const TraceArgs& a, cudaStream_t s) { return launch_trace_t<double>(a, s); }

}  // namespace vt
