// trace_f32.cu -- cells by edge tracing, FP32 form.
#include "trace_impl.cuh"

namespace vt {

cudaError_t launch_trace_f32(const TraceArgs& a, cudaStream_t s) { return launch_trace_t<float>(a, s); }

size_t trace_state_bytes() { return (sizeof(OpenCell) + 15) / 16 * 16; }

cudaError_t launch_keep_tail(const TraceArgs& a, const int32_t* before, uint8_t* kept, int64_t cap, cudaStream_t s)
{
    k_keep_tail<<<304, 256, 0, s>>>(a, before, kept, (int)cap);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_cutters(const TraceArgs& a, cudaStream_t s)
{
    if (a.nq <= 0) return cudaSuccess;
    auto kern = a.g.periodic ? k_cutters<true> : k_cutters<false>;
    unsigned blocks = 1;
    const cudaError_t e = resident_blocks(kern, CUT_BLOCK, 0, a.nq, CUT_BLOCK / 32, blocks);
    if (e != cudaSuccess) return e;
    kern<<<blocks, CUT_BLOCK, 0, s>>>(a);
    count_launch();
    return cudaGetLastError();
}

}  // namespace vt
