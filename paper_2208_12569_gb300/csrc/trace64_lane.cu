// FP64 lattice tracer with one lane per line (trace.cuh's body): the same
// arithmetic as trace64.cuh's groups of eight lanes, bit for bit, for maps so
// large that their longest lines no longer matter. Both forms hold the FP64 pipe
// for the same time a line there; the groups' quotients on the integer pipe then
// cost more than the hardware's, which 32 lines share. Which maps: api.cu,
// line_per_lane. Built without contraction like trace_f64.cu.
#include "trace.cuh"

namespace fqsl {
namespace {
constexpr int kBlock = 128;

// The adaptive scheme's latency wants warps more than registers: 8 blocks (64
// registers, the rest spilled to L1) took 92.5 ms per 1024x1024 map of a
// 256x256x128 cube, 168 registers and 3 blocks 108.9 ms. The fixed step keeps its
// registers (8.9 against 8.5 M Q+Tw/s).
template <bool RECT>
__global__ void __launch_bounds__(kBlock, 8) k_trace64_lane(const TraceArgs A)
{
    trace::trace_body<double, kSrcLattice, true, 0, false, false, RECT>(A, BatchArgs{});
}

template <bool RECT>
__global__ void __launch_bounds__(kBlock) k_trace64_lane_rk38(const TraceArgs A)
{
    trace::trace_body<double, kSrcLattice, true, 0, false, false, RECT, 1>(A, BatchArgs{});
}

typedef void (*Kernel)(const TraceArgs);
Kernel kernel_of(bool rect, int scheme)
{
    if (scheme == 1) return rect ? k_trace64_lane_rk38<true> : k_trace64_lane_rk38<false>;
    return rect ? k_trace64_lane<true> : k_trace64_lane<false>;
}
}  // namespace

cudaError_t launch_trace64_lane(const TraceArgs &a, int grid, cudaStream_t s)
{
    kernel_of(a.f.rect != 0, a.p.scheme)<<<grid, kBlock, 0, s>>>(a);
    return cudaGetLastError();
}

int trace64_lane_blocks_per_sm(bool rect, int scheme)
{
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel_of(rect, scheme), kBlock, 0);
    return b > 0 ? b : 1;
}
}  // namespace fqsl
