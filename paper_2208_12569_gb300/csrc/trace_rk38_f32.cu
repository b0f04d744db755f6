// FP32 tracer instantiations for the fixed-step scheme (Sec. 2.3: Kutta's
// 3/8-rule RK4 with the per-line step of Sec. 4 Eq. step): the persistent
// kernels of trace_f32.cu with trace_body's 4-stage trial, every trial
// accepted. Method I sources (lattice, rotated extra lines, seed lists),
// Method II's two ways of grad(B/|B|) and the taped lattice and extra-line
// tracers of the adjoint's forward pass.
#include "trace.cuh"

#ifndef FQSL_TRACE_F32_MINB
#define FQSL_TRACE_F32_MINB 4
#endif

namespace fqsl {
namespace {
constexpr int kBlock = 128;

template <int SRC, bool ACC, bool FLEX>
__global__ void __launch_bounds__(kBlock, FQSL_TRACE_F32_MINB) k_trace_rk38_f32(const TraceArgs A)
{
    trace::trace_body<float, SRC, ACC, 0, false, false, false, 1, FLEX>(A, BatchArgs{});
}

template <int WAY, bool FLEX>
__global__ void __launch_bounds__(kBlock, FQSL_TRACE_DEV_F32_MINB) k_trace_dev_rk38_f32(const TraceArgs A)
{
    trace::trace_body<float, kSrcLattice, false, WAY, false, false, false, 1, FLEX>(A, BatchArgs{});
}

// batches: many (field, plane) entries in one launch
template <bool ACC, bool FLEX>
__global__ void __launch_bounds__(kBlock, FQSL_TRACE_F32_MINB) k_batch_trace_rk38_f32(const TraceArgs A0,
                                                                                      const BatchArgs B)
{
    trace::trace_body<float, kSrcLattice, ACC, 0, true, false, false, 1, FLEX>(A0, B);
}

// the adjoint's forward pass: lattice or extra lines writing the step tape
template <int SRC, bool ACC>
__global__ void __launch_bounds__(kBlock, FQSL_TRACE_F32_MINB) k_trace_tape_rk38_f32(const TraceArgs A)
{
    trace::trace_body<float, SRC, ACC, 0, false, true, false, 1>(A, BatchArgs{});
}

template <bool ACC>
void launch(const TraceArgs &a, int src, int grid, cudaStream_t s)
{
    const bool flex = a.p.split || a.p.merge;
    if (src == kSrcLattice && flex) k_trace_rk38_f32<kSrcLattice, ACC, true><<<grid, kBlock, 0, s>>>(a);
    else if (src == kSrcLattice) k_trace_rk38_f32<kSrcLattice, ACC, false><<<grid, kBlock, 0, s>>>(a);
    else if (flex) k_trace_rk38_f32<kSrcList, ACC, true><<<grid, kBlock, 0, s>>>(a);
    else k_trace_rk38_f32<kSrcList, ACC, false><<<grid, kBlock, 0, s>>>(a);
}

template <bool ACC>
int blocks(int src)
{
    int b = 0;
    if (src == kSrcLattice)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_rk38_f32<kSrcLattice, ACC, true>, kBlock, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_rk38_f32<kSrcList, ACC, true>, kBlock, 0);
    return b > 0 ? b : 1;
}
}  // namespace

cudaError_t launch_trace_rk38_f32(const TraceArgs &a, int src, int grid, cudaStream_t s, bool acc64)
{
    if (acc64) launch<true>(a, src, grid, s);
    else launch<false>(a, src, grid, s);
    return cudaGetLastError();
}

int trace_rk38_blocks_per_sm_f32(int src, bool acc64) { return acc64 ? blocks<true>(src) : blocks<false>(src); }

cudaError_t launch_batch_trace_rk38_f32(const TraceArgs &a0, const BatchArgs &b, bool acc64, int grid,
                                        cudaStream_t s)
{
    // (the extra lines of rotated seeds run in the same launch: DevParams::merge)
    const bool flex = a0.p.merge != 0;
    if (acc64 && flex) k_batch_trace_rk38_f32<true, true><<<grid, kBlock, 0, s>>>(a0, b);
    else if (acc64) k_batch_trace_rk38_f32<true, false><<<grid, kBlock, 0, s>>>(a0, b);
    else if (flex) k_batch_trace_rk38_f32<false, true><<<grid, kBlock, 0, s>>>(a0, b);
    else k_batch_trace_rk38_f32<false, false><<<grid, kBlock, 0, s>>>(a0, b);
    return cudaGetLastError();
}

int batch_trace_rk38_blocks_per_sm_f32(bool acc64)
{
    int b = 0;
    if (acc64) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_batch_trace_rk38_f32<true, true>, kBlock, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_batch_trace_rk38_f32<false, true>, kBlock, 0);
    return b > 0 ? b : 1;
}

cudaError_t launch_trace_tape_rk38_f32(const TraceArgs &a, int src, int grid, cudaStream_t s, bool acc64)
{
    if (src == kSrcExtra) {
        if (acc64) k_trace_tape_rk38_f32<kSrcExtra, true><<<grid, kBlock, 0, s>>>(a);
        else k_trace_tape_rk38_f32<kSrcExtra, false><<<grid, kBlock, 0, s>>>(a);
    } else {
        if (acc64) k_trace_tape_rk38_f32<kSrcLattice, true><<<grid, kBlock, 0, s>>>(a);
        else k_trace_tape_rk38_f32<kSrcLattice, false><<<grid, kBlock, 0, s>>>(a);
    }
    return cudaGetLastError();
}

int trace_tape_rk38_blocks_per_sm_f32(int src, bool acc64)
{
    int b = 0;
    if (src == kSrcExtra) {
        if (acc64) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_tape_rk38_f32<kSrcExtra, true>, kBlock, 0);
        else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_tape_rk38_f32<kSrcExtra, false>, kBlock, 0);
    } else {
        if (acc64) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_tape_rk38_f32<kSrcLattice, true>, kBlock, 0);
        else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_tape_rk38_f32<kSrcLattice, false>, kBlock, 0);
    }
    return b > 0 ? b : 1;
}

cudaError_t launch_trace_dev_rk38_f32(const TraceArgs &a, int way, int grid, cudaStream_t s)
{
    const bool flex = a.p.split != 0;
    if (way == 1 && flex) k_trace_dev_rk38_f32<1, true><<<grid, kBlock, 0, s>>>(a);
    else if (way == 1) k_trace_dev_rk38_f32<1, false><<<grid, kBlock, 0, s>>>(a);
    else if (flex) k_trace_dev_rk38_f32<2, true><<<grid, kBlock, 0, s>>>(a);
    else k_trace_dev_rk38_f32<2, false><<<grid, kBlock, 0, s>>>(a);
    return cudaGetLastError();
}

int trace_dev_rk38_blocks_per_sm_f32(int way)
{
    int b = 0;
    if (way == 1) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_dev_rk38_f32<1, false>, kBlock, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_dev_rk38_f32<2, false>, kBlock, 0);
    return b > 0 ? b : 1;
}

}  // namespace fqsl
