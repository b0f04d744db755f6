// FP32 instantiations of the persistent tracer: the cube and the line state
// are in float. ACC = false (precision FQSL_F32): error norm in float, length
// and Tw as compensated float sums formed in double per direction. ACC = true
// (FQSL_F32_ACC64): error norm and length/Tw sums accumulated in double. The
// per-line tolerance, footpoints and Bn are double in both.
#include "trace.cuh"

// minimum resident blocks per SM requested from the register allocator
#ifndef FQSL_TRACE_F32_MINB
#define FQSL_TRACE_F32_MINB 4
#endif

namespace fqsl {
namespace {
constexpr int kBlock = 128;

template <int SRC, bool ACC, bool FLEX>
__global__ void __launch_bounds__(kBlock, FQSL_TRACE_F32_MINB) k_trace_f32(const TraceArgs A)
{
    trace::trace_body<float, SRC, ACC, 0, false, false, false, 0, FLEX>(A, BatchArgs{});
}
}  // namespace

namespace {
template <bool ACC>
void launch(const TraceArgs &a, int src, int grid, int block, cudaStream_t s)
{
    const bool flex = a.p.split || a.p.merge;
    if (src == kSrcLattice && flex) k_trace_f32<kSrcLattice, ACC, true><<<grid, block, 0, s>>>(a);
    else if (src == kSrcLattice) k_trace_f32<kSrcLattice, ACC, false><<<grid, block, 0, s>>>(a);
    else if (flex) k_trace_f32<kSrcList, ACC, true><<<grid, block, 0, s>>>(a);
    else k_trace_f32<kSrcList, ACC, false><<<grid, block, 0, s>>>(a);
}

template <bool ACC>
int blocks(int src)
{
    int b = 0;
    if (src == kSrcLattice)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_f32<kSrcLattice, ACC, true>, kBlock, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_f32<kSrcList, ACC, true>, kBlock, 0);
    return b > 0 ? b : 1;
}
}  // namespace

cudaError_t launch_trace_f32(const TraceArgs &a, int src, int grid, int block, cudaStream_t s, bool acc64)
{
    // (extra lines follow the lattice's items: DevParams::merge)
    if (block != kBlock || src == kSrcExtra) return cudaErrorInvalidValue;
    if (a.p.scheme == 1)
        return a.f.rect ? launch_trace_rect_rk38_f32(a, src, grid, s, acc64) : launch_trace_rk38_f32(a, src, grid, s, acc64);
    if (a.f.rect) return launch_trace_rect_f32(a, src, grid, s, acc64);
    if (acc64) launch<true>(a, src, grid, block, s);
    else launch<false>(a, src, grid, block, s);
    return cudaGetLastError();
}

int trace_blocks_per_sm_f32(int src, bool acc64) { return acc64 ? blocks<true>(src) : blocks<false>(src); }

}  // namespace fqsl

namespace fqsl {
namespace {
// Do the seeds of a list lie in order? 512 pairs of neighbours, spread evenly over
// it, are asked whether they are within 1.5 cells (reach) of each other on every
// axis. One block and one pair a thread: the loads' latency and the narrow FP64
// pipe are what it takes (4,096 pairs added 25 us to a list of 1 ms).
__global__ void __launch_bounds__(512) k_list_blocks(const double *__restrict__ seeds, long long n, double3 reach,
                                                     unsigned few, unsigned *__restrict__ blocks)
{
    const double *p = seeds + 3 * ((n - 1) * (int)threadIdx.x / 512);
    const bool near = fabs(p[3] - p[0]) <= reach.x && fabs(p[4] - p[1]) <= reach.y && fabs(p[5] - p[2]) <= reach.z;
    const int count = __syncthreads_count(near);
    if (threadIdx.x == 0) *blocks = 2 * count < 512 ? few : 0xffffffffu;
}
}  // namespace

cudaError_t launch_list_blocks(const TraceArgs &a, unsigned few, cudaStream_t s)
{
    if (a.nitems < 2) return cudaErrorInvalidValue;
    const FieldView &f = a.f;
    const int n[3] = {f.nx, f.ny, f.nz};
    double r[3];  // stretched grid: cells of the mean width
    for (int c = 0; c < 3; c++) r[c] = 1.5 * (f.rect ? (f.hi64[c] - f.lo64[c]) / (n[c] - 1) : f.d[c]);
    k_list_blocks<<<1, 512, 0, s>>>(a.seeds, a.nitems, make_double3(r[0], r[1], r[2]), few, a.q.blocks);
    return cudaGetLastError();
}
}  // namespace fqsl

namespace fqsl {
namespace {
__global__ void __launch_bounds__(256) k_seed_prep_f32(const TraceArgs A, long long n)
{
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x)
        trace::seed_prep_f32(A, idx);
}
}  // namespace

cudaError_t launch_seed_prep_f32(const TraceArgs &a, long long n, cudaStream_t s)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long blocks = (n + 255) / 256;
    if (blocks > (long long)sms * 8) blocks = (long long)sms * 8;
    if (blocks < 1) blocks = 1;
    if (a.f.rect) return launch_seed_prep_rect_f32(a, n, (unsigned)blocks, s);
    k_seed_prep_f32<<<(unsigned)blocks, 256, 0, s>>>(a, n);
    return cudaGetLastError();
}

}  // namespace fqsl

namespace fqsl {
namespace {
__global__ void __launch_bounds__(128) k_extra_prep_f32(const TraceArgs A)
{
    const long long m = 4LL * (long long)*A.q.rot_count;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < m; x += (long long)gridDim.x * blockDim.x)
        trace::extra_prep_f32(A, x);
}

__global__ void __launch_bounds__(128) k_batch_extra_prep_f32(const TraceArgs *__restrict__ desc,
                                                              const long long *__restrict__ xbase, int nent)
{
    const long long total = xbase[nent];
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < total;
         x += (long long)gridDim.x * blockDim.x) {
        int lo = 0, hi = nent - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (xbase[mid] <= x) lo = mid;
            else hi = mid - 1;
        }
        if (x - xbase[lo] < 4LL * (long long)*desc[lo].q.rot_count) trace::extra_prep_f32(desc[lo], x - xbase[lo]);
    }
}

unsigned sm_grid(int per_sm)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (unsigned)(sms * per_sm);
}
}  // namespace

cudaError_t launch_extra_prep_f32(const TraceArgs &a, cudaStream_t s)
{
    if (a.f.rect) return launch_extra_prep_rect_f32(a, sm_grid(4), s);
    k_extra_prep_f32<<<sm_grid(4), 128, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_batch_extra_prep_f32(const TraceArgs *desc, const long long *xbase, int nent, cudaStream_t s)
{
    k_batch_extra_prep_f32<<<sm_grid(4), 128, 0, s>>>(desc, xbase, nent);
    return cudaGetLastError();
}

}  // namespace fqsl

namespace fqsl {
namespace {
template <int WAY, bool FLEX>
__global__ void __launch_bounds__(kBlock, FQSL_TRACE_DEV_F32_MINB) k_trace_dev_f32(const TraceArgs A)
{
    trace::trace_body<float, kSrcLattice, false, WAY, false, false, false, 0, FLEX>(A, BatchArgs{});
}
}  // namespace

cudaError_t launch_trace_dev_f32(const TraceArgs &a, int way, int grid, int block, cudaStream_t s)
{
    if (block != kBlock) return cudaErrorInvalidValue;
    if (a.p.scheme == 1)
        return a.f.rect ? launch_trace_dev_rect_rk38_f32(a, way, grid, s) : launch_trace_dev_rk38_f32(a, way, grid, s);
    if (a.f.rect) return launch_trace_dev_rect_f32(a, way, grid, s);
    const bool flex = a.p.split != 0;
    if (way == 1 && flex) k_trace_dev_f32<1, true><<<grid, block, 0, s>>>(a);
    else if (way == 1) k_trace_dev_f32<1, false><<<grid, block, 0, s>>>(a);
    else if (flex) k_trace_dev_f32<2, true><<<grid, block, 0, s>>>(a);
    else k_trace_dev_f32<2, false><<<grid, block, 0, s>>>(a);
    return cudaGetLastError();
}

int trace_dev_blocks_per_sm_f32(int way)
{
    int b = 0;
    if (way == 1) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_dev_f32<1, false>, kBlock, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_dev_f32<2, false>, kBlock, 0);
    return b > 0 ? b : 1;
}
}  // namespace fqsl

// ---------------------------------------------------------------------------
// batches: many (field, plane) entries in one launch
// ---------------------------------------------------------------------------
namespace fqsl {
namespace {
template <bool ACC, bool FLEX>
__global__ void __launch_bounds__(kBlock, FQSL_TRACE_F32_MINB) k_batch_trace_f32(const TraceArgs A0, const BatchArgs B)
{
    trace::trace_body<float, kSrcLattice, ACC, 0, true, false, false, 0, FLEX>(A0, B);
}

__global__ void __launch_bounds__(256) k_batch_seed_prep_f32(const TraceArgs *__restrict__ desc,
                                                             const long long *__restrict__ nbase, int nent)
{
    const long long total = nbase[nent];
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        int lo = 0, hi = nent - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (nbase[mid] <= idx) lo = mid;
            else hi = mid - 1;
        }
        trace::seed_prep_f32(desc[lo], idx - nbase[lo]);
    }
}

// work-item prefix of the rotated extra lines: 4 per rotated seed, padded to
// whole 32-item chunks per entry
__global__ void k_batch_extra_prefix(const unsigned *__restrict__ rot_counts, int nent, long long *xbase)
{
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    long long acc = 0;
    for (int b = 0; b < nent; b++) {
        xbase[b] = acc;
        acc += (4LL * rot_counts[b] + 31) / 32 * 32;
    }
    xbase[nent] = acc;
}
}  // namespace

cudaError_t launch_batch_seed_prep_f32(const TraceArgs *desc, const long long *nbase, int nent, long long total,
                                       cudaStream_t s)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long blocks = (total + 255) / 256;
    if (blocks > (long long)sms * 8) blocks = (long long)sms * 8;
    if (blocks < 1) blocks = 1;
    k_batch_seed_prep_f32<<<(unsigned)blocks, 256, 0, s>>>(desc, nbase, nent);
    return cudaGetLastError();
}

cudaError_t launch_batch_extra_prefix(const unsigned *rot_counts, int nent, long long *xbase, cudaStream_t s)
{
    k_batch_extra_prefix<<<1, 32, 0, s>>>(rot_counts, nent, xbase);
    return cudaGetLastError();
}

cudaError_t launch_batch_trace_f32(const TraceArgs &a0, const BatchArgs &b, bool acc64, int grid,
                                   cudaStream_t s)
{
    if (a0.p.scheme == 1) return launch_batch_trace_rk38_f32(a0, b, acc64, grid, s);
    // (the extra lines of rotated seeds run in the same launch: DevParams::merge)
    const bool flex = a0.p.merge != 0;
    if (acc64 && flex) k_batch_trace_f32<true, true><<<grid, kBlock, 0, s>>>(a0, b);
    else if (acc64) k_batch_trace_f32<true, false><<<grid, kBlock, 0, s>>>(a0, b);
    else if (flex) k_batch_trace_f32<false, true><<<grid, kBlock, 0, s>>>(a0, b);
    else k_batch_trace_f32<false, false><<<grid, kBlock, 0, s>>>(a0, b);
    return cudaGetLastError();
}

int batch_trace_blocks_per_sm_f32(bool acc64, int scheme)
{
    if (scheme == 1) return batch_trace_rk38_blocks_per_sm_f32(acc64);
    int b = 0;
    if (acc64) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_batch_trace_f32<true, true>, kBlock, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_batch_trace_f32<false, true>, kBlock, 0);
    return b > 0 ? b : 1;
}
}  // namespace fqsl

// ---------------------------------------------------------------------------
// adjoint forward pass: the lattice tracer that also writes the step tape
// ---------------------------------------------------------------------------
namespace fqsl {
namespace {
template <int SRC, bool ACC>
__global__ void __launch_bounds__(kBlock, FQSL_TRACE_F32_MINB) k_trace_tape_f32(const TraceArgs A)
{
    trace::trace_body<float, SRC, ACC, 0, false, true>(A, BatchArgs{});
}
}  // namespace

cudaError_t launch_trace_tape_f32(const TraceArgs &a, int src, int grid, cudaStream_t s, bool acc64)
{
    if (src == kSrcExtra) {
        if (acc64) k_trace_tape_f32<kSrcExtra, true><<<grid, kBlock, 0, s>>>(a);
        else k_trace_tape_f32<kSrcExtra, false><<<grid, kBlock, 0, s>>>(a);
    } else {
        if (acc64) k_trace_tape_f32<kSrcLattice, true><<<grid, kBlock, 0, s>>>(a);
        else k_trace_tape_f32<kSrcLattice, false><<<grid, kBlock, 0, s>>>(a);
    }
    return cudaGetLastError();
}

int trace_tape_blocks_per_sm_f32(int src, bool acc64)
{
    int b = 0;
    if (src == kSrcExtra) {
        if (acc64) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_tape_f32<kSrcExtra, true>, kBlock, 0);
        else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_tape_f32<kSrcExtra, false>, kBlock, 0);
    } else {
        if (acc64) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_tape_f32<kSrcLattice, true>, kBlock, 0);
        else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_trace_tape_f32<kSrcLattice, false>, kBlock, 0);
    }
    return b > 0 ? b : 1;
}
}  // namespace fqsl
