// k_span.cu -- span copies (span.h): permutes that a 16-byte tile cannot take.
//
// A tile whose rows or outputs lie off the 16-byte grid used to move 1 to 8
// bytes per load and store: too few bytes in flight, and (1- and 2-byte cells)
// too many instructions.  Here a unit's input spans are fetched as they lie in
// aligned 16-byte asynchronous copies (no registers, 16 KB in flight per CTA,
// 6 CTAs per SM), the alignment being carried into shared memory, and output
// spans are put together from shared memory in 4-byte words (whole cells from
// 4 bytes up) so that a warp writes 128 contiguous bytes.  Spans' offsets come
// from tables built once per CTA; a CTA's units are gridDim.x apart.
// Bounds: DRAM for cells of 4 bytes and more (251 x 333 x 517 fp32 in order
// 2,0,1: 150 us as narrow tiles, 68 us, 5.1 TB/s; 8-byte cells 5.8 TB/s),
// instruction issue and shared-memory reads (one per cell) below (2-byte 52 us,
// 3.3 TB/s; 1-byte 31 us, 2.8 TB/s).  Units of 16 KB measured against 24 and
// 32 KB: 68, 87, 69 us on the fp32 case, 75, 73, 76 us on 4-channel byte images.
#include <algorithm>
#include <atomic>

#include "launch.h"
#include "span_body.cuh"

namespace rearr {

namespace {

constexpr int kSpanCtas = 6;  // resident CTAs per SM (about 40 registers a thread; 8 spill)

template <int E, bool LUT>
__global__ void __launch_bounds__(kThreads, kSpanCtas) k_span(const __grid_constant__ SpanDesc d)
{
    extern __shared__ __align__(32) unsigned char smem[];
    __shared__ SpanUnit unit[2];
    // The tables read no global memory, so they are built before the wait for
    // the kernel ahead on the stream.
    span_units<E, LUT>(d, blockIdx.x, d.units, gridDim.x, smem, unit, [] {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    });
}

// Span copies of a batch: units of many descriptors handed out `grab` at a
// time; each piece of a descriptor builds its tables anew, so a grab is as
// large as leaves every CTA several, up to kBatchSpanGrab.
constexpr uint64_t kBatchSpanGrab = 16;

template <int E, bool LUT>
__device__ __noinline__ void span_range(const SpanDesc &d, uint32_t u0, uint32_t u1, unsigned char *smem,
                                        SpanUnit (&unit)[2])
{
    span_units<E, LUT>(d, u0, u1, 1, smem, unit, [] {});
}

__global__ void __launch_bounds__(kThreads, kSpanCtas) k_batch_span(const SpanDesc *__restrict__ spans,
                                                                   const uint64_t *__restrict__ prefix, int n,
                                                                   unsigned long long *counter, uint32_t grab)
{
    extern __shared__ __align__(32) unsigned char smem[];
    __shared__ SpanUnit unit[2];
    __shared__ SpanDesc d;
    __shared__ unsigned long long s_start;
    const uint64_t total = prefix[n];
    for (;;) {
        if (threadIdx.x == 0) s_start = atomicAdd(counter, (unsigned long long)grab);
        __syncthreads();
        const uint64_t start = s_start, end = min(total, start + grab);
        if (start >= total) break;
        int lo = 0, hi = n - 1;  // last descriptor with prefix[lo] <= start
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (prefix[mid] <= start) lo = mid;
            else hi = mid - 1;
        }
        for (uint64_t t = start; t < end; ++lo) {
            const uint64_t base = prefix[lo], seg_end = min(end, prefix[lo + 1]);
            for (uint32_t w = threadIdx.x; w < sizeof(SpanDesc) / 4; w += kThreads)
                reinterpret_cast<uint32_t *>(&d)[w] = reinterpret_cast<const uint32_t *>(spans + lo)[w];
            __syncthreads();
            const uint32_t u0 = uint32_t(t - base), u1 = uint32_t(seg_end - base);
            switch (d.E << 1 | d.lut) {
                case 1 << 1 | 0: span_range<1, false>(d, u0, u1, smem, unit); break;
                case 1 << 1 | 1: span_range<1, true>(d, u0, u1, smem, unit); break;
                case 2 << 1 | 0: span_range<2, false>(d, u0, u1, smem, unit); break;
                case 2 << 1 | 1: span_range<2, true>(d, u0, u1, smem, unit); break;
                case 4 << 1 | 0: span_range<4, false>(d, u0, u1, smem, unit); break;
                case 4 << 1 | 1: span_range<4, true>(d, u0, u1, smem, unit); break;
                case 8 << 1 | 0: span_range<8, false>(d, u0, u1, smem, unit); break;
                case 8 << 1 | 1: span_range<8, true>(d, u0, u1, smem, unit); break;
                default: break;
            }
            t = seg_end;
        }
    }
}

template <int E, bool LUT>
cudaError_t launch_span_as(const SpanDesc &d, cudaStream_t s)
{
    // Per device, once: the shared-memory opt-in; SM count.
    static std::atomic<int> sms_of[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int sms = sms_of[dev].load(std::memory_order_acquire);
    if (!sms) {
        e = cudaFuncSetAttribute(k_span<E, LUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSpanSmemMax);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        sms_of[dev].store(sms, std::memory_order_release);
    }
    const uint32_t smem = span_smem_bytes(d);
    const uint32_t per_sm = std::min<uint32_t>(kSpanCtas, std::max<uint32_t>(1, 227u * 1024 / (smem + 1024 + 32)));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::min<uint32_t>(d.units, uint32_t(sms) * per_sm));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_span<E, LUT>, d);
    if (e == cudaSuccess) g_launches.fetch_add(1, std::memory_order_relaxed);
    return e;
}

}  // namespace

cudaError_t launch_batch_spans(const SpanDesc *spans, const uint64_t *prefix, int n, uint64_t units, uint32_t smem,
                               unsigned long long *counter, cudaStream_t s)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_batch_span, cudaFuncAttributeMaxDynamicSharedMemorySize, kSpanSmemMax);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch_span, kThreads, smem);
    if (e != cudaSuccess) return e;
    const uint64_t resident = uint64_t(sms) * uint64_t(std::max(per_sm, 1));
    const uint32_t grab = uint32_t(std::max<uint64_t>(1, std::min(kBatchSpanGrab, units / (4 * resident))));
    const uint64_t grid = std::min<uint64_t>((units + grab - 1) / grab, resident);
    k_batch_span<<<unsigned(std::max<uint64_t>(grid, 1)), kThreads, smem, s>>>(spans, prefix, n, counter, grab);
    return cudaGetLastError();
}

cudaError_t launch_span(const SpanDesc &d, cudaStream_t s)
{
    switch (d.E) {
        case 1: return d.lut ? launch_span_as<1, true>(d, s) : launch_span_as<1, false>(d, s);
        case 2: return d.lut ? launch_span_as<2, true>(d, s) : launch_span_as<2, false>(d, s);
        case 4: return d.lut ? launch_span_as<4, true>(d, s) : launch_span_as<4, false>(d, s);
        case 8: return d.lut ? launch_span_as<8, true>(d, s) : launch_span_as<8, false>(d, s);
        case 16: return d.lut ? launch_span_as<16, true>(d, s) : launch_span_as<16, false>(d, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rearr
