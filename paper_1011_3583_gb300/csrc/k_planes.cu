// k_planes.cu -- permutes of a few planes as a batch of interlaces or
// de-interlaces (plan_planes): the bodies of k_inter_fast, each plane and the
// interlaced array displaced by the batch index of the unit.
//
// A kernel of its own, as the displacements cost registers: with them in
// k_inter_fast as well, plain interlaces of eight planes went from 80 to 108
// and de-interlaces of six from 83 to 107, which is one CTA per SM less
// (80 MB: 28.7 -> 31.1 us, 25.4 -> 27.5).
#include "bodies.cuh"
#include "launch.h"

namespace rearr {

namespace {

template <int E, int K, bool INTER>
__global__ void __launch_bounds__(kThreads) k_planes(const __grid_constant__ InterlaceDesc d, uint32_t n)
{
    pdl_enter();
    __shared__ __align__(16) unsigned char smem[kThreads / 32 * K * 32 * 16];
    for (uint64_t u = blockIdx.x; u < n; u += gridDim.x) {
        uint32_t b, unit, b0, b1;
        fdivmod(uint32_t(u), d.upb, b, unit);
        fdivmod(b, d.b0_div, b1, b0);
        const int64_t ioff = int64_t(b0) * d.b_inter[0] + int64_t(b1) * d.b_inter[1];
        const int64_t poff = int64_t(b0) * d.b_plane[0] + int64_t(b1) * d.b_plane[1];
        if constexpr (INTER) interlace_fast_body<E, K>(d, d.planes, unit, d.upb.d, smem, ioff, poff);
        else deinterlace_fast_body<E, K>(d, d.planes, unit, d.upb.d, smem, ioff, poff);
    }
}

template <int E, int K>
cudaError_t launch_planes_as(const OpDesc &op, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(op.units < 0x7FFFFFFFull ? unsigned(op.units) : 0x7FFFFFFFu);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const uint32_t n = uint32_t(op.units);
    const cudaError_t e = op.cls == OC_INTERLACE ? cudaLaunchKernelEx(&cfg, k_planes<E, K, true>, op.inter, n)
                                                 : cudaLaunchKernelEx(&cfg, k_planes<E, K, false>, op.inter, n);
    if (e == cudaSuccess) g_launches.fetch_add(1, std::memory_order_relaxed);
    return e;
}

template <int E>
cudaError_t launch_planes_k(const OpDesc &op, cudaStream_t s)
{
    switch (op.inter.k) {
        case 2: return launch_planes_as<E, 2>(op, s);
        case 3: return launch_planes_as<E, 3>(op, s);
        case 4: return launch_planes_as<E, 4>(op, s);
        case 5: return launch_planes_as<E, 5>(op, s);
        case 6: return launch_planes_as<E, 6>(op, s);
        case 7: return launch_planes_as<E, 7>(op, s);
        case 8: return launch_planes_as<E, 8>(op, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_planes(const OpDesc &op, cudaStream_t s)
{
    switch (op.inter.elem_bytes) {
        case 1: return launch_planes_k<1>(op, s);
        case 2: return launch_planes_k<2>(op, s);
        case 4: return launch_planes_k<4>(op, s);
        case 8: return launch_planes_k<8>(op, s);
        case 16: return launch_planes_k<16>(op, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rearr
