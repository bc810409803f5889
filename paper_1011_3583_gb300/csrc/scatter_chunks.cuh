// scatter_chunks.cuh -- large scatters dst[idx[i]] = src[i] with every random
// access of the payload in shared memory.
//
// The destination is cut into C chunks that fit one CTA's shared memory (CS
// elements each).
//   lists : each tile of T elements is counting-sorted by chunk in shared
//           memory and appended to the chunks' lists (offset in the chunk, 16
//           bits, and the element): one atomic per tile and chunk reserves
//           the place, consecutive elements of a chunk are written side by
//           side, and the tiles in flight append next to each other, so their
//           partly written sectors are completed in the L2.
//   place : a CTA reads a chunk's list in order, puts the elements in their
//           places in shared memory, marks them in a bitmap, and writes the
//           marked ones out.
// 28 bytes of traffic per 4-byte element (idx 4 twice, src 4, list 6 + 6,
// dst 4) and two kernels; the passes this replaces end in random stores (0.69
// per clock per SM at most).  A list holds CS elements and a slack that covers
// uniformly drawn repeats; a sequence that overflows one sets a flag on which
// the place pass returns and the bucketed passes of k_reorder_l2.cu run.
#pragma once

#include "bodies.cuh"

namespace rearr {

constexpr int kPlaceThreads = 1024;

struct ScatterLists {
    const char *src;
    char *dst;
    const uint32_t *idx;
    uint32_t n, C, CS, cap;        // elements, chunks, elements per chunk, room of a list
    uint32_t cs_mul, cs_shift;     // v / CS = (v * cs_mul) >> (32 + cs_shift), exact for v < 2^29
    uint32_t tiles;
    unsigned long long *near;      // locality sample (k_l2_sample)
    unsigned long long near_threshold;
    uint32_t *over;                // set when a list overflows
    uint32_t *fill;                // [C] elements in the lists, 32 bytes apart
    uint16_t *off;                 // [C][cap]
    char *v;                       // [C][cap]
};

constexpr uint32_t kFillStride = 8;  // words: appends to different lists meet in different sectors

__device__ __forceinline__ bool lists_on(const ScatterLists &p)
{
    return *reinterpret_cast<volatile unsigned long long *>(p.near) < p.near_threshold;
}

// Chunk of an index; clamped so that an index >= n (undefined behaviour for
// the caller) stays inside the arrays.
__device__ __forceinline__ uint32_t list_of(const ScatterLists &p, uint32_t v)
{
    return min(__umulhi(v, p.cs_mul) >> p.cs_shift, p.C - 1);
}

// Four consecutive indices.  Plain loads: a tile's indices are read twice, and
// lines loaded around the L1 (no_allocate) had left the L2 by the second time
// (DRAM reads of 2^27 indices 1.07 against 0.54 GB).
template <bool I64>
__device__ __forceinline__ uint4 list_index4(const uint32_t *idx, uint64_t i)
{
    if constexpr (!I64) {
        return ldg_any<16>(idx + i);
    } else {
        const unsigned long long *q = reinterpret_cast<const unsigned long long *>(idx) + i;
        return make_uint4(uint32_t(__ldg(q)), uint32_t(__ldg(q + 1)), uint32_t(__ldg(q + 2)), uint32_t(__ldg(q + 3)));
    }
}

// Indices of group g (of four) of a tile of m elements; past its end 0xFFFFFFFF.
template <bool I64, bool FULL>
__device__ __forceinline__ uint4 list_group(const ScatterLists &p, uint32_t i0, uint32_t m, uint32_t g)
{
    if (FULL || 4 * g + 4 <= m) return list_index4<I64>(p.idx, uint64_t(i0) + 4 * g);
    uint32_t v[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const uint64_t i = uint64_t(i0) + 4 * g + x;
        v[x] = 4 * g + x >= m ? 0xFFFFFFFFu
               : I64 ? uint32_t(__ldg(reinterpret_cast<const unsigned long long *>(p.idx) + i)) : __ldg(p.idx + i);
    }
    return make_uint4(v[0], v[1], v[2], v[3]);
}

// Exclusive prefix sum of one value per thread over the CTA.
template <int THREADS>
__device__ __forceinline__ uint32_t cta_scan(uint32_t v, uint32_t *warp_sums)
{
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[w] = x;
    __syncthreads();
    if (w == 0) {
        const uint32_t s = lane < THREADS / 32 ? warp_sums[lane] : 0u;
        uint32_t y = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += z;
        }
        if (lane < THREADS / 32) warp_sums[lane] = y - s;
    }
    __syncthreads();
    return warp_sums[w] + x - v;
}

// Shared memory: the sorted tile (elements, then indices), then a word per
// chunk: counts, segment starts, and at last the distance from a segment's
// place in the tile to its place in the lists.  The ranks stay in registers
// between the two passes over the tile's indices.
template <int W, bool I64, int NG, int THREADS, bool FULL>
__device__ __forceinline__ void lists_tile(const ScatterLists &p, uint32_t t, unsigned char *smem, uint32_t *warp_sums)
{
    constexpr uint32_t T = NG * 4 * THREADS;
    constexpr int B = NG % 3 == 0 ? 3 : NG % 4 == 0 ? 4 : NG;  // loads in flight
    uint32_t *sidx = reinterpret_cast<uint32_t *>(smem + size_t(T) * W);
    uint32_t *cnt = sidx + T;
    const uint32_t i0 = t * T, m = FULL ? T : p.n - i0;
    for (uint32_t x = threadIdx.x; x < p.C; x += THREADS) cnt[x] = 0;
    __syncthreads();
    uint32_t rank[NG * 2];
#pragma unroll
    for (int b = 0; b < NG; b += B) {
        uint4 q[B];
#pragma unroll
        for (int j = 0; j < B; ++j) q[j] = list_group<I64, FULL>(p, i0, m, (b + j) * THREADS + threadIdx.x);
#pragma unroll
        for (int j = 0; j < B; ++j) {
            uint32_t r[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const uint32_t k = ((b + j) * THREADS + threadIdx.x) * 4 + x;
                r[x] = FULL || k < m ? atomicAdd(&cnt[list_of(p, word_of(q[j], x))], 1u) : 0u;
            }
            rank[2 * (b + j)] = prmt(r[0], r[1], 0x5410u);
            rank[2 * (b + j) + 1] = prmt(r[2], r[3], 0x5410u);
        }
    }
    __syncthreads();
    // counts -> segment starts; a thread takes neighbouring chunks and, while
    // the tile is sorted, reserves their places in the lists
    constexpr int PER = 8;  // chunks of a thread, at most (C <= PER * THREADS)
    const uint32_t per = (p.C + THREADS - 1) / THREADS;
    const uint32_t x0 = threadIdx.x * per;
    uint32_t have[PER], place[PER], sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        have[j] = uint32_t(j) < per && x0 + j < p.C ? cnt[x0 + j] : 0u;
        sum += have[j];
    }
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        place[j] = 0;
        if (have[j]) place[j] = atomicAdd(&p.fill[size_t(x0 + j) * kFillStride], have[j]);
    }
    uint32_t at = cta_scan<THREADS>(sum, warp_sums);
    const uint32_t at0 = at;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        if (uint32_t(j) < per && x0 + j < p.C) {
            cnt[x0 + j] = at;
            at += have[j];
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < NG; ++b) {
        const uint32_t g = b * THREADS + threadIdx.x;
        const uint4 q = list_group<I64, FULL>(p, i0, m, g);
        typename Word<W>::T val[4];
        const char *s = p.src + (uint64_t(i0) + 4 * g) * W;
        if (FULL || 4 * g + 4 <= m) load4<W>(s, val);
        else {
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (4 * g + x < m) val[x] = ldg_stream<W>(s + x * W);
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            if (FULL || 4 * g + x < m) {
                const uint32_t v = word_of(q, x);
                const uint32_t to = cnt[list_of(p, v)] + ((x & 1) ? rank[2 * b + (x >> 1)] >> 16 : rank[2 * b + (x >> 1)] & 0xFFFFu);
                sidx[to] = v;
                sts<W>(smem + size_t(to) * W, val[x]);
            }
        }
    }
    __syncthreads();
    at = at0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        if (have[j]) {
            const bool fits = place[j] + have[j] <= p.cap;
            if (!fits) *p.over = 1;
            // a segment that does not fit is not written (its elements' places compare past the lists' end)
            cnt[x0 + j] = fits ? (x0 + j) * p.cap + place[j] - at : 0x80000000u;
            at += have[j];
        }
    }
    __syncthreads();
    const uint32_t end = p.C * p.cap;  // < 2^31
#pragma unroll 4
    for (uint32_t q = threadIdx.x; q < m; q += THREADS) {
        const uint32_t v = sidx[q], c = list_of(p, v);
        const uint32_t to = cnt[c] + q;
        if (to < end) {
            p.off[to] = uint16_t(min(v - c * p.CS, p.CS - 1));
            stg<W>(p.v + uint64_t(to) * W, lds<W>(smem + size_t(q) * W));
        }
    }
    __syncthreads();
}

template <int W, bool I64, int NG, int THREADS, int CTAS>
__global__ void __launch_bounds__(THREADS, CTAS) k_scatter_lists(const ScatterLists p)
{
    if (!lists_on(p)) return;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t warp_sums[32];
    constexpr uint32_t T = NG * 4 * THREADS;
    for (uint32_t t = blockIdx.x; t < p.tiles; t += gridDim.x) {
        if ((t + 1) * uint64_t(T) <= p.n) lists_tile<W, I64, NG, THREADS, true>(p, t, smem, warp_sums);
        else lists_tile<W, I64, NG, THREADS, false>(p, t, smem, warp_sums);
    }
}

// A group of Q W-byte values as 16 bytes.
template <int W> union Values16 {
    uint4 u;
    typename Word<W>::T e[16 / W];
    __device__ __forceinline__ Values16() : u(make_uint4(0, 0, 0, 0)) {}
};

template <int W>
__global__ void __launch_bounds__(kPlaceThreads, 1) k_scatter_place(const ScatterLists p)
{
    if (!lists_on(p) || *reinterpret_cast<volatile uint32_t *>(p.over)) return;
    extern __shared__ __align__(16) unsigned char smem[];
    using V = typename Word<W>::T;
    V *chunk = reinterpret_cast<V *>(smem);
    uint32_t *bits = reinterpret_cast<uint32_t *>(smem + size_t(p.CS) * W);
    constexpr uint32_t Q = 16 / W, NV = 8 / Q;  // values per 16 bytes; 16-byte loads of eight values
    const bool vec = (reinterpret_cast<uintptr_t>(p.dst) & 15) == 0;
    for (uint32_t c = blockIdx.x; c < p.C; c += gridDim.x) {
        for (uint32_t x = threadIdx.x; x < p.CS / 32; x += kPlaceThreads) bits[x] = 0;
        const uint32_t have = p.fill[size_t(c) * kFillStride];
        const uint16_t *off = p.off + size_t(c) * p.cap;  // cap is a multiple of 8
        const char *v = p.v + size_t(c) * p.cap * W;
        __syncthreads();
        auto put = [&](uint32_t o, const V &val) {
            chunk[o] = val;
            atomicOr(&bits[o >> 5], 1u << (o & 31));
        };
        for (uint32_t x = threadIdx.x; x < have / 8; x += kPlaceThreads) {
            const uint4 o = ldg_stream<16>(off + 8 * x);
            Values16<W> val[NV];
#pragma unroll
            for (uint32_t k = 0; k < NV; ++k) val[k].u = ldg_stream<16>(v + (uint64_t(8) * x + k * Q) * W);
#pragma unroll
            for (uint32_t k = 0; k < 8; ++k)
                put((word_of(o, k >> 1) >> (16 * (k & 1))) & 0xFFFFu, val[k / Q].e[k % Q]);
        }
        for (uint32_t x = have / 8 * 8 + threadIdx.x; x < have; x += kPlaceThreads) put(off[x], ldg_stream<W>(v + x * W));
        __syncthreads();
        const uint64_t e0 = uint64_t(c) * p.CS;
        const uint32_t m = uint32_t(min(uint64_t(p.CS), uint64_t(p.n) - e0));
        char *o = p.dst + e0 * W;
        for (uint32_t x = threadIdx.x * Q; x < m; x += kPlaceThreads * Q) {
            const uint32_t b = (bits[x >> 5] >> (x & 31)) & ((1u << min(Q, m - x)) - 1);
            if (vec && b == (1u << Q) - 1) {
                stg<16>(o + uint64_t(x) * W, lds<16>(smem + size_t(x) * W));
            } else {
#pragma unroll
                for (uint32_t k = 0; k < Q; ++k)
                    if ((b >> k) & 1) stg<W>(o + uint64_t(x + k) * W, lds<W>(smem + size_t(x + k) * W));
            }
        }
        __syncthreads();
    }
}

}  // namespace rearr
