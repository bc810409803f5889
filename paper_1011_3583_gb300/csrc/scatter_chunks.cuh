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
// 24 bytes of DRAM traffic per 4-byte element (idx 4, its second read in the
// L2; src 4, list 6 + 6, dst 4) and two kernels; the passes this replaces end
// in random stores (0.69 per clock per SM at most).  10^8 x 4 B random: 1160 ->
// 789 us, of which about 3/4 lists (shared-memory wavefronts, 60 % of the pipe's
// cycles: ranking and placing are random accesses; one CTA of 1024 threads per
// SM: before lists had their present length, tiles half as large at two CTAs
// halved the segments and took 1114 us in all instead of 905), 1/4 place.  An element whose list is full is stored at
// once to its place in the destination (which of several elements of one
// destination stays is unspecified).  Where the sample says that many would be,
// the lists set a flag on which the place pass returns and the bucketed passes
// of k_reorder_l2.cu run.
#pragma once

#include "bodies.cuh"

namespace rearr {

constexpr int kListThreads = 1024;

struct ScatterLists {
    const char *src;
    char *dst;
    const uint32_t *idx;
    uint32_t n, C, CS, cap;        // elements, chunks, elements per chunk, room of a list
    uint32_t cs_mul, cs_shift;     // v / CS = (v * cs_mul) >> (32 + cs_shift), exact for v < 2^29
    uint32_t tiles;
    unsigned long long *near;      // locality sample (k_l2_sample)
    unsigned long long near_threshold;
    uint32_t *over;                // set when the sample shows the indices crowded
    uint32_t *fill;                // [C] elements in the lists, 32 bytes apart; beside each the
                                   // sampled indices that fall in the chunk (k_l2_sample)
    uint32_t hits_full, hits_past; // sampled indices that stand for a full list; those beyond, in all, that may be
    uint16_t *off;                 // [C][cap]
    char *v;                       // [C][cap]
};


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
    if constexpr (FULL) {
        return list_index4<I64>(p.idx, uint64_t(i0) + 4 * g);
    } else {
        if (4 * g + 4 <= m) return list_index4<I64>(p.idx, uint64_t(i0) + 4 * g);
        uint32_t v[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const uint64_t i = uint64_t(i0) + 4 * g + x;
            v[x] = 4 * g + x >= m ? 0xFFFFFFFFu
                   : I64 ? uint32_t(__ldg(reinterpret_cast<const unsigned long long *>(p.idx) + i)) : __ldg(p.idx + i);
        }
        return make_uint4(v[0], v[1], v[2], v[3]);
    }
}

// Shared memory: the sorted tile (4-byte elements beside their indices, so that
// a placement is one 8-byte store; wider elements, then the indices), then a
// word per chunk: counts, segment starts, and at last the distance from a segment's
// place in the tile to its place in the lists.  The ranks stay in registers
// between the two passes over the tile's indices.
template <int W, bool I64, int NG, bool FULL>
__device__ __forceinline__ void lists_tile(const ScatterLists &p, uint32_t t, unsigned char *smem, uint32_t *warp_sums)
{
    constexpr uint32_t T = NG * 4 * kListThreads;
    constexpr int B = NG % 3 == 0 ? 3 : NG % 4 == 0 ? 4 : NG;  // loads in flight
    uint32_t *sidx = reinterpret_cast<uint32_t *>(smem + size_t(T) * W);
    uint32_t *cnt = sidx + T;
    const uint32_t i0 = t * T, m = FULL ? T : p.n - i0;
    for (uint32_t x = threadIdx.x; x < p.C; x += kListThreads) cnt[x] = 0;
    __syncthreads();
    uint32_t rank[NG * 2];
#pragma unroll
    for (int b = 0; b < NG; b += B) {
        uint4 q[B];
#pragma unroll
        for (int j = 0; j < B; ++j) q[j] = list_group<I64, FULL>(p, i0, m, (b + j) * kListThreads + threadIdx.x);
#pragma unroll
        for (int j = 0; j < B; ++j) {
            uint32_t r[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const uint32_t k = ((b + j) * kListThreads + threadIdx.x) * 4 + x;
                r[x] = FULL || k < m ? atomicAdd(&cnt[list_of(p, word_of(q[j], x))], 1u) : 0u;
            }
            rank[2 * (b + j)] = prmt(r[0], r[1], 0x5410u);
            rank[2 * (b + j) + 1] = prmt(r[2], r[3], 0x5410u);
        }
    }
    __syncthreads();
    // counts -> segment starts; a thread takes neighbouring chunks and, while
    // the tile is sorted, reserves their places in the lists
    constexpr int PER = kListMaxChunks / kListThreads;  // chunks of a thread, at most
    const uint32_t per = (p.C + kListThreads - 1) / kListThreads;
    const uint32_t x0 = threadIdx.x * per;
    uint32_t place[PER];
    {
        uint32_t have[PER], sum = 0;
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
        uint32_t at = cta_scan<kListThreads>(sum, warp_sums);
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            if (uint32_t(j) < per && x0 + j < p.C) {
                cnt[x0 + j] = at;
                at += have[j];
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < NG; ++b) {
        const uint32_t g = b * kListThreads + threadIdx.x;
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
                if constexpr (W == 4) {
                    sts<8>(smem + size_t(to) * 8, make_uint2(v, val[x]));
                } else {
                    sidx[to] = v;
                    sts<W>(smem + size_t(to) * W, val[x]);
                }
            }
        }
    }
    __syncthreads();
    {
#pragma unroll
        for (int j = 0; j < PER; ++j)
            if (uint32_t(j) < per && x0 + j < p.C) cnt[x0 + j] = (x0 + j) * p.cap + min(place[j], p.cap) - cnt[x0 + j];
    }
    __syncthreads();
#pragma unroll 4
    for (uint32_t q = threadIdx.x; q < m; q += kListThreads) {
        uint32_t v;
        typename Word<W>::T val;
        if constexpr (W == 4) {
            const uint2 x = lds<8>(smem + size_t(q) * 8);
            v = x.x;
            val = x.y;
        } else {
            v = sidx[q];
            val = lds<W>(smem + size_t(q) * W);
        }
        const uint32_t c = list_of(p, v), to = cnt[c] + q;
        if (to < (c + 1) * p.cap) {  // C * cap < 2^31
            p.off[to] = uint16_t(min(v - c * p.CS, p.CS - 1));
            stg<W>(p.v + uint64_t(to) * W, val);
        } else if (v < p.n) {
            stg<W>(p.dst + uint64_t(v) * W, val);
        }
    }
    __syncthreads();
}

template <int W, bool I64, int NG>
__global__ void __launch_bounds__(kListThreads, 1) k_scatter_lists(const ScatterLists p)
{
    pass_enter();
    if (!lists_on(p)) return;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t warp_sums[32], past;
    // Sampled indices beyond full lists: every CTA sees the same counts.
    if (threadIdx.x == 0) past = 0;
    __syncthreads();
    uint32_t mine = 0;
    for (uint32_t c = threadIdx.x; c < p.C; c += kListThreads) {
        const uint32_t h = p.fill[size_t(c) * kFillStride + 1];
        mine += h > p.hits_full ? h - p.hits_full : 0u;
    }
    mine = __reduce_add_sync(0xffffffffu, mine);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&past, mine);
    __syncthreads();
    if (past > p.hits_past) {
        if (threadIdx.x == 0) *p.over = 1;
        return;
    }
    constexpr uint32_t T = NG * 4 * kListThreads;
    for (uint32_t t = blockIdx.x; t < p.tiles; t += gridDim.x) {
        if ((t + 1) * uint64_t(T) <= p.n) lists_tile<W, I64, NG, true>(p, t, smem, warp_sums);
        else lists_tile<W, I64, NG, false>(p, t, smem, warp_sums);
    }
}

// A group of Q W-byte values as 16 bytes.
template <int W> union Values16 {
    uint4 u;
    typename Word<W>::T e[16 / W];
    __device__ __forceinline__ Values16() : u(make_uint4(0, 0, 0, 0)) {}
};

template <int W>
__global__ void __launch_bounds__(kListThreads, 1) k_scatter_place(const ScatterLists p)
{
    pass_enter();
    if (!lists_on(p) || *reinterpret_cast<volatile uint32_t *>(p.over)) return;
    extern __shared__ __align__(16) unsigned char smem[];
    using V = typename Word<W>::T;
    V *chunk = reinterpret_cast<V *>(smem);
    uint32_t *bits = reinterpret_cast<uint32_t *>(smem + size_t(p.CS) * W);
    constexpr uint32_t Q = 16 / W, NV = 8 / Q;  // values per 16 bytes; 16-byte loads of eight values
    const bool vec = (reinterpret_cast<uintptr_t>(p.dst) & 15) == 0;
    for (uint32_t c = blockIdx.x; c < p.C; c += gridDim.x) {
        for (uint32_t x = threadIdx.x; x < p.CS / 32; x += kListThreads) bits[x] = 0;
        const uint32_t have = min(p.fill[size_t(c) * kFillStride], p.cap);
        const uint16_t *off = p.off + size_t(c) * p.cap;  // cap is a multiple of 8
        const char *v = p.v + size_t(c) * p.cap * W;
        __syncthreads();
        auto put = [&](uint32_t o, const V &val) {
            chunk[o] = val;
            atomicOr(&bits[o >> 5], 1u << (o & 31));
        };
        for (uint32_t x = threadIdx.x; x < have / 8; x += kListThreads) {
            const uint4 o = ldg_stream<16>(off + 8 * x);
            Values16<W> val[NV];
#pragma unroll
            for (uint32_t k = 0; k < NV; ++k) val[k].u = ldg_stream<16>(v + (uint64_t(8) * x + k * Q) * W);
#pragma unroll
            for (uint32_t k = 0; k < 8; ++k)
                put((word_of(o, k >> 1) >> (16 * (k & 1))) & 0xFFFFu, val[k / Q].e[k % Q]);
        }
        for (uint32_t x = have / 8 * 8 + threadIdx.x; x < have; x += kListThreads) put(off[x], ldg_stream<W>(v + x * W));
        __syncthreads();
        const uint64_t e0 = uint64_t(c) * p.CS;
        const uint32_t m = uint32_t(min(uint64_t(p.CS), uint64_t(p.n) - e0));
        char *o = p.dst + e0 * W;
        for (uint32_t x = threadIdx.x * Q; x < m; x += kListThreads * Q) {
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
