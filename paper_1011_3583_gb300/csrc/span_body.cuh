// span_body.cuh -- device side of span copies (span.h), shared by the single
// call's kernel and the batched one.
#pragma once

#include "bodies.cuh"
#include "span.h"

namespace rearr {

// Shares n_spans spans out over the CTA: `lanes` neighbouring threads walk one
// span, kThreads / lanes spans at a time (leftover threads idle), so that an
// instruction covers neighbouring chunks (words) of one or a few spans.
struct SpanShare {
    uint32_t group, lane, groups;
    __device__ __forceinline__ explicit SpanShare(const FastDiv &lanes)
    {
        groups = fdiv(kThreads, lanes);
        fdivmod(threadIdx.x, lanes, group, lane);
        if (group >= groups) group = 0xFFFFFFFFu / 2;  // past any span
    }
};

template <int CW>
__device__ __forceinline__ void span_load(const SpanShare &sh, uint32_t lanes, const char *src, uint32_t rows,
                                          uint32_t len, unsigned char *tile, const int64_t *row_in,
                                          const uint32_t *row_sm)
{
    const uint32_t base = uint32_t(reinterpret_cast<uintptr_t>(src) & 15);
    const uint32_t x0 = sh.lane * CW;
#pragma unroll 4
    for (uint32_t row = sh.group; row < rows; row += sh.groups) {
        const uintptr_t g = reinterpret_cast<uintptr_t>(src) + row_in[row];
        const uint32_t left = len + (uint32_t(g) & (CW - 1));  // bytes from the first chunk's start
        const char *p = reinterpret_cast<const char *>(g & ~uintptr_t(CW - 1));
        unsigned char *t = tile + ((base + row_sm[row]) & ~uint32_t(CW - 1));
        if (x0 < left) cp_async<CW>(t + x0, p + x0);
        for (uint32_t x = x0 + lanes * CW; x < left; x += lanes * CW) cp_async<CW>(t + x, p + x);
    }
}

// Spans' offsets from their digits, fastest first.
__device__ __forceinline__ void span_digits(uint32_t q, const FastDiv *ext, const int64_t *stride, const uint32_t *sms,
                                            int64_t &off, uint32_t &sm)
{
    off = 0;
    sm = 0;
#pragma unroll
    for (int i = 0; i < kSpanAxes; ++i) {
        if (ext[i].d == 1) continue;
        uint32_t dig;
        fdivmod(q, ext[i], q, dig);
        off += int64_t(dig) * stride[i];
        sm += dig * sms[i];
    }
}

// A unit's origin and what of a full unit it holds.  One thread works it out
// for the next unit while this one's copies are on their way.
struct SpanUnit {
    const char *src;
    char *dst;
    uint32_t rows, runs, row_bytes, cells;
    bool edge;  // chunks of it reach outside the source
};

// The same for a unit at an end of the source: a chunk that reaches outside it
// is copied cell by cell, what lies inside.  (Chunks no wider than a cell never do.)
template <int CW, int E>
__device__ __noinline__ void span_load_edge(uint32_t group, uint32_t lane, uint32_t groups, const SpanDesc &d,
                                            const SpanUnit &u, unsigned char *tile, const int64_t *row_in,
                                            const uint32_t *row_sm)
{
    const uint32_t base = uint32_t(reinterpret_cast<uintptr_t>(u.src) & 15);
    for (uint32_t row = group; row < u.rows; row += groups) {
        const uintptr_t g = reinterpret_cast<uintptr_t>(u.src) + row_in[row];
        const uint32_t left = u.row_bytes + (uint32_t(g) & (CW - 1));
        const char *p = reinterpret_cast<const char *>(g & ~uintptr_t(CW - 1));
        unsigned char *t = tile + ((base + row_sm[row]) & ~uint32_t(CW - 1));
        for (uint32_t x = lane * CW; x < left; x += d.load_lanes.d * CW) {
            if (p + x >= d.src && p + x + CW <= d.src_end) {
                cp_async<CW>(t + x, p + x);
            } else {
                for (uint32_t k = x; k < x + CW; k += E)
                    if (p + k >= d.src && p + k + E <= d.src_end) sts<E>(t + k, ldg_any<E>(p + k));
            }
        }
    }
}

__device__ __forceinline__ void span_unit(const SpanDesc &d, uint32_t u, SpanUnit &x)
{
    const char *src = d.src;
    char *dst = d.dst;
    uint32_t rows = d.n_rows, runs = d.n_runs, row_bytes = d.row_bytes, cells = d.run_cells;
    int64_t reach = d.reach;
#pragma unroll 1
    for (int i = d.no - 1; i >= 0; --i) {
        uint32_t dig;
        fdivmod(u, d.udiv[i], u, dig);
        src += int64_t(dig) * d.uin[i];
        dst += int64_t(dig) * d.uout[i];
        if (i == d.ua) {
            const uint32_t k = min(d.ka, d.na - dig * d.ka);
            row_bytes = k * d.row_bytes_a;
            if (d.n_runs_a) runs = k * d.n_runs_a;
            if (d.run_cells_a) cells = k * d.run_cells_a;
        }
        if (i == d.ub) {
            const uint32_t k = min(d.kb, d.nb - dig * d.kb);
            if (d.n_rows_b) rows = k * d.n_rows_b;
            if (d.run_cells_b) cells = k * d.run_cells_b;
            reach -= int64_t(d.kb - k) * d.reach_b;
        }
    }
    x.edge = span_at_edge(d, src, reach + row_bytes);
    x.src = src;
    x.dst = dst;
    x.rows = rows;
    x.runs = runs;
    x.row_bytes = row_bytes;
    x.cells = cells;
}

// Offsets of cells p .. p + V - 1 of an output span in shared memory.
template <int V, bool LUT>
__device__ __forceinline__ void span_offsets(const uint16_t *lut, uint32_t p, uint32_t step, uint32_t (&f)[V])
{
    if constexpr (!LUT) {
        f[0] = p * step;
#pragma unroll
        for (int k = 1; k < V; ++k) f[k] = f[k - 1] + step;
    } else if constexpr (V == 4) {
        if ((p & 3) == 0) {
            const uint2 q = lds<8>(lut + p);
            f[0] = q.x & 0xFFFF; f[1] = q.x >> 16; f[2] = q.y & 0xFFFF; f[3] = q.y >> 16;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) f[k] = lut[p + k];
        }
    } else {
#pragma unroll
        for (int k = 0; k < V; ++k) f[k] = lut[p + k];
    }
}

// The word of V cells at s + f[0], s + f[1], ...
template <int E, int V>
__device__ __forceinline__ typename Word<E * V>::T span_word(const unsigned char *s, const uint32_t (&f)[V])
{
    if constexpr (V == 1) return lds<E>(s + f[0]);
    else if constexpr (E == 2) return prmt(lds<2>(s + f[0]), lds<2>(s + f[1]), 0x5410u);
    else return prmt(prmt(lds<1>(s + f[0]), lds<1>(s + f[1]), 0x0040u), prmt(lds<1>(s + f[2]), lds<1>(s + f[3]), 0x0040u),
                     0x5410u);
}

// Units u0, u0 + step, ... below u1 of d, with smem of span_smem_bytes(d) on a
// 32-byte boundary (two chunks of a sector that land in one 32-byte line of
// shared memory are one request: 16 bytes off, 251 x 333 x 517 of 8 bytes in
// order 2,0,1 read 33.0 M sectors from the L2 instead of 22.2 M, 130 against 119
// us), and unit[] in shared memory.  start(): called once the tables stand and
// before anything of the payload is read.  Ends with a barrier.
template <int E, bool LUT, class Start>
__device__ __forceinline__ void span_units(const SpanDesc &d, uint32_t u0, uint32_t u1, uint32_t u_step,
                                           unsigned char *smem, SpanUnit (&unit)[2], Start start)
{
    unsigned char *tile = smem;
    int64_t *row_in = reinterpret_cast<int64_t *>(smem + d.tile_bytes);
    int64_t *run_out = row_in + d.n_rows;
    uint32_t *row_sm = reinterpret_cast<uint32_t *>(run_out + d.n_runs);
    uint32_t *run_sm = row_sm + d.n_rows;
    uint16_t *lut = reinterpret_cast<uint16_t *>(smem + span_lut_offset(d));
    constexpr uint32_t WU = E < 4 ? 4 : E, V = WU / E;

    // The tables hold for every unit; they read no global memory, so they are
    // built before the wait for the kernel ahead on the stream.
    for (uint32_t r = threadIdx.x; r < d.n_rows; r += kThreads)
        span_digits(r, d.row_ext, d.row_in, d.row_sm, row_in[r], row_sm[r]);
    for (uint32_t r = threadIdx.x; r < d.n_runs; r += kThreads)
        span_digits(r, d.run_ext, d.run_out, d.run_sm, run_out[r], run_sm[r]);
    if constexpr (LUT) {
        // a thread's entries are kThreads apart: one decomposition, then steps with carries
        uint32_t dig[kSpanAxes], step[kSpanAxes], ext[kSpanAxes], q = threadIdx.x;
#pragma unroll
        for (int i = 0; i < kSpanAxes; ++i) {
            ext[i] = d.ch_ext[i].d;
            step[i] = d.ch_step[i];
            dig[i] = 0;
            if (ext[i] > 1) fdivmod(q, d.ch_ext[i], q, dig[i]);
        }
        for (uint32_t p = threadIdx.x; p < d.run_cells; p += kThreads) {
            uint32_t sm = 0;
#pragma unroll
            for (int i = 0; i < kSpanAxes; ++i) sm += dig[i] * d.ch_sm[i];
            lut[p] = uint16_t(sm);
            box_advance<kSpanAxes>(dig, step, ext);
        }
    }
    if (threadIdx.x == 0) span_unit(d, u0, unit[0]);
    __syncthreads();
    start();

    const uint32_t ch0 = d.ch_sm[0];
    const SpanShare ld(d.load_lanes), st(d.store_lanes);
    // Output spans that all start on a word boundary and take one pass: the
    // thread's cells have the same offsets in every span of every unit.
    uint32_t fixed[V];
    if (d.fixed && st.lane * V + V <= d.run_cells) span_offsets<V, LUT>(lut, st.lane * V, ch0, fixed);
    uint32_t cur = 0;
    for (uint32_t u = u0; u < u1; u += u_step, cur ^= 1) {
        const SpanUnit x = unit[cur];
        if (E < 16 && x.edge) {
            if (E < 4 && d.chunk == 4) span_load_edge<4, E>(ld.group, ld.lane, ld.groups, d, unit[cur], tile, row_in, row_sm);
            else span_load_edge<16, E>(ld.group, ld.lane, ld.groups, d, unit[cur], tile, row_in, row_sm);
        } else if (d.chunk == 16) span_load<16>(ld, d.load_lanes.d, x.src, x.rows, x.row_bytes, tile, row_in, row_sm);
        else if (d.chunk == 8) span_load<8>(ld, d.load_lanes.d, x.src, x.rows, x.row_bytes, tile, row_in, row_sm);
        else span_load<4>(ld, d.load_lanes.d, x.src, x.rows, x.row_bytes, tile, row_in, row_sm);
        cp_async_commit();
        if (threadIdx.x == 0 && u + u_step < u1) span_unit(d, u + u_step, unit[cur ^ 1]);
        cp_async_wait<0>();
        __syncthreads();

        const unsigned char *cells0 = tile + (reinterpret_cast<uintptr_t>(x.src) & 15);
        const uint32_t cells = x.cells, runs = x.runs;
        if (d.fixed) {
            if (st.lane * V + V <= cells) {
                char *o = x.dst + st.lane * WU;
#pragma unroll 4
                for (uint32_t run = st.group; run < runs; run += st.groups)
                    stg<WU>(o + run_out[run], span_word<E, V>(cells0 + run_sm[run], fixed));
            }
        } else {
            for (uint32_t run = st.group; run < runs; run += st.groups) {
                char *o = x.dst + run_out[run];
                const unsigned char *s = cells0 + run_sm[run];
                const uint32_t head = V > 1 ? (uint32_t(reinterpret_cast<uintptr_t>(o)) & 3) / E : 0;
#pragma unroll 4
                for (uint32_t w = st.lane; w * V < cells + head; w += d.store_lanes.d) {
                    const int32_t p = int32_t(w * V) - int32_t(head);
                    if (p >= 0 && uint32_t(p) + V <= cells) {
                        uint32_t f[V];
                        span_offsets<V, LUT>(lut, p, ch0, f);
                        stg<WU>(o + p * E, span_word<E, V>(s, f));
                    }
                }
            }
        }
        if constexpr (V > 1) {
            // words a span shares with its neighbours at either end: its cells, one a thread
            if (!d.fixed || cells % V != 0) {
                for (uint32_t i = threadIdx.x; i < runs * 2 * (V - 1); i += kThreads) {
                    const uint32_t run = i / (2 * (V - 1)), r = i - run * 2 * (V - 1), k = r >> 1;
                    char *o = x.dst + run_out[run];
                    const uint32_t head = (uint32_t(reinterpret_cast<uintptr_t>(o)) & 3) / E;
                    const uint32_t n = (r & 1) ? (cells + head) % V : (V - head) % V;  // cells of the end's word
                    const uint32_t p = (r & 1) ? cells - 1 - k : k;
                    if (k < n && p < cells)
                        stg<E>(o + p * E, lds<E>(cells0 + run_sm[run] + (LUT ? uint32_t(lut[p]) : p * ch0)));
                }
            }
        }
        __syncthreads();
    }
}

}  // namespace rearr
