// span.h -- descriptor of a span copy: permutes whose accesses on one side
// would be narrow (rows or outputs off the 16-byte grid, thin planes).
#pragma once

#include <stdint.h>

#include "rearr_internal.h"

namespace rearr {

// A work unit is a box of the index space with two chains of axes: along the
// input chain (input-innermost axes) the box is contiguous in the input, along
// the output chain (output-innermost axes) it is contiguous in the output.
// Each chain is whole axes, then at most one axis over a range (the chain's
// partial axis; both chains may end in the same one).  The unit reads input
// spans (one per index of the output chain's axes that the input chain does
// not hold) and writes output spans (one per index of the input chain's axes
// that the output chain does not hold).  Cells are one E-byte word.
//
// The input spans are copied as they lie, in aligned chunks of `chunk` bytes,
// into shared memory at addresses congruent to their global ones modulo
// `chunk` (every shared-memory stride is congruent to its input stride), so
// no span needs an aligned start.  A cell's place in shared memory is linear
// in its digits.  A chunk that would reach past either end of the source (the
// first and the last of an op whose source does not start or end on a chunk)
// is copied cell by cell instead: nothing outside the source is read.
constexpr int kSpanAxes = 4;        // axes of either chain
constexpr int kSpanOuter = 8;       // unit-index digits
constexpr int kSpanMaxSpans = 512;  // input / output spans per unit
constexpr int kSpanSmemMax = 96 * 1024;  // shared memory of a unit, at most (60 KB of spans, then the tables)
constexpr int kSpanMaxLut = 8192;   // cells of an output span that runs over several axes

struct SpanDesc {
    char *dst;
    const char *src;              // the op's first cell, and
    const char *src_end;          // the end of its last
    int64_t row_in[kSpanAxes];    // input spans: digits' input strides, fastest first
    int64_t run_out[kSpanAxes];   // output spans: digits' output strides
    int64_t uin[kSpanOuter], uout[kSpanOuter];
    FastDiv udiv[kSpanOuter];     // unit-index digits, innermost last
    FastDiv row_ext[kSpanAxes], run_ext[kSpanAxes];  // extents
    uint32_t row_sm[kSpanAxes], run_sm[kSpanAxes];   // shared-memory strides
    FastDiv ch_ext[kSpanAxes];                       // the output chain's axes,
    uint32_t ch_sm[kSpanAxes], ch_step[kSpanAxes];   // and the digits of kThreads over them
    uint32_t n_rows, n_runs;      // spans of a full unit
    uint32_t row_bytes;           // bytes of a full input span
    uint32_t run_cells;           // cells of a full output span
    // partial axes: indices per unit, extent, slot among the unit-index digits (-1: none);
    // what a full unit holds per index of the range
    uint32_t ka, na, kb, nb;
    int32_t ua, ub;
    uint32_t row_bytes_a, n_runs_a, run_cells_a;  // per index of the input chain's partial axis (0: not on it)
    uint32_t n_rows_b, run_cells_b;               // per index of the output chain's partial axis (0: not on it)
    int64_t reach;                // bytes from a full unit's origin to its last input span's start
    int64_t reach_b;              // of those, per index of the output chain's partial axis (0: not on it)
    uint32_t chunk;               // bytes of a copy: 16, 8 or 4
    FastDiv load_lanes, store_lanes;  // lanes a span is shared out over when it is copied / stored
    uint32_t tile_bytes;          // shared memory of the staged spans (multiple of 16)
    uint32_t lut;                 // 1: the output chain has several axes (offsets from a table)
    uint32_t fixed;               // 1: every output span starts on a word boundary and fits one pass of the lanes
    uint32_t E;
    int32_t no;
    uint32_t units;
};

// Whether chunks around [src, src + bytes) of a unit reach outside the source.
RH_HD bool span_at_edge(const SpanDesc &d, const char *src, int64_t bytes)
{
    const uintptr_t c = d.chunk - 1;
    return (uintptr_t(src) & ~c) < uintptr_t(d.src) || ((uintptr_t(src) + uintptr_t(bytes) + c) & ~c) > uintptr_t(d.src_end);
}

// Shared memory of a unit: staged spans, the spans' offsets, the table of an
// output span's cells.
RH_HD uint32_t span_lut_offset(const SpanDesc &d) { return (d.tile_bytes + (d.n_rows + d.n_runs) * 12u + 7u) & ~7u; }
RH_HD uint32_t span_smem_bytes(const SpanDesc &d) { return span_lut_offset(d) + (d.lut ? d.run_cells * 2u + 8u : 0u); }

}  // namespace rearr
