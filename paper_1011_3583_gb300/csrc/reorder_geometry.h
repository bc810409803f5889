// reorder_geometry.h -- bucket geometry and scratch layout of the
// L2-resident reorder passes (k_reorder_l2.cu), shared with the host-only
// rearr_reorder_describe.  Source chunks of ~16 MB (at most 512 of them);
// destination chunks of 64 KB (one CTA's shared memory) while the bucket
// count stays within the bound, else the source chunks' size.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace rearr {

constexpr uint32_t kReorderMaxChunks = 512;
constexpr uint64_t kReorderSourceChunkBytes = uint64_t(16) << 20;
constexpr uint32_t kReorderScatterChunkBytes = 64u << 10;
constexpr uint64_t kReorderMaxSmemBuckets = uint64_t(1) << 24;

struct ReorderGeometry {
    uint32_t cs_shift;   // source chunk = 2^cs_shift elements
    uint32_t ds_shift;   // destination chunk = 2^ds_shift elements
    uint32_t C, D;       // source / destination chunks (D = 1 for a scatter)
    bool smem_scatter;   // the gather's last pass through shared memory
    // scratch layout: byte offsets of the arrays and the total
    size_t off_hist, off_row, off_base, off_cur, off_up, off_s, off_i, off_v, off_st, bytes;
};

// n elements of W bytes; scatter: buckets by destination chunk only;
// smem_bucket_limit: the tuned bound on C * D for the shared-memory scatter.
inline ReorderGeometry reorder_geometry(uint64_t n, uint32_t W, bool scatter, uint64_t smem_bucket_limit)
{
    ReorderGeometry g{};
    uint32_t shift = 0;
    while ((uint64_t(1) << shift) * W < kReorderSourceChunkBytes) ++shift;
    while (((n + (uint64_t(1) << shift) - 1) >> shift) > kReorderMaxChunks) ++shift;
    g.cs_shift = shift;
    g.C = uint32_t((n + (uint64_t(1) << shift) - 1) >> shift);
    uint32_t dshift = 0;
    while ((uint64_t(2) << dshift) * W <= kReorderScatterChunkBytes) ++dshift;
    const uint64_t d_small = (n + (uint64_t(1) << dshift) - 1) >> dshift;
    g.smem_scatter = !scatter && uint64_t(g.C) * d_small <= std::min(smem_bucket_limit, kReorderMaxSmemBuckets);
    g.ds_shift = g.smem_scatter ? dshift : shift;
    g.D = scatter ? 1u : g.smem_scatter ? uint32_t(d_small) : g.C;
    const size_t nb = size_t(g.C) * g.D;
    auto al = [](size_t x) { return (x + 255) / 256 * 256; };
    g.off_hist = 256;
    g.off_row = g.off_hist + al(nb * 4);
    g.off_base = g.off_row + al(size_t(g.C) * 4);
    g.off_cur = g.off_base + al(nb * 4);
    g.off_up = g.off_cur + al(nb * 4);
    g.off_s = g.off_up + al((nb + 1) * 4);
    g.off_i = g.off_s + al(size_t(n) * 4);
    g.off_v = g.off_i + al(size_t(n) * 4);
    g.off_st = g.off_v + al(size_t(n) * W);
    // tile-local form: C + 1 segment starts (uint16) per 4096-index tile
    const size_t tiles = size_t((n + 4095) / 4096);
    g.bytes = g.off_st + al(tiles * (size_t(g.C) + 1) * 2);
    return g;
}

// Scatters through chunk lists (scatter_chunks.cuh): destination chunks that
// fit one CTA's shared memory.
constexpr uint32_t kListChunkBytes = 208u << 10;       // shared memory of a chunk
constexpr uint64_t kListMaxElems = uint64_t(1) << 29;  // the chunk division's range
constexpr size_t kListSmem = 231000;                   // shared memory of a CTA, at most

constexpr uint32_t kListMaxChunks = 4096;
constexpr uint32_t kFillStride = 8;  // words per list counter: appends to different lists meet in different sectors
constexpr uint32_t kListMinSegment = 8;  // elements of a tile's segment, on average
constexpr uint32_t kSampleRuns = 4096;       // runs of the locality sample,
constexpr uint32_t kSampleRunHits = 8;       // indices of each that are counted by chunk

struct ListGeometry {
    bool on;
    uint32_t CS, C, cap;         // elements per chunk (a multiple of 32), chunks, room of a list (a multiple of 8)
    uint32_t cs_mul, cs_shift;   // v / CS = (v * cs_mul) >> (32 + cs_shift) for v < 2^29
    uint32_t T;                  // elements of a tile
    uint32_t hits_full;          // sampled indices of a chunk that stand for a full list
    uint32_t hits_past;          // those beyond full lists, in all, that are let through
    size_t smem;                 // shared memory of a CTA
    size_t off_fill, off_off, off_v, end;  // scratch, from `start`
};

// n elements of W bytes; chunks as large as shared memory takes, evened out
// over the sms SMs where each places only a few; scratch from byte `start` to
// byte `limit` of the call's.  Measured against the bucketed passes (random
// permutations, us): 2^25 x 4 B 424 -> 260, 2^26 801 -> 529, 10^8 1160 -> 789,
// 2^27 1537 -> 1130; 2^24 x 8 B 302 -> 212, 2^25 553 -> 418.  Left out, as first
// built: 2^28 x 4 B 3058 -> 3489, 2^26 x 8 B 1056 -> 1127, 2^23 x 16 B 249 -> 240,
// 2^25 x 16 B 895 -> 1148: tiles' segments have to be long enough for their list
// writes to fill sectors, and 16-byte elements (tiles of 8192) gain nothing.
inline ListGeometry list_geometry(uint64_t n, uint32_t W, uint32_t sms, size_t start, size_t limit)
{
    ListGeometry g{};
    if (W > 8 || n > kListMaxElems) return g;
    const uint64_t most = kListChunkBytes / W;
    const uint64_t rounds = (n + most * sms - 1) / (most * sms);
    const uint64_t cs = ((n + rounds * sms - 1) / (rounds * sms) + 31) / 32 * 32;
    g.CS = uint32_t(std::min(most, cs));
    g.C = uint32_t((n + g.CS - 1) / g.CS);
    // With s = floor(log2(CS - 1)) and m = ceil(2^(32 + s) / CS) < 2^32 the error
    // m CS - 2^(32 + s) is below CS <= 2^(s + 1), so v m / 2^(32 + s) is less
    // than 1 / CS above v / CS for v < 2^29 (Granlund & Montgomery, Sec. 4).
    while ((uint64_t(2) << g.cs_shift) < g.CS) ++g.cs_shift;
    const uint64_t two = uint64_t(1) << (32 + g.cs_shift);
    g.cs_mul = uint32_t((two + g.CS - 1) / g.CS);
    // n uniform draws with repeats fill a list to CS with a deviation of
    // sqrt(CS); at least twelve of those are left free.  Sequences that repeat
    // more in some chunks than in others need longer lists: all the room that
    // the call's scratch has (CS twice at 4 bytes, 1.6 times at 8).
    uint32_t root = 1;
    while (uint64_t(root) * root < g.CS) ++root;
    auto al = [](size_t x) { return (x + 255) / 256 * 256; };
    g.off_fill = start;
    g.off_off = g.off_fill + al(size_t(g.C) * kFillStride * 4);
    if (limit < g.off_off + 512) return g;
    const uint64_t room = (limit - g.off_off - 512) / (uint64_t(g.C) * (2 + W));
    g.cap = uint32_t(std::min<uint64_t>(room, 2 * uint64_t(g.CS)) / 8 * 8);
    if (g.cap < g.CS + 12 * root) return g;
    g.T = (W == 4 ? 6 : 4) * 4096;
    g.smem = size_t(g.T) * (W + 4) + size_t(g.C) * 4;
    // A sixteenth beyond full lists: what chance gives uniform draws is a tenth
    // of that, and as many direct stores cost less than the lists gain.
    g.hits_full = uint32_t(uint64_t(kSampleRuns) * kSampleRunHits * g.cap / n);
    g.hits_past = kSampleRuns * kSampleRunHits / 16;
    g.off_v = g.off_off + al(size_t(g.C) * g.cap * 2);
    g.end = g.off_v + al(size_t(g.C) * g.cap * W);
    g.on = g.C <= kListMaxChunks && g.smem <= kListSmem && g.T >= kListMinSegment * g.C && g.end <= limit;
    return g;
}

}  // namespace rearr
