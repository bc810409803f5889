// span_plan.cpp -- host plan of a span copy (span.h).
#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "plan.h"

namespace rearr {

namespace {

constexpr uint64_t kSpanBoxBytes = 16384;    // payload of a unit of a large op
constexpr uint64_t kSpanMinBoxBytes = 4096;  // and of a small one, so that it still fills the GPU
constexpr uint64_t kSpanFillUnits = 608;     // units wanted: four per SM
const FastDiv kOne = make_fastdiv(1);

struct Chain {
    int ax[kSpanAxes];
    int n = 0;
    int64_t run = 0;    // bytes of the span so far
    bool ended = false;
};

}  // namespace

bool plan_span(const std::vector<Axis> &ax, int64_t E, char *dst, const char *src, SpanDesc &d, bool alone, bool lut)
{
    const int R = int(ax.size());
    if (R > kMaxRank || R < 2) return false;
    int64_t os[kMaxRank], K[kMaxRank];  // output strides; indices of the axis in the box (0: outside it)
    uint64_t total = uint64_t(E);
    os[R - 1] = E;
    for (int i = R - 2; i >= 0; --i) os[i] = os[i + 1] * ax[i + 1].extent;
    for (int i = 0; i < R; ++i) {
        K[i] = 0;
        total *= uint64_t(ax[i].extent);
    }
    const uint64_t box = alone ? std::max(kSpanMinBoxBytes, std::min(kSpanBoxBytes, total / kSpanFillUnits)) : kSpanBoxBytes;
    const int64_t vmax = int64_t(box) / E;  // cells of a unit
    int64_t target = E;                     // bytes wanted of each span: an even split of the unit
    while (target * target < vmax * E * E) target *= 2;

    Chain c[2];  // 0: input, 1: output
    c[0].run = c[1].run = E;
    int64_t vol = 1;
    auto next = [&](int s) {
        for (int i = 0; i < R; ++i)
            if ((s == 0 ? ax[i].stride : os[i]) == c[s].run && ax[i].extent > 1) {
                bool on = false;
                for (int j = 0; j < c[s].n; ++j) on |= c[s].ax[j] == i;
                if (!on) return i;
            }
        return -1;
    };
    for (;;) {
        if (!(c[0].ended && c[1].ended)) {
            int s = c[0].run <= c[1].run ? 0 : 1;
            if (c[s].ended) s ^= 1;
            Chain &h = c[s];
            if (h.run >= target && 2 * vol <= vmax) {
                target *= 2;  // long enough, room left: longer ones
                continue;
            }
            if (h.run < target) {
                const int x = h.n < kSpanAxes ? next(s) : -1;
                if (x < 0) { h.ended = true; continue; }
                const int64_t n = ax[x].extent;
                if (K[x] == 0) {
                    const int64_t room = vmax / vol, want = std::max<int64_t>(1, (target + h.run - 1) / h.run);
                    K[x] = n <= room && n <= 2 * want ? n : std::min(n, std::min(room, want));
                    if (K[x] < 2) { K[x] = 0; h.ended = true; continue; }
                    vol *= K[x];
                }
                h.ax[h.n++] = x;
                h.run *= K[x];
                h.ended = K[x] < n;  // a range of an axis ends the chain
                continue;
            }
        }
        // What room is left goes to the partial axes, the one of the shorter
        // span first; a chain whose axis became whole goes on.
        int best = -1;
        int64_t best_run = 0, best_k = 0;
        for (int s = 0; s < 2; ++s) {
            if (!c[s].n) continue;
            const int x = c[s].ax[c[s].n - 1];
            const bool on_out = c[1].n > 1 && c[1].ax[c[1].n - 1] == x;
            const int64_t k = std::min(ax[x].extent, 2 * K[x]);
            if (K[x] < k && vol / K[x] * k <= vmax && !(on_out && c[1].run / E / K[x] * k > kSpanMaxLut) &&
                (best < 0 || c[s].run < best_run)) {
                best = x;
                best_run = c[s].run;
                best_k = k;
            }
        }
        if (best < 0) break;
        for (int s = 0; s < 2; ++s)
            if (c[s].n && c[s].ax[c[s].n - 1] == best) {
                c[s].run = c[s].run / K[best] * best_k;
                c[s].ended = best_k < ax[best].extent;
            }
        vol = vol / K[best] * best_k;
        K[best] = best_k;
    }
    // Ranges of about equal length, in whole 32-byte sectors.
    int part[2] = {-1, -1};
    for (int s = 0; s < 2; ++s) {
        if (!c[s].n) return false;
        const int x = c[s].ax[c[s].n - 1];
        if (K[x] == ax[x].extent) continue;
        part[s] = x;
        if (s == 1 && part[0] == x) continue;  // shared, done
        const int64_t pieces = (ax[x].extent + K[x] - 1) / K[x];
        int64_t k = (ax[x].extent + pieces - 1) / pieces;
        const int64_t q = std::max<int64_t>(1, 32 / E);
        if (K[x] >= q) k = std::min(K[x], (k + q - 1) / q * q);
        for (int t = 0; t < 2; ++t)
            if (c[t].ax[c[t].n - 1] == x) c[t].run = c[t].run / K[x] * k;
        K[x] = k;
    }
    if (c[0].run < 32 || c[1].run < 32) return false;  // spans under a sector: nothing is gained by staging
    if (!lut && c[1].n > 1 && c[1].run > kThreads * std::max<int64_t>(4, E)) return false;

    std::memset(&d, 0, sizeof(d));
    d.dst = dst;
    d.src = src;
    d.src_end = src + E;
    for (int i = 0; i < R; ++i) d.src_end += (ax[i].extent - 1) * ax[i].stride;
    d.E = uint32_t(E);
    d.row_bytes = uint32_t(c[0].run);
    d.run_cells = uint32_t(c[1].run / E);
    d.n_rows = d.n_runs = 1;
    for (int i = 0; i < kSpanAxes; ++i) d.row_ext[i] = d.run_ext[i] = d.ch_ext[i] = kOne;
    auto on = [&](int s, int x) {
        for (int j = 0; j < c[s].n; ++j)
            if (c[s].ax[j] == x) return true;
        return false;
    };
    // Shared-memory strides.  An axis of the input chain keeps its input
    // stride; an input span's axes get the next free stride congruent to
    // theirs modulo the copy width.  Lanes of a store read cells one step of
    // the output's fastest axis apart: when that step is between input spans,
    // an odd number of cells keeps it free of bank conflicts, so where the
    // input stride is even in cells the copies are narrowed to leave the
    // choice.
    int64_t sm[kMaxRank] = {0};
    for (int j = 0; j < c[0].n; ++j) sm[c[0].ax[j]] = ax[c[0].ax[j]].stride;
    const int o1 = c[1].ax[0];
    const bool steps_rows = !on(0, o1) && c[1].n == 1;
    d.chunk = 16;
    if (steps_rows && E < 16 && ax[o1].stride / E % 2 == 0) d.chunk = uint32_t(std::max<int64_t>(4, E));
    int64_t at = c[0].run + 30;  // spans' covering chunks must not overlap
    int nr = 0;
    for (int j = 0; j < c[1].n; ++j) {
        const int x = c[1].ax[j];
        if (on(0, x)) continue;
        const int64_t cw = d.chunk, want = ax[x].stride % cw;
        int64_t s = at + ((want - at) % cw + cw) % cw;
        if (j == 0 && steps_rows) {  // the fewest factors of two (in cells) among the next few
            int64_t best = s;
            auto twos = [&](int64_t v) {
                int t = 0;
                while (t < 5 && v / E % (2 << t) == 0) ++t;
                return t;
            };
            for (int m = 1; m < 4; ++m)
                if (twos(s + m * cw) < twos(best)) best = s + m * cw;
            s = best;
        }
        sm[x] = s;
        d.row_ext[nr] = make_fastdiv(uint32_t(K[x]));
        d.row_in[nr] = ax[x].stride;
        d.row_sm[nr] = uint32_t(s);
        ++nr;
        d.n_rows *= uint32_t(K[x]);
        d.reach += (K[x] - 1) * ax[x].stride;
        at = s * K[x];
    }
    d.tile_bytes = uint32_t((at + 32 + 15) / 16 * 16);
    if (d.tile_bytes > 60000) return false;  // table entries are 16-bit
    int nu = 0;
    for (int j = 0; j < c[0].n; ++j) {
        const int x = c[0].ax[j];
        if (on(1, x)) continue;
        d.run_ext[nu] = make_fastdiv(uint32_t(K[x]));
        d.run_out[nu] = os[x];
        d.run_sm[nu] = uint32_t(sm[x]);
        ++nu;
        d.n_runs *= uint32_t(K[x]);
    }
    if (d.n_rows > uint32_t(kSpanMaxSpans) || d.n_runs > uint32_t(kSpanMaxSpans)) return false;
    d.lut = c[1].n > 1;
    uint32_t step = kThreads;
    for (int j = 0; j < c[1].n; ++j) {
        d.ch_sm[j] = uint32_t(sm[c[1].ax[j]]);
        if (!d.lut) continue;
        d.ch_ext[j] = make_fastdiv(uint32_t(K[c[1].ax[j]]));
        fdivmod(step, d.ch_ext[j], step, d.ch_step[j]);
    }
    if (d.lut && d.run_cells > uint32_t(kSpanMaxLut)) return false;
    // Unit index: the input chain's range innermost, then the output chain's,
    // then the other axes in output order.
    d.ua = d.ub = -1;
    int no = 0;
    uint64_t units = 1;
    auto digit = [&](int64_t count, int64_t in, int64_t out) {
        if (no >= kSpanOuter || count > 0x7FFFFFFF) return false;
        d.udiv[no] = make_fastdiv(uint32_t(count));
        d.uin[no] = in;
        d.uout[no] = out;
        ++no;
        units *= uint64_t(count);
        return units < 0xFFFFFFFFull;
    };
    for (int i = 0; i < R; ++i)
        if (K[i] == 0 && !digit(ax[i].extent, ax[i].stride, os[i])) return false;
    auto range = [&](int x, int32_t &slot, uint32_t &k, uint32_t &n) {
        slot = no;
        k = uint32_t(K[x]);
        n = uint32_t(ax[x].extent);
        return ax[x].extent <= 0x7FFFFFFF &&
               digit((ax[x].extent + K[x] - 1) / K[x], K[x] * ax[x].stride, K[x] * os[x]);
    };
    if (part[1] >= 0 && part[1] != part[0] && !range(part[1], d.ub, d.kb, d.nb)) return false;
    if (part[0] >= 0 && !range(part[0], d.ua, d.ka, d.na)) return false;
    if (part[0] >= 0) {
        d.row_bytes_a = uint32_t(c[0].run / K[part[0]]);
        if (on(1, part[0])) d.run_cells_a = uint32_t(c[1].run / E / K[part[0]]);
        else d.n_runs_a = d.n_runs / uint32_t(K[part[0]]);
    }
    if (part[1] >= 0 && part[1] != part[0]) {
        d.run_cells_b = uint32_t(c[1].run / E / K[part[1]]);
        if (!on(0, part[1])) {
            d.n_rows_b = d.n_rows / uint32_t(K[part[1]]);
            d.reach_b = ax[part[1]].stride;
        }
    }
    d.no = no;
    d.units = uint32_t(units);
    const int64_t word = std::max<int64_t>(4, E);
    uint64_t out_or = uint64_t(uintptr_t(dst));
    for (int i = 0; i < nu; ++i) out_or |= uint64_t(d.run_out[i]);
    for (int i = 0; i < no; ++i) out_or |= uint64_t(d.uout[i]);
    const bool on_words = out_or % uint64_t(word) == 0;
    const int64_t chunks = (c[0].run - 1 + d.chunk - 1) / d.chunk + 1;
    const int64_t words = on_words ? (c[1].run + word - 1) / word : (c[1].run - 1 + word - 1) / word + 1;
    // Lanes a span is shared out over: the fewest steps of the CTA.
    auto lanes = [](uint32_t items, uint32_t spans) {
        uint32_t best = kThreads, cost = 0xFFFFFFFFu;
        const uint32_t least = uint32_t((uint64_t(items) * spans + kThreads - 1) / kThreads);
        for (uint32_t passes = (items + kThreads - 1) / kThreads; passes <= 64; ++passes) {
            const uint32_t l = (items + passes - 1) / passes, groups = kThreads / l;
            const uint32_t steps = passes * ((spans + groups - 1) / groups);
            if (steps < cost) {
                cost = steps;
                best = l;
                if (steps <= least) break;
            }
            if (l <= 8) break;
        }
        return best;
    };
    d.load_lanes = make_fastdiv(lanes(uint32_t(chunks), d.n_rows));
    d.store_lanes = make_fastdiv(lanes(uint32_t(words), d.n_runs));
    d.fixed = on_words && words <= int64_t(d.store_lanes.d);
    return true;
}

// Host run of a span descriptor as the kernel walks it, checking what the
// kernel relies on: copies aligned on both sides, inside the source array and
// the staged area, each at an address no other span's chunk takes, holding at
// least one byte of the span; every cell read from a byte some copy delivered;
// every store inside the destination.
static bool span_emulate(const SpanDesc &d, char *dst0, size_t dst_bytes, const char *src0, size_t src_bytes,
                         std::string &err)
{
    const int E = int(d.E), cw = int(d.chunk);
    auto digits = [&](uint32_t q, const FastDiv *ext, const uint32_t *sm, const int64_t *st, int64_t &off) {
        uint32_t s = 0;
        off = 0;
        for (int i = 0; i < kSpanAxes; ++i) {
            const uint32_t dig = q % ext[i].d;
            q /= ext[i].d;
            s += dig * sm[i];
            if (st) off += int64_t(dig) * st[i];
        }
        return s;
    };
    std::vector<unsigned char> tile(d.tile_bytes);
    std::vector<int> owner(d.tile_bytes);
    for (uint32_t u = 0; u < d.units; ++u) {
        const char *src = d.src;
        char *dst = d.dst;
        uint32_t rows = d.n_rows, runs = d.n_runs, len = d.row_bytes, cells = d.run_cells, q = u;
        int64_t reach = d.reach;
        for (int i = d.no - 1; i >= 0; --i) {
            uint32_t dig;
            fdivmod(q, d.udiv[i], q, dig);
            src += int64_t(dig) * d.uin[i];
            dst += int64_t(dig) * d.uout[i];
            if (i == d.ua) {
                const uint32_t k = std::min(d.ka, d.na - dig * d.ka);
                len = k * d.row_bytes_a;
                if (d.n_runs_a) runs = k * d.n_runs_a;
                if (d.run_cells_a) cells = k * d.run_cells_a;
            }
            if (i == d.ub) {
                const uint32_t k = std::min(d.kb, d.nb - dig * d.kb);
                if (d.n_rows_b) rows = k * d.n_rows_b;
                if (d.run_cells_b) cells = k * d.run_cells_b;
                reach -= int64_t(d.kb - k) * d.reach_b;
            }
        }
        const bool edge = span_at_edge(d, src, reach + len);
        const uintptr_t lo = uintptr_t(src0), hi = lo + src_bytes;
        std::fill(tile.begin(), tile.end(), 0xCD);
        std::fill(owner.begin(), owner.end(), -1);
        const uint32_t base = uint32_t(uintptr_t(src) & 15);
        for (uint32_t r = 0; r < rows; ++r) {
            int64_t off;
            const uint32_t sm = digits(r, d.row_ext, d.row_sm, d.row_in, off);
            const uintptr_t g = uintptr_t(src) + off;
            for (uint32_t ch = 0;; ++ch) {
                const uintptr_t p = (g & ~uintptr_t(cw - 1)) + ch * cw;
                if (p >= g + len) break;
                const uint32_t at = ((base + sm) & ~uint32_t(cw - 1)) + ch * cw;
                if ((g - (base + sm)) % uintptr_t(cw)) { err = "span: shared-memory address not congruent"; return false; }
                if (at + cw > d.tile_bytes) { err = "span: copy outside the staged area"; return false; }
                const bool cut = edge && (p < uintptr_t(d.src) || p + cw > uintptr_t(d.src_end));  // copied cell by cell
                for (int k = 0; k < cw; ++k) {
                    if (cut && (p + k < uintptr_t(d.src) || p + k >= uintptr_t(d.src_end))) continue;
                    if (p + k < lo || p + k >= hi) { err = "span: read outside the source"; return false; }
                    if (owner[at + k] >= 0) { err = "span: two copies overlap"; return false; }
                    owner[at + k] = int(r);
                    // bytes of the chunk outside the span are whatever lies there
                    tile[at + k] = p + k >= g && p + k < g + len ? *reinterpret_cast<const unsigned char *>(p + k) : 0xEE;
                }
            }
        }
        for (uint32_t r = 0; r < runs; ++r) {
            int64_t off;
            const uint32_t sm = digits(r, d.run_ext, d.run_sm, d.run_out, off);
            char *o = dst + off;
            for (uint32_t p = 0; p < cells; ++p) {
                int64_t none;
                const uint32_t f = d.lut ? digits(p, d.ch_ext, d.ch_sm, nullptr, none) : p * d.ch_sm[0];
                const uint32_t at = base + sm + f;
                if (at + E > d.tile_bytes) { err = "span: cell outside the staged area"; return false; }
                if (at % uint32_t(E)) { err = "span: cell misaligned"; return false; }
                for (int k = 0; k < E; ++k)
                    if (owner[at + k] < 0) { err = "span: cell not staged"; return false; }
                if (o + int64_t(p) * E < dst0 || o + int64_t(p + 1) * E > dst0 + dst_bytes) {
                    err = "span: store outside the destination";
                    return false;
                }
                std::memcpy(o + int64_t(p) * E, &tile[at], E);
            }
        }
    }
    return true;
}

// Host run of interlaces planned for a permute: every cell of every plane.
static bool planes_emulate(const OpDesc &op, char *dst0, size_t dst_bytes, std::string &err)
{
    const InterlaceDesc &d = op.inter;
    const int E = int(d.elem_bytes);
    const uint64_t upb = d.upb.d, groups = d.n * E / 16;
    if (d.n * E % 16 != 0 || upb * d.unit_groups < groups) { err = "planes: units do not cover a plane"; return false; }
    for (uint64_t b = 0; b < op.units / upb; ++b) {
        const int64_t b0 = int64_t(b % d.b0_div.d), b1 = int64_t(b / d.b0_div.d);
        char *iv = d.inter + b0 * d.b_inter[0] + b1 * d.b_inter[1];
        const int64_t poff = b0 * d.b_plane[0] + b1 * d.b_plane[1];
        for (uint32_t j = 0; j < d.k; ++j)
            for (uint64_t i = 0; i < d.n; ++i) {
                char *c = iv + (i * d.k + j) * E, *pl = d.planes[j] + poff + i * E;
                char *to = op.cls == OC_INTERLACE ? c : pl;
                if (i == 0 && (uintptr_t(iv) % 16 || uintptr_t(pl) % 16)) { err = "planes: off the 16-byte grid"; return false; }
                if (to < dst0 || to + E > dst0 + dst_bytes) { err = "planes: store outside the destination"; return false; }
                std::memcpy(to, op.cls == OC_INTERLACE ? pl : c, E);
            }
    }
    return true;
}

bool selftest_span(std::string &err)
{
    uint64_t x = 0x9E3779B97F4A7C15ull;
    auto rnd = [&](uint64_t n) {
        x ^= x << 13; x ^= x >> 7; x ^= x << 17;
        return x % n;
    };
    int plans = 0, partial = 0, luts = 0, shared = 0, narrow = 0, planes = 0, inter = 0, full = 0;
    for (int t = 0; t < 12000 && (plans < 500 || planes < 60 || full < 200); ++t) {
        const int rank = 2 + int(rnd(5));
        const int E = 1 << rnd(5);
        // units as those of a batch, of 16 KB whatever the op's size, in half
        // of the draws, on arrays that are long enough for some of them
        const bool alone = rnd(2) == 0;
        int64_t dims[kMaxRank];
        uint64_t total = 1;
        for (int i = 0; i < rank; ++i) {
            dims[i] = rnd(4) == 0 ? 1 + int64_t(rnd(3000)) : 1 + int64_t(rnd(rnd(2) ? 12 : 60));
            if (rnd(3) == 0) dims[i] = rnd(2) ? (dims[i] + 15) / 16 * 16 : 2 + int64_t(rnd(4));
            total *= uint64_t(dims[i]);
        }
        if (total > (uint64_t(1) << (alone ? 16 : 17)) || total < 64) continue;
        int perm[kMaxRank];
        for (int i = 0; i < rank; ++i) perm[i] = i;
        for (int i = rank - 1; i > 0; --i) std::swap(perm[i], perm[rnd(uint64_t(i) + 1)]);
        // a box of the array (the N-to-M reorder's strides) in a third of the draws
        int64_t range[kMaxRank];
        const bool boxed = rnd(3) == 0;
        uint64_t out_total = 1;
        for (int i = 0; i < rank; ++i) {
            range[i] = boxed ? 1 + int64_t(rnd(uint64_t(dims[i]))) : dims[i];
            out_total *= uint64_t(range[i]);
        }
        const size_t bytes = size_t(total) * E, out_bytes = size_t(out_total) * E;
        std::vector<char> sbuf(bytes + 64), dbuf(out_bytes + 64), want(out_bytes);
        char *src = sbuf.data() + ((16 - uintptr_t(sbuf.data()) % 16) % 16) + (rnd(3) == 0 ? E * rnd(16 / E) : 0);
        char *dst = dbuf.data() + ((16 - uintptr_t(dbuf.data()) % 16) % 16) + (rnd(3) == 0 ? E * rnd(16 / E) : 0);
        for (size_t i = 0; i < bytes; ++i) src[i] = char(rnd(256));
        int64_t s[kMaxRank];
        s[rank - 1] = E;
        for (int i = rank - 2; i >= 0; --i) s[i] = s[i + 1] * dims[i + 1];
        for (uint64_t o = 0; o < out_total; ++o) {
            uint64_t r = o;
            int64_t in = 0;
            for (int i = rank - 1; i >= 0; --i) {
                const int64_t ext = range[perm[i]];
                in += int64_t(r % uint64_t(ext)) * s[perm[i]];
                r /= uint64_t(ext);
            }
            std::memcpy(&want[o * E], src + in, E);
        }
        std::vector<Axis> ax;
        for (int i = 0; i < rank; ++i) {
            const Axis cur{range[perm[i]], s[perm[i]]};
            if (cur.extent == 1) continue;
            if (!ax.empty() && ax.back().stride == cur.stride * cur.extent) {
                ax.back().extent *= cur.extent;
                ax.back().stride = cur.stride;
            } else {
                ax.push_back(cur);
            }
        }
        if (ax.size() < 2 || ax.back().stride == E) continue;
        auto same = [&](const char *what) {
            if (std::memcmp(dst, want.data(), out_bytes) == 0) return true;
            err = std::string(what) + " of a rank-" + std::to_string(rank) + " permute of " + std::to_string(E) +
                  "-byte cells differ from the permute";
            return false;
        };
        OpDesc op;
        if (plan_planes(ax, E, dst, src, op)) {
            ++planes;
            inter += op.cls == OC_INTERLACE;
            std::memset(dst, 0, out_bytes);
            if (!planes_emulate(op, dst, out_bytes, err) || !same("interlaces")) return false;
        }
        SpanDesc d;
        if (!plan_span(ax, E, dst, src, d, alone)) continue;
        ++plans;
        partial += d.ua >= 0 || d.ub >= 0;
        luts += d.lut;
        shared += d.ua >= 0 && d.run_cells_a;
        narrow += d.chunk < 16;
        full += uint64_t(d.n_rows) * d.row_bytes > 2 * kSpanMinBoxBytes;
        std::memset(dst, 0, out_bytes);
        if (!span_emulate(d, dst, out_bytes, src, bytes, err) || !same("the spans")) return false;
    }
    if (plans < 300 || partial < 50 || luts < 50 || shared < 10 || narrow < 20 || inter < 10 || planes - inter < 10 ||
        full < 100) {
        err = "span self-test planned " + std::to_string(plans) + " copies (" + std::to_string(partial) + " partial, " +
              std::to_string(luts) + " of several axes, " + std::to_string(shared) + " sharing a range, " +
              std::to_string(narrow) + " in narrow copies, " + std::to_string(full) + " of full units) and " +
              std::to_string(planes) + " interlaces";
        return false;
    }
    return true;
}

}  // namespace rearr
