// plan.cpp -- host plan compiler of librearr.
//
// A permute is brought to canonical form in the spirit of the paper's
// "offset/striding approach" (arXiv:1011.3583 Sec. III.B):
//   1. extent-1 axes are dropped;
//   2. output axes that are adjacent and in order in the input are merged
//      (stride[i] == stride[i+1] * extent[i+1]);
//   3. an unmoved innermost axis (input stride 1 on the output's last axis)
//      is folded into a wider cell; after that the output's fastest axis
//      always differs from the input's fastest axis;
//   4. the op is classified: a plain copy, long contiguous runs, or a tiled
//      transpose on the plane of the input's fastest and the output's fastest
//      axes with the other axes as batch (Sec. III.B: the 2-D plane of the
//      fastest dimensions of the original and the desired order).
#include "plan.h"
#include "reorder_geometry.h"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>

#include "tuning.h"
#include "variants.h"

namespace rearr {

namespace {

constexpr int64_t kMaxExtent = (int64_t(1) << 31) - 1;
constexpr int64_t kRunMinBytes = 128;     // cells this large are copied as runs
constexpr int64_t kRunUnitBytes = 32768;  // payload of one runs work unit
constexpr uint64_t kReorderL2MinBytes = uint64_t(128) << 20;  // reorder sources this large use L2 passes
constexpr uint64_t kMaxUnits = 0xFFFFFFFFull;
constexpr uint64_t kSpanMinCells = uint64_t(3) << 18;  // smaller thin-plane ops stay strided copies
constexpr int64_t kPlaneMinCells = 576;  // shorter planes are no interlaces: see plan_planes()
constexpr uint64_t kSpanLutCells = uint64_t(12) << 20; // thin planes whose spans need a table: see span_thin()

bool mul_overflows(uint64_t a, uint64_t b, uint64_t &out)
{
    if (a != 0 && b > UINT64_MAX / a) return true;
    out = a * b;
    return false;
}

bool ranges_overlap(uintptr_t a, uint64_t na, uintptr_t b, uint64_t nb)
{
    if (na == 0 || nb == 0) return false;
    return a < b + nb && b < a + na;
}

}  // namespace

int pow2_align(uint64_t a, uint64_t b, uint64_t c, uint64_t d)
{
    const uint64_t v = a | b | c | d | 16;
    return int(v & (~v + 1));  // lowest set bit, at most 16
}

// Shape of a fully vectorised fast tile: staged row bytes (128/256/512) and
// payload (16 KB, or the 8 KB half tile where an element size has one).  The
// shape that fills the DA x DB plane best is chosen (ragged last tiles waste
// bandwidth), ties broken toward full tiles and then toward equal input-row
// and output-row bytes.  An autotuned table may override the choice per
// (E, DA, DB) class.
static TileShape choose_shape(int E, int64_t DA, int64_t DB)
{
    std::vector<TileShape> cands = {{128, kTileBytes}, {256, kTileBytes}};
    if (E != 1) cands.push_back({512, kTileBytes});
    if (half_tile_vout(E)) cands.push_back({128, kTileBytes / 2});
    TileShape best{default_rowb(E), kTileBytes};
    double best_util = -1.0, best_bal = 1e9;
    for (const TileShape &c : cands) {
        const int64_t TA = c.rowb / E, TB = c.tbytes / c.rowb;
        const double ua = double(DA) / double(((DA + TA - 1) / TA) * TA);
        const double ub = double(DB) / double(((DB + TB - 1) / TB) * TB);
        const double util = ua * ub;
        // a half tile must fill clearly better to be chosen
        const double bal = std::fabs(std::log2(double(c.rowb)) - std::log2(double(TB * E))) +
                           (c.tbytes < kTileBytes ? 8.0 : 0.0);
        if (util > best_util + 0.01 || (util > best_util - 0.01 && bal < best_bal)) {
            best = c;
            best_util = std::max(best_util, util);
            best_bal = bal;
        }
    }
    TileShape tuned;
    if (tuned_shape(E, DA, DB, false, tuned) && (tuned.tbytes != kTileBytes / 2 || half_tile_vout(E))) return tuned;
    return best;
}

// The tile descriptor of plane (A = axis p, B = axis R-1) with the other
// axes as batch.  qa / qb (-1: none) are the batch axes that A / B absorb
// (a widened plane): A then spans DA * extent(qa) cells, B DB * extent(qb).
// Tile shape of a widened plane (see choose_widening): the candidate that
// fills the DA x DB plane (extents after widening) best, then the one whose
// shorter side -- input rows of ROWB bytes or output runs of TB * E bytes,
// each at most what the plane offers -- is longest (up to 512 bytes), then
// the smaller tile.  32 KB tiles exist for the shapes of double_tile_ok().
static TileShape choose_wide_shape(int E, int64_t DA0, int64_t DB0, int64_t DA, int64_t DB)
{
    TileShape tuned;
    if (tuned_shape(E, DA0, DB0, true, tuned)) return tuned;
    TileShape best{default_rowb(E), kTileBytes};
    double best_util = -1.0;
    int64_t best_run = -1;
    for (int rowb : {128, 256, 512}) {
        if (E == 1 && rowb == 512) continue;
        for (int tbytes : {kTileBytes, 2 * kTileBytes}) {
            if (tbytes > kTileBytes && !double_tile_ok(E, rowb)) continue;
            const int64_t TA = rowb / E, TB = tbytes / rowb;
            const double ua = double(DA) / double(((DA + TA - 1) / TA) * TA);
            const double ub = double(DB) / double(((DB + TB - 1) / TB) * TB);
            const double util = ua * ub;
            const int64_t run = std::min<int64_t>({int64_t(rowb), DA * E, TB * E, DB * E, 512});
            if (util > best_util + 0.01 || (util > best_util - 0.01 && run > best_run)) {
                best = {rowb, tbytes};
                best_util = std::max(best_util, util);
                best_run = run;
            }
        }
    }
    return best;
}

// A transpose plane whose input rows (DA cells of A) or output runs (DB cells
// of B) are short leaves DRAM with short bursts scattered far apart: every
// tile reads DB rows of DA*E bytes at the stride of B and writes DA runs of
// DB*E bytes at the stride of A.  Such a side is widened over the axis that
// continues it -- A over the batch axis of input stride DA cells (the input
// stays contiguous across the planes), B over the output axis just before it
// (the output stays contiguous) -- so one tile spans several planes and both
// its reads and its writes come in runs of up to 512 bytes.  Sides of at
// least wide_min_bytes() are left alone; an axis that continues both sides
// widens the shorter one.  Fast tiles only (one element per cell).  When DA
// is not a multiple of a 16-byte chunk's elements, the store phase splits
// every element's coordinate on its own (tile_fast_body).
static void choose_widening(const std::vector<Axis> &ax, int p, int64_t cell, int &qa, int &qb)
{
    const int R = int(ax.size());
    const uint64_t lim = wide_min_bytes();
    qa = qb = -1;
    if (R < 3) return;
    const int64_t DA = ax[p].extent, DB = ax[R - 1].extent;
    if (uint64_t(DA * cell) < lim)
        for (int i = 0; i < R - 1; ++i)
            if (i != p && ax[i].stride == DA * cell && DA * ax[i].extent <= kMaxExtent) qa = i;
    if (uint64_t(DB * cell) < lim && R - 2 != p && DB * ax[R - 2].extent <= kMaxExtent) qb = R - 2;
    if (qa >= 0 && qa == qb) {
        if (DA <= DB) qb = -1;
        else qa = -1;
    }
}

static void fill_tile_common(TileDesc &t, const std::vector<Axis> &ax, int p, int64_t cell, int qa, int qb,
                             char *dst, const char *src)
{
    const int R = int(ax.size());
    // Output strides (cells) of the canonical output axes, row-major.
    int64_t os[kMaxRank];
    os[R - 1] = 1;
    for (int i = R - 2; i >= 0; --i) os[i] = os[i + 1] * ax[i + 1].extent;
    const int64_t DA = ax[p].extent, DB = ax[R - 1].extent;
    t.dst = dst;
    t.src = src;
    t.sb_in = ax[R - 1].stride;
    t.sa_out = os[p] * cell;
    t.DA = uint32_t(qa >= 0 ? DA * ax[qa].extent : DA);
    t.DB = uint32_t(qb >= 0 ? DB * ax[qb].extent : DB);
    t.da_split = make_fastdiv(uint32_t(DA));
    t.db_split = make_fastdiv(uint32_t(DB));
    t.sa1_out = qa >= 0 ? os[qa] * cell : 0;
    t.sb1_in = qb >= 0 ? ax[qb].stride : 0;
    int nb = 0;
    for (int i = 0; i < R; ++i) {
        if (i == p || i == R - 1 || i == qa || i == qb) continue;
        t.bin[nb] = ax[i].stride;
        t.bout[nb] = os[i] * cell;
        t.bdiv[nb] = make_fastdiv(uint32_t(ax[i].extent));
        ++nb;
    }
    for (int i = nb; i < kMaxBatch; ++i) {
        t.bin[i] = 0;
        t.bout[i] = 0;
        t.bdiv[i] = make_fastdiv(1);
    }
    t.nb = nb;
}

// Box plan of a thin-plane permute with cells of one aligned E-byte word (see
// BoxDesc).  The unit's sub-box U grows from the input-innermost and the
// output-innermost axes: each step takes the axis that continues the shorter
// of the two runs (the input chain's next axis has an input stride equal to
// the chain's length, the output chain's an output stride equal to its),
// else the other side's, whole while the unit fits kBoxBytes.  When neither
// fits whole, the first becomes the partial axis over K indices (the last
// step).  Growth stops once both runs reach box_run_bytes() and the unit holds
// half a tile.  False when the box needs more axes than the descriptor holds,
// a run stays shorter than box_min_run_bytes(), or its stores would be
// narrower than 4 bytes.
static bool plan_box(const std::vector<Axis> &ax, int64_t E, uintptr_t da, uintptr_t sa, char *dst,
                     const char *src, OpDesc &op, rearr_permute_info &info)
{
    const int R = int(ax.size());
    std::vector<int64_t> os(R);  // output strides in bytes
    os[R - 1] = E;
    for (int i = R - 2; i >= 0; --i) os[i] = os[i + 1] * ax[i + 1].extent;
    const int64_t cap = kBoxBytes / E;
    std::vector<int> U;
    int kax = -1;
    int64_t K = 1, prod = 1;
    auto in_u = [&](int i) { return std::find(U.begin(), U.end(), i) != U.end(); };
    // One side's chain: its run in bytes, the axes on it and the next axis (-1: none).
    auto chain = [&](bool input, int64_t &run, std::vector<int> &on, int &next) {
        run = E;
        on.clear();
        next = -1;
        for (;;) {
            int hit = -1;
            for (int i = 0; i < R; ++i)
                if ((input ? ax[i].stride : os[i]) == run) hit = i;
            if (hit < 0) return;
            if (!in_u(hit)) {
                next = hit;
                return;
            }
            on.push_back(hit);
            if (hit == kax) {
                run *= K;
                return;
            }
            run *= ax[hit].extent;
        }
    };
    int64_t rin = E, rout = E;
    std::vector<int> on_in, on_out;
    const int64_t target = int64_t(box_run_bytes());
    for (;;) {
        int nin, nout;
        chain(true, rin, on_in, nin);
        chain(false, rout, on_out, nout);
        if (kax >= 0 || int(U.size()) == kMaxBoxAxes) break;
        if (rin >= target && rout >= target && 2 * prod * E >= kBoxBytes) break;
        const int first = rin <= rout ? (nin >= 0 ? nin : nout) : (nout >= 0 ? nout : nin);
        const int second = first == nin ? nout : nin;
        if (first < 0) break;
        if (prod * ax[first].extent <= cap) {
            U.push_back(first);
            prod *= ax[first].extent;
            continue;
        }
        if (second >= 0 && prod * ax[second].extent <= cap) {
            U.push_back(second);
            prod *= ax[second].extent;
            continue;
        }
        int64_t k = cap / prod;
        // range starts stay 16-byte aligned on both sides where K allows
        const int64_t m = std::max(16 / std::min<int64_t>(16, ax[first].stride & -ax[first].stride),
                                   16 / std::min<int64_t>(16, os[first] & -os[first]));
        if (k >= 2 * m) k -= k % m;
        if (k < 2) break;
        U.push_back(first);
        kax = first;
        K = k;
        prod *= k;
    }
    if (rin < int64_t(box_min_run_bytes()) || rout < int64_t(box_min_run_bytes())) return false;
    // unit-index axes: the others in output order, the partial axis as its range index
    struct Slot {
        int64_t ext, in, out;
    };
    std::vector<Slot> outer;
    int kunit = -1;
    for (int i = 0; i < R; ++i) {
        if (i == kax) {
            kunit = int(outer.size());
            outer.push_back({(ax[i].extent + K - 1) / K, K * ax[i].stride, K * os[i]});
        } else if (!in_u(i)) {
            outer.push_back({ax[i].extent, ax[i].stride, os[i]});
        }
    }
    if (int(outer.size()) > kMaxBoxOuter) return false;
    uint64_t units = 1;
    for (const Slot &o : outer) units *= uint64_t(o.ext);
    if (units >= kMaxUnits) return false;
    // widest loads / stores: within a run, and every run start aligned
    auto width = [&](bool input) {
        const std::vector<int> &on = input ? on_in : on_out;
        uint64_t bits = uint64_t(input ? rin : rout) | uint64_t(input ? sa : da) | 16;
        for (int i : U)
            if (std::find(on.begin(), on.end(), i) == on.end()) bits |= uint64_t(input ? ax[i].stride : os[i]);
        for (const Slot &o : outer) bits |= uint64_t(input ? o.in : o.out);
        const uint64_t v = bits & (~bits + 1);
        return uint32_t(std::max<uint64_t>(v, uint64_t(E)));
    };
    BoxDesc b;
    std::memset(&b, 0, sizeof(b));
    b.dst = dst;
    b.src = src;
    std::vector<int> by_in = U, by_out = U;
    std::sort(by_in.begin(), by_in.end(), [&](int x, int y) { return ax[x].stride < ax[y].stride; });
    std::sort(by_out.begin(), by_out.end(), [&](int x, int y) { return os[x] < os[y]; });
    const int nu = int(U.size());
    std::vector<int64_t> sm(R, 0);  // shared-memory strides, dense in input order
    int64_t acc = E;
    for (int j = 0; j < nu; ++j) {
        const int i = by_in[j];
        const int64_t ext = i == kax ? K : ax[i].extent;
        b.iext[j] = make_fastdiv(uint32_t(ext));
        b.iin[j] = ax[i].stride;
        sm[i] = acc;
        acc *= ext;
    }
    for (int j = 0; j < nu; ++j) {
        const int i = by_out[j];
        b.oext[j] = make_fastdiv(uint32_t(i == kax ? K : ax[i].extent));
        b.oout[j] = os[i];
        b.osm[j] = uint32_t(sm[i]);
    }
    for (int j = nu; j < kMaxBoxAxes; ++j) b.iext[j] = b.oext[j] = make_fastdiv(1);
    const int no = int(outer.size());
    for (int j = 0; j < kMaxBoxOuter; ++j) {
        b.udiv[j] = make_fastdiv(j < no ? uint32_t(outer[j].ext) : 1u);
        b.uin[j] = j < no ? outer[j].in : 0;
        b.uout[j] = j < no ? outer[j].out : 0;
    }
    b.nu = int8_t(nu);
    b.no = int8_t(no);
    b.kin = b.kout = -1;
    for (int j = 0; j < nu; ++j) {
        if (by_in[j] == kax) b.kin = int8_t(j);
        if (by_out[j] == kax) b.kout = int8_t(j);
    }
    b.kunit = int8_t(kunit);
    b.K = uint32_t(K);
    b.kfull = uint32_t(kax >= 0 ? ax[kax].extent : 1);
    b.vin = width(true);
    b.vout = width(false);
    // byte or 2-byte stores of short cells: the strided copy writes its
    // contiguous output 16 bytes at a time instead
    if (b.vout < 4) return false;
    b.cells = uint32_t(prod);
    op.cls = OC_BOX;
    op.word = uint32_t(E);
    op.box = b;
    op.units = units;
    info.kind = REARR_KIND_BOX;
    info.word_bytes = int(E);
    info.tile_a = int(rin / E);
    info.tile_b = int(rout / E);
    info.vec_in = int(b.vin);
    info.vec_out = int(b.vout);
    info.wide_a = info.wide_b = -1;
    info.n_tiles = int64_t(units);
    return true;
}

// Output spans of 1- and 2-byte cells over several axes, the first of them across
// input spans of a stride that is a multiple of 16 bytes: how many lanes of a
// store read different words of one bank (lanes are 4 / E cells apart, so they
// meet n0 / gcd(n0, 4 / E) of the n0 input spans); 1 for other plans.
static uint32_t span_bank_lanes(const SpanDesc &d)
{
    if (!d.lut || d.fixed || d.E > 2 || d.ch_sm[0] % 16 != 0) return 1;
    uint32_t g = 4 / d.E;
    while (d.ch_ext[0].d % g != 0) g /= 2;
    const uint32_t spans = std::min(32u, d.ch_ext[0].d / g);
    uint32_t banks = 32;
    for (uint32_t words = g * d.ch_sm[0] / 4; banks > 1 && words % 2 == 0; words /= 2) banks /= 2;
    return spans / std::min(banks, spans);
}

// From this many on the strided copy is faster (us, strided against spans).  In
// a call of its own, last two axes swapped: with four lanes 200 x 16 x 4096
// bytes 13.8, 14.2; eight 200 x 32 x 4096 21.6, 33.5; twelve 512 x 48 x 512
// 13.2, 23.8, of 2 bytes 15.6, 21.6.  In a batch of 800 MB the span units run in
// one kernel with nothing beside them: with eight 64 x 32 x 512 bytes 1024, 970,
// 64 x 512 x 8 of 2 bytes 1595, 533; twelve 64 x 48 x 512 bytes 810, 1309, of 2
// bytes 591, 629.
constexpr uint32_t kSpanBankLanes = 8;
constexpr uint32_t kSpanBankLanesBatch = 12;

// Whether a thin plane's span copy beats its strided copy (us, strided against
// span).  Output spans over several axes take their offsets from a table and
// their words one by one: that pays where every span fits one pass of the lanes
// on word boundaries (fixed), or from kSpanLutCells cells on, several units per
// CTA (1 byte: 9 x 3 x 340 x 1550 in order 0,2,3,1 18.3, 13.0, but 18 x 2 x 193
// x 597 7.0, 8.0; 2 bytes: 34 x 3 x 372 x 511 24.4, 17.6, but 36 x 6 x 557 x 35
// 6.8, 9.5; 4 bytes: 12 x 2 x 363 x 273 4.3, 6.0, 57 x 4 x 151 x 829 39.2, 39.4).
// A span of 32 words or more whose words all lie in one bank takes a cycle a
// lane (4 x 1168 x 2416 bytes reversed 43.7, 51.5; 64 x 512 x 32 of 2 bytes 6.2,
// 8.0; single bytes along one axis still gain, 512 x 512 x 32 41.5, 34.7).
// Taking every third 4-byte cell apart is near the copy rate either way
// (1817 x 1490 x 3 10.3, 12.4), every fourth is not (28 x 31 x 1218 x 4 11.1,
// 7.2).
static bool span_thin(const SpanDesc &d, bool lut)
{
    if (d.lut && !d.fixed) return lut && span_bank_lanes(d) < kSpanBankLanes;
    const bool one_bank = d.store_lanes.d >= 32 && d.ch_sm[0] * (4 / d.E) % 128 == 0;
    if (one_bank && (d.lut || d.E == 2)) return false;
    return d.lut || d.E < 4 || d.ch_sm[0] >= 16;
}

// Plans a gather of `total` elements of elem_bytes whose output axes are
// given in order (slowest first) with their input byte strides; src already
// points at the element of output index 0.  The output is contiguous.
static rearr_status plan_axes(void *dst, const char *src, size_t elem_bytes, const std::vector<Axis> &in_axes,
                              uint64_t total, PermPlan &pl, std::string &err, PlanFor what)
{
    rearr_permute_info &info = pl.info;
    const uint64_t bytes = total * elem_bytes;
    // Axes with extent > 1, merged where adjacent and in order.
    std::vector<Axis> ax;
    ax.reserve(in_axes.size());
    for (const Axis &cur : in_axes) {
        if (cur.extent == 1) continue;
        if (!ax.empty() && ax.back().stride == cur.stride * cur.extent) {
            ax.back().extent *= cur.extent;
            ax.back().stride = cur.stride;
        } else {
            ax.push_back(cur);
        }
    }
    int64_t cell = int64_t(elem_bytes);
    const uintptr_t da = uintptr_t(dst), sa = uintptr_t(src);

    auto set_copy = [&]() {
        info.kind = REARR_KIND_COPY;
        info.rank = 1;
        info.dims[0] = int64_t(total);
        info.in_strides[0] = 1;
        info.cell_bytes = int64_t(elem_bytes);
        const int W = pow2_align(da, sa, bytes);
        info.word_bytes = W;
        OpDesc &op = pl.op;
        op.cls = OC_COPY;
        op.word = uint32_t(W);
        op.copy.dst = static_cast<char *>(dst);
        op.copy.src = src;
        op.copy.bytes = bytes;
        op.copy.unit_bytes = uint64_t(kThreads) * 4 * W;
        op.units = (bytes + op.copy.unit_bytes - 1) / op.copy.unit_bytes;
        info.n_tiles = int64_t(op.units);
    };

    if (ax.empty() || (ax.size() == 1 && ax[0].stride == cell)) {  // one contiguous range
        set_copy();
        return REARR_OK;
    }
    // Fold an unmoved (input-contiguous) innermost axis into the cell.
    if (ax.back().stride == cell) {
        cell *= ax.back().extent;
        ax.pop_back();
        if (ax.empty() || (ax.size() == 1 && ax[0].stride == cell)) {
            set_copy();
            return REARR_OK;
        }
    }
    const int R = int(ax.size());
    uint64_t strides_or = 0;
    info.rank = R;
    for (int i = 0; i < R; ++i) {
        info.dims[i] = ax[i].extent;
        info.in_strides[i] = ax[i].stride / cell;
        strides_or |= uint64_t(ax[i].stride);
    }
    info.cell_bytes = cell;
    int p = -1;  // output axis along which input cells are contiguous
    for (int i = 0; i < R; ++i)
        if (ax[i].stride == cell) p = i;

    // Every output cell copied on its own (one cell is one W-byte word), 16/W
    // consecutive cells per thread written with one 16-byte store.
    auto set_strided = [&](int W, uint64_t n_cells) {
        StridedDesc sd;
        std::memset(&sd, 0, sizeof(sd));
        sd.dst = static_cast<char *>(dst);
        sd.src = src;
        sd.nd = R;
        for (int i = 0; i < kMaxRank; ++i) {
            sd.in_stride[i] = i < R ? ax[i].stride : 0;
            sd.div[i] = make_fastdiv(i < R ? uint32_t(ax[i].extent) : 1u);
        }
        sd.n_cells = n_cells;
        sd.vec = (da % 16 == 0) ? 1u : 0u;
        const uint64_t per_unit = uint64_t(kThreads) * (16 / W) * kStridedSteps;
        OpDesc &op = pl.op;
        op.cls = OC_STRIDED;
        op.word = uint32_t(W);
        op.strided = sd;
        op.units = (n_cells + per_unit - 1) / per_unit;
        info.kind = REARR_KIND_STRIDED;
        info.tile_a = info.tile_b = 0;
        info.wide_a = info.wide_b = -1;
        info.word_bytes = W;
        info.vec_in = W;
        info.vec_out = sd.vec ? 16 : W;
        info.n_tiles = int64_t(op.units);
    };

    // A box with no input-contiguous axis and cells of one aligned word (the
    // input's fastest axis dropped): every read is a scattered word, so each
    // cell is gathered on its own and the output written 16 bytes at a time.
    if (p < 0 && cell <= 16) {
        const int W = pow2_align(da, sa, uint64_t(cell), strides_or);
        const uint64_t n_cells = bytes / uint64_t(cell);
        bool fits = n_cells < kMaxUnits;
        for (int i = 0; i < R; ++i) fits &= ax[i].extent < int64_t(kMaxUnits);
        if (W == cell && fits) {
            set_strided(W, n_cells);
            return REARR_OK;
        }
    }

    // Cells of 128 bytes or more are copied as runs, and so are boxes with no
    // input-contiguous axis (there both sides cannot be coalesced).  Runs
    // shorter than runs_tile_max_bytes() on a transpose plane are copied in
    // blocks of cells instead (tile_runs_body), for long runs on both sides.
    const bool blocked_runs = p >= 0 && cell >= kRunMinBytes && uint64_t(cell) < runs_tile_max_bytes();
    if ((cell >= kRunMinBytes && !blocked_runs) || p < 0) {
        const int W = pow2_align(da, sa, uint64_t(cell), strides_or);
        uint64_t n_runs = 1;
        for (int i = 0; i < R; ++i) n_runs *= uint64_t(ax[i].extent);
        if (n_runs > kMaxUnits) { err = "too many runs"; return REARR_EINVAL; }
        for (int i = 0; i < R; ++i)
            if (ax[i].extent > int64_t(kMaxUnits)) { err = "a collapsed axis has 2^32 or more elements"; return REARR_EINVAL; }
        info.kind = REARR_KIND_RUNS;
        info.word_bytes = W;
        OpDesc &op = pl.op;
        op.cls = OC_RUNS;
        op.word = uint32_t(W);
        RunsDesc &r = op.runs;
        r.dst = static_cast<char *>(dst);
        r.src = src;
        r.run_bytes = cell;
        r.nd = R;
        for (int i = 0; i < kMaxRank; ++i) {
            r.in_stride[i] = i < R ? ax[i].stride : 0;
            r.div[i] = make_fastdiv(i < R ? uint32_t(ax[i].extent) : 1u);
        }
        r.n_runs = n_runs;
        const uint64_t wpr = uint64_t(cell) / W;
        if (wpr > 0xFFFFFFFFull) { err = "a run has 2^32 or more words"; return REARR_EINVAL; }
        r.wpr_div = make_fastdiv(uint32_t(wpr));
        if (cell > kRunUnitBytes) {
            // long runs: units are chunks of kRunUnitBytes
            const uint64_t cw = kRunUnitBytes / W;
            const uint64_t cpr = (wpr + cw - 1) / cw;
            if (n_runs * cpr > kMaxUnits) { err = "too many run chunks"; return REARR_EINVAL; }
            r.chunk_words = uint32_t(cw);
            r.cpr_div = make_fastdiv(uint32_t(cpr));
            r.runs_per_unit = 1;
            op.units = n_runs * cpr;
        } else {
            r.chunk_words = uint32_t(wpr);
            r.cpr_div = make_fastdiv(1);
            r.runs_per_unit = uint32_t(std::min<int64_t>(kMaxRunsPerUnit, std::max<int64_t>(1, kRunUnitBytes / cell)));
            op.units = (n_runs + r.runs_per_unit - 1) / r.runs_per_unit;
            // Short runs of a dense input may be walked in input order: the
            // reads become sequential and each run is written whole.
            if (uint64_t(cell) <= runs_mirror_max_bytes()) {
                std::vector<int> by_in(R);
                for (int i = 0; i < R; ++i) by_in[i] = i;
                std::sort(by_in.begin(), by_in.end(), [&](int a, int b) { return ax[a].stride > ax[b].stride; });
                bool dense = true;
                int64_t expect = cell;
                for (int k = R - 1; k >= 0; --k) {
                    dense &= ax[by_in[k]].stride == expect;
                    expect *= ax[by_in[k]].extent;
                }
                if (dense) {
                    std::vector<int64_t> out_stride(R);
                    int64_t os = cell;
                    for (int i = R - 1; i >= 0; --i) {
                        out_stride[i] = os;
                        os *= ax[i].extent;
                    }
                    r.mirror = 1;
                    for (int k = 0; k < kMaxRank; ++k) {
                        r.in_stride[k] = k < R ? out_stride[by_in[k]] : 0;
                        r.div[k] = make_fastdiv(k < R ? uint32_t(ax[by_in[k]].extent) : 1u);
                    }
                }
            }
        }
        info.n_tiles = int64_t(op.units);
        return REARR_OK;
    }

    info.plane_a = p;
    const int64_t DA = ax[p].extent, DB = ax[R - 1].extent;
    for (int i = 0; i < R; ++i)
        if (ax[i].extent > kMaxExtent) { err = "a collapsed axis has 2^31 or more elements"; return REARR_EINVAL; }

    OpDesc &op = pl.op;
    TileDesc &t = op.tile;
    const int W = pow2_align(da, sa, uint64_t(cell), strides_or);
    info.word_bytes = W;
    int vin = 0, vout = 0, qa = -1, qb = -1;
    bool narrow = false;  // a fast tile that moves less than 16 bytes at a time on a side
    if (W == cell) {
        const int E = int(cell);
        // Widest legal global access on each side.  Input rows start at src
        // plus sums of the input strides of the axes other than A (and other
        // than the axis a widened A absorbs: the widened row is contiguous
        // over DA * extent(qa) cells, so the load width follows that row
        // length); output rows start at multiples of DB*E bytes from dst.
        choose_widening(ax, p, cell, qa, qb);
        uint64_t in_or = 0;
        for (int i = 0; i < R; ++i)
            if (i != p && i != qa) in_or |= uint64_t(ax[i].stride);
        const int64_t DAw = qa >= 0 ? DA * ax[qa].extent : DA;
        const int vcap = tile_vector_bytes();
        vin = E;
        for (int v : {16, 4}) {
            if (v > E && v <= vcap && (uint64_t(DAw) * E) % v == 0 && sa % v == 0 && in_or % v == 0) { vin = v; break; }
        }
        vout = E;
        const int vmax = std::min(std::min(16, 4 * E), vcap);
        for (int v : {vmax, 4}) {
            if (v > E && (uint64_t(DB) * E) % v == 0 && da % v == 0) { vout = v; break; }
        }
    }
    fill_tile_common(t, ax, p, cell, qa, qb, static_cast<char *>(dst), src);
    info.wide_a = qa;
    info.wide_b = qb;
    uint64_t batch = 1;
    for (int i = 0; i < t.nb; ++i) batch *= t.bdiv[i].d;

    if (W == cell) {
        // Fast tile: one power-of-two element per cell.
        const int E = int(cell);
        // Tile shape: the default for the element size, or for the fully
        // vectorised widths the shape that fills the plane best (a widened
        // plane: the shape with the longest runs on both sides).
        TileShape shape{default_rowb(E), kTileBytes};
        narrow = vin < 16 || vout < std::min(16, 4 * E);
        if (!narrow) {
            shape = (qa >= 0 || qb >= 0) ? choose_wide_shape(E, DA, DB, t.DA, t.DB) : choose_shape(E, DA, DB);
            if (shape.tbytes < kTileBytes) vout = half_tile_vout(E);
        }
        t.TA = uint32_t(shape.rowb / E);
        t.TB = uint32_t(shape.tbytes / shape.rowb);
        info.kind = REARR_KIND_TILE;
        info.vec_in = vin;
        info.vec_out = vout;
        t.variant = tile_variant(E, vin, vout, shape.rowb, shape.tbytes);
        t.c = 1;
        t.pitch = 0;
        op.cls = OC_TILE;
    } else if (blocked_runs) {
        const int64_t c = cell / W;
        const int64_t side = std::max<int64_t>(int64_t(runs_tile_cells()), int64_t(runs_tile_side_bytes()) / cell);
        const int64_t nbk = std::max<int64_t>(1, std::min<int64_t>(side, 64));
        const int64_t TA = std::min<int64_t>(DA, nbk), TB = std::min<int64_t>(DB, nbk);
        if (TB * TA * c > int64_t(kMaxUnits)) { err = "a runs block has 2^32 or more words"; return REARR_EINVAL; }
        info.kind = REARR_KIND_TILE_CELLS;
        t.TA = uint32_t(TA);
        t.TB = uint32_t(TB);
        t.c = uint32_t(c);
        t.pitch = 0;  // no staging: blocked runs
        t.rowwords_div = make_fastdiv(uint32_t(TA * c));
        t.outwords_div = make_fastdiv(uint32_t(TB * c));
        t.c_div = make_fastdiv(uint32_t(c));
        t.variant = uint32_t(W);
        op.cls = OC_TILE_CELLS;
    } else {
        const int64_t c = cell / W;
        int64_t TA = std::max<int64_t>(1, std::min<int64_t>(DA, 256 / cell));
        int64_t TB = std::max<int64_t>(1, std::min<int64_t>(DB, 16384 / (TA * cell)));
        if (TB == DB) TA = std::max<int64_t>(1, std::min<int64_t>(DA, 16384 / (TB * cell)));
        auto pitch_of = [&](int64_t ta) {
            const int64_t rw = ta * c;
            const int64_t pad = ((c - rw) % 32 + 32) % 32;
            return rw + pad;
        };
        while (TB > 1 && TB * pitch_of(TA) * W > kSmemBytes) --TB;
        while (TA > 1 && TB * pitch_of(TA) * W > kSmemBytes) --TA;
        info.kind = REARR_KIND_TILE_CELLS;
        t.TA = uint32_t(TA);
        t.TB = uint32_t(TB);
        t.c = uint32_t(c);
        t.pitch = uint32_t(pitch_of(TA));
        t.rowwords_div = make_fastdiv(uint32_t(TA * c));
        t.outwords_div = make_fastdiv(uint32_t(TB * c));
        t.c_div = make_fastdiv(uint32_t(c));
        t.variant = uint32_t(W);
        op.cls = OC_TILE_CELLS;
    }
    info.tile_a = int(t.TA);
    info.tile_b = int(t.TB);
    const uint64_t ta_tiles = (uint64_t(t.DA) + t.TA - 1) / t.TA;
    const uint64_t tb_tiles = (uint64_t(t.DB) + t.TB - 1) / t.TB;
    const uint64_t units = ta_tiles * tb_tiles * batch;
    if (units > kMaxUnits || ta_tiles > kMaxUnits || tb_tiles > kMaxUnits) {
        err = "too many tiles";
        return REARR_EINVAL;
    }
    t.ta_div = make_fastdiv(uint32_t(ta_tiles));
    t.tb_div = make_fastdiv(uint32_t(tb_tiles));
    op.word = uint32_t(W);
    op.units = units;
    info.n_tiles = int64_t(units);

    // Thin planes (DA x DB far below a tile): every output cell copied on its
    // own (one cell is one W-byte word) when the tiles would carry little
    // payload on average -- a tile costs a whole load / store round trip
    // whatever its fill.  Decided after the tile plan so that the tile count
    // is the one the tile kernel would run; the thresholds are tuning knobs.
    // A 32 KB tile halves the CTA count: small ops keep the 16 KB tile of the
    // same row length so that they still fill the GPU.
    if (op.cls == OC_TILE && bytes < double_tile_min_bytes()) {
        tile_to_single_width(op);
        info.tile_b = int(t.TB);
        info.n_tiles = int64_t(op.units);
    }
    const uint64_t n_cells = bytes / uint64_t(cell);
    const ThinTuning thin_rule = thin_tuning();
    // (a threshold above what a tile holds means: every under-filled tile;
    // ops whose tiles are all full stay tiles)
    const uint64_t cells_rule = std::min<uint64_t>(thin_rule.tile_cells, uint64_t(t.TA) * t.TB);
    const bool thin_plane = bytes < op.units * thin_rule.tile_bytes ||
                            (bytes <= thin_rule.l2_bytes && n_cells < op.units * cells_rule);
    if (W == cell && thin_plane && n_cells < kMaxUnits &&
        !(uint64_t(cell) <= box_max_cell_bytes() && plan_box(ax, cell, da, sa, static_cast<char *>(dst), src, op, info)))
        set_strided(W, n_cells);
    // What a single call runs instead (the batched kernel keeps the op above).
    // Interlaces of a few planes, on 16-byte boundaries: the warp-staged
    // kernel moves 16 bytes at a time on every side.  32 x 3 x 1024^2 NCHW ->
    // NHWC, against the strided copy: 1-byte cells 106 -> 32 us, 2-byte 111 ->
    // 61, 4-byte 138 -> 119; 2^20-odd cells of 8 bytes in short planes gain
    // nothing below kSpanMinCells.
    // Span copies, against what else ran (measured on 510 random permutes of
    // 0.1 to 256 MB whose op is such a tile or a thin plane):
    // - tiles without 16-byte loads: 1.1 to 25 times as fast at any fill
    //   (251 x 333 x 517 in order 2,0,1: 1-byte cells 112 -> 31 us, 2-byte 139
    //   -> 52, 4-byte 150 -> 68, 8-byte 136 -> 120).  Tiles with 16-byte loads
    //   and narrower stores are faster than spans as long as they are full
    //   enough (4-byte cells, tiles a half to full 0.35 to 0.96; 1-byte ones
    //   three eighths full 0.33), so the line is a fill below which spans won
    //   at each cell size (32 x 16 x 4 x 3520 x 4 fp32 in order 1,0,4,2,3: 219
    //   -> 38 us at 6 %).
    // - thin planes of 1- to 4-byte cells from kSpanMinCells on, by span_thin().
    //   Strided copies of 8 and 16 bytes run at the copy rate already, and
    //   smaller ones are over before a span copy has its tables (1479 x 381
    //   2-byte cells: 4.7 against 5.2 us; 1001 x 999 bytes: 6.7 against 5.1).
    if (what == PlanFor::kOp || W != cell || op.cls == OC_BOX || tile_vector_bytes() != 16) return REARR_OK;
    const bool tile = op.cls == OC_TILE;
    const uint64_t held = op.units * uint64_t(t.TA) * t.TB;  // cells of full tiles
    const uint64_t least_fill = cell == 1 ? 12 : cell == 2 ? 33 : cell == 4 ? 40 : 45;  // per cent
    const bool span_tile = tile && (vin < 16 || 100 * n_cells < least_fill * held);
    const bool thin = op.cls == OC_STRIDED && n_cells >= kSpanMinCells;
    char *d = static_cast<char *>(dst);
    if (what == PlanFor::kBatch) {
        pl.use_batch_span = cell <= 8 && (op.cls == OC_STRIDED || span_tile) &&
                            plan_span(ax, cell, d, src, pl.span, false) &&
                            span_bank_lanes(pl.span) < kSpanBankLanesBatch;
        return REARR_OK;
    }
    pl.use_planes = (thin || narrow || (tile && 3 * n_cells < 2 * held)) && plan_planes(ax, cell, d, src, pl.planes_op);
    if (pl.use_planes) return REARR_OK;
    if (span_tile) {
        pl.use_span = plan_span(ax, cell, d, src, pl.span);
    } else if (thin && (cell < 4 || (cell == 4 && ax.back().extent >= 32 && ax.back().stride >= 16))) {
        const bool lut = cell < 4 && n_cells >= kSpanLutCells;
        pl.use_span = plan_span(ax, cell, d, src, pl.span, true, lut) && span_thin(pl.span, lut);
    }
    return REARR_OK;
}

// 16-byte groups per plane and unit of a fast interlace / de-interlace of k
// planes, `bytes` in all.  Four steps of the CTA per unit left an operation of
// 50 MB less than one wave of CTAs.  us at four, two, one: interlaced 4096^2 x
// 3 bytes 18.5, 17.2, 16.7, 2^23 x 5 fp32 53.9, 50.7, 49.9, 2^26 x 4 fp32 313,
// 309, 306, but 2^25 x 8 fp32 313, 313, 317; split 4096^2 x 3 bytes 17.7, 17.4,
// 17.1, 2^23 x 6 of 2 bytes 34.6, 33.9, 34.8, and 2^26 x 4 fp32 315, 316, 325
// (a large split writes longer runs per plane with four).
static uint64_t inter_unit_groups(bool inter, uint32_t k, uint64_t bytes)
{
    const uint64_t steps = inter ? (k <= 6 ? 1 : 2) : bytes <= (uint64_t(256) << 20) ? 2 : kInterSteps;
    return uint64_t(kThreads) * steps;
}

// Interlace: the output's fastest axis steps over k planes that are dense in
// the input along the axis before it.  De-interlace: the mirror image, k cells
// dense in the input, spread over k output planes dense along the output's
// fastest axis.  The other axes (after collapsing, at most two) are a batch.
// k_planes moves 16-byte groups on both sides, so everything has to lie on
// 16-byte boundaries, and a CTA works on one batch index at a time, so planes
// have to be long (20 MB, us, strided copies against interlaces: 2 planes of
// 128 fp32 7.2, 21.3, of 228 7.2, 12.5, of 336 7.2, 9.2; split into 6 of 64
// 8-byte cells 6.8, 19.8, of 168 7.2, 9.1; 2 of 256 2-byte cells 11.4, 21.2, of
// 456 11.4, 12.5; 8 of 512 bytes 17.4, 18.7).  From kPlaneMinCells cells on
// planes of 1 to 4 bytes won by 1.03 to 5 times, of 8 bytes by 0.9 to 2.3.
bool plan_planes(const std::vector<Axis> &ax, int64_t E, char *dst, const char *src, OpDesc &op)
{
    const int R = int(ax.size());
    int64_t os[kMaxRank];
    os[R - 1] = E;
    for (int i = R - 2; i >= 0; --i) os[i] = os[i + 1] * ax[i + 1].extent;
    int ik = -1, ip = -1;  // the axis over planes, the axis along them
    const bool inter = ax[R - 1].extent <= kInlineK && ax[R - 2].stride == E;
    if (inter) {
        ik = R - 1;
        ip = R - 2;
    } else {
        for (int i = 0; i < R - 1; ++i)
            if (ax[i].stride == E && ax[i].extent <= kInlineK && ax[R - 1].stride == E * ax[i].extent) ik = i;
        if (ik < 0) return false;
        ip = R - 1;
    }
    if (R > 4) return false;
    const int64_t k = ax[ik].extent, n = ax[ip].extent;
    const int64_t plane = inter ? ax[ik].stride : os[ik];
    if (n < kPlaneMinCells || (n * E) % 16 != 0) return false;
    std::memset(&op, 0, sizeof(op));
    InterlaceDesc &d = op.inter;
    uint64_t align = uint64_t(uintptr_t(dst)) | uint64_t(uintptr_t(src)) | uint64_t(plane), batch = 1;
    int nb = 0;
    for (int i = R - 1; i >= 0; --i) {
        if (i == ik || i == ip) continue;
        d.b_inter[nb] = inter ? os[i] : ax[i].stride;
        d.b_plane[nb] = inter ? ax[i].stride : os[i];
        align |= uint64_t(os[i]) | uint64_t(ax[i].stride);
        if (nb == 0) d.b0_div = make_fastdiv(uint32_t(ax[i].extent));
        batch *= uint64_t(ax[i].extent);
        ++nb;
    }
    if (nb == 0) d.b0_div = make_fastdiv(1);
    if (align % 16 != 0) return false;
    op.cls = inter ? OC_INTERLACE : OC_DEINTERLACE;
    op.word = uint32_t(E);
    d.inter = inter ? dst : const_cast<char *>(src);
    for (int j = 0; j < kInlineK; ++j)
        d.planes[j] = j < k ? (inter ? const_cast<char *>(src) : dst) + j * plane : nullptr;
    d.n = uint64_t(n);
    d.k = uint32_t(k);
    d.c = 1;
    d.elem_bytes = uint32_t(E);
    d.fast = 1;
    const uint64_t groups = uint64_t(n) * E / 16;
    d.unit_groups = inter_unit_groups(inter, uint32_t(k), uint64_t(n) * k * E * batch);
    const uint64_t upb = (groups + d.unit_groups - 1) / d.unit_groups;
    if (upb * batch >= kMaxUnits) return false;
    d.upb = make_fastdiv(uint32_t(upb));
    op.units = upb * batch;
    return true;
}

// The parts of a plan that its flags do not cover, zeroed.
static void clear(PermPlan &pl)
{
    std::memset(&pl.info, 0, sizeof(pl.info));
    std::memset(&pl.op, 0, sizeof(pl.op));
    pl.use_planes = pl.use_span = pl.use_batch_span = false;
}

rearr_status plan_permute(void *dst, const void *src, size_t elem_bytes, int rank, const int64_t *dims,
                          const int *perm, PermPlan &pl, std::string &err, PlanFor what)
{
    clear(pl);
    rearr_permute_info &info = pl.info;
    info.plane_a = -1;
    info.wide_a = info.wide_b = -1;
    if (elem_bytes == 0) { err = "elem_bytes must be >= 1"; return REARR_EINVAL; }
    if (rank < 1 || rank > kMaxRank) { err = "rank must be in [1, 8]"; return REARR_EINVAL; }
    if (!dims || !perm) { err = "dims and perm must not be NULL"; return REARR_EINVAL; }
    bool seen[kMaxRank] = {false};
    for (int i = 0; i < rank; ++i) {
        if (dims[i] < 0) { err = "dims must be >= 0"; return REARR_EINVAL; }
        if (perm[i] < 0 || perm[i] >= rank || seen[perm[i]]) {
            err = "perm is not a permutation of 0..rank-1";
            return REARR_EINVAL;
        }
        seen[perm[i]] = true;
    }
    uint64_t total = 1;
    for (int i = 0; i < rank; ++i)
        if (mul_overflows(total, uint64_t(dims[i]), total)) { err = "element count overflows"; return REARR_EINVAL; }
    uint64_t bytes;
    if (mul_overflows(total, elem_bytes, bytes) || bytes > (uint64_t(1) << 62)) {
        err = "byte count overflows";
        return REARR_EINVAL;
    }
    if (total == 0) {
        info.kind = REARR_KIND_NOOP;
        pl.op.units = 0;
        return REARR_OK;
    }
    if (!dst || !src) { err = "dst and src must not be NULL"; return REARR_EINVAL; }
    if (ranges_overlap(uintptr_t(dst), bytes, uintptr_t(src), bytes)) {
        err = "dst overlaps src (in-place permute is not supported)";
        return REARR_EINVAL;
    }
    // Row-major input strides in bytes; output axis i is input axis perm[i].
    int64_t s[kMaxRank];
    s[rank - 1] = int64_t(elem_bytes);
    for (int i = rank - 2; i >= 0; --i) s[i] = s[i + 1] * dims[i + 1];
    std::vector<Axis> ax;
    ax.reserve(size_t(rank));
    for (int i = 0; i < rank; ++i) ax.push_back(Axis{dims[perm[i]], s[perm[i]]});
    return plan_axes(dst, static_cast<const char *>(src), elem_bytes, ax, total, pl, err, what);
}

rearr_status plan_reorder_nm(void *dst, const void *src, size_t elem_bytes, int rank_in, const int64_t *dims,
                             int rank_out, const int *order, const int64_t *base, const int64_t *range,
                             PermPlan &pl, std::string &err, PlanFor what)
{
    clear(pl);
    pl.info.plane_a = -1;
    pl.info.wide_a = pl.info.wide_b = -1;
    if (elem_bytes == 0) { err = "elem_bytes must be >= 1"; return REARR_EINVAL; }
    if (rank_in < 1 || rank_in > kMaxRank) { err = "rank_in must be in [1, 8]"; return REARR_EINVAL; }
    if (rank_out < 1 || rank_out > rank_in) { err = "rank_out must be in [1, rank_in]"; return REARR_EINVAL; }
    if (!dims || !order || !base || !range) { err = "dims, order, base and range must not be NULL"; return REARR_EINVAL; }
    bool kept[kMaxRank] = {false};
    for (int i = 0; i < rank_out; ++i) {
        const int a = order[i];
        if (a < 0 || a >= rank_in || kept[a]) { err = "order must list distinct input axes"; return REARR_EINVAL; }
        kept[a] = true;
    }
    uint64_t total = 1, in_total = 1;
    for (int a = 0; a < rank_in; ++a) {
        if (dims[a] < 0 || base[a] < 0) { err = "dims and base must be >= 0"; return REARR_EINVAL; }
        if (kept[a]) {
            if (range[a] < 0 || base[a] + range[a] > dims[a]) { err = "a kept axis range leaves the input"; return REARR_EINVAL; }
            if (mul_overflows(total, uint64_t(range[a]), total)) { err = "element count overflows"; return REARR_EINVAL; }
        } else if (base[a] >= dims[a]) {
            err = "a dropped axis base index is out of range";
            return REARR_EINVAL;
        }
        if (mul_overflows(in_total, uint64_t(dims[a]), in_total)) { err = "element count overflows"; return REARR_EINVAL; }
    }
    uint64_t bytes, in_bytes;
    if (mul_overflows(total, elem_bytes, bytes) || mul_overflows(in_total, elem_bytes, in_bytes) ||
        in_bytes > (uint64_t(1) << 62)) {
        err = "byte count overflows";
        return REARR_EINVAL;
    }
    if (total == 0) {
        pl.info.kind = REARR_KIND_NOOP;
        pl.op.units = 0;
        return REARR_OK;
    }
    if (!dst || !src) { err = "dst and src must not be NULL"; return REARR_EINVAL; }
    if (ranges_overlap(uintptr_t(dst), bytes, uintptr_t(src), in_bytes)) {
        err = "dst overlaps src";
        return REARR_EINVAL;
    }
    int64_t s[kMaxRank];
    s[rank_in - 1] = int64_t(elem_bytes);
    for (int a = rank_in - 2; a >= 0; --a) s[a] = s[a + 1] * dims[a + 1];
    int64_t off = 0;
    for (int a = 0; a < rank_in; ++a) off += base[a] * s[a];
    std::vector<Axis> ax;
    ax.reserve(size_t(rank_out));
    for (int i = 0; i < rank_out; ++i) ax.push_back(Axis{range[order[i]], s[order[i]]});
    return plan_axes(dst, static_cast<const char *>(src) + off, elem_bytes, ax, total, pl, err, what);
}

// Groups of four elements per thread in a unit of an index gather or scatter of
// n elements of one W-byte word (vec: the body of 16-byte index loads, which
// holds two groups in flight).  One up to 2^23 elements and two beyond: with
// eight, 3M elements were 367 CTAs for 152 SMs (us at one, two, four, eight:
// 3,000,017 x 8 B random gather 17.6, 17.4, 20.3, 20.7, 65,536 x 4 B 2.3, 2.7,
// 3.7, 5.2; 16M x 4 B 70.0, 68.3, 69.5, 70.5).  Where that is not enough work
// for a CTA, or too much for an SM:
// - 1- and 2-byte elements in local order read 4 to 8 KB a unit of 1024: 8M x
//   1 B in shuffled blocks 9.7, 6.4, 6.0, 6.6, 40M 44.7, 33.5, 31.8, 33.2, 40M
//   x 2 B 73.6, 59.5, 57.4, 58.2 (also by 64-bit indices: 162, 156, 153, 158);
//   in random order the four are within 1 % from 3M on, below it one is ahead
//   (1.5M x 1 B 7.3, 9.4).
// - scatters of 8-byte elements write quarters of 32-byte sectors, which an SM
//   joins only while one CTA does it: a CTA per SM as long as eight groups last
//   (600,000 in shuffled blocks 5.0, 3.6, 2.9 (four), 4.3, 1.05M 6.0, 8.5, 5.8,
//   4.4; in random order 5.4, 4.5, 4.7, 6.8 and 7.0, 9.2, 7.2, 7.0).
static uint32_t gather_groups(uint64_t n, uint32_t W, bool vec, bool scatter)
{
    const uint64_t unit = uint64_t(kThreads) * 4, sms = 152;
    if (vec && scatter && W == 8 && n <= 8 * unit * sms) return uint32_t((n + unit * sms - 1) / (unit * sms));
    if (n > uint64_t(1) << 23) return W == 2 || (vec && W == 1) ? 4 : 2;
    return vec && W <= 2 && n > uint64_t(5) << 19 ? 2 : 1;
}

rearr_status plan_reorder(void *dst, const void *src, const uint32_t *idx, size_t n, size_t elem_bytes,
                          OpDesc &op, std::string &err, int idx_bytes, bool scatter)
{
    std::memset(&op, 0, sizeof(op));
    if (elem_bytes == 0) { err = "elem_bytes must be >= 1"; return REARR_EINVAL; }
    uint64_t bytes;
    if (mul_overflows(n, elem_bytes, bytes) || bytes > (uint64_t(1) << 62)) {
        err = "byte count overflows";
        return REARR_EINVAL;
    }
    if (idx_bytes == 4 && n > 0xFFFFFFFFull + 1) { err = "n exceeds the uint32 index range"; return REARR_EINVAL; }
    if (n == 0) { op.units = 0; return REARR_OK; }
    if (!dst || !src || !idx) { err = "dst, src and idx must not be NULL"; return REARR_EINVAL; }
    const uintptr_t da = uintptr_t(dst), sa = uintptr_t(src), ia = uintptr_t(idx);
    if (ranges_overlap(da, bytes, sa, bytes) || ranges_overlap(da, bytes, ia, uint64_t(n) * idx_bytes)) {
        err = "dst overlaps src or idx";
        return REARR_EINVAL;
    }
    if (ia % uintptr_t(idx_bytes) != 0) { err = "idx must be aligned to its index size"; return REARR_EINVAL; }
    const int W = pow2_align(da, sa, elem_bytes);
    op.cls = OC_GATHER;
    op.word = uint32_t(W);
    GatherDesc &g = op.gather;
    g.dst = static_cast<char *>(dst);
    g.src = static_cast<const char *>(src);
    g.idx = idx;
    g.n = n;
    g.c = uint32_t(elem_bytes / W);
    g.idx64 = idx_bytes == 8 ? 1u : 0u;
    g.scatter = scatter ? 1u : 0u;
    // the contiguous side (dst of a gather, src of a scatter) in groups of 4
    const uintptr_t contiguous = scatter ? sa : da;
    g.vec = (g.c == 1 && idx_bytes == 4 && ia % 16 == 0 && contiguous % uint64_t(std::min(16, 4 * W)) == 0) ? 1u : 0u;
    g.unit_elems = uint32_t(kThreads) * 4 * gather_groups(n, uint32_t(W), g.vec != 0, scatter);
    op.units = (uint64_t(n) + g.unit_elems - 1) / g.unit_elems;
    // Sources much larger than the L2 go through the bucketed passes (which
    // fall back to this direct gather on the device if the indices turn out
    // to be local).
    // (64-bit indices too: every valid one is < n < 2^32)
    const bool l2_ok = g.vec || (g.c == 1 && idx_bytes == 8 && contiguous % uint64_t(std::min(16, 4 * W)) == 0);
    g.l2 = (l2_ok && (W == 4 || W == 8 || W == 16) && bytes >= kReorderL2MinBytes && n <= 0xFFFFFFFFull) ? 1u : 0u;
    return REARR_OK;
}

rearr_status plan_interlace(bool inter, char *interlaced, char *const *planes, int k, size_t n,
                            size_t elem_bytes, InterlacePlan &pl, std::string &err)
{
    std::memset(&pl.op, 0, sizeof(pl.op));
    pl.planes.clear();
    if (elem_bytes == 0) { err = "elem_bytes must be >= 1"; return REARR_EINVAL; }
    if (k < 1 || k > kMaxK) { err = "k must be in [1, 256]"; return REARR_EINVAL; }
    if (!planes) { err = "the plane pointer array must not be NULL"; return REARR_EINVAL; }
    uint64_t pbytes, ibytes;
    if (mul_overflows(n, elem_bytes, pbytes) || mul_overflows(pbytes, uint64_t(k), ibytes) ||
        ibytes > (uint64_t(1) << 62)) {
        err = "byte count overflows";
        return REARR_EINVAL;
    }
    if (n == 0) { pl.op.units = 0; return REARR_OK; }
    if (!interlaced) { err = "the interlaced array pointer must not be NULL"; return REARR_EINVAL; }
    uint64_t align_or = uintptr_t(interlaced);
    for (int j = 0; j < k; ++j) {
        if (!planes[j]) { err = "a plane pointer is NULL"; return REARR_EINVAL; }
        if (ranges_overlap(uintptr_t(planes[j]), pbytes, uintptr_t(interlaced), ibytes)) {
            err = "a plane overlaps the interlaced array";
            return REARR_EINVAL;
        }
        align_or |= uintptr_t(planes[j]);
        pl.planes.push_back(planes[j]);
    }
    if (!inter) {  // de-interlace writes the planes: they must not overlap each other
        std::vector<std::pair<uintptr_t, int>> order;
        for (int j = 0; j < k; ++j) order.push_back({uintptr_t(planes[j]), j});
        std::sort(order.begin(), order.end());
        for (int j = 1; j < k; ++j)
            if (order[j - 1].first + pbytes > order[j].first) {
                err = "destination planes overlap";
                return REARR_EINVAL;
            }
    }
    OpDesc &op = pl.op;
    InterlaceDesc &d = op.inter;
    op.cls = inter ? OC_INTERLACE : OC_DEINTERLACE;
    d.inter = interlaced;
    for (int j = 0; j < kInlineK; ++j) d.planes[j] = j < k ? planes[j] : nullptr;
    d.planes_dev = nullptr;
    d.n = n;
    d.k = uint32_t(k);
    d.elem_bytes = uint32_t(elem_bytes);
    const bool pow2e = elem_bytes == 1 || elem_bytes == 2 || elem_bytes == 4 || elem_bytes == 8 ||
                       elem_bytes == 16;
    d.fast = (pow2e && k <= 8 && align_or % 16 == 0) ? 1u : 0u;
    if (d.fast) {
        const uint64_t groups = uint64_t(n) * elem_bytes / 16;
        op.word = uint32_t(elem_bytes);
        d.c = 1;
        d.unit_groups = inter_unit_groups(inter, uint32_t(k), ibytes);
        op.units = std::max<uint64_t>(1, (groups + d.unit_groups - 1) / d.unit_groups);
    } else {
        const int W = pow2_align(align_or, elem_bytes);
        op.word = uint32_t(W);
        d.c = uint32_t(elem_bytes / W);
        const uint64_t kc = uint64_t(k) * d.c;
        if (kc > 0xFFFFFFFFull) { err = "k * elem_bytes too large"; return REARR_EINVAL; }
        d.unit_groups = std::max<uint64_t>(1, 8192 / kc);
        d.kc_div = make_fastdiv(uint32_t(kc));
        d.c_div = make_fastdiv(d.c);
        op.units = (uint64_t(n) + d.unit_groups - 1) / d.unit_groups;
    }
    return REARR_OK;
}

void tile_to_single_width(OpDesc &op)
{
    if (op.cls != OC_TILE) return;
    TileDesc &t = op.tile;
    const uint32_t v = t.variant;
    const int tbytes = int((v >> 22) & 0xFu) * 8192;
    if (tbytes <= kTileBytes) return;
    const int E = int(v & 0x3Fu), vin = int((v >> 6) & 0x3Fu), vout = int((v >> 12) & 0x3Fu);
    const int rowb = int((v >> 18) & 0xFu) * 128;
    t.TB = uint32_t(kTileBytes / rowb);
    t.variant = tile_variant(E, vin, vout, rowb, kTileBytes);
    uint64_t batch = 1;
    for (int i = 0; i < t.nb; ++i) batch *= t.bdiv[i].d;
    const uint64_t ta_tiles = t.ta_div.d;
    const uint64_t tb_tiles = (uint64_t(t.DB) + t.TB - 1) / t.TB;
    t.tb_div = make_fastdiv(uint32_t(tb_tiles));
    op.units = ta_tiles * tb_tiles * batch;
}

// Host run of a box descriptor over the cells the device body visits
// (box_body), checking what the body relies on: every load and store inside
// its buffer and aligned to its width, the cells of one load (store)
// consecutive in the input (output) and inside the partial axis' range, every
// shared-memory access inside the unit, and the odometer's slot equal to the
// one decomposed from the cell's index.  Shared memory is poisoned before
// each unit.
static bool box_emulate(const OpDesc &op, const char *src0, size_t src_bytes, char *dst0, size_t dst_bytes, int E,
                        std::string &err)
{
    const BoxDesc &d = op.box;
    std::vector<unsigned char> smem(kBoxBytes);
    auto in_cell = [&](uint32_t c, int64_t &off, uint32_t &kd) {
        off = 0;
        kd = 0;
        for (int i = 0; i < d.nu; ++i) {
            uint32_t dig;
            fdivmod(c, d.iext[i], c, dig);
            off += int64_t(dig) * d.iin[i];
            if (i == d.kin) kd = dig;
        }
    };
    auto out_cell = [&](uint32_t c, uint32_t *dig, uint32_t &sm, int64_t &off, uint32_t &kd) {
        sm = 0;
        off = 0;
        kd = 0;
        for (int i = 0; i < d.nu; ++i) {
            fdivmod(c, d.oext[i], c, dig[i]);
            sm += dig[i] * d.osm[i];
            off += int64_t(dig[i]) * d.oout[i];
            if (i == d.kout) kd = dig[i];
        }
    };
    if (uint64_t(d.cells) * E > uint64_t(kBoxBytes)) { err = "box unit larger than its shared memory"; return false; }
    for (uint64_t unit = 0; unit < op.units; ++unit) {
        std::memset(smem.data(), 0xCD, smem.size());
        uint32_t q = uint32_t(unit), keff = d.K;
        int64_t bin = 0, bout = 0;
        for (int i = d.no - 1; i >= 0; --i) {
            uint32_t dig;
            fdivmod(q, d.udiv[i], q, dig);
            bin += int64_t(dig) * d.uin[i];
            bout += int64_t(dig) * d.uout[i];
            if (i == d.kunit) keff = std::min(d.K, d.kfull - dig * d.K);
        }
        const uint32_t vin = keff < d.K ? uint32_t(E) : d.vin, vout = keff < d.K ? uint32_t(E) : d.vout;
        for (uint32_t x = 0; x < d.cells * uint32_t(E); x += vin) {
            int64_t off;
            uint32_t kd;
            in_cell(x / E, off, kd);
            if (kd >= keff) continue;
            const char *g = d.src + bin + off;
            if (uintptr_t(g) % vin) { err = "box load misaligned"; return false; }
            if (g < src0 || g + vin > src0 + src_bytes) { err = "box load outside the source"; return false; }
            for (uint32_t k = 1; k < vin / uint32_t(E); ++k) {
                int64_t o2;
                uint32_t k2;
                in_cell(x / E + k, o2, k2);
                if (o2 != off + int64_t(k) * E || k2 >= keff) { err = "box load spans two runs"; return false; }
            }
            std::memcpy(&smem[x], g, vin);
        }
        const uint32_t V = vout / uint32_t(E);
        for (uint32_t y = 0; y < d.cells; y += V) {
            uint32_t dig[kMaxBoxAxes], sm, kd;
            int64_t off;
            out_cell(y, dig, sm, off, kd);
            if (kd >= keff) continue;
            char *g = d.dst + bout + off;
            if (uintptr_t(g) % vout) { err = "box store misaligned"; return false; }
            if (g < dst0 || g + vout > dst0 + dst_bytes) { err = "box store outside the destination"; return false; }
            for (uint32_t k = 0; k < V; ++k) {
                uint32_t dig2[kMaxBoxAxes], sm2, kd2;
                int64_t off2;
                out_cell(y + k, dig2, sm2, off2, kd2);
                if (sm2 != sm || off2 != off + int64_t(k) * E || kd2 >= keff) { err = "box store spans two runs"; return false; }
                if (uint64_t(sm) + E > uint64_t(d.cells) * E) { err = "box slot outside the unit"; return false; }
                std::memcpy(g + k * E, &smem[sm], E);
                for (int i = 0; i < d.nu; ++i) {  // the device body's odometer step
                    sm += d.osm[i];
                    if (++dig[i] < d.oext[i].d) break;
                    sm -= d.oext[i].d * d.osm[i];
                    dig[i] = 0;
                }
            }
        }
    }
    return true;
}

// Box plans of pseudo-random permutes (ranks 2-6, extents up to a few
// thousand, cells of 1-16 bytes, aligned and unaligned pointers) run on the
// host by box_emulate and compared with the permute written out directly.
static bool selftest_box(std::string &err)
{
    uint64_t x = 0x2545F4914F6CDD1Dull;
    auto rnd = [&](uint64_t n) {
        x ^= x << 13; x ^= x >> 7; x ^= x << 17;
        return x % n;
    };
    int boxes = 0, partial = 0;
    for (int t = 0; t < 2000 && boxes < 300; ++t) {
        const int rank = 2 + int(rnd(5));
        const int E = 1 << rnd(5);
        int64_t dims[kMaxRank];
        uint64_t total = 1;
        for (int i = 0; i < rank; ++i) {
            dims[i] = rnd(4) == 0 ? 1 + int64_t(rnd(3000)) : 1 + int64_t(rnd(rnd(2) ? 12 : 60));
            total *= uint64_t(dims[i]);
        }
        if (total > (uint64_t(1) << 17) || total < 2) continue;
        int perm[kMaxRank];
        for (int i = 0; i < rank; ++i) perm[i] = i;
        for (int i = rank - 1; i > 0; --i) std::swap(perm[i], perm[rnd(uint64_t(i) + 1)]);
        const size_t bytes = size_t(total) * E;
        const int so = rnd(3) == 0 ? E : 0, dof = rnd(3) == 0 ? E : 0;
        std::vector<char> sbuf(bytes + 64), dbuf(bytes + 64), want(bytes);
        char *src = sbuf.data() + ((16 - uintptr_t(sbuf.data()) % 16) % 16) + so;
        char *dst = dbuf.data() + ((16 - uintptr_t(dbuf.data()) % 16) % 16) + dof;
        for (size_t i = 0; i < bytes; ++i) src[i] = char(rnd(256));
        // the permute written out: output cell o (row-major over dims[perm])
        int64_t s[kMaxRank];
        s[rank - 1] = E;
        for (int i = rank - 2; i >= 0; --i) s[i] = s[i + 1] * dims[i + 1];
        for (uint64_t o = 0; o < total; ++o) {
            uint64_t r = o;
            int64_t in = 0;
            for (int i = rank - 1; i >= 0; --i) {
                const int64_t ext = dims[perm[i]];
                in += int64_t(r % uint64_t(ext)) * s[perm[i]];
                r /= uint64_t(ext);
            }
            std::memcpy(&want[o * E], src + in, E);
        }
        // canonical axes as plan_axes forms them
        std::vector<Axis> ax;
        for (int i = 0; i < rank; ++i) {
            const Axis cur{dims[perm[i]], s[perm[i]]};
            if (cur.extent == 1) continue;
            if (!ax.empty() && ax.back().stride == cur.stride * cur.extent) {
                ax.back().extent *= cur.extent;
                ax.back().stride = cur.stride;
            } else {
                ax.push_back(cur);
            }
        }
        if (ax.size() < 2 || ax.back().stride == E) continue;  // a copy or an unmoved inner axis
        bool has_a = false;
        for (const Axis &a : ax) has_a |= a.stride == E;
        if (!has_a) continue;
        OpDesc op;
        std::memset(&op, 0, sizeof(op));
        rearr_permute_info info;
        std::memset(&info, 0, sizeof(info));
        if (!plan_box(ax, E, uintptr_t(dst), uintptr_t(src), dst, src, op, info)) continue;
        ++boxes;
        partial += op.box.kunit >= 0;
        std::memset(dst, 0, bytes);
        if (!box_emulate(op, src, bytes, dst, bytes, E, err)) return false;
        if (std::memcmp(dst, want.data(), bytes) != 0) {
            char buf[160];
            std::snprintf(buf, sizeof buf, "box plan of a rank-%d permute of %d-byte cells differs from the permute",
                          rank, E);
            err = buf;
            return false;
        }
    }
    if (boxes < 100 || partial < 10) {
        char buf[96];
        std::snprintf(buf, sizeof buf, "box self-test planned only %d boxes (%d partial)", boxes, partial);
        err = buf;
        return false;
    }
    return true;
}

// Geometry of the scatter's chunk lists: within the call's scratch, with room
// for half as many elements again as a chunk has, and an exact chunk division.
static bool selftest_lists(std::string &err)
{
    int on = 0;
    for (uint32_t W : {4u, 8u})
        for (uint32_t sms : {148u, 152u, 160u})
            for (uint64_t n = kReorderL2MinBytes / W; n <= kListMaxElems; n += n / 7 + 3) {
                const ReorderGeometry gm = reorder_geometry(n, W, true, kReorderMaxSmemBuckets);
                const ListGeometry g = list_geometry(n, W, sms, gm.off_s, gm.bytes);
                if (!g.on) continue;
                ++on;
                bool ok = 2 * uint64_t(g.cap) >= 3 * uint64_t(g.CS) && g.cap % 8 == 0 && g.CS % 32 == 0 &&
                          g.end <= gm.bytes && uint64_t(g.C) * g.cap < (uint64_t(1) << 31) &&
                          size_t(g.CS) * W + g.CS / 8 <= kListSmem;
                for (uint64_t c = 1; c <= g.C; ++c)
                    for (uint64_t v : {c * g.CS - 1, c * g.CS})
                        if (v < n) ok &= (uint64_t(uint32_t(v)) * g.cs_mul >> (32 + g.cs_shift)) == v / g.CS;
                if (!ok) {
                    err = "chunk lists of " + std::to_string(n) + " elements of " + std::to_string(W) + " bytes: " +
                          std::to_string(g.C) + " chunks of " + std::to_string(g.CS) + ", lists of " +
                          std::to_string(g.cap);
                    return false;
                }
            }
    if (on < 30) err = "chunk lists planned for " + std::to_string(on) + " sizes only";
    return on >= 30;
}

// The forms a permute is planned in, by what it is planned for.
static bool selftest_plan_for(std::string &err)
{
    const int64_t ragged[3] = {251, 333, 517}, planes[3] = {32, 3, 65536};
    const int rotated[3] = {2, 0, 1}, swapped[3] = {0, 2, 1};
    void *dst = reinterpret_cast<void *>(uintptr_t(1) << 47);
    const void *src = reinterpret_cast<const void *>(uintptr_t(1) << 46);
    for (int i = 0; i < 6; ++i) {
        const bool inter = i >= 3;
        const PlanFor what[3] = {PlanFor::kCall, PlanFor::kBatch, PlanFor::kOp};
        const PlanFor w = what[i % 3];
        PermPlan pl;
        if (plan_permute(dst, src, 4, 3, inter ? planes : ragged, inter ? swapped : rotated, pl, err, w) != REARR_OK)
            return false;
        const bool call = w == PlanFor::kCall;
        if (pl.op.units == 0 || pl.use_planes != (call && inter) || pl.use_span != (call && !inter) ||
            pl.use_batch_span != (w == PlanFor::kBatch)) {
            err = "a permute is planned in forms that are not asked for";
            return false;
        }
    }
    return true;
}

// Routes of single calls on either side of the lines drawn in plan_axes():
// what: 0 the op itself, 1 a span copy, 2 interlaces.
static bool selftest_routes(std::string &err)
{
    struct Case {
        int what, elem, rank;
        int64_t dims[4];
        int perm[4];
    };
    static const Case cases[] = {
        {1, 4, 3, {251, 333, 517}, {2, 0, 1}},        // tiles without 16-byte loads
        {1, 1, 3, {2027, 37, 630}, {0, 2, 1}},
        {1, 4, 4, {8, 441, 1247, 8}, {0, 3, 1, 2}},   // tiles an eighth full
        {0, 1, 4, {4, 416, 1600, 48}, {0, 3, 1, 2}},  // tiles with 16-byte loads, three eighths to half full
        {0, 2, 3, {1056, 1328, 32}, {0, 2, 1}},
        {0, 4, 3, {258, 134, 648}, {0, 2, 1}},
        {0, 4, 3, {243, 418, 100}, {0, 2, 1}},        // full ones
        {0, 2, 3, {791, 61, 408}, {0, 2, 1}},
        {1, 4, 4, {28, 31, 1218, 4}, {0, 3, 1, 2}},   // thin planes, spans along one axis
        {0, 4, 3, {1817, 1490, 3}, {0, 2, 1}},
        {1, 2, 4, {15, 263, 204, 3}, {0, 3, 1, 2}},
        {1, 1, 4, {9, 3, 340, 1550}, {0, 2, 3, 1}},   // along several: enough cells
        {1, 2, 4, {34, 3, 372, 511}, {0, 2, 3, 1}},
        {0, 1, 4, {18, 2, 193, 597}, {0, 2, 3, 1}},   // too few
        {0, 2, 4, {36, 6, 557, 35}, {0, 2, 3, 1}},
        {0, 4, 4, {12, 2, 363, 273}, {0, 2, 3, 1}},   // 4-byte cells
        {0, 1, 3, {4, 1168, 2416}, {2, 1, 0}},        // words of a span in one bank
        {0, 2, 3, {64, 512, 32}, {0, 2, 1}},
        {0, 1, 3, {512, 48, 512}, {0, 2, 1}},         // of many spans
        {0, 4, 3, {20480, 2, 128}, {0, 2, 1}},        // short planes
        {0, 8, 3, {6826, 64, 6}, {0, 2, 1}},
        {2, 4, 3, {2048, 3, 1024}, {0, 2, 1}},        // long ones
        {2, 1, 4, {32, 3, 1024, 1024}, {0, 2, 3, 1}},
        {2, 2, 4, {32, 1024, 1024, 3}, {0, 3, 1, 2}},
    };
    for (const Case &c : cases) {
        PermPlan pl;
        if (plan_permute(reinterpret_cast<void *>(uintptr_t(1) << 47), reinterpret_cast<const void *>(uintptr_t(1) << 46),
                         size_t(c.elem), c.rank, c.dims, c.perm, pl, err) != REARR_OK)
            return false;
        const int got = pl.use_planes ? 2 : pl.use_span ? 1 : 0;
        if (got != c.what) {
            err = "route " + std::to_string(got) + " instead of " + std::to_string(c.what) + " for " +
                  std::to_string(c.dims[0]) + " x " + std::to_string(c.dims[1]) + " ... of " + std::to_string(c.elem) + " bytes";
            return false;
        }
    }
    return true;
}

bool selftest_host(std::string &err)
{
    // Fast division against the hardware divide on divisors and dividends
    // near powers of two, small values and pseudo-random values.
    std::vector<uint32_t> ds, ns;
    for (uint32_t v = 1; v < 300; ++v) ds.push_back(v);
    for (int b = 1; b < 32; ++b) {
        const uint32_t p = uint32_t(1) << b;
        ds.push_back(p - 1); ds.push_back(p); ds.push_back(p + 1);
    }
    ds.push_back(0xFFFFFFFFu); ds.push_back(0xFFFFFFFEu); ds.push_back(0x80000001u);
    uint64_t x = 0x9E3779B97F4A7C15ull;
    for (int i = 0; i < 200; ++i) {
        x ^= x << 13; x ^= x >> 7; x ^= x << 17;
        ds.push_back(uint32_t(x) | 1u);
        ds.push_back(uint32_t(x >> 40) + 1u);
        ns.push_back(uint32_t(x >> 3));
    }
    for (uint32_t v = 0; v < 1000; ++v) ns.push_back(v);
    for (int b = 1; b < 32; ++b) {
        const uint32_t p = uint32_t(1) << b;
        ns.push_back(p - 1); ns.push_back(p); ns.push_back(p + 1);
    }
    ns.push_back(0xFFFFFFFFu); ns.push_back(0xFFFFFFFEu);
    for (uint32_t d : ds) {
        const FastDiv f = make_fastdiv(d);
        for (uint32_t n : ns) {
            uint32_t q, r;
            fdivmod(n, f, q, r);
            if (q != n / d || r != n % d) {
                char buf[128];
                std::snprintf(buf, sizeof buf, "fastdiv %u / %u gave %u r %u", n, d, q, r);
                err = buf;
                return false;
            }
        }
        // every multiple boundary of small quotients
        for (uint64_t m = 1; m < 5; ++m) {
            const uint64_t n = m * d;
            if (n > 0xFFFFFFFFull) break;
            for (int off = -1; off <= 1; ++off) {
                const uint64_t nn = n + off;
                if (nn > 0xFFFFFFFFull) continue;
                uint32_t q, r;
                fdivmod(uint32_t(nn), f, q, r);
                if (q != uint32_t(nn / d) || r != uint32_t(nn % d)) { err = "fastdiv boundary"; return false; }
            }
        }
    }
    if (pow2_align(0) != 16 || pow2_align(12) != 4 || pow2_align(1024, 6) != 2 || pow2_align(3) != 1) {
        err = "pow2_align";
        return false;
    }
    return selftest_box(err) && selftest_lists(err) && selftest_plan_for(err) && selftest_routes(err) && selftest_span(err);
}

}  // namespace rearr
