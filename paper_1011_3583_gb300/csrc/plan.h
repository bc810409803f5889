// plan.h -- host plan compiler of librearr: validates an operation, reduces
// it to canonical form and fills the work-list descriptor of its kernel.
#pragma once

#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/librearr.h"
#include "rearr_internal.h"
#include "span.h"

namespace rearr {

struct Axis {
    int64_t extent;
    int64_t stride;  // input stride in bytes
};

// What a permute is planned for: a single call, an op of a captured batch, or
// the op alone (the server's requests, a pipeline's direct ops, the describe
// calls).
enum class PlanFor { kCall, kBatch, kOp };

struct PermPlan {
    rearr_permute_info info;  // what rearr_permute_describe reports: op and its geometry
    OpDesc op;                // descriptor of the work-list body
    // kCall: what runs instead, if there is one: interlaces of a few planes, or
    // a span copy.
    bool use_planes, use_span;
    OpDesc planes_op;
    SpanDesc span;
    // kBatch: whether a batch large enough for a kernel of span copies runs
    // `span` instead of op.
    bool use_batch_span;
};

struct InterlacePlan {
    OpDesc op;
    std::vector<char *> planes;  // all k plane pointers
};

// Each returns REARR_OK or REARR_EINVAL (with a message in err).  A plan with
// op.units == 0 is a no-op.
rearr_status plan_permute(void *dst, const void *src, size_t elem_bytes, int rank,
                          const int64_t *dims, const int *perm, PermPlan &pl, std::string &err,
                          PlanFor what = PlanFor::kCall);
rearr_status plan_reorder_nm(void *dst, const void *src, size_t elem_bytes, int rank_in, const int64_t *dims,
                             int rank_out, const int *order, const int64_t *base, const int64_t *range,
                             PermPlan &pl, std::string &err, PlanFor what = PlanFor::kCall);
// Gather dst[i] = src[idx[i]] (or, with scatter, dst[idx[i]] = src[i]) with
// idx_bytes-byte (4 or 8) indices.
rearr_status plan_reorder(void *dst, const void *src, const uint32_t *idx, size_t n,
                          size_t elem_bytes, OpDesc &op, std::string &err, int idx_bytes = 4,
                          bool scatter = false);
rearr_status plan_interlace(bool inter, char *interlaced, char *const *planes, int k, size_t n,
                            size_t elem_bytes, InterlacePlan &pl, std::string &err);

// A permute of the canonical axes as a batch of interlaces or de-interlaces
// (false: it is none, or not on 16-byte boundaries).
bool plan_planes(const std::vector<Axis> &ax, int64_t E, char *dst, const char *src, OpDesc &op);

// Span copy of the canonical axes (output order, slowest first; input strides
// in bytes; one E-byte word a cell): false where it does not apply.  alone: the
// op has the GPU to itself, so a small one is cut into units that fill it.  lut:
// output spans over several axes may be longer than one pass of the lanes.
bool plan_span(const std::vector<Axis> &ax, int64_t E, char *dst, const char *src, SpanDesc &d, bool alone = true,
               bool lut = true);

// A fast tile planned with the 32 KB payload re-planned with the 16 KB tile of
// the same row length (the batched kernel holds two 16 KB tiles per CTA).
void tile_to_single_width(OpDesc &op);

// Largest power of two <= 16 dividing every argument.
int pow2_align(uint64_t a, uint64_t b = 0, uint64_t c = 0, uint64_t d = 0);

// Span plans of pseudo-random permutes run on the host against the permute.
bool selftest_span(std::string &err);

// Host self-checks of the integer helpers (fast division, alignment).
bool selftest_host(std::string &err);

}  // namespace rearr
