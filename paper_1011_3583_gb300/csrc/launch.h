// launch.h -- kernel launchers of librearr (host side).
#pragma once

#include <cuda_runtime.h>

#include <atomic>

#include "plan.h"
#include "rearr_internal.h"

namespace rearr {

// Kernels launched by this library so far (graph replays add their kernels).
extern std::atomic<uint64_t> g_launches;

// Launch the one-op kernel of `op` on stream s.  planes_all holds the k plane
// pointers of an interlace / de-interlace (ignored otherwise).
cudaError_t launch_single(const OpDesc &op, char *const *planes_all, cudaStream_t s);

// A planned permute or N-to-M box as a single call: as interlaces (k_planes.cu)
// or a span copy (k_span.cu) if it has such a plan, else the kernel of its op.
cudaError_t launch_planes(const OpDesc &op, cudaStream_t s);
cudaError_t launch_span(const SpanDesc &d, cudaStream_t s);
inline cudaError_t launch_permute(const PermPlan &pl, cudaStream_t s)
{
    if (pl.use_planes) return launch_planes(pl.planes_op, s);
    return pl.use_span ? launch_span(pl.span, s) : launch_single(pl.op, nullptr, s);
}

// The span copies of a batch (device arrays of n descriptors and of the prefix
// sums of their units; smem: the largest descriptor's shared memory; counter
// zeroed before).
cudaError_t launch_batch_spans(const SpanDesc *spans, const uint64_t *prefix, int n, uint64_t units, uint32_t smem,
                               unsigned long long *counter, cudaStream_t s);

// The L2-resident bucketed reorder (k_reorder_l2.cu) of a gather op with l2 set.
cudaError_t launch_reorder_l2(const OpDesc &op, cudaStream_t s);

// Number of the n indices (idx_bytes 4 or 8) that are >= bound, counted on the
// device; waits for the count on stream s (k_check.cu).
cudaError_t count_bad_indices(const void *idx, size_t n, int idx_bytes, uint64_t bound, uint64_t *n_bad,
                              cudaStream_t s);

}  // namespace rearr
