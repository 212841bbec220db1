// Which mode a tuned batch keeps. Host code, no CUDA.
#pragma once

namespace demag {

// Batch modes, in the order of demag_batch_set_mode.
enum { kBatchPersistent = 0, kBatchBranches = 1, kBatchPasses = 2 };

// t: ms per call of each mode (1e30: not available). The fastest; the
// pass-batched launches in place of the branch graph where that is less than a
// tenth faster: the branch graph is rebuilt whenever a call brings other buffers (6 ms
// for 64 states against a call of 1.4 ms), the other modes upload a table.
inline int batch_pick_mode(const double t[3])
{
    int best = t[kBatchPersistent] < t[kBatchBranches] ? kBatchPersistent : kBatchBranches;
    if (t[kBatchPasses] < t[best]) best = kBatchPasses;
    if (best == kBatchBranches && 0.9 * t[kBatchPasses] <= t[kBatchBranches]) best = kBatchPasses;
    return best;
}

}  // namespace demag
