// Swap deltas from bit planes (lpf_swap.cu), called by lpf_delta_swap.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

struct lpf_paths;

namespace lpf {
struct DeltaArgs;
// Whether segments are short enough (255 pixels) and the planes fit in shared
// memory.  d: geometry after delta_prepare.
bool swap_planes_apply(const DeltaArgs& d);
// Parts that a chunk's vectors are best cut into (by the cell and window alone,
// so that sums do not depend on how many candidates a call has).
int swap_planes_split(const DeltaArgs& d);
// Enqueue count changes (dcounts [K][2][n_canon], or null) and error changes
// per part of a chunk (partial [n_chunks * split][K], or null) of K exchanges.
// first: the call's first round (the handle's timing starts there).  d: the cell's
// geometry and tables after delta_prepare, target and counts when partial is
// given, selection in the extended layout.
int swap_planes_run(const uint8_t* img_dev, lpf_paths* paths, const int32_t* pairs_dev, int K, int32_t* dcounts_dev,
                    float* partial_dev, const DeltaArgs& d, int split, bool first, cudaStream_t s);
// Allow the kernels the opt-in shared memory; *max_static gets the larger of
// its value and their static shared memory.
int swap_planes_attributes(int optin, int* max_static);
}  // namespace lpf
