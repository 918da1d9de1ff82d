// Swap deltas from bit planes (lpf_swap.cu), called by lpf_delta_swap.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

struct lpf_paths;

namespace lpf {
struct DeltaArgs;
// Whether the handle's segments are short enough (255 pixels).
bool swap_planes_apply(const lpf_paths* p);
// Enqueue count changes (dcounts [K][2][n_canon], or null) and per-chunk error
// changes (partial [n_chunks][K], or null) of K exchanges.  d: the cell's
// geometry and tables after delta_prepare, target and counts when partial is
// given, selection in the extended layout.
int swap_planes_run(const uint8_t* img_dev, lpf_paths* paths, const int32_t* pairs_dev, int K, int32_t* dcounts_dev,
                    float* partial_dev, const DeltaArgs& d, cudaStream_t s);
// Allow the kernels the opt-in shared memory; *max_static gets the larger of
// its value and their static shared memory.
int swap_planes_attributes(int optin, int* max_static);
}  // namespace lpf
