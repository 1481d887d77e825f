// step_launch.h -- the launches of step_kernels.cu, one set per capacity (the
// namespaces), for the C ABI (relaysum.cu), which has checked the arguments.
#pragma once

namespace relaysum {

// launch_counts         the counter kernel over `windows` (1 or 2) handles
// launch_step           the step kernel (the node-parallel one or the walk);
//                       after_counts: as the programmatic dependent of the
//                       counter kernel just enqueued
// launch_step_windows   the walk over two handles' windows
// launch_steps          several steps in one launch
// launch_steps_counts   the counters behind it
#define RELAY_STEP_LAUNCHES(SPACE)                                                                                \
    namespace SPACE {                                                                                             \
    int launch_counts(const relay_handle* const* hs, int32_t* const* counts, int windows, cudaStream_t stream);   \
    int launch_step(const relay_handle* h, const ModelArgs& a, bool nodes, cudaStream_t stream,                   \
                    bool after_counts);                                                                           \
    int launch_step_windows(const relay_handle* const* hs, const ModelArgs* as, cudaStream_t stream,              \
                            bool after_counts);                                                                   \
    int launch_steps(const relay_handle* h, const ModelArgs& a, FusedSteps& fs, cudaStream_t stream);             \
    int launch_steps_counts(const relay_handle* h, int32_t* counts, int k, cudaStream_t stream,                   \
                            bool after_models);                                                                   \
    }
RELAY_STEP_LAUNCHES(small)
RELAY_STEP_LAUNCHES(large)
#undef RELAY_STEP_LAUNCHES

}  // namespace relaysum
