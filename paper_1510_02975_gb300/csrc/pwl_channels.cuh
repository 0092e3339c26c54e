// pwl_channels.cuh -- internal interface of the channel-wise kernels.
#pragma once

#include "pwl_table.cuh"

namespace pwl {

struct ChanArgs {
    const float* knots;   // [C, N+1] FP32
    const float* values;  // [C, N+1] FP32
    int64_t C, R;         // channels, rows
    int N, K;             // intervals, cells per channel
    int cluster;          // CTAs per cluster
    int64_t passes;       // passes of the CTA over all rows: ceil(R / rows per pass)
    int64_t work;         // tile groups (of a cluster's CTAs) x passes
    int* status;          // device word: bit 0 set if a channel's knots are not strictly increasing
};

}  // namespace pwl
