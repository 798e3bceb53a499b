// F-stage kernels of fengine_wide.cu, called by fengine.cu where fwide_takes says so: transforms of 32 points and
// more, filterbanks of at most 8 taps.
#pragma once

#include <vector>

#include "corr_internal.h"

namespace corr {

struct FWideArgs {
    int kind, log2L, n_inputs, n_frames, n_taps, n_sm;
    const void* d_in;      // packed samples [frame][L][n_inputs]
    void* d_out;           // float2 [frame][channel][n_inputs]
    const void* d_tw;      // fwide_tables(kind, log2L) on the device
    const float* d_taps;   // filterbank prototype, n_taps x L values (null: plain transform)
};

bool fwide_takes(int kind, int log2L, int n_inputs, int n_taps, int n_frames, int n_sm);   // n_taps = 0: plain transform
std::vector<float2> fwide_tables(int kind, int log2L);
cudaError_t launch_fwide(const FWideArgs& p, cudaStream_t s);

}  // namespace corr
