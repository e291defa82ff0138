// Whole steps that are short of work: two launches on one stream (small_step.cu).
#pragma once

#include "dp_common.cuh"

namespace dpg {

// Whether a checked DP_STEP_ALL call takes them; small_step.cu says where the line lies.
bool small_step_fits(const dp_step_desc& S);
dp_status launch_small_step(const dp_step_desc& S, cudaStream_t st);

}  // namespace dpg
