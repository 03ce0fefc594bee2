// Dense-stream kernel for the rows of a grouped call (internal header).
#pragma once

#include "scap_fc.cuh"

namespace scap {

cudaError_t launch_fc_ds_grouped(bool bf16, const FcArgs &a, cudaStream_t st);  // up to 32 rows, plain sparse FC (scap_fc_tc.cu)

}  // namespace scap
