// Quantised weights on the tensor cores (scap_fc_qm.cu): interface for the 8-bit and 4-bit entry points (internal header).
#pragma once

#include "scap_fc.cuh"

namespace scap {

struct QmArgs {
    FcArgs f;                   // f.wscale: 8-bit weights only
    const float *scale;         // 4-bit weights: [ceil(K / group), N]
    const unsigned char *zero;  // 4-bit weights: same shape
    int group;                  // 4-bit weights: input channels per group (a multiple of 32)
    int sg;                     // 4-bit weights: scale groups that the shared memory of a CTA holds (set by the launcher)
};

// Whether the kernel can take the call (alignment of its vector loads, groups of a rank in shared memory).
bool qm_applicable(int wbits, const QmArgs &a);
// Blocks of 16 channels that a warp of the kernel works through (at up to four rows).
int qm_blocks_per_warp(const QmArgs &a);
// wbits: 8 or 4; xkind: 0 fp16, 1 bf16.  Chooses the split-K factor itself.
cudaError_t launch_fc_qm(int wbits, int mode, int xkind, QmArgs a, cudaStream_t st);

// 8-bit weights on the 5th-generation tensor cores in integers (scap_fc_i8.cu).
int i8_split(const FcArgs &a);                    // split-K factor
int i8_blocks_per_rank(const FcArgs &a, int S);  // blocks of 128 channels
bool i8_applicable(const FcArgs &a, int blocks_per_rank);
cudaError_t launch_fc_i8(int mode, int xkind, FcArgs a, cudaStream_t st);  // a.S: the split-K factor

}  // namespace scap
