// Host-side entry to the split-operand tcgen05 kernels (codec_split_project.cuh, codec_split_expand.cuh).
#pragma once

#include <cuda_runtime.h>

#include "generic_kernels.cuh"

namespace ssn {

constexpr int kSplitMaxRank = 128;   // coordinates the split kernels take

// Projection only (a.src, no a.dst) and expansion only (a.zin, a.dst) of either element type, any
// alignment, leading dimension, position form and width; cudaErrorNotSupported, with nothing
// launched, for ranks above kSplitMaxRank, for both halves in one call and for the row statistic.
cudaError_t launch_codec_split_project(const TokenArgs &a, int32_t dtype, int sm_count, cudaStream_t stream);
cudaError_t launch_codec_split_expand(const TokenArgs &a, int32_t dtype, int sm_count, cudaStream_t stream);

}  // namespace ssn
