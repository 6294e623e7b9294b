// On-chip FP32 kernels of sides 64 and 128 (fp32_block.cu).
#pragma once

#include <cuda_runtime.h>

#include "bdct_internal.h"

namespace bdct {

// Fill the kernels' constant tables on the current device; d_table holds the
// FP32 cosine table (called by fused_init_device).
cudaError_t block_init_device(const float *d_table);
// 64 x 128, 128 x 64 and 128 x 128 (64 x 64 runs in fp32_ring.cu).
bool block_supported(int rows, int cols);
// Contiguous, indexed and tiled batches.  sc is ignored for the round trip
// and the spectral direction (orthonormal both); the spectral direction takes
// the plain diagonal in g.lam.
cudaError_t block_launch(int rows, int cols, Dir dir, const DirScales &sc, const ExecGeom &g, unsigned int *status,
                         cudaStream_t stream);

}  // namespace bdct
