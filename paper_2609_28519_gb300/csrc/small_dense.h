// On-chip dense route for small arrays (small_dense.cu).
#pragma once

#include <cuda_runtime.h>

#include "bdct_internal.h"

namespace bdct {

// Both sides at most 64 and the width a multiple of 4.
bool small_dense_supported(int h, int w);

// Half-operator tables (dense_gen_table) of the passes a direction runs:
// forward fw, fh; inverse ih, iw; round trip and spectral all four.
struct SmallTables {
    const float *fw, *fh, *ih, *iw;
};

// One direction over the arrays of `g`, in shared memory; lam is the h x w
// diagonal of the spectral direction.  The arrays are a contiguous batch,
// indexed arrays (element offsets) or the tiles of an image (leading
// dimensions multiples of 4).  In place is allowed.
cudaError_t small_dense_run(int h, int w, Dir dir, const SmallTables &t, const float *lam, const ExecGeom &g,
                            cudaStream_t stream);

}  // namespace bdct
