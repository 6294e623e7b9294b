// Separable dense passes through a workspace, any shape (dense_passes.cu).
#pragma once

#include <cuda_runtime.h>

namespace bdct {

// The n x n operator of one direction (1 forward, 2 inverse) and
// normalization, generated in FP64, as the passes read it: its even and odd
// halves (dense_table_floats(n) floats, 16-byte aligned).
size_t dense_table_floats(int n);
cudaError_t dense_gen_table(float *t, int n, int direction, int norm, cudaStream_t stream);

// One pass over `count` h x w arrays: every row (rows = true, length w) or
// every column (length h) multiplied by the table's operator; `inverse` as
// the table's direction.  in_off / out_off index the arrays (element offsets)
// or are null for contiguous ones; lam, if not null (forward columns only),
// multiplies output (k, l) by lam[k * w + l]: the spectrum times the diagonal
// (Prop. 1, Eq. 4).  w is a multiple of 4, every array 16-byte aligned; in
// and out are distinct.
struct DensePass {
    const float *in;
    float *out;
    const float *table;
    int h, w;
    long long count;
    bool rows, inverse;
    const long long *in_off = nullptr, *out_off = nullptr;
    const float *lam = nullptr;
};
cudaError_t dense_pass(const DensePass &d, cudaStream_t stream);

}  // namespace bdct
