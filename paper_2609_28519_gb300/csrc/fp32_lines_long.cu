// The line engine's kernels of 1024 points and more.
#include <cuda_runtime.h>

#include "fp32_lines_kernel.cuh"

namespace bdct {

cudaError_t lines_long_init_table(const float *d_table) { return init_cos_table(d_table); }
cudaError_t lines_long_init_table3(const float *d_table) { return init_cos_table3(d_table); }

cudaError_t lines_long_pass(int n, LinesMode mode, const LinesCall &c, cudaStream_t stream)
{
    switch (n) {
        case 1024: return lines_run<1024>(mode, c, stream);
        case 1536: return lines_run<1536>(mode, c, stream);
        case 2048: return lines_run<2048>(mode, c, stream);
        case 4096: return lines_run<4096>(mode, c, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace bdct
