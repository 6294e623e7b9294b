// Allocation-free entry point: the separable route with fixed scratch.
//
// Every other entry point needs a plan, and creating a plan calls cudaMalloc
// for its tables and workspace.  Some callers cannot do that: a process whose
// device memory is entirely handed out by another allocator (a framework's
// caching allocator, a pre-reserved pool), code that must not trigger the
// device-wide synchronization that cudaMalloc/cudaFree can imply, or a
// deployment that must know its full device-memory footprint at load time.
// For them this file offers one entry point that needs no plan and allocates
// nothing: it runs the separable dense route (operator matrices, then a row
// pass and a column pass through an intermediate buffer) with all of its
// scratch -- the operator tables and the intermediates -- in one
// file-scope device array of fixed size.
//
// Host code may not pass that array's name to a kernel: on the host the name
// is only a stand-in, not a device address.  The first call on each device
// therefore looks the address up once with cudaGetSymbolAddress (with that
// device current) and every launch receives that pointer.
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "bdct_internal.h"
#include "dense_passes.h"

namespace bdct {

// 8 MiB of scratch per device, held by every GPU that loads the library
// until the process exits.
constexpr size_t kNoAllocScratchFloats = size_t(2) << 20;
constexpr int kNoAllocMaxSide = 512;

static __device__ __align__(256) float g_noalloc_scratch[kNoAllocScratchFloats];

static std::mutex g_noalloc_mutex;
static float *g_noalloc_ptr[64];

// Device address of the scratch array for the current device (set up on the
// first call per device).
static cudaError_t noalloc_scratch(int dev, float **out)
{
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = static_cast<float *>(p);
    }
    *out = g_noalloc_ptr[dev];
    return cudaSuccess;
}

}  // namespace bdct

extern "C" int bdct_execute_noalloc(int rows, int cols, unsigned kind, int norm, const float *in, float *out,
                                    size_t batch, void *stream)
{
    using namespace bdct;
    if (rows < 1 || cols < 1) return BDCT_ERR_INVALID_ARG;
    if (kind != BDCT_FORWARD && kind != BDCT_INVERSE && kind != BDCT_ROUNDTRIP) return BDCT_ERR_INVALID_ARG;
    if (norm != BDCT_NORM_ORTHO && norm != BDCT_NORM_NONE) return BDCT_ERR_INVALID_ARG;
    if (rows > kNoAllocMaxSide || cols > kNoAllocMaxSide || cols % 4 != 0) return BDCT_ERR_UNSUPPORTED_SHAPE;
    if (batch == 0) return BDCT_OK;
    if (!in || !out) return BDCT_ERR_INVALID_ARG;
    if (((uintptr_t)in | (uintptr_t)out) & 15u) return BDCT_ERR_ALIGN;
    const size_t hw = (size_t)rows * cols;
    if (batch > (size_t)INT64_MAX / (hw * sizeof(float))) return BDCT_ERR_INVALID_ARG;
    {
        const uintptr_t a = (uintptr_t)in, b = (uintptr_t)out, n = batch * hw * sizeof(float);
        if (a != b && a < b + n && b < a + n) return BDCT_ERR_ALIAS;
    }

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return BDCT_ERR_CUDA;
    float *scratch = nullptr;
    e = noalloc_scratch(dev, &scratch);
    if (e != cudaSuccess) return BDCT_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;

    // scratch layout: operator tables first, then the intermediates
    const size_t th = dense_table_floats(rows), per_dir = th + dense_table_floats(cols);
    const bool rt = kind == BDCT_ROUNDTRIP;
    const size_t mats = rt ? 2 * per_dir : per_dir;
    const int nbuf = rt ? 2 : 1;
    const size_t room = kNoAllocScratchFloats - mats;
    const long long chunk = (long long)(room / (hw * nbuf));
    if (chunk < 1) return BDCT_ERR_UNSUPPORTED_SHAPE;
    float *op_h = scratch, *op_w = scratch + th;
    float *w1 = scratch + mats, *w2 = w1 + (size_t)chunk * hw;

    // The tables are regenerated by every call (FP64 cosines, rounded once
    // to FP32), so nothing left by an earlier call is ever read; no part of
    // the scratch needs to start at zero.
    if (!rt) {
        const int direction = kind == BDCT_FORWARD ? 1 : 2;
        e = dense_gen_table(op_h, rows, direction, norm, s);
        if (e == cudaSuccess) e = dense_gen_table(op_w, cols, direction, norm, s);
    } else {
        // the round trip is normalized: orthonormal forward core, then its adjoint
        e = dense_gen_table(op_h, rows, 1, BDCT_NORM_ORTHO, s);
        if (e == cudaSuccess) e = dense_gen_table(op_w, cols, 1, BDCT_NORM_ORTHO, s);
        if (e == cudaSuccess) e = dense_gen_table(op_h + per_dir, rows, 2, BDCT_NORM_ORTHO, s);
        if (e == cudaSuccess) e = dense_gen_table(op_w + per_dir, cols, 2, BDCT_NORM_ORTHO, s);
    }
    if (e != cudaSuccess) return BDCT_ERR_CUDA;

    for (long long b0 = 0; b0 < (long long)batch; b0 += chunk) {
        const long long nb = ((long long)batch - b0) < chunk ? ((long long)batch - b0) : chunk;
        const float *src = in + b0 * (long long)hw;
        float *dst = out + b0 * (long long)hw;
        const bool inv = kind == BDCT_INVERSE;
        e = dense_pass({src, w1, op_w, rows, cols, nb, true, inv}, s);
        if (!rt) {
            if (e == cudaSuccess) e = dense_pass({w1, dst, op_h, rows, cols, nb, false, inv}, s);
        } else {
            if (e == cudaSuccess) e = dense_pass({w1, w2, op_h, rows, cols, nb, false, false}, s);
            if (e == cudaSuccess) e = dense_pass({w2, w1, op_h + per_dir, rows, cols, nb, false, true}, s);
            if (e == cudaSuccess) e = dense_pass({w1, dst, op_w + per_dir, rows, cols, nb, true, true}, s);
        }
        if (e != cudaSuccess) return BDCT_ERR_CUDA;
    }
    return BDCT_OK;
}
