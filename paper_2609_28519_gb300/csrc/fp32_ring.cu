// FP32 ring kernel for 64x64 arrays (the other shapes of sides 64 and 128 run
// in fp32_block.cu, which measured 0.77 / 0.77 / 0.44 / 0.40 of HBM on 64x64
// against 0.90 / 0.91 / 0.76 / 0.60 here: forward, inverse, round trip,
// spectral, 512 MiB).
//
// What is computed: Eq. 2 of the BRiDCT paper, C(X) = Q_h X Q_w^T (forward,
// DCT-II), C^{-1}(Y) = Q_h^T Y Q_w (inverse, DCT-III) and the normalized
// round trip (Prop. 1: forward core, E_n^2, adjoint core per axis), one read
// and one write of every element, both passes on chip.
//
// Organization (warp-specialized, one persistent CTA per SM):
//  * one producer warp keeps a ring of S shared-memory slots full, one array
//    per slot.  Contiguous batches and image tiles move by TMA tensor copies
//    (boxes of 32 columns x all rows, 128-byte swizzle), completing on the
//    slot's mbarrier, and leave by TMA tensor stores; the producer refills a
//    slot with the array S positions ahead once its stores have read it.
//    Indexed batches (ragged classes, arrays at arbitrary offsets) move by
//    16-byte cp.async copies placed at the same swizzled positions and leave
//    by vector stores;
//  * NG consumer groups (named barriers, no CTA-wide synchronization) take
//    the slots round robin, about three slots per group (two for the round
//    trips, which run more groups), so each group's next arrays are in
//    flight while it computes; a group transforms every row of its array,
//    then every column, in place.
//
// Slot layout (the GPU counterpart of the paper's padded stride, Section
// 3.2): columns 32b .. 32b+31 of all rows form box b; row r of a box is 128
// bytes, whose 16-byte chunk k sits at chunk position k XOR (r mod 8).  Eight
// consecutive rows at one logical chunk, and 32 consecutive columns of one
// row, then fall into distinct banks, so the row pass (one row per thread,
// 16-byte accesses) and the column pass (one column per thread) are both
// free of bank conflicts.
//
// Each line runs whole in one thread (dct_cores.cuh).
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>

#include "bdct_internal.h"
#include "dct_cores.cuh"
#include "ptx.cuh"

namespace bdct {

cudaError_t ring_init_table(const float *d_table) { return init_cos_table(d_table); }

bool ring_supported(int rows, int cols)
{
    return rows == 64 && cols == 64;
}

constexpr int kRingMaxSmem = 232448;  // 227 KiB, the opt-in limit per CTA

// The group count depends on the direction; the group, slot and box sizes do
// not, and the helpers that use only those take the default.
template <int DIR = DIR_FWD>
struct RingCfg {
    static constexpr int H = 64, W = 64;
    static constexpr int GT = 64;       // threads per consumer group (one line each)
    static constexpr int GW = GT / 32;  // warps per consumer group
    static constexpr int SLOT_BYTES = H * W * 4;
    static constexpr int SLOT_FLOATS = H * W;
    static constexpr int BOX_BYTES = H * 128;  // 32 columns x H rows
    // spectral direction: the folded diagonal staged once per CTA
    static constexpr int LAM_BYTES = DIR == DIR_SPEC ? H * W * 4 : 0;
    static constexpr int S_MAX = (kRingMaxSmem - 2048 - LAM_BYTES) / SLOT_BYTES;
    // about three slots per group, so that a group's next arrays load while
    // it computes; the slot count is a multiple of the group count (a group
    // always reuses slots it consumed itself, which the slot barriers' parity
    // tracking relies on)
    // (round trips, twice the arithmetic per array, run seven groups over two
    // slots each: 0.67 -> 0.76 of HBM, while forward and inverse measured
    // 0.90 -> 0.81 that way; the spectral direction, four 1D cores per line
    // pair like the round trip plus the diagonal, six over the thirteen slots
    // left beside the diagonal)
    static constexpr int NG = DIR == DIR_RT ? 7 : DIR == DIR_SPEC ? 6 : S_MAX / 3;
    static constexpr int S = (S_MAX / NG) * NG;
    static constexpr int PROD_WARP = NG * GW;
    static constexpr int THREADS = (NG * GW + 1) * 32;
    // slots start 1024-byte aligned (128-byte swizzle atoms)
    static constexpr size_t SMEM = 1024 + (size_t)S * SLOT_BYTES + (size_t)2 * S * 8 + LAM_BYTES;
    static_assert(GT % 32 == 0 && S >= 2 && S % NG == 0, "ring shape");
    static_assert(SMEM <= (size_t)kRingMaxSmem, "shared memory");
    static_assert(BOX_BYTES % 1024 == 0, "swizzle atoms");
};

// Named barrier over the threads of one consumer group.
__device__ __forceinline__ void group_sync(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Named barrier that also ANDs a predicate over the group.
__device__ __forceinline__ bool group_and(int id, int nthreads, bool v)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.and.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v), "r"(id), "r"(nthreads)
        : "memory");
    return r != 0;
}

// Slot byte offset of 16-byte chunk k (k < W/4) of row r.
template <int H>
__device__ __forceinline__ uint32_t sw_chunk(int r, int k)
{
    return (uint32_t)((k >> 3) * (H * 128) + r * 128 + (((k & 7) ^ (r & 7)) << 4));
}

// Row view: chunk k of a fixed row r is at base + (k / 8) * BOX_BYTES + o[k % 8].
struct RowView {
    uint32_t o[8];
    __device__ __forceinline__ explicit RowView(int r)
    {
#pragma unroll
        for (int t = 0; t < 8; ++t) o[t] = (uint32_t)(r * 128 + ((t ^ (r & 7)) << 4));
    }
};

// Column view: the float at slot position p of row i is at base + i * 128 + o[i % 8].
template <int H>
struct ColView {
    uint32_t o[8];
    __device__ __forceinline__ explicit ColView(int p)
    {
        const int pc = p >> 2;
#pragma unroll
        for (int t = 0; t < 8; ++t) o[t] = (uint32_t)((pc >> 3) * (H * 128) + (((pc & 7) ^ t) << 4) + (p & 3) * 4);
    }
};

template <typename T>
__device__ __forceinline__ T &at(char *base, uint32_t off)
{
    return *reinterpret_cast<T *>(base + off);
}

// ---------------------------------------------------------------- one array
// The two passes run in one loop, so that the 1D cores (the largest part of
// the code) exist once: pass 0 takes rows, pass 1 columns, in place.
//
// The spectral direction (64 x 64, Prop. 1 / Eq. 4 with a general diagonal)
// takes three passes with the unscaled cores: rows forward; columns forward,
// times the column's entries of the folded diagonal lam_s (E_h Lambda E_w
// with every scale of both axes in it), adjoint; rows adjoint.
template <int DIR>
__device__ __forceinline__ void ring_array(char *slot, int gt, int bar, const DirScales &sc, const float *lam_s)
{
    using C = RingCfg<>;
    constexpr int BB = C::BOX_BYTES;
    constexpr int NPASS = DIR == DIR_SPEC ? 3 : 2;
#pragma unroll 1
    for (int pass = 0; pass < NPASS; ++pass) {
        const AxisScale s = (pass & 1) ? sc.h : sc.w;
        // one thread per line; row r (passes 0 and 2) or column c (pass 1)
        float x[64];
        if ((pass & 1) == 0) {
            const RowView rv(gt);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const float4 t = at<float4>(slot, (k >> 3) * BB + rv.o[k & 7]);
                x[4 * k] = t.x; x[4 * k + 1] = t.y; x[4 * k + 2] = t.z; x[4 * k + 3] = t.w;
            }
        } else {
            const ColView<64> cv(gt);
#pragma unroll
            for (int i = 0; i < 64; ++i) x[i] = at<float>(slot, i * 128 + cv.o[i & 7]);
        }
        if constexpr (DIR == DIR_SPEC) {
            if (pass == 1) {
                line_op<64, CORE_FWD>(x, s);
#pragma unroll
                for (int k = 0; k < 64; ++k) x[k] *= lam_s[k * 64 + gt];
                line_op<64, CORE_INV>(x, s);
            } else if (pass == 0) {
                line_op<64, CORE_FWD>(x, s);
            } else {
                line_op<64, CORE_INV>(x, s);
            }
        } else {
            line_op<64, DIR>(x, s);
        }
        if ((pass & 1) == 0) {
            const RowView rv(gt);
#pragma unroll
            for (int k = 0; k < 16; ++k)
                at<float4>(slot, (k >> 3) * BB + rv.o[k & 7]) =
                    make_float4(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3]);
        } else {
            const ColView<64> cv(gt);
#pragma unroll
            for (int i = 0; i < 64; ++i) at<float>(slot, i * 128 + cv.o[i & 7]) = x[i];
        }
        group_sync(bar, C::GT);
    }
}

// ---------------------------------------------------------------- kernel
struct RingParams {
    CUtensorMap map_in, map_out;  // contiguous and tiled batches (TMA)
    const float *in;
    float *out;
    long long count;          // arrays or tiles
    int tiles_per_row;        // tiled only
    int tiled;
    int indexed;              // arrays at in + in_off[a], out + out_off[a] (cp.async path)
    long long ld_in, ld_out;  // tiled only (floats)
    DirScales sc;
    unsigned int *status;
    const long long *in_off, *out_off;
    const float *lam;         // spectral direction: the folded diagonal (H x W), else null
};

// TMA coordinates (x: column, y: row) of the first element of array or tile a.
template <int H, int W>
__device__ __forceinline__ void ring_coords(const RingParams &p, long long a, int &x, int &y)
{
    if (p.tiled) {
        const long long br = a / p.tiles_per_row, bc = a - br * p.tiles_per_row;
        x = (int)(bc * W);
        y = (int)(br * H);
    } else {
        x = 0;
        y = (int)(a * H);
    }
}

template <int DIR>
__global__ void __launch_bounds__(RingCfg<DIR>::THREADS, 1) k_ring(const __grid_constant__ RingParams p)
{
    using C = RingCfg<DIR>;
    constexpr int H = C::H, W = C::W;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // 1024-byte aligned slots
    const uint32_t raw = smem_u32(smem_raw);
    char *smem = reinterpret_cast<char *>(smem_raw) + (((raw + 1023u) & ~1023u) - raw);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + C::S * C::SLOT_BYTES);
    uint64_t *done = full + C::S;
    float *lam_s = reinterpret_cast<float *>(done + C::S);  // spectral only (16-byte aligned)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long grid = gridDim.x;
    const long long first = blockIdx.x;
    const int n = first < p.count ? (int)((p.count - first + grid - 1) / grid) : 0;

    if (tid == 0) {
        for (int s = 0; s < C::S; ++s) {
            mbar_init(&full[s], p.indexed ? 32 : 1);  // 32 lane arrivals (cp.async) or one expect_tx
            mbar_init(&done[s], 1);
        }
        fence_mbar_init();
    }
    pdl_launch_dependents();
    pdl_wait_prerequisites();
    if constexpr (DIR == DIR_SPEC) {
        for (int e = tid; e < H * W; e += C::THREADS) lam_s[e] = __ldg(p.lam + e);
    }
    __syncthreads();

    if (warp == C::PROD_WARP) {
        // ---------------- producer
        bool ok = true;
        int filled = 0, consumed = 0;
        if (!p.indexed) {
            // TMA tensor copies issued by lane 0
            auto fill = [&](int j) {
                const int s = j % C::S;
                char *slot = smem + s * C::SLOT_BYTES;
                int x, y;
                ring_coords<H, W>(p, first + (long long)j * grid, x, y);
                mbar_arrive_expect_tx(&full[s], (uint32_t)C::SLOT_BYTES);
#pragma unroll
                for (int b = 0; b < W / 32; ++b) tensor_load_2d(slot + b * C::BOX_BYTES, &p.map_in, x + 32 * b, y, &full[s]);
            };
            if (lane == 0) {
                const int pro = n < C::S ? n : C::S;
                for (int j = 0; j < pro; ++j) fill(j);
                filled = pro;
                for (int j = 0; j < n; ++j) {
                    const int s = j % C::S;
                    if (!mbar_wait_bounded(&done[s], (uint32_t)((j / C::S) & 1))) {
                        record_timeout(p.status);
                        ok = false;
                        break;
                    }
                    consumed = j + 1;
                    const char *slot = smem + s * C::SLOT_BYTES;
                    int x, y;
                    ring_coords<H, W>(p, first + (long long)j * grid, x, y);
#pragma unroll
                    for (int b = 0; b < W / 32; ++b) tensor_store_2d(&p.map_out, x + 32 * b, y, slot + b * C::BOX_BYTES);
                    bulk_commit();
                    // refill the slot stored one step earlier once its stores have read it
                    if (j >= 1 && j - 1 + C::S < n) {
                        bulk_wait_read<1>();
                        fill(j - 1 + C::S);
                        filled = j + C::S;
                    }
                }
                bulk_wait<0>();
            }
        } else {
            // 16-byte cp.async copies by all lanes, at the swizzled positions
            constexpr int Q = W / 4;  // chunks per row
            auto fill = [&](int j) {
                const long long a = first + (long long)j * grid;
                const int s = j % C::S;
                char *slot = smem + s * C::SLOT_BYTES;
                const float *src = p.in + p.in_off[a];
#pragma unroll 8
                for (int t = lane; t < H * Q; t += 32) {
                    const int r = t / Q, k = t - r * Q;
                    cp_async16(slot + sw_chunk<H>(r, k), src + r * W + 4 * k);
                }
                cp_async_mbar_arrive(&full[s]);
            };
            const int pro = n < C::S ? n : C::S;
            for (int j = 0; j < pro; ++j) fill(j);
            filled = pro;
            for (int j = 0; j < n; ++j) {
                const int s = j % C::S;
                ok = __all_sync(0xffffffffu, mbar_wait_bounded(&done[s], (uint32_t)((j / C::S) & 1)));
                if (!ok) {
                    if (lane == 0) record_timeout(p.status);
                    break;
                }
                consumed = j + 1;
                const long long a = first + (long long)j * grid;
                float *dst = p.out + p.out_off[a];
                const char *slot = smem + s * C::SLOT_BYTES;
#pragma unroll 8
                for (int t = lane; t < H * Q; t += 32) {
                    const int r = t / Q, k = t - r * Q;
                    *reinterpret_cast<float4 *>(dst + r * W + 4 * k) =
                        *reinterpret_cast<const float4 *>(slot + sw_chunk<H>(r, k));
                }
                __syncwarp();  // every lane's reads of the slot done before any lane refills it
                if (j + C::S < n) {
                    fill(j + C::S);
                    filled = j + C::S + 1;
                }
            }
            cp_async_wait_all();
        }
        if (!__all_sync(0xffffffffu, ok)) {
            // loads issued for arrays never consumed land (bounded) before the CTA exits
            if (lane == 0)
                for (int j = consumed; j < filled; ++j)
                    if (!mbar_wait_bounded(&full[j % C::S], (uint32_t)((j / C::S) & 1))) break;
        }
        return;
    }

    // ---------------- consumers
    const int g = warp / C::GW;
    const int gt = tid - g * C::GT;
    const int bar = 1 + g;
    for (int j = g; j < n; j += C::NG) {
        const int s = j % C::S;
        bool ok = mbar_wait_bounded(&full[s], (uint32_t)((j / C::S) & 1));
        ok = group_and(bar, C::GT, ok);
        if (!ok) {
            if (gt == 0) record_timeout(p.status);
            break;
        }
        char *slot = smem + s * C::SLOT_BYTES;
        ring_array<DIR>(slot, gt, bar, p.sc, lam_s);  // ends with a group barrier
        fence_proxy_async_smem();  // the TMA store reads the slot through the async proxy
        group_sync(bar, C::GT);
        if (gt == 0) mbar_arrive(&done[s]);
    }
}

// ---------------------------------------------------------------- host side
template <int DIR>
static cudaError_t ring_launch_one(const DirScales &sc, const ExecGeom &g, unsigned int *status,
                                   cudaStream_t stream)
{
    using C = RingCfg<DIR>;
    constexpr int H = C::H, W = C::W;
    auto kern = k_ring<DIR>;
    static DeviceLaunchCache cache;
    int dev = 0, bps_dev = 0, num_sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cache.get(
        dev,
        [&](int d, int &bps, int &sms) {
            cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
            if (r == cudaSuccess) r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, C::THREADS, C::SMEM);
            if (r == cudaSuccess && bps < 1) r = cudaErrorInvalidConfiguration;
            if (r == cudaSuccess) r = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d);
            if (r == cudaSuccess && debug_enabled())
                fprintf(stderr, "[bdct] k_ring<%d>: %d slots of %d B, %d groups x %d warps + producer, smem %zu B\n", DIR,
                        C::S, C::SLOT_BYTES, C::NG, C::GW, C::SMEM);
            return r;
        },
        &bps_dev, &num_sms);
    if (e != cudaSuccess) return e;
    (void)bps_dev;
    if (g.count <= 0) return cudaSuccess;
    RingParams p{};
    p.in = g.in;
    p.out = g.out;
    p.count = g.count;
    p.tiled = g.tiled;
    p.tiles_per_row = g.tiles_per_row;
    p.ld_in = g.ld_in;
    p.ld_out = g.ld_out;
    p.sc = sc;
    p.status = status;
    p.in_off = g.in_off;
    p.out_off = g.out_off;
    p.lam = g.lam;
    if (DIR == DIR_SPEC && !g.lam) return cudaErrorInvalidValue;
    p.indexed = (g.in_off != nullptr || g.out_off != nullptr) ? 1 : 0;
    if (p.indexed) {
        if (!g.in_off || !g.out_off) return cudaErrorInvalidValue;
    } else if (g.tiled) {
        const unsigned long long rows = (unsigned long long)(g.count / g.tiles_per_row) * H;
        const unsigned long long cols = (unsigned long long)g.tiles_per_row * W;
        e = tma_map_2d(&p.map_in, g.in, rows, cols, (unsigned long long)g.ld_in, H);
        if (e == cudaSuccess) e = tma_map_2d(&p.map_out, g.out, rows, cols, (unsigned long long)g.ld_out, H);
        if (e != cudaSuccess) return e;
    } else {
        const unsigned long long rows = (unsigned long long)g.count * H;
        e = tma_map_2d(&p.map_in, g.in, rows, W, W, H);
        if (e == cudaSuccess) e = tma_map_2d(&p.map_out, g.out, rows, W, W, H);
        if (e != cudaSuccess) return e;
    }
    long long grid = num_sms;
    if (grid > g.count) grid = g.count;
    if ((g.count + grid - 1) / grid > 0x7fffff00LL) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(C::THREADS);
    cfg.dynamicSmemBytes = C::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p);
}

cudaError_t ring_launch(Dir dir, const DirScales &sc, const ExecGeom &g, unsigned int *status, cudaStream_t stream)
{
    switch (dir) {
        case DIR_FWD: return ring_launch_one<DIR_FWD>(sc, g, status, stream);
        case DIR_INV: return ring_launch_one<DIR_INV>(sc, g, status, stream);
        case DIR_SPEC: return ring_launch_one<DIR_SPEC>(sc, g, status, stream);
        default: return ring_launch_one<DIR_RT>(sc, g, status, stream);
    }
}

}  // namespace bdct
