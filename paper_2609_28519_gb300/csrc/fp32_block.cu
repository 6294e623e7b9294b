// On-chip FP32 kernels for sides 64 and 128: 128 x 128, 64 x 128 and 128 x 64
// arrays, one read and one write of every element.
//
// What is computed: Eq. 2 of the BRiDCT paper, C(X) = Q_h X Q_w^T (forward,
// DCT-II), C^{-1}(Y) = Q_h^T Y Q_w (inverse, DCT-III), the normalized round
// trip and the spectral composition (Prop. 1), with the line steps of
// line_steps.cuh along both axes.
//
// Organization: a CTA holds one array in shared memory.  The forward's row
// pass reads the rows where bulk copies put them, exchanges in place and
// writes its coefficients transposed over the same buffer; the column pass
// runs on those rows the same way and stores its outputs straight to global
// memory, a warp writing 32 consecutive coefficients of one row.  The inverse
// runs the transposed steps: coefficients straight into registers, the column
// pass, the row pass, and one bulk store per row.  The spectral direction joins
// the two in the middle: the column pass's coefficients stay in registers, take
// the diagonal, and go back through the adjoint steps in place.  The round trip
// runs forward and back along the rows, is transposed, and the same along the
// columns: one transposition, and the range of one axis (joined in the middle
// as the spectral direction is, a constant 128 x 128 array overflowed from
// 2^118, this way from 2^121).
//
// Every thread has exactly one couple of the last step (two short FFTs of 8
// points in packed halves, 32 values), so the transposed write needs no
// second buffer: all units are in registers before any coefficient is
// written.  512 threads at 64 registers, two CTAs per SM for 128 x 128: one
// array's copies overlap the other's arithmetic.
//
// What bounds it: 40 bytes of shared-memory traffic and about 30
// multiply-adds per element, against 8 bytes of HBM traffic, and the latency
// between the barriers of one array (shared wavefronts 40-50%, FMA pipe 39-57%).
// Against the form before it (one CTA of eight warps per SM over a ring of
// arrays), 512 MiB, us: 128 x 128 forward 424 -> 215, inverse 506 -> 245, round
// trip 868 -> 324, spectral 974 -> 386; 64 x 128 272 -> 207, 340 -> 206, 536 ->
// 309, 642 -> 347.  64 x 64 is faster in fp32_ring.cu.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <type_traits>

#include "bdct_internal.h"
#include "fp32_block.h"
#include "fp32_lines.h"
#include "line_steps.cuh"
#include "ptx.cuh"

namespace bdct {

namespace {

// Tables of 64 and 128 points, for the orthonormal scale and the unnormalized
// pair's.  A warp's 32 lanes take 32 lines of one couple, so every entry is
// uniform over the warp and comes through the constant cache: in shared memory
// the tables took a quarter of its wavefronts (128 x 128 forward 242 -> 220 us,
// round trip 437 -> 375, 8192 arrays).
constexpr int kTabMax = LineSplit<128>::TAB;
__constant__ float4 c_line[4 * kTabMax];  // [plain][64 or 128]

template <int H, int W>
struct BlockCfg {
    using AW = LineSplit<W>;
    using AH = LineSplit<H>;
    static constexpr int THREADS = H * (AW::C / 2);  // one couple of the last step each, in both passes
    static constexpr int GW = THREADS / H, GH = THREADS / W;  // threads per line
    static constexpr int NB = 1024 / THREADS;  // CTAs per SM: 64 registers a thread
    static constexpr int PW = W + 4, PH = H + 4;  // row pitch before and after the transposition (floats)
    static constexpr int BUF = H * PW > W * PH ? H * PW : W * PH;
    static constexpr size_t SMEM = (size_t)BUF * 4 + 16;
    static_assert(GH == AH::C / 2 && GW == AW::C / 2, "one couple each");
    static_assert(THREADS >= H && H % 32 == 0 && W % 32 == 0, "lanes");
    static_assert(AW::R2 == 1 && AH::R2 == 1, "two steps");
};

struct BlockParams {
    const float *in;
    float *out;
    long long count;          // arrays or tiles
    int tiles_per_row;        // tiled only
    long long ld_in, ld_out;  // tiled only (floats)
    const long long *in_off, *out_off;
    DirScales sc;             // twice the scales of the forward's outputs or the inverse's inputs
    const float *lam;         // spectral: Lambda (H x W), else null
    unsigned int *status;
    int plain;                // the unnormalized pair's scales
};

// First step of this thread's couples of line `row` (in place), and its transpose.
template <int N, int G>
__device__ __forceinline__ void first_step(float4 *row, int g, const float4 *t1)
{
    using S = LineSplit<N>;
#pragma unroll
    for (int cc = g; cc < S::M1 / 2; cc += G) {
        float4 x[S::R1 / 2], y[S::R1 / 2];
#pragma unroll
        for (int j = 0; j < S::R1 / 2; ++j) {
            x[j] = row[cc + S::M1 * j];
            y[j] = row[S::M1 - 1 - cc + S::M1 * j];
        }
        step_forward<S::R1, S::M1, true>(x, y, t1 + cc);
#pragma unroll
        for (int j = 0; j < S::R1 / 2; ++j) {
            row[cc + S::M1 * j] = x[j];
            row[S::M1 - 1 - cc + S::M1 * j] = y[j];
        }
    }
}

template <int N, int G>
__device__ __forceinline__ void first_step_adjoint(float4 *row, int g, const float4 *t1)
{
    using S = LineSplit<N>;
#pragma unroll
    for (int cc = g; cc < S::M1 / 2; cc += G) {
        float4 x[S::R1 / 2], y[S::R1 / 2];
#pragma unroll
        for (int j = 0; j < S::R1 / 2; ++j) {
            x[j] = row[cc + S::M1 * j];
            y[j] = row[S::M1 - 1 - cc + S::M1 * j];
        }
        step_adjoint<S::R1, S::M1, true>(x, y, t1 + cc);
#pragma unroll
        for (int j = 0; j < S::R1 / 2; ++j) {
            row[cc + S::M1 * j] = x[j];
            row[S::M1 - 1 - cc + S::M1 * j] = y[j];
        }
    }
}

// The line's first-step adjoint with its results handed on instead: read() once
// every unit of this thread's couples is in registers, put(i, v) for element i.
template <int N, int G, typename R, typename P>
__device__ __forceinline__ void first_step_adjoint_out(const float4 *row, int g, const float4 *t1, R &&read, P &&put)
{
    using S = LineSplit<N>;
    constexpr int NC = S::M1 / 2 / G;
    static_assert(NC * G == S::M1 / 2, "couples");
    float4 x[NC][S::R1 / 2], y[NC][S::R1 / 2];
#pragma unroll
    for (int i = 0; i < NC; ++i)
#pragma unroll
        for (int j = 0; j < S::R1 / 2; ++j) {
            x[i][j] = row[g + G * i + S::M1 * j];
            y[i][j] = row[S::M1 - 1 - g - G * i + S::M1 * j];
        }
    read();
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        step_adjoint<S::R1, S::M1, true>(x[i], y[i], t1 + g + G * i);
#pragma unroll
        for (int j = 0; j < S::R1 / 2; ++j) {
            const int p = 4 * (g + G * i + S::M1 * j), q = 4 * (S::M1 - 1 - g - G * i + S::M1 * j);
            put(p, x[i][j].x); put(p + 1, x[i][j].y); put(p + 2, x[i][j].z); put(p + 3, x[i][j].w);
            put(q, y[i][j].x); put(q + 1, y[i][j].y); put(q + 2, y[i][j].z); put(q + 3, y[i][j].w);
        }
    }
}

// Units of couple c: columns c and C - c (C/2 for c = 0).
template <int N>
__device__ __forceinline__ void couple_units(float4 *row, int c, float4 *&px, float4 *&pw)
{
    using S = LineSplit<N>;
    px = row + S::M1 * c;
    pw = row + S::M1 - 1 + S::M1 * ((c ? S::C - c : S::C / 2) - S::R1 / 2);
}

// The couple's coefficients and back, in place: the middle of a line's round trip.
template <int N>
__device__ __forceinline__ void couple_round_trip(float4 *row, int c, SplitTable ts, AxisScale sc)
{
    using S = LineSplit<N>;
    float4 x[4], w[4], *px, *pw;
    couple_units<N>(row, c, px, pw);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        x[m] = px[m];
        w[m] = pw[-m];
    }
    float2 dr[8], di[8], a[8], b[8];
    last_forward<8>(x, w, dr, di);
    split_forward<8, S::C>(c, dr, di, ts, sc, a, b);
    split_adjoint<8, S::C>(c, a, b, ts, sc, dr, di);
    last_adjoint<8>(x, w, dr, di);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        px[m] = x[m];
        pw[-m] = w[m];
    }
}

template <int H, int W, int DIR, bool TILED>
__global__ void __launch_bounds__(BlockCfg<H, W>::THREADS, BlockCfg<H, W>::NB) k_block(const BlockParams p)
{
    using C = BlockCfg<H, W>;
    using AW = LineSplit<W>;
    using AH = LineSplit<H>;
    constexpr bool FWD = DIR != DIR_INV, INV = DIR != DIR_FWD;
    extern __shared__ __align__(128) float bsm[];
    const float4 *tw = c_line + (2 * p.plain + (W == 128)) * kTabMax, *th = c_line + (2 * p.plain + (H == 128)) * kTabMax;
    uint64_t *bar = reinterpret_cast<uint64_t *>(bsm + C::BUF);
    const int tid = threadIdx.x;
    // row pass: row rw, couple gw; column pass: column rh, couple gh
    const int rw = tid % H, gw = __shfl_sync(0xffffffffu, tid / H, 0), rh = tid % W, gh = __shfl_sync(0xffffffffu, tid / W, 0);
    float4 *row_w = reinterpret_cast<float4 *>(bsm + rw * C::PW);
    float4 *row_h = reinterpret_cast<float4 *>(bsm + rh * C::PH);
    const SplitTable sw{tw + AW::U1, reinterpret_cast<const float2 *>(tw + AW::U1 + AW::L / 2)};
    const SplitTable sh{th + AH::U1, reinterpret_cast<const float2 *>(th + AH::U1 + AH::L / 2)};

    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    pdl_launch_dependents();
    pdl_wait_prerequisites();
    __syncthreads();

    using Ld = typename std::conditional<TILED, long long, int>::type;  // offsets fold into the instructions for arrays
    const Ld ldi = TILED ? (Ld)p.ld_in : W, ldo = TILED ? (Ld)p.ld_out : W;
    auto src_of = [&](long long a) -> const float * {
        if (TILED) return p.in + (a / p.tiles_per_row) * H * p.ld_in + (a % p.tiles_per_row) * W;
        return p.in_off ? p.in + p.in_off[a] : p.in + a * (H * W);
    };
    auto dst_of = [&](long long a) -> float * {
        if (TILED) return p.out + (a / p.tiles_per_row) * H * p.ld_out + (a % p.tiles_per_row) * W;
        return p.out_off ? p.out + p.out_off[a] : p.out + a * (H * W);
    };
    // one bulk copy per row
    auto load = [&](long long a) {
        if (tid < H) {
            if (tid == 0) mbar_arrive_expect_tx(bar, H * W * 4);
            bulk_load(bsm + tid * C::PW, src_of(a) + (long long)tid * ldi, W * 4, bar);
        }
    };
    if (FWD && (long long)blockIdx.x < p.count) load(blockIdx.x);

    uint32_t phase = 0;
    for (long long ar = blockIdx.x; ar < p.count; ar += gridDim.x) {
        const long long next = ar + gridDim.x;
        float2 a[8], b[8];  // the couple's coefficients (R3 = 8 for both lengths)
        // the inverse's next array into L2: its loads go straight to registers
        // (128 x 128 251 -> 243 us; the other directions gain nothing)
        if (DIR == DIR_INV && !TILED && tid == 0 && next < p.count) bulk_prefetch_l2(src_of(next), H * W * 4);
        if constexpr (FWD) {
            const bool ok = mbar_wait_bounded(bar, phase);
            phase ^= 1;
            first_step<W, C::GW>(row_w, gw, tw);
            if (!__syncthreads_and(ok)) {
                // the load did not land in time: record it, give the copies one
                // more bounded wait, and stop
                if (tid == 0) {
                    record_timeout(p.status);
                    mbar_wait_bounded(bar, phase ^ 1);
                }
                return;
            }
            if constexpr (DIR == DIR_RT) {
                // each axis forward and back in turn, so that no coefficient is
                // larger than its own axis makes it
                couple_round_trip<W>(row_w, gw, sw, p.sc.w);
                __syncthreads();
                first_step_adjoint_out<W, C::GW>(
                    row_w, gw, tw, [] { __syncthreads(); }, [&](int i, float v) { bsm[i * C::PH + rw] = v; });
                __syncthreads();
                first_step<H, C::GH>(row_h, gh, th);
                __syncthreads();
                couple_round_trip<H>(row_h, gh, sh, p.sc.h);
                __syncthreads();
                float *o = dst_of(ar) + rh;
                first_step_adjoint_out<H, C::GH>(
                    row_h, gh, th,
                    [&] {  // the next array may land
                        fence_proxy_async_smem();
                        __syncthreads();
                        if (next < p.count) load(next);
                    },
                    [&](int i, float v) { o[i * ldo] = v; });
                continue;
            }
            {
                float4 x[4], w[4], *px, *pw;
                couple_units<W>(row_w, gw, px, pw);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    x[m] = px[m];
                    w[m] = pw[-m];
                }
                __syncthreads();  // every unit read: the coefficients go over them, transposed
                float2 dr[8], di[8];
                last_forward<8>(x, w, dr, di);
                split_forward<8, AW::C>(gw, dr, di, sw, p.sc.w, a, b);
                const SlotIndex<AW> at(gw);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    bsm[at.ax(k) * C::PH + rw] = a[k].x;
                    bsm[at.ay(k) * C::PH + rw] = a[k].y;
                    bsm[at.bx(k) * C::PH + rw] = b[k].x;
                    bsm[at.by(k) * C::PH + rw] = b[k].y;
                }
            }
            __syncthreads();
            first_step<H, C::GH>(row_h, gh, th);
            __syncthreads();
            float4 x[4], w[4], *px, *pw;
            couple_units<H>(row_h, gh, px, pw);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                x[m] = px[m];
                w[m] = pw[-m];
            }
            if constexpr (DIR == DIR_FWD) {
                // the next array may land
                fence_proxy_async_smem();
                __syncthreads();
                if (next < p.count) load(next);
            }
            float2 dr[8], di[8];
            last_forward<8>(x, w, dr, di);
            split_forward<8, AH::C>(gh, dr, di, sh, p.sc.h, a, b);
        }
        const SlotIndex<AH> at(gh);
        if constexpr (DIR == DIR_FWD) {
            float *o = dst_of(ar) + rh;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                o[at.ax(k) * ldo] = a[k].x;
                o[at.ay(k) * ldo] = a[k].y;
                o[at.bx(k) * ldo] = b[k].x;
                o[at.by(k) * ldo] = b[k].y;
            }
            continue;
        }
        if constexpr (DIR == DIR_INV) {
            const float *q = src_of(ar) + rh;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                a[k].x = __ldcg(q + at.ax(k) * ldi);
                a[k].y = __ldcg(q + at.ay(k) * ldi);
                b[k].x = __ldcg(q + at.bx(k) * ldi);
                b[k].y = __ldcg(q + at.by(k) * ldi);
            }
            // the previous array's stores must have read the buffer
            if (tid < H) bulk_wait_read<0>();
            __syncthreads();
        }
        if constexpr (DIR == DIR_SPEC) {
            const float *l = p.lam + rh;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                a[k].x *= __ldg(l + at.ax(k) * W);
                a[k].y *= __ldg(l + at.ay(k) * W);
                b[k].x *= __ldg(l + at.bx(k) * W);
                b[k].y *= __ldg(l + at.by(k) * W);
            }
        }
        if constexpr (INV) {
            {
                float2 dr[8], di[8];
                float4 x[4], w[4], *px, *pw;
                couple_units<H>(row_h, gh, px, pw);
                split_adjoint<8, AH::C>(gh, a, b, sh, p.sc.h, dr, di);
                last_adjoint<8>(x, w, dr, di);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    px[m] = x[m];
                    pw[-m] = w[m];
                }
            }
            __syncthreads();
            first_step_adjoint<H, C::GH>(row_h, gh, th);
            __syncthreads();
            {
                const SlotIndex<AW> aw(gw);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    a[k].x = bsm[aw.ax(k) * C::PH + rw];
                    a[k].y = bsm[aw.ay(k) * C::PH + rw];
                    b[k].x = bsm[aw.bx(k) * C::PH + rw];
                    b[k].y = bsm[aw.by(k) * C::PH + rw];
                }
                __syncthreads();  // every coefficient read: the units go over them
                float2 dr[8], di[8];
                float4 x[4], w[4], *px, *pw;
                couple_units<W>(row_w, gw, px, pw);
                split_adjoint<8, AW::C>(gw, a, b, sw, p.sc.w, dr, di);
                last_adjoint<8>(x, w, dr, di);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    px[m] = x[m];
                    pw[-m] = w[m];
                }
            }
            __syncthreads();
            first_step_adjoint<W, C::GW>(row_w, gw, tw);
            fence_proxy_async_smem();  // the stores read the buffer through the async proxy
            __syncthreads();
            if (tid < H) {
                bulk_store(dst_of(ar) + (long long)tid * ldo, bsm + tid * C::PW, W * 4);
                bulk_commit();
                if (FWD && next < p.count) bulk_wait_read<0>();
            }
            if constexpr (FWD) {
                // each thread's row lands where its own store has read
                if (next < p.count) load(next);
            }
        }
    }
    if ((DIR == DIR_INV || DIR == DIR_SPEC) && tid < H) bulk_wait<0>();
}

template <int H, int W, int DIR, bool TILED>
cudaError_t block_launch_one(const DirScales &sc, const ExecGeom &g, unsigned int *status, cudaStream_t stream)
{
    using C = BlockCfg<H, W>;
    auto kern = k_block<H, W, DIR, TILED>;
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
                fprintf(stderr, "[bdct] k_block<%d,%d,%d,%d>: %d CTAs/SM x %d threads, smem %zu B\n", H, W, DIR,
                        (int)TILED, bps, C::THREADS, C::SMEM);
            return r;
        },
        &bps_dev, &num_sms);
    if (e != cudaSuccess) return e;
    if (g.count <= 0) return cudaSuccess;
    BlockParams p{};
    p.in = g.in;
    p.out = g.out;
    p.count = g.count;
    p.tiles_per_row = g.tiles_per_row;
    p.ld_in = g.ld_in;
    p.ld_out = g.ld_out;
    p.in_off = g.in_off;
    p.out_off = g.out_off;
    p.sc = sc;
    if (DIR == DIR_RT || DIR == DIR_SPEC) {
        // the orthonormal pair, whatever the plan's normalization
        auto ortho = [](int n) { return AxisScale{(float)std::sqrt(1.0 / n), (float)std::sqrt(2.0 / n)}; };
        p.sc = DirScales{ortho(H), ortho(W)};
    }
    p.lam = g.lam;
    p.plain = p.sc.w.s1 == 2.0f;
    for (AxisScale *a : {&p.sc.h, &p.sc.w}) *a = AxisScale{2.0f * a->s0, 2.0f * a->s1};  // the first steps halve
    p.status = status;
    if (DIR == DIR_SPEC && !g.lam) return cudaErrorInvalidValue;
    long long grid = (long long)bps_dev * num_sms;
    if (grid > g.count) grid = g.count;
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

template <int H, int W, int DIR>
cudaError_t block_tiled(const DirScales &sc, const ExecGeom &g, unsigned int *st, cudaStream_t s)
{
    return g.tiled ? block_launch_one<H, W, DIR, true>(sc, g, st, s) : block_launch_one<H, W, DIR, false>(sc, g, st, s);
}

template <int H, int W>
cudaError_t block_dir(Dir dir, const DirScales &sc, const ExecGeom &g, unsigned int *st, cudaStream_t s)
{
    switch (dir) {
        case DIR_FWD: return block_tiled<H, W, DIR_FWD>(sc, g, st, s);
        case DIR_INV: return block_tiled<H, W, DIR_INV>(sc, g, st, s);
        case DIR_RT: return block_tiled<H, W, DIR_RT>(sc, g, st, s);
        default: return block_tiled<H, W, DIR_SPEC>(sc, g, st, s);
    }
}

}  // namespace

cudaError_t block_init_device(const float *d_table)
{
    cudaError_t e = init_cos_table(d_table);
    float4 *tmp = nullptr;
    const size_t bytes = sizeof(float4) * 4 * kTabMax;
    if (e == cudaSuccess) e = cudaMalloc(&tmp, bytes);
    if (e != cudaSuccess) return e;
    LineTable tables[4];
    for (int i = 0; i < 4; ++i) {
        const int n = i % 2 ? 128 : 64;
        tables[i] = {tmp + i * kTabMax, n, 1, i / 2 ? 2.0 : std::sqrt(2.0 / n)};
    }
    e = cudaMemset(tmp, 0, bytes);
    if (e == cudaSuccess) e = lines_gen_tables(tables, 4, 0);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_line, tmp, bytes, 0, cudaMemcpyDeviceToDevice);
    cudaFree(tmp);
    return e;
}

bool block_supported(int rows, int cols)
{
    return (rows == 64 || rows == 128) && (cols == 64 || cols == 128) && !(rows == 64 && cols == 64);
}

cudaError_t block_launch(int rows, int cols, Dir dir, const DirScales &sc, const ExecGeom &g, unsigned int *status,
                         cudaStream_t stream)
{
    if (rows == 64 && cols == 128) return block_dir<64, 128>(dir, sc, g, status, stream);
    if (rows == 128 && cols == 64) return block_dir<128, 64>(dir, sc, g, status, stream);
    if (rows == 128 && cols == 128) return block_dir<128, 128>(dir, sc, g, status, stream);
    return cudaErrorInvalidValue;
}

}  // namespace bdct
