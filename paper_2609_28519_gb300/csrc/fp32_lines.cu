// FFT-based FP32 line engine: one separable pass of the 2D DCT for long
// lines (64 .. 4096 points, powers of two, and 192, 384, 768, 1536 =
// 3 * 2^6 .. 3 * 2^9).
//
// What is computed: the 1D factor of Eq. 2 of the BRiDCT paper along every
// line of a batch of arrays -- y_k = s_k sum_j x_j cos(pi (2j+1) k / (2N))
// (forward), its adjoint x_j = sum_k s_k y_k cos(...) (inverse), or the
// forward, a diagonal and the adjoint in one pass (round trip and spectral
// composition, Prop. 1).  The forward reads rows and writes its result
// transposed, the inverse reads transposed and writes rows, so two passes
// give the 2D transform in natural layout.
//
// The length-N DCT-II of a real line is evaluated exactly through a complex
// FFT of L = N/2 points (Makhoul's reordering): z_m = (x_{4m}, x_{4m+2}) and
// z_{L-1-m} = (x_{4m+3}, x_{4m+1}) for m < L/2, Z = FFT_L(z), then with
// E = Z_k + conj Z_{L-k}, O = -i (Z_k - conj Z_{L-k}), P = exp(-2 pi i k/N) O,
// V = E + P, V' = conj(E - P) and W_k = exp(-i pi k / (2N)) / 2:
//   y_k = Re(W_k V),  y_{N-k} = -Im(W_k V),
//   y_{L-k} = Re(W_{L-k} V'),  y_{L+k} = -Im(W_{L-k} V').
// The FFT takes two or three steps, L = R1 R2 R3 (R2 = 1 for two), each a set
// of short FFTs in registers with one exchange through shared memory between
// steps.  The DCT-III is the exact transpose of those steps in reverse order.
//
// Packed pairs.  A thread transforms two short FFTs ("a couple") at once in
// the halves of float2 registers (one packed instruction serves both): column
// cc and its mirror MC-1-cc, taken in reversed order with real and imaginary
// parts swapped.  In that form one aligned float4 of the line, (x_{4q} ..
// x_{4q+3}), is exactly one element of both halves, so nothing is shuffled to
// form the pairs, and so is one float4 of every exchange (a "unit").  The
// last step pairs column c with C-c, conjugated, which puts Z_k and
// conj Z_{L-k} in the two halves of one register.  Phases that the mirrored
// and the conjugated halves pick up are part of the twiddle tables: the
// mirrored half of column cc takes exp(2 pi i k (cc+1) / (R MC)), and the
// step before the last uses signed k in [-R/2, R/2).
//
// Shared memory.  A CTA holds a panel of PR lines, one line per lane: line l
// at pitch N + 4 floats, which puts the lanes' float4 of one index on
// distinct banks in every phase.  A step writes its results over the units it
// read, so there is one panel buffer, and the only barriers are one between
// steps.  The transposed side goes straight between registers and global
// memory: at a fixed index the PR lanes hold PR consecutive elements.  The
// row side moves by one bulk copy (TMA) per line.
//
// What bounds it: 16 bytes of shared-memory traffic per element, pass and
// exchange (37 TB/s on the chip) and about 16 multiply-adds, against 8 bytes
// of HBM traffic per element and pass.
#include <cuda_runtime.h>

#include <cstdio>

#include "line_steps.cuh"
#include "ptx.cuh"
#include "fp32_lines.h"

namespace bdct {

cudaError_t lines_init_table(const float *d_table) { return init_cos_table(d_table); }
cudaError_t lines_init_table3(const float *d_table) { return init_cos_table3(d_table); }

bool lines_supported(int n)
{
    return n == 64 || n == 128 || n == 256 || n == 512 || n == 1024 || n == 2048 || n == 4096 || n == 192 ||
           n == 384 || n == 768 || n == 1536;
}

namespace {

// LinesMode as the kernel's parameter: forward and inverse, rows ->
// transposed; forward and adjoint in one pass, rows -> transposed or (with the
// diagonal) rows -> rows; inverse, transposed -> rows
enum Mode { MODE_F = 0, MODE_J = 1, MODE_P = 2, MODE_RR = 3, MODE_I = 4 };

// Lines per panel (PR), threads per line (G) and resident CTAs per SM that the
// registers are held to (NB), by mode: the best of a sweep over radices and
// these at 256 MiB, where one CTA more or half the lines per panel cost
// 10-30%.  Panels of 8 lines (32-byte pieces on the transposed side) only
// where shared memory holds no more.
constexpr int set_of(int mode) { return mode == MODE_F ? 0 : mode == MODE_J || mode == MODE_P ? 1 : 2; }

template <int N, int MODE>
struct LineCfg : LineSplit<N, set_of(MODE)> {
    static constexpr int SET = set_of(MODE);
    static constexpr int G = N <= 192 ? (N == 128 ? 4 : 2) : N == 256 ? (SET ? 4 : 8) : N == 384 ? (SET == 1 ? 4 : 8)
                           : N == 512 ? 8 : N == 768 ? (SET == 1 ? 8 : 12) : N == 1024 ? (SET == 1 ? 8 : 16)
                           : N == 1536 ? (SET ? 16 : 24) : N == 2048 ? 32 : 64;
    static constexpr int PR = N <= 192 || (N == 256 && SET) || (N == 384 && SET == 1) ? 32 : N <= 1024 ? 16 : 8;
    static constexpr int THREADS = PR * G;
    static constexpr int NB = N == 64 ? 12 : N == 128 ? 6 : N == 192 ? 8 : N == 256 ? (SET == 0 ? 6 : SET == 1 ? 4 : 5)
                            : N == 384 ? (SET == 0 ? 6 : SET == 1 ? 3 : 4) : N == 512 ? 4 : N == 768 ? (SET ? 3 : 2)
                            : N == 1024 ? (SET == 1 ? 3 : 2) : N == 1536 ? (SET ? 3 : 2) : N == 2048 ? 2 : 1;
    static constexpr int PT = N + (PR >= 8 ? 4 : 32 / PR);  // line pitch (floats)
    // the tables are staged in shared memory (the split's read through L1
    // instead: 1024 points inverse 0.328 -> 0.275 of HBM)
    static constexpr size_t SMEM = (size_t)PR * PT * 4 + (size_t)LineSplit<N, SET>::TAB * 16 + 16;
    static_assert(THREADS % 32 == 0 && PR <= 32 && PR % 4 == 0, "lanes");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

struct LinesParams {
    const float *src;
    float *dst;
    int rows;                            // lines per array
    int npanels;
    AxisScale sc;                        // forward: output scales, inverse: input scales (both when both run)
    const long long *src_off, *dst_off;  // indexed arrays (element offsets), or null
    const float4 *tw;                    // the plan's table for N (lines_gen_table)
    const float *lam;                    // MODE_RR, or null: output k of line r times lam[k * rows + r]
    unsigned int *status;
    int reverse;                         // take panels last to first (the pass then starts with
                                         // what the previous pass wrote last, still in L2)
};

// Member m (0 .. 3: a.x, a.y, b.x, b.y) of slot k.
template <int R>
__device__ __forceinline__ float &member(float2 (&a)[R], float2 (&b)[R], int k, int m)
{
    return m == 0 ? a[k].x : m == 1 ? a[k].y : m == 2 ? b[k].x : b[k].y;
}

// Unit q = c + m j of a column (elements 4q .. 4q + 3, ld floats apart).
__device__ __forceinline__ const char *unit_at(const float *p, int ld, int c, int m, int j, int i)
{
    const unsigned row = 4u * (unsigned)ld;
    return mad_wide(4u * (unsigned)m * row, j, mad_wide(row, 4 * c + i, reinterpret_cast<const char *>(p)));
}
__device__ __forceinline__ void store_unit(float *p, int ld, int c, int m, int j, float4 v)
{
    auto at = [&](int i) { return reinterpret_cast<float *>(const_cast<char *>(unit_at(p, ld, c, m, j, i))); };
    __stcg(at(0), v.x);
    __stcg(at(1), v.y);
    __stcg(at(2), v.z);
    __stcg(at(3), v.w);
}

// Unit slot of first-step result k1: base and direction (k1 < R1/2 kept its
// column's slots, the others the mirror's).
template <typename C>
__device__ __forceinline__ int sub_base(int k1, int &sgn)
{
    const bool e = k1 >= C::R1 / 2;
    sgn = e ? -1 : 1;
    return e ? C::M1 - 1 + C::M1 * (k1 - C::R1 / 2) : C::M1 * k1;
}

template <int N, int MODE>
__global__ void __launch_bounds__(LineCfg<N, MODE>::THREADS, LineCfg<N, MODE>::NB) k_lines(const LinesParams p)
{
    using C = LineCfg<N, MODE>;
    constexpr int R1 = C::R1, R2 = C::R2, R3 = C::R3, M1 = C::M1, CC = C::C, PR = C::PR, G = C::G;
    constexpr bool ROWS_IN = MODE != MODE_I;
    constexpr bool ROWS_OUT = MODE == MODE_I || MODE == MODE_RR;
    constexpr bool FWD = MODE != MODE_I && MODE != MODE_J, INV = MODE != MODE_F;
    extern __shared__ __align__(128) float lsm[];
    float4 *tab = reinterpret_cast<float4 *>(lsm + PR * C::PT);
    uint64_t *bar = reinterpret_cast<uint64_t *>(tab + C::TAB);
    const float4 *t1 = tab, *t2 = tab + C::U1;
    const SplitTable ts{t2 + C::U2, reinterpret_cast<const float2 *>(t2 + C::U2 + C::L / 2)};
    const int tid = threadIdx.x, line = tid % PR, g = tid / PR;
    float4 *row = reinterpret_cast<float4 *>(lsm + line * C::PT);

    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    // the tables are plan data, written before any transform was queued
    for (int r = tid; r < C::TAB; r += C::THREADS) tab[r] = __ldg(p.tw + r);
    pdl_wait_prerequisites();
    __syncthreads();

    auto panel_at = [&](int pn, long long &b, int &r0) {
        if (p.reverse) pn = p.npanels - 1 - pn;
        const long long r = (long long)pn * PR;
        b = r / p.rows;  // panels never straddle two arrays
        r0 = (int)(r - b * p.rows);
    };
    auto src_of = [&](long long b) { return p.src_off ? p.src + p.src_off[b] : p.src + b * (long long)N * p.rows; };
    auto dst_of = [&](long long b) { return p.dst_off ? p.dst + p.dst_off[b] : p.dst + b * (long long)N * p.rows; };
    // warp 0: one bulk copy per line of the panel
    auto load_panel = [&](int pn) {
        long long b;
        int r0;
        panel_at(pn, b, r0);
        if (tid == 0) mbar_arrive_expect_tx(bar, PR * N * 4);
        __syncwarp();
        if (tid < PR) bulk_load(lsm + tid * C::PT, src_of(b) + (long long)(r0 + tid) * N, N * 4, bar);
    };
    if (ROWS_IN && tid < 32 && (int)blockIdx.x < p.npanels) load_panel(blockIdx.x);

    uint32_t phase = 0;
    for (int pn = blockIdx.x; pn < p.npanels; pn += gridDim.x) {
        long long b;
        int r0;
        panel_at(pn, b, r0);
        const int next = pn + (int)gridDim.x;
        // let the next kernel in only for the last panels: its CTAs, of another
        // size, would hold registers and shared memory all along (128 x 512
        // forward 434 -> 350 us, 256^2 spectral 725 -> 593 us)
        if (next >= p.npanels) pdl_launch_dependents();
        bool ok = true;
        if constexpr (ROWS_IN) {
            ok = mbar_wait_bounded(bar, phase);
            phase ^= 1;
        }
        constexpr int ROUNDS = (CC / 2 + G - 1) / G;  // couples of the last step per thread
        float2 ya[MODE == MODE_J ? ROUNDS : 1][R3], yb[MODE == MODE_J ? ROUNDS : 1][R3];
        if constexpr (MODE == MODE_J) {
            // ---- every coefficient of this thread's couples, before units go over the rows
#pragma unroll
            for (int rd = 0; rd < ROUNDS; ++rd) {
                const int c = g + rd * G;
                if ((CC / 2) % G == 0 || c < CC / 2)
                    walk_row<C>(reinterpret_cast<const float *>(row), c,
                                [&](const float *q, int k, int m) { member(ya[rd], yb[rd], k, m) = *q; });
            }
        }
        if constexpr (FWD) {
            // ---- first step
#pragma unroll 1
            for (int cc = g; cc < M1 / 2; cc += G) {
                float4 x[R1 / 2], y[R1 / 2];
#pragma unroll
                for (int j = 0; j < R1 / 2; ++j) {
                    x[j] = row[cc + M1 * j];
                    y[j] = row[M1 - 1 - cc + M1 * j];
                }
                step_forward<R1, M1>(x, y, t1 + cc);
#pragma unroll
                for (int j = 0; j < R1 / 2; ++j) {
                    row[cc + M1 * j] = x[j];
                    row[M1 - 1 - cc + M1 * j] = y[j];
                }
            }
        }
        if constexpr (ROWS_IN) {
            if (!__syncthreads_and(ok)) {
                // the load did not land in time: record it, give the copies
                // one more bounded wait, and stop
                if (tid == 0) {
                    record_timeout(p.status);
                    mbar_wait_bounded(bar, phase ^ 1);
                }
                return;
            }
        }
        if constexpr (FWD) {
            // ---- middle step
            if constexpr (R2 > 1) {
#pragma unroll 1
                for (int q = g; q < R1 * R3 / 2; q += G) {
                    int sgn;
                    const int k1 = q / (R3 / 2), m3 = q % (R3 / 2);
                    const int qb = sub_base<C>(k1, sgn);
                    float4 *px = row + qb + sgn * m3, *py = row + qb + sgn * (R3 - 1 - m3);
                    float4 x[R2 / 2], y[R2 / 2];
#pragma unroll
                    for (int j = 0; j < R2 / 2; ++j) {
                        x[j] = px[sgn * R3 * j];
                        y[j] = py[sgn * R3 * j];
                    }
                    step_forward<R2, R3>(x, y, t2 + m3);
#pragma unroll
                    for (int j = 0; j < R2 / 2; ++j) {
                        px[sgn * R3 * j] = x[j];
                        py[sgn * R3 * j] = y[j];
                    }
                }
                __syncthreads();
            }
        }
        // ---- last step, split, and the transposed side
        {
            const float *src = MODE == MODE_I ? src_of(b) + r0 + line : nullptr;
            float *dst = MODE == MODE_F ? dst_of(b) + r0 + line : nullptr;
            const float *lam = MODE == MODE_RR && p.lam ? p.lam + r0 + line : nullptr;
#pragma unroll(MODE == MODE_J ? ROUNDS : 1)
            for (int rd = 0; rd < ROUNDS; ++rd) {
                const int c = g + rd * G;
                const bool active = (CC / 2) % G == 0 || c < CC / 2;
                // the couple's columns: c and C-c (C/2 for c = 0)
                float4 *px, *pw;
                int sx = 1, sw = -1;
                if constexpr (R2 == 1) {
                    px = row + M1 * c;
                    pw = row + M1 - 1 + M1 * ((c ? CC - c : CC / 2) - R1 / 2);
                } else {
                    const int k1 = c % R1, k2 = c / R1;
                    px = row + sub_base<C>(k1, sx) + sx * (R3 * k2);
                    const int k1p = k1 ? R1 - k1 : 0;
                    const int k2p = k1 ? R2 - 1 - k2 : (c ? R2 - k2 : R2 / 2);
                    pw = row + sub_base<C>(k1p, sw) + sw * (R3 - 1 + R3 * (k2p - R2 / 2));
                    sw = -sw;
                }
                float4 x[R3 / 2], w[R3 / 2];
                float2 dr[R3], di[R3], a[R3], bb[R3];
                if constexpr (FWD) {
                    if (active) {
#pragma unroll
                        for (int m = 0; m < R3 / 2; ++m) {
                            x[m] = px[sx * m];
                            w[m] = pw[sw * m];
                        }
                    }
                    if constexpr (MODE == MODE_F) {
                        if (rd == ROUNDS - 1) {
                            // every unit of the panel is in registers: the next panel may land
                            fence_proxy_async_smem();
                            __syncthreads();
                            if (tid < 32 && next < p.npanels) load_panel(next);
                        }
                    }
                    if (active) {
                        last_forward<R3>(x, w, dr, di);
                        split_forward<R3, CC>(c, dr, di, ts, p.sc, a, bb);
                    }
                } else if constexpr (MODE == MODE_J) {
#pragma unroll
                    for (int k = 0; k < R3; ++k) {
                        a[k] = ya[rd][k];
                        bb[k] = yb[rd][k];
                    }
                } else {
                    if (active) {
                        walk_slots<C>(src, c, p.rows, [&](const char *q, int k, int m) {
                            member(a, bb, k, m) = __ldcg(reinterpret_cast<const float *>(q));
                        });
                    }
                    if (rd == 0) {
                        // the previous panel's stores must have read the buffer
                        if (tid < PR) bulk_wait_read<0>();
                        __syncthreads();
                    }
                }
                if constexpr (MODE == MODE_F) {
                    if (active) {
                        walk_slots<C>(dst, c, p.rows, [&](const char *q, int k, int m) {
                            __stcg(reinterpret_cast<float *>(const_cast<char *>(q)), member(a, bb, k, m));
                        });
                    }
                }
                if constexpr (MODE == MODE_RR) {
                    if (active && lam) {
                        walk_slots<C>(lam, c, p.rows, [&](const char *q, int k, int m) {
                            member(a, bb, k, m) *= __ldg(reinterpret_cast<const float *>(q));
                        });
                    }
                }
                if constexpr (INV) {
                    if (active) {
                        split_adjoint<R3, CC>(c, a, bb, ts, p.sc, dr, di);
                        last_adjoint<R3>(x, w, dr, di);
#pragma unroll
                        for (int m = 0; m < R3 / 2; ++m) {
                            px[sx * m] = x[m];
                            pw[sw * m] = w[m];
                        }
                    }
                }
            }
        }
        if constexpr (INV) {
            __syncthreads();
            if constexpr (R2 > 1) {
#pragma unroll 1
                for (int q = g; q < R1 * R3 / 2; q += G) {
                    int sgn;
                    const int k1 = q / (R3 / 2), m3 = q % (R3 / 2);
                    const int qb = sub_base<C>(k1, sgn);
                    float4 *px = row + qb + sgn * m3, *py = row + qb + sgn * (R3 - 1 - m3);
                    float4 x[R2 / 2], y[R2 / 2];
#pragma unroll
                    for (int j = 0; j < R2 / 2; ++j) {
                        x[j] = px[sgn * R3 * j];
                        y[j] = py[sgn * R3 * j];
                    }
                    step_adjoint<R2, R3>(x, y, t2 + m3);
#pragma unroll
                    for (int j = 0; j < R2 / 2; ++j) {
                        px[sgn * R3 * j] = x[j];
                        py[sgn * R3 * j] = y[j];
                    }
                }
                __syncthreads();
            }
            // ---- first step: rows in place, or the transposed side
            constexpr int ROUNDS1 = (M1 / 2 + G - 1) / G;
            float *dst = ROWS_OUT ? nullptr : dst_of(b) + r0 + line;
#pragma unroll 1
            for (int rd = 0; rd < ROUNDS1; ++rd) {
                const int cc = g + rd * G;
                const bool active = (M1 / 2) % G == 0 || cc < M1 / 2;
                float4 x[R1 / 2], y[R1 / 2];
                if (active) {
#pragma unroll
                    for (int j = 0; j < R1 / 2; ++j) {
                        x[j] = row[cc + M1 * j];
                        y[j] = row[M1 - 1 - cc + M1 * j];
                    }
                }
                if (!ROWS_OUT && rd == ROUNDS1 - 1) {
                    // every unit of the panel is in registers: the next panel may land
                    fence_proxy_async_smem();
                    __syncthreads();
                    if (tid < 32 && next < p.npanels) load_panel(next);
                }
                if (!active) continue;
                step_adjoint<R1, M1>(x, y, t1 + cc);
#pragma unroll
                for (int j = 0; j < R1 / 2; ++j) {
                    if constexpr (ROWS_OUT) {
                        row[cc + M1 * j] = x[j];
                        row[M1 - 1 - cc + M1 * j] = y[j];
                    } else {
                        store_unit(dst, p.rows, cc, M1, j, x[j]);
                        store_unit(dst, p.rows, M1 - 1 - cc, M1, j, y[j]);
                    }
                }
            }
            if constexpr (ROWS_OUT) {
                fence_proxy_async_smem();  // the stores read the panel through the async proxy
                __syncthreads();
                if (tid < PR) {
                    bulk_store(dst_of(b) + (long long)(r0 + tid) * N, lsm + tid * C::PT, N * 4);
                    bulk_commit();
                }
                if constexpr (MODE == MODE_RR) {
                    if (tid < 32 && next < p.npanels) {
                        if (tid < PR) bulk_wait_read<0>();
                        __syncwarp();
                        load_panel(next);
                    }
                }
            }
        }
    }
    if constexpr (ROWS_OUT) {
        if (tid < PR) bulk_wait<0>();
    }
}

template <int N, int MODE>
cudaError_t lines_launch(const LinesParams &p0, long long nrows, cudaStream_t stream)
{
    using C = LineCfg<N, MODE>;
    auto kern = k_lines<N, MODE>;
    static DeviceLaunchCache cache;
    int dev = 0, blocks_per_sm = 0, num_sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cache.get(
        dev,
        [&](int d, int &bps, int &sms) {
            cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
            if (r == cudaSuccess) r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, C::THREADS, C::SMEM);
            if (r == cudaSuccess) r = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d);
            if (r == cudaSuccess && bps < 1) r = cudaErrorInvalidConfiguration;
            if (r == cudaSuccess && debug_enabled())
                fprintf(stderr, "[bdct] k_lines<%d,%d>: %d CTAs/SM x %d threads, panel %d lines, smem %zu B\n", N, MODE,
                        bps, C::THREADS, C::PR, C::SMEM);
            return r;
        },
        &blocks_per_sm, &num_sms);
    if (e != cudaSuccess) return e;
    LinesParams p = p0;
    if (p.rows % C::PR != 0) return cudaErrorInvalidValue;  // panels never straddle two arrays
    const long long np = nrows / C::PR;
    if (np <= 0) return cudaSuccess;
    if (np > 0x7ff00000LL) return cudaErrorInvalidValue;
    p.npanels = (int)np;
    long long grid = (long long)blocks_per_sm * num_sms;
    if (grid > np) grid = np;
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

template <int N>
cudaError_t lines_mode(LinesMode mode, const LinesParams &p, long long nrows, cudaStream_t s)
{
    switch (mode) {
        case LINES_FORWARD: return lines_launch<N, MODE_F>(p, nrows, s);
        case LINES_INVERSE: return lines_launch<N, MODE_J>(p, nrows, s);
        case LINES_PAIR: return lines_launch<N, MODE_P>(p, nrows, s);
        case LINES_PAIR_ROWS: return lines_launch<N, MODE_RR>(p, nrows, s);
        default: return lines_launch<N, MODE_I>(p, nrows, s);
    }
}

// The tables of length n = 2L, in FP64 with every angle reduced exactly in
// integers; layout as LineCfg (first step, middle step, split).
struct TableShape {
    int n, r1, r2, r3;
};

__device__ void cos_sin_2pi(long long m, long long d, double &c, double &s)  // of 2 pi m / d
{
    m %= d;
    if (m < 0) m += d;
    sincospi(2.0 * (double)m / (double)d, &s, &c);
}

// All tables of a plan in one launch, blockIdx.y the table.
constexpr int kMaxTables = 12;
struct TableJobs {
    float4 *dst[kMaxTables];
    TableShape shape[kMaxTables];
    double s1[kMaxTables];
};

__global__ void k_gen_line_tw(const TableJobs jobs)
{
    float4 *t = jobs.dst[blockIdx.y];
    const TableShape q = jobs.shape[blockIdx.y];
    const double s1 = jobs.s1[blockIdx.y];
    const int L = q.n / 2, m1 = L / q.r1, c3 = L / q.r3;
    const int u1 = q.r1 * (m1 / 2), u2 = q.r2 > 1 ? q.r2 * (q.r3 / 2) : 0;
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    double ca, sa, cb, sb;
    if (r < u1 + u2) {
        // entry (k, cc): exp(-2 pi i cc k / (R MC)) and exp(2 pi i (cc+1) k / (R MC)),
        // k signed in the step before the last
        const bool first = r < u1;
        const int R = first ? q.r1 : q.r2, mc = first ? m1 : q.r3;
        const int e = first ? r : r - u1;
        int k = e / (mc / 2);
        const int cc = e % (mc / 2);
        if ((q.r2 == 1 || !first) && k >= R / 2) k -= R;
        const long long d = (long long)R * mc;
        cos_sin_2pi((long long)cc * k, d, ca, sa);
        cos_sin_2pi((long long)(cc + 1) * k, d, cb, sb);
        t[r] = make_float4((float)ca, (float)cb, (float)sa, (float)sb);
    } else if (r < u1 + u2 + L / 2) {
        const int e = r - u1 - u2;
        const int k3 = e / (c3 / 2), c = e % (c3 / 2);
        const int k = c3 * k3 + (c || k3 < q.r3 / 2 ? c : c3 / 2 - L / 2);
        const double f = 0.5 * s1;
        double cw, sw;
        cos_sin_2pi(k, q.n, cw, sw);
        cos_sin_2pi(k, 4ll * q.n, ca, sa);       // W_k = exp(-i pi k / (2n))
        cos_sin_2pi(L - k, 4ll * q.n, cb, sb);   // W_{L-k}
        float4 *o = t + u1 + u2;
        o[e] = make_float4((float)cw, (float)sw, (float)(f * ca), (float)(f * cb));
        reinterpret_cast<float2 *>(o + L / 2)[e] = make_float2((float)(f * sa), (float)(f * sb));
    }
}

template <int N, int SET>
TableShape shape_of()
{
    using S = LineSplit<N, SET>;
    return TableShape{N, S::R1, S::R2, S::R3};
}

template <int N>
bool shape_of_set(int set, TableShape *q)
{
    *q = set == 0 ? shape_of<N, 0>() : set == 1 ? shape_of<N, 1>() : shape_of<N, 2>();
    return true;
}

bool table_shape(int n, int set, TableShape *q)
{
    switch (n) {
        case 64: return shape_of_set<64>(set, q);
        case 128: return shape_of_set<128>(set, q);
        case 192: return shape_of_set<192>(set, q);
        case 256: return shape_of_set<256>(set, q);
        case 384: return shape_of_set<384>(set, q);
        case 512: return shape_of_set<512>(set, q);
        case 768: return shape_of_set<768>(set, q);
        case 1024: return shape_of_set<1024>(set, q);
        case 1536: return shape_of_set<1536>(set, q);
        case 2048: return shape_of_set<2048>(set, q);
        case 4096: return shape_of_set<4096>(set, q);
        default: return false;
    }
}

}  // namespace

size_t lines_table_elems(int n, int set)
{
    TableShape q;
    if (!table_shape(n, set, &q)) return 0;
    const int L = n / 2;
    return (size_t)q.r1 * (L / q.r1 / 2) + (q.r2 > 1 ? (size_t)q.r2 * (q.r3 / 2) : 0) + L / 2 + L / 4;
}

cudaError_t lines_gen_tables(const LineTable *tables, int count, cudaStream_t s)
{
    if (count < 1 || count > kMaxTables) return cudaErrorInvalidValue;
    TableJobs jobs{};
    int most = 0;
    for (int i = 0; i < count; ++i) {
        if (!table_shape(tables[i].n, tables[i].set, &jobs.shape[i])) return cudaErrorInvalidValue;
        jobs.dst[i] = tables[i].dst;
        jobs.s1[i] = tables[i].s1;
        const int e = (int)lines_table_elems(tables[i].n, tables[i].set);
        if (e > most) most = e;
    }
    k_gen_line_tw<<<dim3((most + 127) / 128, count), 128, 0, s>>>(jobs);
    return cudaGetLastError();
}

cudaError_t lines_pass(const float *src, float *dst, int rows, int n, long long count, LinesMode mode, AxisScale sc,
                       const float4 *tw, const float *lam, unsigned int *status, cudaStream_t stream,
                       const long long *src_off, const long long *dst_off, bool reverse)
{
    LinesParams p{};
    p.src = src;
    p.dst = dst;
    p.rows = rows;
    p.sc = sc;
    p.src_off = src_off;
    p.dst_off = dst_off;
    p.tw = tw;
    p.lam = lam;
    p.status = status;
    p.reverse = reverse ? 1 : 0;
    const long long nrows = (long long)rows * count;
    switch (n) {
        case 64: return lines_mode<64>(mode, p, nrows, stream);
        case 128: return lines_mode<128>(mode, p, nrows, stream);
        case 192: return lines_mode<192>(mode, p, nrows, stream);
        case 256: return lines_mode<256>(mode, p, nrows, stream);
        case 384: return lines_mode<384>(mode, p, nrows, stream);
        case 512: return lines_mode<512>(mode, p, nrows, stream);
        case 768: return lines_mode<768>(mode, p, nrows, stream);
        case 1024: return lines_mode<1024>(mode, p, nrows, stream);
        case 1536: return lines_mode<1536>(mode, p, nrows, stream);
        case 2048: return lines_mode<2048>(mode, p, nrows, stream);
        case 4096: return lines_mode<4096>(mode, p, nrows, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace bdct
