// FFT-based FP32 line engine: one separable pass of the 2D DCT for long
// lines (64 .. 4096 points, powers of two, and 192, 384, 768, 1536 =
// 3 * 2^6 .. 3 * 2^9).
//
// What is computed: the 1D factor of Eq. 2 of the BRiDCT paper along every
// line of a batch of arrays -- y_k = s_k sum_j x_j cos(pi (2j+1) k / (2N))
// (forward), its adjoint x_j = sum_k s_k y_k cos(...) (inverse), or the
// forward, a diagonal and the adjoint in one pass (round trip and spectral
// composition, Prop. 1).  A pass reads rows and writes its result
// transposed, so two of them give the 2D transform in natural layout; only the
// last of the spectral composition's three passes writes rows.
//
// The length-N DCT-II of a real line is evaluated exactly through a complex
// FFT of L = N/2 points (Makhoul's reordering): z_m = (x_{4m}, x_{4m+2}) and
// z_{L-1-m} = (x_{4m+3}, x_{4m+1}) for m < L/2, Z = FFT_L(z), then with
// E = Z_k + conj Z_{L-k}, O = -i (Z_k - conj Z_{L-k}), P = exp(-2 pi i k/N) O,
// V = E + P, V' = conj(E - P) and W_k = exp(-i pi k / (2N)) / 2:
//   y_k = Re(W_k V),  y_{N-k} = -Im(W_k V),
//   y_{L-k} = Re(W_{L-k} V'),  y_{L+k} = -Im(W_{L-k} V').
// (The factor 1/2 of W_k is in the first step's twiddles, ahead of the sums.)
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
// What bounds it: up to 512 points the two passes' HBM traffic, 16 bytes per
// element (256^2 forward: 0.92 of the copy rate over the bytes it moves);
// beyond that, and in the pair modes, the chain of shared-memory exchanges (16
// bytes per element, pass and exchange) and the multiply-adds, with 12 to 16
// warps per SM at full registers.  The form before this one ran four-step FFTs
// with one sub-FFT per thread, unpacked, 33 instructions per element and pass
// where this takes 18 to 26 one way.  512 MiB, before -> now, us:
//                 forward      inverse      round trip   spectral
//   256^2         469 -> 345   543 -> 355   758 -> 411   1053 -> 583
//   768 x 1024    556 -> 361   652 -> 376   979 -> 569   1303 -> 699
//   1024^2        525 -> 369   575 -> 362   872 -> 553   1185 -> 706
//   2048^2        638 -> 422   671 -> 439   992 -> 651   1445 -> 820
//   4 x 4096^2    395 -> 232   414 -> 243   639 -> 361    917 -> 510
#pragma once

#include <cuda_runtime.h>

#include <cstdio>

#include "line_steps.cuh"
#include "ptx.cuh"
#include "fp32_lines.h"

namespace bdct {

namespace {

// LinesMode as the kernel's parameter: forward, inverse, forward and adjoint in
// one pass, the same with a diagonal between (its own mode: a test of a null
// diagonal in MODE_P cost 1024^2 round trips 577 -> 592 us), each rows ->
// transposed; inverse, rows -> rows
enum Mode { MODE_F = 0, MODE_I = 1, MODE_P = 2, MODE_D = 3, MODE_R = 4 };

// Lines per panel (PR), threads per line (G) and resident CTAs per SM that the
// registers are held to (NB), by mode: the best of a sweep over radices and
// these at 256 MiB, where one CTA more or half the lines per panel cost
// 10-30%.  Panels of 8 lines (32-byte pieces on the transposed side) only
// where shared memory holds no more.
constexpr int set_of(int mode) { return mode == MODE_F ? 0 : 1; }

// FEW: a call with few panels lasts as long as one panel's chain of steps, so its
// panels are 8 lines and a step is one couple per thread, with the short radices
// of set 2 (a single 1024 x 768 array, forward and inverse: 24.9 -> 15.2 us).
constexpr bool has_few(int n) { return n >= 192 && n < 4096; }
// Lines per panel of the ordinary form.
constexpr int panel_lines(int n, int set) { return n <= 192 || (n <= 384 && set) ? 32 : n <= 1024 ? 16 : 8; }
template <int N, int MODE, bool FEW>
struct LineCfg;

template <int N, int MODE>
struct LineCfg<N, MODE, true> : LineSplit<N, 2> {
    static constexpr int G = N <= 512 ? 8 : N == 768 ? 24 : N == 1024 ? 32 : N == 1536 ? 48 : 64;
    static constexpr int PR = 8;
    static constexpr int THREADS = PR * G;
    static constexpr int NB = THREADS >= 384 ? 1 : 2;
    // registers as for 256 threads: at 128 a panel of the next pass, of another
    // length, fits beside one of this pass and starts under it (1 x 1024 x 768
    // round trip 13.0 us with 136 registers at 768 points, 10.1 with 128)
    static constexpr int BOUND = THREADS == 192 ? 256 : THREADS;
    static constexpr int PT = N + 4;  // line pitch (floats)
    static constexpr size_t SMEM = (size_t)PR * PT * 4 + (size_t)LineSplit<N, 2>::TAB * 16 + 16;
};

template <int N, int MODE>
struct LineCfg<N, MODE, false> : LineSplit<N, set_of(MODE)> {
    static constexpr int SET = set_of(MODE);
    static constexpr int G = N <= 192 ? (N == 128 ? 4 : 2) : N == 256 || N == 384 ? (SET ? 4 : 8) : N == 512 ? 8
                           : N == 768 ? (SET ? 8 : 12) : N == 1024 ? (SET ? 8 : 16) : N == 1536 ? (SET ? 16 : 24)
                           : N == 2048 ? 32 : 64;
    static constexpr int PR = panel_lines(N, SET);
    static constexpr int THREADS = PR * G, BOUND = THREADS;
    static constexpr int NB = N == 64 ? 12 : N == 128 ? 6 : N == 192 ? 8 : N == 256 ? (SET ? 4 : 6) : N == 384 ? (SET ? 3 : 6)
                            : N == 512 ? 4 : N == 768 || N == 1024 || N == 1536 ? (SET ? 3 : 2) : N == 2048 ? 2 : 1;
    static constexpr int PT = N + 4;  // line pitch (floats)
    // the tables are staged in shared memory (the split's read through L1
    // instead: 1024 points inverse 0.328 -> 0.275 of HBM)
    static constexpr size_t SMEM = (size_t)PR * PT * 4 + (size_t)LineSplit<N, SET>::TAB * 16 + 16;
    static_assert(THREADS % 32 == 0 && PR <= 32 && PR % 4 == 0, "lanes");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

// Shared memory of an SM, of that a CTA's own share, and the most a CTA can ask for.
constexpr long long kSmemPerSm = 228 * 1024, kSmemReserved = 1024, kSmemMax = kSmemPerSm - kSmemReserved;

struct LinesParams {
    const float *src;
    float *dst;
    int rows;                            // lines per array
    int npanels;
    AxisScale sc;                        // twice the forward's output scales or the inverse's input scales (both when both run)
    const long long *src_off, *dst_off;  // indexed arrays (element offsets), or null
    const float4 *tw;                    // the plan's table for N and the modes' set
    const float4 *tw_few;                // and of set 2
    const float *lam;                    // MODE_D: coefficient k of line r times lam[k * rows + r]
    unsigned int *status;
    int beside_set;                      // table set of the pass along the other axis
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

template <int N, int MODE, bool FEW>
__global__ void __launch_bounds__(LineCfg<N, MODE, FEW>::BOUND, LineCfg<N, MODE, FEW>::NB) k_lines(const LinesParams p)
{
    using C = LineCfg<N, MODE, FEW>;
    constexpr int R1 = C::R1, R2 = C::R2, R3 = C::R3, M1 = C::M1, CC = C::C, PR = C::PR, G = C::G;
    constexpr bool ROWS_OUT = MODE == MODE_R;
    constexpr bool FWD = MODE == MODE_F || MODE == MODE_P || MODE == MODE_D, INV = MODE != MODE_F;
    extern __shared__ __align__(128) float lsm[];
    float4 *tab = reinterpret_cast<float4 *>(lsm + PR * C::PT);
    uint64_t *bar = reinterpret_cast<uint64_t *>(tab + C::TAB);
    const float4 *t1 = tab, *t2 = tab + C::U1;
    const SplitTable ts{t2 + C::U2, reinterpret_cast<const float2 *>(t2 + C::U2 + C::L / 2)};
    const int tid = threadIdx.x, line = tid % PR, g = tid / PR;
    float4 *row = reinterpret_cast<float4 *>(lsm + line * C::PT);
    // the inverse's last step reads single coefficients of its rows: there a
    // warp takes 8 lines of 4 couples (pitch 4 mod 32: 32 lines of one couple
    // would meet on 8 banks; 512 MiB inverse, 768 x 1024 398 -> 384 us, 384^2 379
    // -> 363, 1024^2 398 -> 384, spectral 256^2 618 -> 594).  Not for the
    // lengths whose inverse is at its limit of 128 registers, where the extra
    // indices cost more: 256^2 358 -> 368, 512^2 367 -> 381.
    constexpr bool FULL = FWD || PR <= 8 || (MODE == MODE_I && !FEW && (N == 192 || N == 256 || N == 512));
    constexpr int CG = FULL ? 32 / PR : G < 4 ? G : 4, CL = 32 / CG;
    const int cline = FULL ? line : tid % CL + CL * (tid / 32 % (PR / CL));
    const int cg = FULL ? g : tid / CL % CG + CG * (tid / 32 / (PR / CL));
    float4 *crow = reinterpret_cast<float4 *>(lsm + cline * C::PT);

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
    if (tid < 32 && (int)blockIdx.x < p.npanels) load_panel(blockIdx.x);

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
        const bool ok = mbar_wait_bounded(bar, phase);
        phase ^= 1;
        constexpr int ROUNDS = (CC / 2 + G - 1) / G;  // couples of the last step per thread
        float2 ya[!FWD ? ROUNDS : 1][R3], yb[!FWD ? ROUNDS : 1][R3];
        if constexpr (!FWD) {
            // ---- every coefficient of this thread's couples, before units go over the rows
#pragma unroll
            for (int rd = 0; rd < ROUNDS; ++rd) {
                const int c = cg + rd * G;
                if ((CC / 2) % G == 0 || c < CC / 2)
                    walk_row<C>(reinterpret_cast<const float *>(crow), c,
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
                step_forward<R1, M1, true>(x, y, t1 + cc);
#pragma unroll
                for (int j = 0; j < R1 / 2; ++j) {
                    row[cc + M1 * j] = x[j];
                    row[M1 - 1 - cc + M1 * j] = y[j];
                }
            }
        }
        if (!__syncthreads_and(ok)) {
            // the load did not land in time: record it, give the copies one
            // more bounded wait, and stop
            if (tid == 0) {
                record_timeout(p.status);
                mbar_wait_bounded(bar, phase ^ 1);
            }
            return;
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
                    step_forward<R2, R3, false>(x, y, t2 + m3);
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
            float *dst = MODE == MODE_F ? dst_of(b) + r0 + line : nullptr;
            const float *lam = MODE == MODE_D ? p.lam + r0 + line : nullptr;
#pragma unroll(!FWD ? ROUNDS : 1)
            for (int rd = 0; rd < ROUNDS; ++rd) {
                const int c = cg + rd * G;
                const bool active = (CC / 2) % G == 0 || c < CC / 2;
                // the couple's columns: c and C-c (C/2 for c = 0)
                float4 *px, *pw;
                int sx = 1, sw = -1;
                if constexpr (R2 == 1) {
                    px = crow + M1 * c;
                    pw = crow + M1 - 1 + M1 * ((c ? CC - c : CC / 2) - R1 / 2);
                } else {
                    const int k1 = c % R1, k2 = c / R1;
                    px = crow + sub_base<C>(k1, sx) + sx * (R3 * k2);
                    const int k1p = k1 ? R1 - k1 : 0;
                    const int k2p = k1 ? R2 - 1 - k2 : (c ? R2 - k2 : R2 / 2);
                    pw = crow + sub_base<C>(k1p, sw) + sw * (R3 - 1 + R3 * (k2p - R2 / 2));
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
                } else {
#pragma unroll
                    for (int k = 0; k < R3; ++k) {
                        a[k] = ya[rd][k];
                        bb[k] = yb[rd][k];
                    }
                }
                if constexpr (MODE == MODE_F) {
                    if (active) {
                        walk_slots<C>(dst, c, p.rows, [&](const char *q, int k, int m) {
                            __stcg(reinterpret_cast<float *>(const_cast<char *>(q)), member(a, bb, k, m));
                        });
                    }
                }
                if constexpr (MODE == MODE_D) {
                    if (active) {
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
                    step_adjoint<R2, R3, false>(x, y, t2 + m3);
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
                step_adjoint<R1, M1, true>(x, y, t1 + cc);
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
                if (tid < 32 && next < p.npanels) {
                    if (tid < PR) bulk_wait_read<0>();
                    __syncwarp();
                    load_panel(next);
                }
            }
        }
    }
    if constexpr (ROWS_OUT) {
        if (tid < PR) bulk_wait<0>();
    }
}

template <int N, int MODE, bool FEW = false>
cudaError_t lines_launch(const LinesParams &p0, long long nrows, cudaStream_t stream)
{
    using C = LineCfg<N, MODE, FEW>;
    auto kern = k_lines<N, MODE, FEW>;
    static DeviceLaunchCache cache;
    int dev = 0, blocks_per_sm = 0, num_sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cache.get(
        dev,
        [&](int d, int &bps, int &sms) {
            cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
            if (r == cudaSuccess) r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, C::THREADS, C::SMEM);
            if (r == cudaSuccess) r = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d);
            if (r == cudaSuccess && bps < 1) r = cudaErrorInvalidConfiguration;
            if (r == cudaSuccess && debug_enabled())
                fprintf(stderr, "[bdct] k_lines<%d,%d,%d>: %d CTAs/SM x %d threads, panel %d lines, smem %zu B\n", N, MODE,
                        (int)FEW, bps, C::THREADS, C::PR, C::SMEM);
            return r;
        },
        &blocks_per_sm, &num_sms);
    if (e != cudaSuccess) return e;
    LinesParams p = p0;
    if (p.rows % C::PR != 0) return cudaErrorInvalidValue;  // panels never straddle two arrays
    const long long np = nrows / C::PR;
    if (np <= 0) return cudaSuccess;
    // fewer panels than SMs: the short chain.  At half the line and at the line
    // (2048 lines of 512 points) 512 x 512 x 2 takes 6.6 us with it and 7.4 with the
    // ordinary form inverse, 11.1 and 11.0 round trip, 512 x 512 x 4 8.0 and 8.2,
    // 12.8 and 12.3; 192 x 64 x 24 (48 panels) forward 6.0 and 9.9.  At 2048 points
    // the pair modes spill in this form (220 to 300 bytes): up to 16 panels the
    // ordinary one is the faster (2048 x 64 round trip 12.7 us, 11.3), from 32 on
    // this one (13.2, 16.6).  4096 points have one form; at 64 and 128 the forms
    // differ by less than 10% of calls of 6 us.
    if constexpr (has_few(N) && !FEW) {
        if (np < num_sms) {
            LinesParams few = p;
            few.tw = p.tw_few;
            return lines_launch<N, MODE, true>(few, nrows, stream);
        }
    }
    if (np > 0x7ff00000LL) return cudaErrorInvalidValue;
    p.npanels = (int)np;
    long long grid = (long long)blocks_per_sm * num_sms;
    if (grid > np) grid = np;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(C::THREADS);
    cfg.dynamicSmemBytes = C::SMEM;
    // More panels than SMs but fewer than fit at once: the CTAs ask for so much
    // shared memory that an SM holds no more than its share.  They start while the
    // pass before them still drains and would otherwise pile up on the SMs it has
    // left (192 x 128 x 48 inverse 13.0 -> 9.9 us, 512 x 256 x 16 forward 14.1 ->
    // 10.7, 192 x 1024 x 12 14.9 -> 11.2).  Not beside a pass of fewer than 3/4 panels
    // per SM, whose small CTAs fit in anywhere and would wait (1024 x 64 x 8 round
    // trip 8.8 us, 11.1), but for 192 points, whose own chain is the longer (192 x
    // 1024 x 8 inverse 16.4 -> 11.6).
    const bool beside_few =  // of the pass along the other axis
        N != 192 && has_few(p.rows) && 4 * (nrows / p.rows * N / panel_lines(p.rows, p.beside_set)) < 3 * num_sms;
    if (!FEW && !beside_few && np > num_sms && np < (long long)blocks_per_sm * num_sms) {
        const long long share = kSmemPerSm / ((np + num_sms - 1) / num_sms) - kSmemReserved;
        if (share > (long long)C::SMEM) cfg.dynamicSmemBytes = (size_t)share / 128 * 128;
    }
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p);
}

template <int N>
cudaError_t lines_run(LinesMode mode, const LinesCall &c, cudaStream_t s)
{
    LinesParams p{};
    p.src = c.src;
    p.dst = c.dst;
    p.rows = c.rows;
    p.sc = AxisScale{2.0f * c.sc.s0, 2.0f * c.sc.s1};  // the first step halves
    p.src_off = c.src_off;
    p.dst_off = c.dst_off;
    p.tw = c.tw;
    p.tw_few = c.tw_few;
    p.lam = c.lam;
    p.status = c.status;
    p.beside_set = c.beside == LINES_FORWARD ? 0 : 1;
    p.reverse = c.reverse ? 1 : 0;
    const long long nrows = (long long)c.rows * c.count;
    switch (mode) {
        case LINES_FORWARD: return lines_launch<N, MODE_F>(p, nrows, s);
        case LINES_INVERSE: return lines_launch<N, MODE_I>(p, nrows, s);
        case LINES_PAIR: return lines_launch<N, MODE_P>(p, nrows, s);
        case LINES_PAIR_DIAGONAL: return lines_launch<N, MODE_D>(p, nrows, s);
        default: return lines_launch<N, MODE_R>(p, nrows, s);
    }
}

}  // namespace

}  // namespace bdct
