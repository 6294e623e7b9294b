// On-chip dense route for small arrays of any side up to 64 that the fused
// kernels do not cover (non-power-of-two sides such as 24, 26, 40 or 48).
//
// What is computed: Eq. 2 of the BRiDCT paper as the sandwich M_h X M_w^T
// (M = Q_n forward, Q_n^T inverse, Eq. 1; Section 7.1 makes h and w
// independent); the round trip is the forward pair then the inverse pair of
// the orthonormal operators (Prop. 1 with Lambda = I), and the spectral
// direction puts Lambda between them (Eq. 4).  One read and one write of
// every element; every pass runs in shared memory on the half products of
// dense_passes.cu: n/2 multiply-adds per point, the even and the odd product
// in the halves of packed pairs, operand pairs (s, d) = half the sums and
// differences of mirrored elements (forward; half_pair, ptx.cuh) or (y_2k,
// y_2k+1) (inverse).
//
// Organization.  A CTA of four warps transforms G arrays at a time, G chosen
// so that one tile of 8 lines x 4 output pairs per thread covers them
// (about 8192 elements), or, in a call of few arrays, of eight warps with tiles
// of 2 lines.  Every pass stores what the next one contracts,
// already paired, from registers:
//  * along w, forward: a thread's lines are mirrored rows (i, h-1-i), whose
//    sum and difference is the pair the pass along h needs;
//  * along h, forward: coefficient rows 2o and 2o + 1 come out as one pair,
//    which the adjoint pass along h contracts (times Lambda), or go to global
//    memory;
//  * along h, inverse: a thread's lines are neighbouring columns (2q, 2q+1),
//    the pair of the inverse along w;
// so there is no conversion pass, and a pass costs one read and one write of
// shared memory per element beyond the products' operands.  Lanes are laid
// out as in dense_passes.cu (16-byte reads in two wavefronts); short sides
// give the lanes to lines instead of outputs.  Sums of more than 16 terms are
// taken in blocks of 16 added to the running total, as in the dense passes.
//
// What bounds it: multiply-adds and the reads of their operands with 12 warps
// per SM (FMA pipe 41-44%).  Against 4 x 4 tiles over the whole operators, 256
// MiB, us, forward / round trip: 12 x 12 343 / 585 -> 167 / 267, 26 x 32 382 /
// 704 -> 197 / 339, 48 x 48 573 / 1081 -> 396 / 718, 60 x 60 750 / 1414 -> 329 /
// 575.
#include <cuda_runtime.h>

#include <cstdio>
#include <type_traits>

#include "bdct_internal.h"
#include "dense_passes.h"
#include "ptx.cuh"
#include "small_dense.h"

namespace bdct {

namespace {

// Threads per CTA, by the line pairs I per thread and tile: 4, or 1 for calls
// of few arrays (small_dense_run).
template <int I>
constexpr int kThreadsOf = I == 1 ? 256 : 128;
constexpr int kMaxSide = 64;
constexpr int kMaxArrays = 64;
constexpr int kSlack = 256;    // pairs past a buffer that an edge tile may read

// Calls of at most this many elements per SM take tiles of 2 lines and eight
// warps: such a call lasts as long as one CTA's chain of passes, which large
// tiles and arrays packed into few CTAs only lengthen, and the short code of
// small tiles is fetched sooner (333 arrays of 12 x 12 forward 4.7 -> 2.9 us,
// round trip 7.7 -> 4.1; one 60 x 60 array 6.6 -> 4.9; 1000 of 20 x 20 6.0 ->
// 4.6).  From about 7000 the large tiles' fewer operand reads win (1000 arrays
// of 40 x 40, 10526 an SM, 14.3 us with small tiles, 13.1 with large; 2000 of
// 24 x 24, 7579 an SM, 8.9 and 8.2).
constexpr long long kFew = 6144;

// Elements per CTA: one tile of 2 I lines x 8 outputs per thread.
template <int I>
constexpr int kTarget = kThreadsOf<I> * 16 * I;

// Exact quotients of small unsigned values by a fixed divisor.
struct FastDiv {
    unsigned d, m;
    __host__ FastDiv(unsigned d_ = 1) : d(d_), m((unsigned)(((1ull << 32) + d_ - 1) / d_)) {}
    __device__ __forceinline__ unsigned div(unsigned x) const { return d == 1 ? x : __umulhi(x, m); }
};

// One axis of the products: half length (outputs pairs and contraction), lane
// layout.
struct Axis {
    int nh, tc, np;   // pairs, output quads, table row (pairs)
    int tcl;          // output quads per warp: 4, 2 or 1; 2 where 4 would idle two more of
                      // them (5 and 6 quads: 40 x 40 forward 368 -> 360 us, 48 x 48 408 -> 400,
                      // 36 x 36 393 -> 383, 256 MiB), but not 1 for 3 quads (24 x 24 inverse
                      // 194 -> 206: every lane then reads its own lines)
    __host__ __device__ explicit Axis(int n = 2)
        : nh((n + 1) / 2), tc((nh + 3) / 4), np(4 * tc), tcl(tc <= 2 ? tc : tc == 5 || tc == 6 ? 2 : 4)
    {
    }
    __host__ __device__ int line_block(int I) const { return 64 * I / tcl; }  // lines of a warp's tile
};

struct SmallParams {
    const float *in;
    float *out;
    const long long *in_off, *out_off;  // indexed arrays (element offsets), or null
    int tpr;                            // image tiles: tiles per image row (0: arrays)
    long long ld_in, ld_out;            // row strides (floats)
    long long count;
    int h, w;
    int G;                           // arrays per iteration
    int buf0, buf1, tabs;            // buffer and table sizes (pairs)
    const float2 *fw, *fh, *ih, *iw;  // tables of the passes used (dense_gen_table)
    const float *lam;                // spectral: Lambda (h x w), or null
    FastDiv div_h, div_w4, div_hp, div_wq, div_kh;
    long long groups;
};

__host__ __device__ constexpr int even2(int n) { return (n + 3) / 4 * 4 + 2; }  // pitch: 2 mod 4 pairs

// Pitches (pairs) of the operand buffers.
__host__ __device__ inline int pitch_fw(int h, int G) { return even2(2 * ((h + 1) / 2) * G); }
__host__ __device__ inline int pitch_h(int w, int G) { return even2(w * G); }
__host__ __device__ inline int pitch_iw(int h, int G) { return even2(h * G); }

// This lane's place in a warp tile of an axis: output quad and line group.
__device__ __forceinline__ void lane_place(const Axis &x, int lane, int &tq, int &la)
{
    if (x.tcl == 4) {
        tq = (lane & 1) + (lane >> 1 & 2);
        la = (lane >> 1 & 1) + (lane >> 2 & 6);
    } else if (x.tcl == 2) {
        tq = lane & 1;
        la = lane >> 1;
    } else {
        tq = 0;
        la = lane;
    }
}

// Products of lines l0 + i * ls (+ 1), i < I, and output pairs 4 tc .. 4 tc + 3:
// acc[2i + r][o] = (even, odd) sums over k < K of a[k][line] * t[k][o].
template <bool LONG, int I>
__device__ __forceinline__ void products(const float2 *a, int pitch, int ls, const float2 *t, int np, int K,
                                         float2 (&acc)[2 * I][4])
{
#pragma unroll
    for (int r = 0; r < 2 * I; ++r)
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[r][o] = make_float2(0.f, 0.f);
    auto step = [&](float2 (&sum)[2 * I][4]) {
        float2 x[2 * I], m[4];
#pragma unroll
        for (int i = 0; i < I; ++i) {
            const float4 v = *reinterpret_cast<const float4 *>(a + i * ls);
            x[2 * i] = make_float2(v.x, v.y);
            x[2 * i + 1] = make_float2(v.z, v.w);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float4 v = *reinterpret_cast<const float4 *>(t + 2 * i);
            m[2 * i] = make_float2(v.x, v.y);
            m[2 * i + 1] = make_float2(v.z, v.w);
        }
        a += pitch;
        t += np;
#pragma unroll
        for (int r = 0; r < 2 * I; ++r)
#pragma unroll
            for (int o = 0; o < 4; ++o) sum[r][o] = __ffma2_rn(x[r], m[o], sum[r][o]);
    };
    if constexpr (!LONG) {
#pragma unroll 2
        for (int k = 0; k < K; ++k) step(acc);
    } else {
        for (int k0 = 0; k0 < K; k0 += 16) {
            const int kn = min(16, K - k0);
            float2 part[2 * I][4];
#pragma unroll
            for (int r = 0; r < 2 * I; ++r)
#pragma unroll
                for (int o = 0; o < 4; ++o) part[r][o] = make_float2(0.f, 0.f);
#pragma unroll 2
            for (int k = 0; k < kn; ++k) step(part);
#pragma unroll
            for (int r = 0; r < 2 * I; ++r)
#pragma unroll
                for (int o = 0; o < 4; ++o) acc[r][o] = __fadd2_rn(acc[r][o], part[r][o]);
        }
    }
}

// DIR: DIR_FWD, DIR_INV, or DIR_RT for both pairs (Lambda between if set).
template <int DIR, bool LONG, int I>
__global__ void __launch_bounds__(kThreadsOf<I>, I == 1 ? 2 : LONG ? 2 : 3) k_small(const SmallParams p)
{
    constexpr int kThreads = kThreadsOf<I>;
    constexpr bool FWD = DIR != DIR_INV, INV = DIR != DIR_FWD;
    extern __shared__ __align__(16) float2 ssm[];
    float2 *buf[2] = {ssm, ssm + p.buf0};
    const int h = p.h, w = p.w, G = p.G, tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    const Axis aw(w), ah(h);
    const int kw = aw.nh, kh = ah.nh;
    float2 *tab = ssm + p.buf0 + p.buf1;
    float2 *t_fw = tab, *t_fh = t_fw + (FWD ? kw * aw.np : 0), *t_ih = t_fh + (FWD ? kh * ah.np : 0),
           *t_iw = t_ih + (INV ? kh * ah.np : 0);
    __shared__ long long base_in[kMaxArrays], base_out[kMaxArrays];
    // offsets of every row of the group: in global memory (the input's for the
    // first forward pass, the output's for the last inverse one) and, fixed, the
    // place of a row beside its mirror
    long long *row_off = reinterpret_cast<long long *>(tab + p.tabs);
    int *row_at = reinterpret_cast<int *>(row_off + G * h);
    if (FWD) {
        for (int l = tid; l < G * h; l += kThreads) {
            const int a = p.div_h.div(l), r = l - a * h, m = h - 1 - r;
            row_at[l] = 2 * (a * kh + min(r, m)) + (r > m);
        }
    }

    pdl_launch_dependents();
    // the tables are plan data, written before any transform was queued
    auto stage = [&](float2 *t, const float2 *src, int n) {
        for (int e = tid; e < n; e += kThreads) t[e] = __ldg(src + e);
    };
    if (FWD) {
        stage(t_fw, p.fw, kw * aw.np);
        stage(t_fh, p.fh, kh * ah.np);
    }
    if (INV) {
        stage(t_ih, p.ih, kh * ah.np);
        stage(t_iw, p.iw, kw * aw.np);
    }
    pdl_wait_prerequisites();

    int tqw, law, tqh, lah;
    lane_place(aw, lane, tqw, law);
    lane_place(ah, lane, tqh, lah);
    const int pfw = pitch_fw(h, G), ph = pitch_h(w, G), piw = pitch_iw(h, G);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);

    for (long long grp = blockIdx.x; grp < p.groups; grp += gridDim.x) {
        const long long a0 = grp * G;
        const int na = (int)(p.count - a0 < G ? p.count - a0 : G);
        __syncthreads();  // the last group's stores have taken their bases
        if (tid < na) {
            const long long a = a0 + tid;
            if (p.tpr) {
                const long long br = a / p.tpr, bc = a - br * p.tpr;
                base_in[tid] = br * h * p.ld_in + bc * w;
                base_out[tid] = br * h * p.ld_out + bc * w;
            } else {
                base_in[tid] = p.in_off ? p.in_off[a] : a * (long long)h * w;
                base_out[tid] = p.out_off ? p.out_off[a] : a * (long long)h * w;
            }
        }
        __syncthreads();
        for (int l = tid; l < na * h; l += kThreads) {
            const int a = p.div_h.div(l), r = l - a * h;
            row_off[l] = FWD ? base_in[a] + r * p.ld_in : base_out[a] + r * p.ld_out;
        }
        __syncthreads();

        // ---- the arrays, paired for the first pass, four tasks in flight a thread
        if constexpr (FWD) {
            // four elements from the front of a row and their mirrors
            const int Q = (w + 7) / 8, tasks = na * h * Q;
            for (int e0 = tid; e0 < tasks; e0 += 4 * kThreads) {
                float4 x[4], y[4];
                int at[4], kq[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int e = e0 + u * kThreads;
                    x[u] = y[u] = zero;
                    at[u] = -1;
                    if (e < tasks) {
                        const int row = p.div_wq.div(e), q = e - row * Q;
                        const float *g = p.in + row_off[row];
                        x[u] = __ldcg(reinterpret_cast<const float4 *>(g + 4 * q));
                        y[u] = __ldcg(reinterpret_cast<const float4 *>(g + w - 4 - 4 * q));
                        at[u] = row_at[row];
                        kq[u] = 4 * q;
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (at[u] < 0) continue;
                    float2 *o = buf[0] + kq[u] * pfw + at[u];
                    const float f[4] = {x[u].x, x[u].y, x[u].z, x[u].w}, b[4] = {y[u].w, y[u].z, y[u].y, y[u].x};
                    // w/2 is even: all four pairs, or the middle two
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (i < 2 || kq[u] + 4 <= kw) o[i * pfw] = half_pair(f[i], b[i]);
                }
            }
        } else {
            // coefficient rows 2k and 2k + 1, four columns
            const int W4 = w / 4, tasks = na * kh * W4;
            for (int e0 = tid; e0 < tasks; e0 += 4 * kThreads) {
                float4 x[4], y[4];
                int at[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int e = e0 + u * kThreads;
                    x[u] = y[u] = zero;
                    at[u] = -1;
                    if (e < tasks) {
                        const int row = p.div_w4.div(e), c = 4 * (e - row * W4);
                        const int a = p.div_kh.div(row), k = row - a * kh;
                        const float *g = p.in + base_in[a] + 2 * k * p.ld_in + c;
                        x[u] = __ldcg(reinterpret_cast<const float4 *>(g));
                        if (2 * k + 1 < h) y[u] = __ldcg(reinterpret_cast<const float4 *>(g + p.ld_in));
                        at[u] = k * ph + a * w + c;
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (at[u] < 0) continue;
                    float4 *o = reinterpret_cast<float4 *>(buf[0] + at[u]);
                    o[0] = make_float4(x[u].x, y[u].x, x[u].y, y[u].y);
                    o[1] = make_float4(x[u].z, y[u].z, x[u].w, y[u].w);
                }
            }
        }
        __syncthreads();

        float2 acc[2 * I][4];
        // tiles of a pass: line blocks x groups of tcl output quads, a warp each
        auto for_tiles = [&](const Axis &x, int lines, int tq, int la, auto &&tile) {
            const int lb = x.line_block(I), nlb = (lines + lb - 1) / lb, nt = nlb * ((x.tc + x.tcl - 1) / x.tcl);
            for (int t = warp; t < nt; t += kThreads / 32) {
                const int tg = t / nlb;
                const int q = tg * x.tcl + tq;
                tile((t - tg * nlb) * lb + 2 * la, lb / I, q < x.tc ? q : x.tc - 1, q < x.tc);
            }
        };

        if constexpr (FWD) {
            // ---- along w: rows (i, h-1-i) of an array
            for_tiles(aw, 2 * kh * na, tqw, law, [&](int l0, int ls, int tc, bool live) {
                products<LONG, I>(buf[0] + l0, pfw, ls, t_fw + 4 * tc, aw.np, kw, acc);
                if (!live) return;
#pragma unroll
                for (int i = 0; i < I; ++i) {
                    const int pr = (l0 + i * ls) / 2;
                    const int a = p.div_hp.div(pr), r = pr - a * kh;
                    if (a >= na) continue;
                    const bool mid = 2 * r + 1 == h;  // an odd height's middle row, its own mirror
                    float4 *o = reinterpret_cast<float4 *>(buf[1] + r * ph + a * w + 8 * tc);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (c >= 2 && 4 * tc + 4 > kw) continue;  // w/2 is even
                        const float2 u = acc[2 * i][c], v = acc[2 * i + 1][c];
                        const float2 e = half_pair(u.x, v.x), d = half_pair(u.y, v.y);
                        o[c] = mid ? make_float4(0.5f * u.x, 0.f, 0.5f * u.y, 0.f) : make_float4(e.x, e.y, d.x, d.y);
                    }
                }
            });
            __syncthreads();
            // ---- along h: neighbouring columns; coefficient rows 2o, 2o + 1
            for_tiles(ah, w * na, tqh, lah, [&](int l0, int ls, int tc, bool live) {
                products<LONG, I>(buf[1] + l0, ph, ls, t_fh + 4 * tc, ah.np, kh, acc);
                if (!live) return;
#pragma unroll
                for (int i = 0; i < I; ++i) {
                    const int l = l0 + i * ls;
                    const int a = p.div_w4.div(l / 4), c = l - a * w;
                    if (a >= na) continue;
                    if constexpr (DIR == DIR_FWD) {
                        // up to eight coefficient rows, one after the other
                        float *g = p.out + base_out[a] + c + 8 * tc * p.ld_out;
                        const int rows = h - 8 * tc;
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float2 u = acc[2 * i][q / 2], v = acc[2 * i + 1][q / 2];
                            if (q < rows) *reinterpret_cast<float2 *>(g) = q % 2 ? make_float2(u.y, v.y) : make_float2(u.x, v.x);
                            g += p.ld_out;
                        }
                    } else {
#pragma unroll
                        for (int o = 0; o < 4; ++o) {
                            const int k = 2 * (4 * tc + o);
                            if (k >= h) continue;
                            float2 u = acc[2 * i][o], v = acc[2 * i + 1][o];
                            if (p.lam) {
                                const float2 l0v = __ldg(reinterpret_cast<const float2 *>(p.lam + k * w + c));
                                u.x *= l0v.x;
                                v.x *= l0v.y;
                                if (k + 1 < h) {
                                    const float2 l1v = __ldg(reinterpret_cast<const float2 *>(p.lam + (k + 1) * w + c));
                                    u.y *= l1v.x;
                                    v.y *= l1v.y;
                                }
                            }
                            *reinterpret_cast<float4 *>(buf[0] + (k / 2) * ph + l) = make_float4(u.x, u.y, v.x, v.y);
                        }
                    }
                }
            });
            if constexpr (DIR == DIR_RT) __syncthreads();
        }
        if constexpr (INV) {
            // ---- along h, inverse: rows j and h-1-j of neighbouring columns
            for_tiles(ah, w * na, tqh, lah, [&](int l0, int ls, int tc, bool live) {
                products<LONG, I>(buf[0] + l0, ph, ls, t_ih + 4 * tc, ah.np, kh, acc);
                if (!live) return;
#pragma unroll
                for (int i = 0; i < I; ++i) {
                    const int l = l0 + i * ls;
                    const int a = p.div_w4.div(l / 4), c = l - a * w;
                    if (a >= na) continue;
                    float2 *b = buf[1] + (c / 2) * piw + a * h;
#pragma unroll
                    for (int o = 0; o < 4; ++o) {
                        const int j = 4 * tc + o;
                        if (j >= kh) continue;
                        const float2 u = acc[2 * i][o], v = acc[2 * i + 1][o];
                        b[j] = make_float2(u.x + u.y, v.x + v.y);
                        b[h - 1 - j] = make_float2(u.x - u.y, v.x - v.y);
                    }
                }
            });
            if constexpr (DIR == DIR_RT) {
                for (int l = tid; l < na * h; l += kThreads) {
                    const int a = p.div_h.div(l), r = l - a * h;
                    row_off[l] = base_out[a] + r * p.ld_out;
                }
            }
            __syncthreads();
            // ---- along w, inverse: rows to global memory
            for_tiles(aw, h * na, tqw, law, [&](int l0, int ls, int tc, bool live) {
                products<LONG, I>(buf[1] + l0, piw, ls, t_iw + 4 * tc, aw.np, kw, acc);
                if (!live) return;
                const int o0 = 4 * tc;
#pragma unroll
                for (int i = 0; i < I; ++i)
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        const int l = l0 + i * ls + s;
                        if (l >= na * h) continue;
                        float *g = p.out + row_off[l];
                        const float2 *v = acc[2 * i + s];
                        if (o0 + 4 <= kw) {
                            *reinterpret_cast<float4 *>(g + o0) =
                                make_float4(v[0].x + v[0].y, v[1].x + v[1].y, v[2].x + v[2].y, v[3].x + v[3].y);
                            *reinterpret_cast<float4 *>(g + w - 4 - o0) =
                                make_float4(v[3].x - v[3].y, v[2].x - v[2].y, v[1].x - v[1].y, v[0].x - v[0].y);
                        } else {
                            // the two middle pairs (w a multiple of 4, w/2 not): one float4
                            *reinterpret_cast<float4 *>(g + o0) =
                                make_float4(v[0].x + v[0].y, v[1].x + v[1].y, v[1].x - v[1].y, v[0].x - v[0].y);
                        }
                    }
            });
        }
    }
}

template <int DIR, bool LONG, int I>
cudaError_t launch(SmallParams p, int sms, cudaStream_t stream)
{
    constexpr int kThreads = kThreadsOf<I>;
    const Axis aw(p.w), ah(p.h);
    constexpr bool FWD = DIR != DIR_INV, INV = DIR != DIR_FWD;
    // arrays per iteration: about kTarget elements but no more than spread the
    // call over the SMs, and among the counts near it the one whose warp tiles
    // fill the four warps best (the larger on a tie)
    auto tiles = [](const Axis &x, int lines) {
        return (lines + x.line_block(I) - 1) / x.line_block(I) * ((x.tc + x.tcl - 1) / x.tcl);
    };
    long long gmax = kTarget<I> / (p.h * p.w);
    if (gmax > (p.count + sms - 1) / sms) gmax = (p.count + sms - 1) / sms;
    if (gmax < 1) gmax = 1;
    if (gmax > kMaxArrays) gmax = kMaxArrays;
    int G = 1;
    double best = 0.0;
    for (int g = (int)gmax; g >= 1 && 2 * g >= gmax; --g) {
        auto rounds = [&](int t) { return (t + kThreads / 32 - 1) / (kThreads / 32); };
        const int r = rounds(tiles(aw, FWD ? 2 * ah.nh * g : p.h * g)) + rounds(tiles(ah, p.w * g));
        const double per = (double)g / r;
        if (per > best * 1.02) {
            best = per;
            G = g;
        }
    }
    p.G = G;
    const int fw = aw.nh * pitch_fw(p.h, G) + kSlack, hh = ah.nh * pitch_h(p.w, G) + kSlack,
              iw = aw.nh * pitch_iw(p.h, G) + kSlack;
    p.buf0 = FWD ? (INV && hh > fw ? hh : fw) : hh;
    p.buf1 = FWD ? (INV && iw > hh ? iw : hh) : iw;
    p.buf0 = (p.buf0 + 1) / 2 * 2;
    p.buf1 = (p.buf1 + 1) / 2 * 2;
    const int tabs = (FWD + INV) * (aw.nh * aw.np + ah.nh * ah.np);
    p.tabs = tabs;
    const size_t smem = ((size_t)p.buf0 + p.buf1 + tabs) * sizeof(float2) + (size_t)G * p.h * 12;
    if (smem > 220 * 1024) return cudaErrorInvalidValue;
    p.groups = (p.count + G - 1) / G;

    auto kern = k_small<DIR, LONG, I>;
    static DeviceLaunchCache cache;
    int dev = 0, bps = 0, unused = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cache.get(
        dev,
        [&](int, int &b, int &n) {
            b = n = 1;
            return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
        },
        &bps, &unused);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    long long grid = (long long)per_sm * sms;
    if (grid > p.groups) grid = p.groups;
    if (debug_enabled()) {
        // once per configuration, not per launch
        static std::mutex mu;
        static long long last = -1;
        const long long key = ((long long)p.h << 20) | ((long long)p.w << 8) | (DIR * 8 + I);
        std::lock_guard<std::mutex> lock(mu);
        if (key != last) {
            last = key;
            fprintf(stderr, "[bdct] k_small<%d,%d,%d> %dx%d: %d arrays per iteration, %d CTAs/SM, smem %zu B\n", DIR,
                    (int)LONG, I, p.h, p.w, G, per_sm, smem);
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p);
}

}  // namespace

bool small_dense_supported(int h, int w)
{
    return h >= 1 && w >= 4 && h <= kMaxSide && w <= kMaxSide && w % 4 == 0;
}

cudaError_t small_dense_run(int h, int w, Dir dir, const SmallTables &t, const float *lam, const ExecGeom &g,
                            cudaStream_t stream)
{
    if (!small_dense_supported(h, w)) return cudaErrorInvalidValue;
    if (g.count <= 0) return cudaSuccess;
    SmallParams p{};
    p.in = g.in;
    p.out = g.out;
    p.in_off = g.in_off;
    p.out_off = g.out_off;
    p.tpr = g.tiled ? g.tiles_per_row : 0;
    p.ld_in = g.tiled ? g.ld_in : w;
    p.ld_out = g.tiled ? g.ld_out : w;
    p.count = g.count;
    p.h = h;
    p.w = w;
    p.fw = reinterpret_cast<const float2 *>(t.fw);
    p.fh = reinterpret_cast<const float2 *>(t.fh);
    p.ih = reinterpret_cast<const float2 *>(t.ih);
    p.iw = reinterpret_cast<const float2 *>(t.iw);
    p.lam = dir == DIR_SPEC ? lam : nullptr;
    p.div_h = FastDiv(h);
    p.div_w4 = FastDiv(w / 4);
    p.div_hp = FastDiv((h + 1) / 2);
    p.div_wq = FastDiv((w + 7) / 8);
    p.div_kh = FastDiv((h + 1) / 2);
    static DeviceLaunchCache cache;
    int dev = 0, bps = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cache.get(
        dev,
        [&](int d, int &b, int &n) {
            b = 1;
            return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, d);
        },
        &bps, &sms);
    if (e != cudaSuccess) return e;
    const bool is_long = h > 32 || w > 32;  // more than 16 pairs on an axis
    const bool few = g.count * (long long)(h * w) <= kFew * sms;
    auto run = [&](auto dir_c) {
        constexpr int D = decltype(dir_c)::value;
        if (few) return is_long ? launch<D, true, 1>(p, sms, stream) : launch<D, false, 1>(p, sms, stream);
        return is_long ? launch<D, true, 4>(p, sms, stream) : launch<D, false, 4>(p, sms, stream);
    };
    if (dir == DIR_FWD) return run(std::integral_constant<int, DIR_FWD>{});
    if (dir == DIR_INV) return run(std::integral_constant<int, DIR_INV>{});
    return run(std::integral_constant<int, DIR_RT>{});
}

}  // namespace bdct
