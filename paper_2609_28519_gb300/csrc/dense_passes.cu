// Separable dense passes: the general-shape FP32 route.
//
// Eq. 2 of the BRiDCT paper is the sandwich M_h X M_w^T, with M = Q_n for the
// forward transform (Eq. 1) and M = Q_n^T for the inverse; Section 7.1 makes
// h and w independent.  Here the two 1D operators are applied as two FP32
// matrix products, one pass along each axis, through a plan-owned workspace:
// the route of shapes without a fast kernel (sides above 64 with other
// factors, which Eq. 1 defines for any n) and of the allocation-free entry
// point.
//
// Half products.  cos(pi (2j+1) k / (2n)) is even about the middle of the
// line for even k and odd for odd k, so with s_j = (x_j + x_{n-1-j}) / 2 and
// d_j = (x_j - x_{n-1-j}) / 2 (j < n/2; half_pair, ptx.cuh) the even outputs are
// a product with s and the odd ones a product with d, each half as long: n/2
// multiply-adds per point instead of n.  The inverse runs it backwards: a from the even coefficients,
// b from the odd ones, x_j = a_j + b_j, x_{n-1-j} = a_j - b_j.
//
// Tiles.  The two products run in the halves of packed pairs: (s_j, d_j) of a
// line times (M_even, M_odd) of an output pair is one instruction, and neither
// operand has to be duplicated or moved to form its pair.  A CTA takes 64
// lines and up to 64 output pairs, a thread 8 lines x 4 pairs.  Per contraction
// index it reads six float4 for 64 multiply-adds; a warp's lanes are 8 lines
// by 4 output quads, so each of those reads is two shared-memory wavefronts
// and the multiply-adds, not the reads, bound the loop.  The outputs are dealt
// to the tiles evenly in steps of 4, so a side of 100 fills 52 columns for its
// 50 pairs.  Sums and differences are formed once, as a chunk of 16 indices
// goes from global to shared memory; the next chunk's loads are in flight
// during the current products.  Each chunk's products are summed on their own
// and added to the running total, so the rounding error grows like 16 + n/32
// rather than n/2.
//
// What bounds it: multiply-adds, with eight warps per SM (FMA pipe 46-49%).
// Against whole operators in 64 x 64 tiles, us: 100 x 100, 256 MiB, forward 1696
// -> 528, inverse 1696 -> 510, round trip 3392 -> 1037; 16 arrays of 1000 x
// 1000, forward 2431 -> 728.  Three CTAs per SM (168 registers, spills), the
// products split by warps and a persistent form were 7-23% slower.
#include <cuda_runtime.h>

#include "bdct_internal.h"
#include "dense_passes.h"
#include "ptx.cuh"

namespace bdct {

// cos(pi m / (2n)) for integer m, reduced exactly, evaluated in FP64.
__device__ double cos_half_turns(long long m, long long n)
{
    const long long d = 2 * n;  // angle = pi m / d
    long long r = m % (2 * d);
    if (r < 0) r += 2 * d;
    if (r > d) r = 2 * d - r;  // [0, d]
    double sign = 1.0;
    if (2 * r > d) { r = d - r; sign = -1.0; }  // [0, d/2]
    if (r == 0) return sign;
    if (2 * r == d) return 0.0;
    return sign * cospi((double)r / (double)d);
}

// s_k cos(pi (2j+1) k / (2n))
// norm 0 (orthonormal): s_k = alpha_k of Eq. 1
// norm 1 (REDFT pair):  forward (direction 1) s_k = 2, inverse s_0 = 1, s_k = 2
__device__ double operator_entry(int k, int j, int n, int direction, int norm)
{
    double s;
    if (norm == 0) s = (k == 0) ? sqrt(1.0 / n) : sqrt(2.0 / n);
    else if (direction == 1) s = 2.0;
    else s = (k == 0) ? 1.0 : 2.0;
    return s * cos_half_turns((2LL * j + 1) * k, n);
}

namespace {

constexpr int kThreads = 128;
constexpr int kLines = 64;          // lines per CTA
constexpr int kChunk = 16;          // contraction indices per stage
constexpr int kPitch = kLines + 2;  // stage row pitch (pairs)
constexpr int kMaxTile = 64;        // output pairs per CTA at most
constexpr int kResident = 2;        // CTAs per SM: no spills (three, with 168 registers, 1134 us where two take 1057)

// Half operators of side n: pairs (even, odd) [kp][np], zero in the padding;
// kp, np = n/2 rounded up to whole chunks and tiles.
struct DenseShape {
    int n, nh, tiles, tc, np, kp;
    __host__ __device__ explicit DenseShape(int n_)
        : n(n_), nh((n_ + 1) / 2), tiles((nh + kMaxTile - 1) / kMaxTile),
          tc(((nh + tiles - 1) / tiles + 3) / 4), np(tiles * tc * 4), kp((nh + kChunk - 1) / kChunk * kChunk)
    {
    }
};

// forward: t[j][o] = 2 M[2o + e][j]; inverse: t[o][j] = M^T[j][2o + e], e the half.
// One warp per block and one entry per thread: FP64 runs at two lanes a cycle,
// so the warps are spread over the SMs.
__global__ void k_gen_half(float *t, DenseShape q, int direction, int norm)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 2ll * q.kp * q.np) return;
    const int r = (int)(idx / 2 / q.np), c = (int)(idx / 2 % q.np), e = (int)(idx & 1);
    const int k = 2 * (direction == 1 ? c : r) + e, j = direction == 1 ? r : c;
    const double f = direction == 1 ? 2.0 : 1.0;
    t[idx] = j < q.nh && k < q.n ? (float)(f * operator_entry(k, j, q.n, direction, norm)) : 0.f;
}

struct DenseParams {
    const float *in;
    float *out;
    const float2 *table;
    const long long *in_off, *out_off;  // indexed arrays (element offsets), or null
    const float *lam;                   // columns, forward: output (k, l) times lam[k * w + l]; or null
    long long lines;                    // rows or columns of all arrays
    int h, w;
};

// ROWS: lines are rows (contiguous); else columns, four neighbours at a time.
template <bool ROWS, bool INV>
__global__ void __launch_bounds__(kThreads, kResident) k_dense(const DenseParams p)
{
    __shared__ __align__(16) float2 as[2][kChunk][kPitch];
    __shared__ __align__(16) float2 bs[2][kChunk][kMaxTile];
    const int n = ROWS ? p.w : p.h, w = p.w;
    const DenseShape q(n);
    const int tid = threadIdx.x;
    const long long per = ROWS ? p.h : p.w;  // lines per array
    const int tile = blockIdx.x % q.tiles;
    const long long line0 = (long long)(blockIdx.x / q.tiles) * kLines;

    pdl_launch_dependents();
    pdl_wait_prerequisites();

    // where the CTA's lines begin (a column's first element), in the input and
    // the output: the divisions are done once per line, not per use
    __shared__ long long off_in[kLines], off_out[kLines];
    if (tid < kLines && line0 + tid < p.lines) {
        const long long b = (line0 + tid) / per, i = line0 + tid - b * per;
        const long long in_array = ROWS ? i * w : i, packed = b * (long long)p.h * w;
        off_in[tid] = (p.in_off ? p.in_off[b] : packed) + in_array;
        off_out[tid] = (p.out_off ? p.out_off[b] : packed) + in_array;
    }
    __syncthreads();

    // ---- this thread's two tasks of a chunk: two float4 each
    const float *pa[2], *pb[2];  // of the next chunk: moved on by each fetch
    int kk[2], ln[2];
    bool live[2];
    const long long step_a = ROWS ? (INV ? 2 * kChunk : kChunk) : (INV ? 2 * kChunk : kChunk) * (long long)w;
    const long long step_b = INV ? step_a : -step_a;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        if (ROWS) {
            kk[u] = 4 * (tid % 4);  // four contraction indices of one line
            ln[u] = tid / 4 + 32 * u;
        } else {
            kk[u] = tid / 16 + 8 * u;  // one contraction index of four columns
            ln[u] = 4 * (tid % 16);
        }
        live[u] = line0 + ln[u] < p.lines;
        const float *base = live[u] ? p.in + off_in[ln[u]] : p.in;
        // forward: index k and its mirror; inverse: coefficients 2k and 2k + 1 (rows: eight from 2k)
        pa[u] = base + (INV ? 2 * kk[u] : kk[u]) * (ROWS ? 1ll : (long long)w);
        pb[u] = base + (INV ? (ROWS ? 2 * kk[u] + 4 : 2 * kk[u] + 1) : (ROWS ? n - 4 - kk[u] : n - 1 - kk[u])) *
                           (ROWS ? 1ll : (long long)w);
    }
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 va[2], vb[2];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int k = k0 + kk[u];
            const bool a = live[u] && (INV ? 2 * k < n : k < q.nh);
            const bool b = live[u] && (INV ? (ROWS ? 2 * k + 4 : 2 * k + 1) < n : k < q.nh);
            va[u] = a ? __ldcg(reinterpret_cast<const float4 *>(pa[u])) : zero;
            vb[u] = b ? __ldcg(reinterpret_cast<const float4 *>(pb[u])) : zero;
            pa[u] += step_a;
            pb[u] += step_b;
        }
    };
    auto put = [&](int st, int k0) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float4 a = va[u], b = vb[u];
            if (ROWS) {
                float2 v[4];
                if (!INV) {
                    const float x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.w, b.z, b.y, b.x};
#pragma unroll
                    for (int i = 0; i < 4; ++i)  // past the middle: the mirrored pairs again, left out
                        v[i] = k0 + kk[u] + i < q.nh ? half_pair(x[i], y[i]) : make_float2(0.f, 0.f);
                } else {
                    v[0] = make_float2(a.x, a.y); v[1] = make_float2(a.z, a.w);
                    v[2] = make_float2(b.x, b.y); v[3] = make_float2(b.z, b.w);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) as[st][kk[u] + i][ln[u]] = v[i];
            } else {
                float2 v0 = make_float2(a.x, b.x), v1 = make_float2(a.y, b.y), v2 = make_float2(a.z, b.z),
                       v3 = make_float2(a.w, b.w);
                if (!INV) {
                    if (2 * (k0 + kk[u]) + 1 == n) {  // the middle of an odd length, its own mirror
                        v0 = make_float2(0.5f * a.x, 0.f);
                        v1 = make_float2(0.5f * a.y, 0.f);
                        v2 = make_float2(0.5f * a.z, 0.f);
                        v3 = make_float2(0.5f * a.w, 0.f);
                    } else {
                        v0 = half_pair(a.x, b.x);
                        v1 = half_pair(a.y, b.y);
                        v2 = half_pair(a.z, b.z);
                        v3 = half_pair(a.w, b.w);
                    }
                }
                float4 *o = reinterpret_cast<float4 *>(&as[st][kk[u]][ln[u]]);
                o[0] = make_float4(v0.x, v0.y, v1.x, v1.y);
                o[1] = make_float4(v2.x, v2.y, v3.x, v3.y);
            }
        }
    };
    const float2 *tab = p.table + tile * (q.tc * 4);
    auto fetch_op = [&](int st, int k0) {
        // eight threads a row, 16 bytes at a time
        const int r = tid / 8;
        const float2 *g = tab + (long long)(k0 + r) * q.np;
        for (int c = tid % 8; c < 2 * q.tc; c += 8) cp_async16(&bs[st][r][2 * c], g + 2 * c);
        cp_async_commit();
    };
    static_assert(kThreads == 8 * kChunk, "operator rows");

    // ---- compute role: lines 2 la + 16 i and the next (i < 4), output pairs 4 tc ..
    // lanes: output quad from bits 0 and 2, lines from bits 1, 3 and 4, so that
    // lanes i and i^1 read the same lines and lanes i and i^2 the same outputs
    // (a 16-byte read then takes two wavefronts instead of four)
    const int lane = tid % 32;
    const int tc = tid / 32 * 4 + (lane & 1) + (lane >> 1 & 2), la = (lane >> 1 & 1) + (lane >> 2 & 6);
    const bool active = tc < q.tc;
    float2 acc[8][4];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[r][o] = make_float2(0.f, 0.f);
    fetch_op(0, 0);
    fetch(0);
    put(0, 0);
    cp_async_wait_group<0>();
    __syncthreads();
    for (int k0 = 0, st = 0; k0 < q.nh; k0 += kChunk, st ^= 1) {
        const bool more = k0 + kChunk < q.nh;
        if (more) {
            fetch_op(st ^ 1, k0 + kChunk);
            fetch(k0 + kChunk);
        }
        if (active) {
            float2 part[8][4];
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int o = 0; o < 4; ++o) part[r][o] = make_float2(0.f, 0.f);
            auto step = [&](int k) {
                float2 x[8], m[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 v = *reinterpret_cast<const float4 *>(&as[st][k][2 * la + 16 * i]);
                    x[2 * i] = make_float2(v.x, v.y);
                    x[2 * i + 1] = make_float2(v.z, v.w);
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float4 v = *reinterpret_cast<const float4 *>(&bs[st][k][4 * tc + 2 * i]);
                    m[2 * i] = make_float2(v.x, v.y);
                    m[2 * i + 1] = make_float2(v.z, v.w);
                }
#pragma unroll
                for (int r = 0; r < 8; ++r)
#pragma unroll
                    for (int o = 0; o < 4; ++o) part[r][o] = __ffma2_rn(x[r], m[o], part[r][o]);
            };
            if (k0 + kChunk <= q.nh) {
#pragma unroll
                for (int k = 0; k < kChunk; ++k) step(k);
            } else {
                const int last = (q.nh - k0 + 1) / 2;  // the padding is zero
#pragma unroll 1
                for (int k = 0; k < last; ++k) {
                    step(2 * k);
                    step(2 * k + 1);
                }
            }
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int o = 0; o < 4; ++o) acc[r][o] = __fadd2_rn(acc[r][o], part[r][o]);
        }
        if (more) {
            put(st ^ 1, k0 + kChunk);
            cp_async_wait_group<0>();
            __syncthreads();
        }
    }
    if (!active) return;
    const int o0 = 4 * (tile * q.tc + tc);  // first output pair of this thread
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const long long line = line0 + 2 * la + 16 * i;
        if (line >= p.lines) continue;
        if (!ROWS) {
            // two neighbouring columns (w is a multiple of 4, so they share an array)
            float *dst = p.out + off_out[2 * la + 16 * i];
            const float *lam = !INV && p.lam ? p.lam + line % w : nullptr;
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const float2 u = acc[2 * i][o], v = acc[2 * i + 1][o];
                const int j = o0 + o;
                if (j >= q.nh) continue;
                float2 a, b;
                int ka, kb;
                if (!INV) {
                    a = make_float2(u.x, v.x);
                    b = make_float2(u.y, v.y);
                    ka = 2 * j;
                    kb = 2 * j + 1;
                } else {
                    a = make_float2(u.x + u.y, v.x + v.y);
                    b = make_float2(u.x - u.y, v.x - v.y);
                    ka = j;
                    kb = n - 1 - j;
                }
                if (!INV && lam) {
                    const float2 l = __ldg(reinterpret_cast<const float2 *>(lam + (long long)ka * w));
                    a = make_float2(a.x * l.x, a.y * l.y);
                    if (kb < n) {
                        const float2 m = __ldg(reinterpret_cast<const float2 *>(lam + (long long)kb * w));
                        b = make_float2(b.x * m.x, b.y * m.y);
                    }
                }
                *reinterpret_cast<float2 *>(dst + (long long)ka * w) = a;
                if (kb < n) *reinterpret_cast<float2 *>(dst + (long long)kb * w) = b;
            }
        } else {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                if (line + r >= p.lines) continue;
                float *dst = p.out + off_out[2 * la + 16 * i + r];
                const float2 *v = acc[2 * i + r];
                if (!INV) {
                    // coefficients 2 o0 .. 2 o0 + 7
                    if (2 * o0 < n) *reinterpret_cast<float4 *>(dst + 2 * o0) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
                    if (2 * o0 + 4 < n)
                        *reinterpret_cast<float4 *>(dst + 2 * o0 + 4) = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
                } else if (o0 + 4 <= q.nh) {
                    *reinterpret_cast<float4 *>(dst + o0) =
                        make_float4(v[0].x + v[0].y, v[1].x + v[1].y, v[2].x + v[2].y, v[3].x + v[3].y);
                    *reinterpret_cast<float4 *>(dst + n - 4 - o0) =
                        make_float4(v[3].x - v[3].y, v[2].x - v[2].y, v[1].x - v[1].y, v[0].x - v[0].y);
                } else {
#pragma unroll
                    for (int o = 0; o < 4; ++o)
                        if (o0 + o < q.nh) {
                            dst[o0 + o] = v[o].x + v[o].y;
                            dst[n - 1 - o0 - o] = v[o].x - v[o].y;
                        }
                }
            }
        }
    }
}

template <bool ROWS, bool INV>
cudaError_t launch(const DenseParams &p, cudaStream_t stream)
{
    const DenseShape q(ROWS ? p.w : p.h);
    const long long blocks = (p.lines + kLines - 1) / kLines * q.tiles;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_dense<ROWS, INV>, p);
}

}  // namespace

size_t dense_table_floats(int n)
{
    const DenseShape q(n);
    return (size_t)2 * q.kp * q.np;
}

cudaError_t dense_gen_table(float *t, int n, int direction, int norm, cudaStream_t stream)
{
    const long long total = (long long)dense_table_floats(n);
    k_gen_half<<<(unsigned)((total + 31) / 32), 32, 0, stream>>>(t, DenseShape(n), direction, norm);
    return cudaGetLastError();
}

cudaError_t dense_pass(const DensePass &d, cudaStream_t stream)
{
    if (d.count <= 0) return cudaSuccess;
    DenseParams p{d.in, d.out, reinterpret_cast<const float2 *>(d.table), d.in_off, d.out_off, d.lam, d.count * (d.rows ? d.h : d.w), d.h, d.w};
    if (d.rows) return d.inverse ? launch<true, true>(p, stream) : launch<true, false>(p, stream);
    return d.inverse ? launch<false, true>(p, stream) : launch<false, false>(p, stream);
}

}  // namespace bdct
