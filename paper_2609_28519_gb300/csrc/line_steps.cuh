// Steps of the FFT evaluation of a DCT line on packed couples, shared by the
// line engine (fp32_lines_kernel.cuh) and the on-chip kernels of sides 64 and 128
// (fp32_block.cu).  fp32_lines_kernel.cuh's header derives the factorization and the
// packed form; this file holds its short FFTs, twiddles and the split.
//
// Rounding.  A rotation and the sums that take it run as one chain of
// multiply-adds, the smaller product first (a product or a sum is rounded at
// its own size), and an eighth of a turn as a sum times 1/sqrt 2; that costs no
// more instructions than rotating first.  With the mean of the rounded roots
// taken back in the last factor (line_error, fp32_lines.cu) the relative L2 of
// 1e6 uniform values fell from 1.66 to 1.42e-7 (192 x 192 forward), 2.57 to 2.10
// (its round trip), 1.82 to 1.57 (768 x 768 forward), 1.45 to 1.33 (128 x 128
// forward), times by 0-3%.
#pragma once

#include <cuda_runtime.h>

#include "dct_cores.cuh"

namespace bdct {

// Radices of a line of N points: L = N/2 = R1 R2 R3 (R2 = 1: two steps), for
// the line engine's forward passes (set 0), its others (1) and every pass over
// few lines (2).  The best of a sweep: fewer, larger steps move less through
// shared memory (1024 points inverse: 32 x 16 runs 0.398 of HBM where 8 x 8 x 8
// runs 0.356), but the adjoint also holds its coefficients in registers; few
// lines want the shortest chain.  Sides 64, 128 and 192 split alike in all.
template <int N, int SET = 1>
struct LineSplit {
    static constexpr int L = N / 2;
    static constexpr int R1 = N == 64 ? 4 : N == 128 || N == 192 ? 8
                            : SET == 0 ? (N == 256 || N == 384 || N == 1536 ? 8 : N == 768 ? 24 : 16)
                            : SET == 1 ? (N == 384 || N == 768 ? 24 : N == 1024 ? 32 : N == 1536 ? 12 : 16)
                                       : (N == 768 || N == 1024 || N == 1536 ? 8 : 16);
    static constexpr int R3 = N == 64 || N == 128 ? 8 : N == 192 ? 12
                            : SET == 0 ? (N == 256 || N == 512 ? 8 : N == 384 ? 6 : 16)
                            : SET == 1 ? (N == 512 || N == 1024 ? 16 : 8)
                                       : (N == 384 ? 12 : N == 512 ? 16 : 8);
    static constexpr int R2 = L / (R1 * R3);
    static constexpr int M1 = L / R1;  // columns of the first step
    static constexpr int C = L / R3;   // columns of the last step
    static constexpr int U1 = R1 * (M1 / 2);               // twiddle entries (float4) of the first step,
    static constexpr int U2 = R2 > 1 ? R2 * (R3 / 2) : 0;  // of the middle step,
    static constexpr int US = L / 2 + L / 4;               // and of the split (L/2 slots of 24 bytes)
    static constexpr int TAB = U1 + U2 + US;
    static_assert(R1 * R2 * R3 == L && R1 % 2 == 0 && R3 % 2 == 0 && M1 % 2 == 0 && C % 2 == 0, "split");
    static_assert(R2 == 1 || R2 % 2 == 0, "split");
};

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// cos and sin of 2 pi j / R, R a power of two or three times one.
template <int R>
__device__ __forceinline__ void unit_root(int j, float &c, float &s)
{
    c = R % 3 == 0 ? cospi3_md(2 * j, R) : cospi_md(2 * j, R);
    s = R % 3 == 0 ? sinpi3_md(2 * j, R) : sinpi_md(2 * j, R);
}

// (a, b) -> (a + w b, a - w b), w = exp(-2 pi i k / R), 0 <= k < R/2, the
// rotation inside the sums.
template <int R>
__device__ __forceinline__ void butterfly(float2 ar, float2 ai, float2 br, float2 bi, int k, float2 &pr, float2 &pi,
                                          float2 &mr, float2 &mi)
{
    using O = VOps<float2>;
    if (k == 0) {
        pr = O::add(ar, br); pi = O::add(ai, bi);
        mr = O::sub(ar, br); mi = O::sub(ai, bi);
        return;
    }
    if (4 * k == R) {
        pr = O::add(ar, bi); pi = O::sub(ai, br);
        mr = O::sub(ar, bi); mi = O::add(ai, br);
        return;
    }
    float c, s;
    unit_root<R>(k, c, s);
    if (8 * k == R || 8 * k == 3 * R) {
        // w = (+-1 - i) / sqrt 2: two sums, then one instruction each
        const float2 t = 8 * k == R ? O::add(br, bi) : O::sub(bi, br), u = 8 * k == R ? O::sub(bi, br) : O::add(br, bi);
        const float v = 8 * k == R ? s : -s;
        pr = O::fma(t, s, ar); pi = O::fma(u, v, ai);
        mr = O::fma(t, -s, ar); mi = O::fma(u, -v, ai);
        return;
    }
    if (8 * k < R || 8 * k > 3 * R) {  // the smaller product first: its sum is rounded at the smaller value
        pr = O::fma(br, c, O::fma(bi, s, ar));
        pi = O::fma(bi, c, O::fma(br, -s, ai));
        mr = O::fma(br, -c, O::fma(bi, -s, ar));
        mi = O::fma(bi, -c, O::fma(br, s, ai));
    } else {
        pr = O::fma(bi, s, O::fma(br, c, ar));
        pi = O::fma(br, -s, O::fma(bi, c, ai));
        mr = O::fma(bi, -s, O::fma(br, -c, ar));
        mi = O::fma(br, s, O::fma(bi, -c, ai));
    }
}

// Outputs k, k + R/3, k + 2R/3 of a radix-3 stage of R points: the 3-point DFT
// of (a, w^k b, w^2k c), w = exp(-2 pi i / R).
template <int R>
__device__ __forceinline__ void fft3(float2 ar, float2 ai, float2 br, float2 bi, float2 cr, float2 ci, int k, float2 &xr,
                                     float2 &xi, float2 &yr, float2 &yi, float2 &zr, float2 &zi)
{
    using O = VOps<float2>;
    float2 pr = br, pi = bi, qr = cr, qi = ci;
    if (k != 0) {
        rot3(br, bi, k, R, pr, pi);
        rot3(cr, ci, 2 * k, R, qr, qi);
    }
    const float2 tr = O::add(pr, qr), ti = O::add(pi, qi), sr = O::sub(pr, qr), si = O::sub(pi, qi);
    const float2 mr = O::fma(tr, -0.5f, ar), mi = O::fma(ti, -0.5f, ai);
    const float h = cospi3_md(256, 1536);  // sqrt(3) / 2
    xr = O::add(ar, tr); xi = O::add(ai, ti);
    yr = O::fma(si, h, mr); yi = O::fma(sr, -h, mi);
    zr = O::fma(si, -h, mr); zi = O::fma(sr, h, mi);
}

// FFT of R points a_j given u_j = a_j + a_{j+R/2} and v_j = a_j - a_{j+R/2}:
// decimation in time, the pairs its first stage.
template <int R>
__device__ __forceinline__ void fft_from_uv(const float2 (&ur)[R / 2], const float2 (&ui)[R / 2],
                                            const float2 (&vr)[R / 2], const float2 (&vi)[R / 2], float2 (&dr)[R],
                                            float2 (&di)[R])
{
    using O = VOps<float2>;
    if constexpr (R == 2) {
        dr[0] = ur[0]; di[0] = ui[0];
        dr[1] = vr[0]; di[1] = vi[0];
    } else {
        constexpr int Q = R % 3 == 0 ? 3 : 2, M = R / Q;
        float2 er[Q][M], ei[Q][M];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            float2 pr[M / 2], pi[M / 2], mr[M / 2], mi[M / 2];
#pragma unroll
            for (int j = 0; j < M / 2; ++j) {
                pr[j] = ur[Q * j + q]; pi[j] = ui[Q * j + q];
                mr[j] = vr[Q * j + q]; mi[j] = vi[Q * j + q];
            }
            fft_from_uv<M>(pr, pi, mr, mi, er[q], ei[q]);
        }
#pragma unroll
        for (int k = 0; k < M; ++k) {
            if constexpr (Q == 2)
                butterfly<R>(er[0][k], ei[0][k], er[1][k], ei[1][k], k, dr[k], di[k], dr[k + M], di[k + M]);
            else
                fft3<R>(er[0][k], ei[0][k], er[1][k], ei[1][k], er[2][k], ei[2][k], k, dr[k], di[k], dr[k + M], di[k + M],
                        dr[k + 2 * M], di[k + 2 * M]);
        }
    }
}

// FFT of R points in place.
template <int R>
__device__ __forceinline__ void fft_packed(float2 (&re)[R], float2 (&im)[R])
{
    using O = VOps<float2>;
    if constexpr (R == 3) {
        const float2 xr[3] = {re[0], re[1], re[2]}, xi[3] = {im[0], im[1], im[2]};
        fft3<3>(xr[0], xi[0], xr[1], xi[1], xr[2], xi[2], 0, re[0], im[0], re[1], im[1], re[2], im[2]);
    } else if constexpr (R > 1) {
        float2 ur[R / 2], ui[R / 2], vr[R / 2], vi[R / 2];
#pragma unroll
        for (int j = 0; j < R / 2; ++j) {
            ur[j] = O::add(re[j], re[j + R / 2]); ui[j] = O::add(im[j], im[j + R / 2]);
            vr[j] = O::sub(re[j], re[j + R / 2]); vi[j] = O::sub(im[j], im[j + R / 2]);
        }
        fft_from_uv<R>(ur, ui, vr, vi, re, im);
    }
}

// Conjugate FFT of R points up to its last butterflies: u of the even inputs,
// v of the odd ones (the last butterflies are adjoint_out's).
template <int R>
__device__ __forceinline__ void uv_from_fft(const float2 (&dr)[R], const float2 (&di)[R], float2 (&ur)[R / 2],
                                            float2 (&ui)[R / 2], float2 (&vr)[R / 2], float2 (&vi)[R / 2])
{
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
        ur[k] = dr[2 * k]; ui[k] = di[2 * k];
        vr[k] = dr[2 * k + 1]; vi[k] = di[2 * k + 1];
    }
    fft_packed<R / 2>(ui, ur);
    fft_packed<R / 2>(vi, vr);
}

// u + conj(w) v and u - conj(w) v, w = exp(-2 pi i j / R), the outer
// instruction of every sum scalar (its halves go to different places).
template <int R>
__device__ __forceinline__ void adjoint_out(float2 ur, float2 ui, float2 vr, float2 vi, int j, float2 &pr, float2 &pi,
                                            float2 &mr, float2 &mi)
{
    using O = VOps<float2>;
    if (j == 0) {
        pr = make_float2(ur.x + vr.x, ur.y + vr.y); pi = make_float2(ui.x + vi.x, ui.y + vi.y);
        mr = make_float2(ur.x - vr.x, ur.y - vr.y); mi = make_float2(ui.x - vi.x, ui.y - vi.y);
        return;
    }
    if (4 * j == R) {
        pr = make_float2(ur.x - vi.x, ur.y - vi.y); pi = make_float2(ui.x + vr.x, ui.y + vr.y);
        mr = make_float2(ur.x + vi.x, ur.y + vi.y); mi = make_float2(ui.x - vr.x, ui.y - vr.y);
        return;
    }
    float c, s;
    unit_root<R>(j, c, s);
    if (8 * j == R || 8 * j == 3 * R) {
        // conj(w) = (+-1 + i) / sqrt 2
        const bool first = 8 * j == R;
        const float2 t = first ? O::sub(vr, vi) : O::add(vr, vi), u = first ? O::add(vr, vi) : O::sub(vr, vi);
        const float z = first ? s : -s;
        pr = make_float2(fmaf(t.x, z, ur.x), fmaf(t.y, z, ur.y));
        mr = make_float2(fmaf(t.x, -z, ur.x), fmaf(t.y, -z, ur.y));
        pi = make_float2(fmaf(u.x, s, ui.x), fmaf(u.y, s, ui.y));
        mi = make_float2(fmaf(u.x, -s, ui.x), fmaf(u.y, -s, ui.y));
        return;
    }
    // the smaller product first
    if (8 * j < R || 8 * j > 3 * R) {
        const float2 a = O::fma(vi, -s, ur), b = O::fma(vi, s, ur), d = O::fma(vr, s, ui), e = O::fma(vr, -s, ui);
        pr = make_float2(fmaf(vr.x, c, a.x), fmaf(vr.y, c, a.y));
        mr = make_float2(fmaf(vr.x, -c, b.x), fmaf(vr.y, -c, b.y));
        pi = make_float2(fmaf(vi.x, c, d.x), fmaf(vi.y, c, d.y));
        mi = make_float2(fmaf(vi.x, -c, e.x), fmaf(vi.y, -c, e.y));
    } else {
        const float2 a = O::fma(vr, c, ur), b = O::fma(vr, -c, ur), d = O::fma(vi, c, ui), e = O::fma(vi, -c, ui);
        pr = make_float2(fmaf(vi.x, -s, a.x), fmaf(vi.y, -s, a.y));
        mr = make_float2(fmaf(vi.x, s, b.x), fmaf(vi.y, s, b.y));
        pi = make_float2(fmaf(vr.x, s, d.x), fmaf(vr.y, s, d.y));
        mi = make_float2(fmaf(vr.x, -s, e.x), fmaf(vr.y, -s, e.y));
    }
}

// ------------------------------------------------------- first and middle steps
// The couple of columns cc and MC-1-cc: x holds units cc + MC j, y units
// MC-1-cc + MC j (j < R/2).  Results k: into x (k < R/2) and y, the slots
// they came from, times the twiddles tw[k * (MC/2)].  The sine goes first: most
// angles are small.
// HALF (the first step): the twiddles hold a factor 1/2, which the last factor
// would carry otherwise, so that the split's sums are no larger than their
// results (without it a forward's range ends a binade earlier, and the
// inverse's products lose a bit of subnormal values).
template <int R, int MC, bool HALF>
__device__ __forceinline__ void step_forward(float4 (&x)[R / 2], float4 (&y)[R / 2], const float4 *tw)
{
    float2 ur[R / 2], ui[R / 2], vr[R / 2], vi[R / 2], dr[R], di[R];
#pragma unroll
    for (int j = 0; j < R / 2; ++j) {
        const float4 a = x[j], b = y[R / 2 - 1 - j];
        ur[j] = make_float2(a.x + b.w, a.y + b.z);
        ui[j] = make_float2(a.z + b.y, a.w + b.x);
        vr[j] = make_float2(a.x - b.w, a.y - b.z);
        vi[j] = make_float2(a.z - b.y, a.w - b.x);
    }
    fft_from_uv<R>(ur, ui, vr, vi, dr, di);
#pragma unroll
    for (int k = 0; k < R; ++k) {
        float2 re = dr[k], im = di[k];
        if (HALF && k == 0) {
            re = VOps<float2>::mul(re, 0.5f);
            im = VOps<float2>::mul(im, 0.5f);
        }
        if (k > 0) {
            const float4 t = tw[k * (MC / 2)];
            const float2 c = make_float2(t.x, t.y), s = make_float2(t.z, t.w);
            re = __ffma2_rn(dr[k], c, __fmul2_rn(di[k], s));
            im = __ffma2_rn(di[k], c, __fmul2_rn(neg2(dr[k]), s));
        }
        const float4 o = make_float4(re.x, re.y, im.x, im.y);
        if (k < R / 2) x[k] = o;
        else y[k - R / 2] = o;
    }
}

template <int R, int MC, bool HALF>
__device__ __forceinline__ void step_adjoint(float4 (&x)[R / 2], float4 (&y)[R / 2], const float4 *tw)
{
    float2 dr[R], di[R], ur[R / 2], ui[R / 2], vr[R / 2], vi[R / 2];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const float4 o = k < R / 2 ? x[k < R / 2 ? k : 0] : y[k < R / 2 ? 0 : k - R / 2];
        const float2 re = make_float2(o.x, o.y), im = make_float2(o.z, o.w);
        dr[k] = HALF ? VOps<float2>::mul(re, 0.5f) : re;
        di[k] = HALF ? VOps<float2>::mul(im, 0.5f) : im;
        if (k > 0) {
            const float4 t = tw[k * (MC / 2)];
            const float2 c = make_float2(t.x, t.y), s = make_float2(t.z, t.w);
            dr[k] = __ffma2_rn(re, c, __fmul2_rn(neg2(im), s));
            di[k] = __ffma2_rn(im, c, __fmul2_rn(re, s));
        }
    }
    uv_from_fft<R>(dr, di, ur, ui, vr, vi);
#pragma unroll
    for (int j = 0; j < R / 2; ++j) {
        float2 pr, pi, mr, mi;
        adjoint_out<R>(ur[j], ui[j], vr[j], vi[j], j, pr, pi, mr, mi);
        x[j] = make_float4(pr.x, pr.y, pi.x, pi.y);
        y[R / 2 - 1 - j] = make_float4(mi.y, mi.x, mr.y, mr.x);
    }
}

// ---------------------------------------------------------------- last step
// Columns c (units x, index m) and its partner C-c (units w): D_k's halves
// become Z_{c + C k} and conj Z_{L - c - C k}.
template <int R>
__device__ __forceinline__ void last_forward(const float4 (&x)[R / 2], const float4 (&w)[R / 2], float2 (&dr)[R],
                                             float2 (&di)[R])
{
    float2 ur[R / 2], ui[R / 2], vr[R / 2], vi[R / 2];
#pragma unroll
    for (int j = 0; j < R / 2; ++j) {
        const float4 a = x[j], b = x[R / 2 - 1 - j], p = w[j], q = w[R / 2 - 1 - j];
        ur[j] = make_float2(a.x + b.w, p.x + q.w);
        ui[j] = make_float2(a.z + b.y, -p.z - q.y);
        vr[j] = make_float2(a.x - b.w, p.x - q.w);
        vi[j] = make_float2(a.z - b.y, q.y - p.z);
    }
    fft_from_uv<R>(ur, ui, vr, vi, dr, di);
}

template <int R>
__device__ __forceinline__ void last_adjoint(float4 (&x)[R / 2], float4 (&w)[R / 2], const float2 (&dr)[R],
                                             const float2 (&di)[R])
{
    float2 ur[R / 2], ui[R / 2], vr[R / 2], vi[R / 2];
    uv_from_fft<R>(dr, di, ur, ui, vr, vi);
#pragma unroll
    for (int j = 0; j < R / 2; ++j) {
        const int m = R / 2 - 1 - j;
        float2 pr, pi, mr, mi;
        adjoint_out<R>(ur[j], ui[j], vr[j], vi[j], j, pr, pi, mr, mi);
        x[j].x = pr.x;
        x[m].w = mr.x;
        x[j].z = pi.x;
        x[m].y = mi.x;
        w[j].x = pr.y;
        w[m].w = mr.y;
        w[j].z = -pi.y;
        w[m].y = -mi.y;
    }
}

// ---------------------------------------------------------------- the split
// Four outputs from Z_k = (ar, ai) and conj Z_{L-k} = (br, bi): a = (y_k,
// y_{L-k}), b = (y_{N-k}, y_{L+k}).  The table holds exp(-2 pi i k/N) = t.x -
// i t.y and, times s_1, the pairs over (k, L-k) of Re W (t.z, t.w) and
// -Im W (nwi).
// Whether |cos| is the smaller of the split's angle pi (k + x) / R, 0 <= x < 1/2 (of slot k).
template <int R>
__device__ __forceinline__ constexpr bool cos_first(int k)
{
    return 4 * k + 1 > R && 4 * k + 1 < 3 * R;
}

__device__ __forceinline__ void split_one(float ar, float ai, float br, float bi, const float4 t, const float2 nwi,
                                          bool cos_first, float2 &a, float2 &b)
{
    const float er = ar + br, ei = ai + bi, orr = ai - bi, oi = br - ar;
    const float p0 = cos_first ? orr : oi, p1 = cos_first ? oi : orr, q0 = cos_first ? oi : -orr, q1 = cos_first ? -orr : oi;
    const float f0 = cos_first ? t.x : t.y, f1 = cos_first ? t.y : t.x;
    const float2 vr = make_float2(fmaf(p1, f1, fmaf(p0, f0, er)), fmaf(-p1, f1, fmaf(-p0, f0, er)));
    const float2 vi = make_float2(fmaf(q1, f1, fmaf(q0, f0, ei)), fmaf(q1, f1, fmaf(q0, f0, -ei)));
    const float2 wr = make_float2(t.z, t.w);
    a = __ffma2_rn(vr, wr, __fmul2_rn(vi, nwi));
    b = __ffma2_rn(neg2(vi), wr, __fmul2_rn(vr, nwi));
}

__device__ __forceinline__ void split_one_adjoint(float2 a, float2 b, const float4 t, const float2 nwi, bool cos_first, float &ar,
                                                  float &ai, float &br, float &bi)
{
    const float2 wr = make_float2(t.z, t.w);
    const float2 vr = __ffma2_rn(a, wr, __fmul2_rn(b, nwi));
    const float2 vi = __ffma2_rn(neg2(b), wr, __fmul2_rn(a, nwi));
    const float er = vr.x + vr.y, pr = vr.x - vr.y, ei = vi.x - vi.y, pi = vi.x + vi.y;
    const float p0 = cos_first ? pi : pr, p1 = cos_first ? pr : pi, q0 = cos_first ? -pr : pi, q1 = cos_first ? pi : -pr;
    const float f0 = cos_first ? t.x : t.y, f1 = cos_first ? t.y : t.x;
    ar = fmaf(-p1, f1, fmaf(-p0, f0, er));
    br = fmaf(p1, f1, fmaf(p0, f0, er));
    ai = fmaf(-q1, f1, fmaf(-q0, f0, ei));
    bi = fmaf(q1, f1, fmaf(q0, f0, ei));
}

// The split's table by slot (k3 * (C/2) + c).
struct SplitTable {
    const float4 *ta;
    const float2 *tb;
    __device__ __forceinline__ float4 a(int i) const { return ta[i]; }
    __device__ __forceinline__ float2 b(int i) const { return tb[i]; }
};

constexpr float kCos8 = 0.92387953251128675613f, kSin8 = 0.38268343236508977173f;  // of pi / 8
constexpr float kRoot = 0.70710678118654752440f;

// The outputs of couple c in slot order: slot k3 of c > 0 is k = c + C k3; of
// c = 0, k = C k3 (k3 < R/2) and k = C/2 + C (k3 - R/2), with slot 0 holding
// a = (y_0, y_L), b = (y_{L/2}, y_{3L/2}).  Column 0 pairs k3 with R - k3 in
// its own half and column C/2 pairs k3 with R-1-k3, so each is one split.
template <int R, int C>
__device__ __forceinline__ void split_forward(int c, const float2 (&dr)[R], const float2 (&di)[R], SplitTable ts,
                                              AxisScale s, float2 (&a)[R], float2 (&b)[R])
{
    if (c != 0) {
#pragma unroll
        for (int k = 0; k < R; ++k)
            split_one(dr[k].x, di[k].x, dr[k].y, di[k].y, ts.a(k * (C / 2) + c), ts.b(k * (C / 2) + c), cos_first<R>(k), a[k], b[k]);
    } else {
        a[0] = make_float2((dr[0].x + di[0].x) * s.s0, (dr[0].x - di[0].x) * (kRoot * s.s1));
        const float hr = dr[R / 2].x * s.s1, hi = di[R / 2].x * s.s1;
        b[0] = make_float2(fmaf(hr, kCos8, -hi * kSin8), fmaf(hr, kSin8, hi * kCos8));
#pragma unroll
        for (int k = 1; k < R / 2; ++k)
            split_one(dr[k].x, di[k].x, dr[R - k].x, -di[R - k].x, ts.a(k * (C / 2)), ts.b(k * (C / 2)), cos_first<R>(k), a[k], b[k]);
#pragma unroll
        for (int k = 0; k < R / 2; ++k)
            split_one(dr[R - 1 - k].y, -di[R - 1 - k].y, dr[k].y, di[k].y, ts.a((R / 2 + k) * (C / 2)),
                      ts.b((R / 2 + k) * (C / 2)), cos_first<R>(k), a[R / 2 + k], b[R / 2 + k]);
    }
}

template <int R, int C>
__device__ __forceinline__ void split_adjoint(int c, const float2 (&a)[R], const float2 (&b)[R], SplitTable ts,
                                              AxisScale s, float2 (&dr)[R], float2 (&di)[R])
{
    if (c != 0) {
#pragma unroll
        for (int k = 0; k < R; ++k)
            split_one_adjoint(a[k], b[k], ts.a(k * (C / 2) + c), ts.b(k * (C / 2) + c), cos_first<R>(k), dr[k].x, di[k].x, dr[k].y, di[k].y);
    } else {
        const float u = a[0].x * s.s0, v = a[0].y * (kRoot * s.s1);
        dr[0].x = u + v;
        di[0].x = u - v;
        const float p = b[0].x * s.s1, q = b[0].y * s.s1;
        dr[R / 2].x = fmaf(p, kCos8, q * kSin8);
        di[R / 2].x = fmaf(q, kCos8, -p * kSin8);
#pragma unroll
        for (int k = 1; k < R / 2; ++k) {
            float im;
            split_one_adjoint(a[k], b[k], ts.a(k * (C / 2)), ts.b(k * (C / 2)), cos_first<R>(k), dr[k].x, di[k].x, dr[R - k].x, im);
            di[R - k].x = -im;
        }
#pragma unroll
        for (int k = 0; k < R / 2; ++k) {
            float im;
            split_one_adjoint(a[R / 2 + k], b[R / 2 + k], ts.a((R / 2 + k) * (C / 2)), ts.b((R / 2 + k) * (C / 2)), cos_first<R>(k), dr[R - 1 - k].y, im, dr[k].y,
                              di[k].y);
            di[R - 1 - k].y = -im;
        }
    }
}

// ------------------------------------------------------------ transposed side
// The coefficient index of every member of a couple's slots: slot k3 holds
// k = C k3 + c (for c = 0 the upper half of the slots C/2 + C (k3 - R3/2)) in
// a.x, L - k in a.y, N - k in b.x, L + k in b.y; slot 0 of c = 0 holds L/2 and
// 3L/2 in b.
template <typename C>
struct SlotIndex {
    static constexpr int N = 2 * C::L;
    int lo, hi;   // first index of the lower and the upper half of the slots, minus C k3
    bool zero;
    __device__ __forceinline__ explicit SlotIndex(int c)
        : lo(c), hi(c ? c : C::C / 2 - C::L / 2), zero(c == 0)
    {
    }
    __device__ __forceinline__ int k(int k3) const { return C::C * k3 + (k3 < C::R3 / 2 ? lo : hi); }
    __device__ __forceinline__ int ax(int k3) const { return k(k3); }
    __device__ __forceinline__ int ay(int k3) const { return C::L - k(k3); }
    __device__ __forceinline__ int bx(int k3) const { return (k3 == 0 && zero) ? C::L / 2 : N - k(k3); }
    __device__ __forceinline__ int by(int k3) const { return (k3 == 0 && zero) ? 3 * C::L / 2 : C::L + k(k3); }
};

// visit(address, slot, member) for every slot of couple c of a line in shared
// memory (consecutive coefficients): constant steps from four bases.
template <typename C, typename F>
__device__ __forceinline__ void walk_row(const float *p, int c, F &&visit)
{
    constexpr int N = 2 * C::L, H = C::R3 / 2;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int k0 = half == 0 ? c : C::C * H + (c ? c : C::C / 2 - C::L / 2);
        const float *ax = p + k0, *ay = p + C::L - k0, *bx = p + N - k0, *by = p + C::L + k0;
#pragma unroll
        for (int t = 0; t < H; ++t) {
            const int k3 = half * H + t;
            const bool zero = k3 == 0 && c == 0;
            visit(ax + C::C * t, k3, 0);
            visit(ay - C::C * t, k3, 1);
            visit(zero ? p + C::L / 2 : bx - C::C * t, k3, 2);
            visit(zero ? p + 3 * C::L / 2 : by + C::C * t, k3, 3);
        }
    }
}

// a + b * c, one instruction
__device__ __forceinline__ const char *mad_wide(unsigned b, unsigned c, const char *a)
{
    unsigned long long r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(b), "r"(c), "l"(a));
    return reinterpret_cast<const char *>(r);
}

// visit(address, member) for every slot of couple c in an array whose
// consecutive coefficients lie ld floats apart from p on.  The four members of
// a half of the slots step evenly (two up, two down), so an address is one
// multiply-add from one of four bases (a 64-bit index times ld each took six
// instructions per element, a quarter of a 256-point forward pass).
// ld < 2^26 / C.
template <typename C, typename F>
__device__ __forceinline__ void walk_slots(const float *p, int c, int ld, F &&visit)
{
    constexpr int N = 2 * C::L;
    constexpr int H = C::R3 / 2;
    const unsigned step = 4u * C::C * (unsigned)ld;  // bytes per slot
    const char *base = reinterpret_cast<const char *>(p);
    const unsigned row = 4u * (unsigned)ld;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int k0 = half == 0 ? c : C::C * H + (c ? c : C::C / 2 - C::L / 2);  // of the half's first slot
        const char *ax = mad_wide(row, k0, base), *by = mad_wide(row, C::L + k0, base);
        // downward members from their lowest, the half's last slot
        const char *ay = mad_wide(row, C::L - C::C * (H - 1) - k0, base), *bx = mad_wide(row, N - C::C * (H - 1) - k0, base);
#pragma unroll
        for (int t = 0; t < H; ++t) {
            const int k3 = half * H + t;
            visit(mad_wide(step, t, ax), k3, 0);
            visit(mad_wide(step, H - 1 - t, ay), k3, 1);
            const char *x = mad_wide(step, H - 1 - t, bx), *y = mad_wide(step, t, by);
            if (k3 == 0 && c == 0) {
                x = mad_wide(row, C::L / 2, base);
                y = mad_wide(row, 3 * C::L / 2, base);
            }
            visit(x, k3, 2);
            visit(y, k3, 3);
        }
    }
}

}  // namespace bdct
