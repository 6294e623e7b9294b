// Entry points of the line engine (fp32_lines.cu).
#pragma once

#include <cuda_runtime.h>

#include "bdct_internal.h"

namespace bdct {

// What one separable pass does with arrays of `rows` lines of n points (r the
// line, k or j the index along it):
//   LINES_FORWARD       src[r][j] -> dst[k][r]   DCT-II, output scales
//   LINES_INVERSE       src[r][k] -> dst[j][r]   DCT-III, input scales
//   LINES_PAIR          src[r][j] -> dst[j][r]   DCT-II, DCT-III (round trip)
//   LINES_PAIR_DIAGONAL src[r][j] -> dst[j][r]   DCT-II, diagonal, DCT-III (Prop. 1)
//   LINES_INVERSE_ROWS  src[r][k] -> dst[r][j]   DCT-III, input scales
// Two transposing passes, along w and then along h (the intermediate is w x
// h), give the 2D transform in natural layout; the spectral composition is a
// forward along w, the pair along h, an inverse of the rows along w.  That
// way every pass reads by bulk copies; the other order (the pair rows to rows,
// then an inverse from the transposed side, gathered through registers) is
// slower from 512 points on (spectral, 512 MiB: 1024^2 777 -> 728 us, 2048^2
// 909 -> 829, 16 arrays of 1024^2 112 -> 104; 256^2 594 -> 616).
enum LinesMode { LINES_FORWARD, LINES_INVERSE, LINES_PAIR, LINES_PAIR_DIAGONAL, LINES_INVERSE_ROWS };

// Copy the cosine tables (device buffers) into the line engine's constant
// memory (called by fused_init_device).
cudaError_t lines_init_table(const float *d_table);
cudaError_t lines_init_table3(const float *d_table);
// True if n has an FFT-based line engine: powers of two 64..4096, and 192,
// 384, 768, 1536.
bool lines_supported(int n);
// A twiddle table of length n (lines_table_elems float4 entries) for a set of
// modes that split the line alike: 0 LINES_FORWARD, 1 the others, 2 every mode
// on few lines; s1 is the scale of every index above 0, folded in.
struct LineTable {
    float4 *dst;
    int n, set;
    double s1;
};
// Entries of a table: 0 for set 2 of a length without a few-panel form.
size_t lines_table_elems(int n, int set);
// Generate up to 12 tables in FP64, one launch.
cudaError_t lines_gen_tables(const LineTable *tables, int count, cudaStream_t s);
// One pass over `count` arrays of `rows` lines.  sc holds the scales of the
// pass (sc.s1 the tables' s1; the pair modes apply them twice, so they take the
// orthonormal ones); tw is the table of the mode's set, tw_few the one of set 2
// with the same scale, which a call with few lines uses; lam is the
// diagonal of LINES_PAIR_DIAGONAL: coefficient k of line r is multiplied by
// lam[k * rows + r].  src_off / dst_off index the arrays (element offsets) or
// are null for contiguous arrays; reverse takes the lines last to first.
// src == dst is allowed for LINES_INVERSE_ROWS only, the other modes read
// what other CTAs write.
struct LinesCall {
    const float *src;
    float *dst;
    int rows;
    long long count;
    AxisScale sc;
    const float4 *tw, *tw_few;
    unsigned int *status;
    const long long *src_off = nullptr, *dst_off = nullptr;
    bool reverse = false;
    LinesMode beside = LINES_FORWARD;  // what the call's pass along the other axis does
    const float *lam = nullptr;
};
cudaError_t lines_pass(const LinesCall &c, int n, LinesMode mode, cudaStream_t stream);

}  // namespace bdct
