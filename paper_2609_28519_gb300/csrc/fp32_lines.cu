// The line engine's tables and entry points, and its kernels up to 768 points
// (fp32_lines_kernel.cuh; the longer lengths compile beside it in
// fp32_lines_long.cu).
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>

#include "fp32_lines_kernel.cuh"

namespace bdct {

// fp32_lines_long.cu
cudaError_t lines_long_init_table(const float *d_table);
cudaError_t lines_long_init_table3(const float *d_table);
cudaError_t lines_long_pass(int n, LinesMode mode, const LinesCall &c, cudaStream_t stream);

cudaError_t lines_init_table(const float *d_table)
{
    const cudaError_t e = init_cos_table(d_table);
    return e == cudaSuccess ? lines_long_init_table(d_table) : e;
}
cudaError_t lines_init_table3(const float *d_table)
{
    const cudaError_t e = init_cos_table3(d_table);
    return e == cudaSuccess ? lines_long_init_table3(d_table) : e;
}

bool lines_supported(int n)
{
    return n == 64 || n == 128 || n == 256 || n == 512 || n == 1024 || n == 2048 || n == 4096 || n == 192 ||
           n == 384 || n == 768 || n == 1536;
}

namespace {

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
        const double h = first ? 0.5 : 1.0;  // step_forward's HALF
        t[r] = make_float4((float)(h * ca), (float)(h * cb), (float)(h * sa), (float)(h * sb));
    } else if (r < u1 + u2 + L / 2) {
        const int e = r - u1 - u2;
        const int k3 = e / (c3 / 2), c = e % (c3 / 2);
        const int k = c3 * k3 + (c || k3 < q.r3 / 2 ? c : c3 / 2 - L / 2);
        double cw, sw;
        cos_sin_2pi(k, q.n, cw, sw);
        cos_sin_2pi(k, 4ll * q.n, ca, sa);       // W_k = exp(-i pi k / (2n))
        cos_sin_2pi(L - k, 4ll * q.n, cb, sb);   // W_{L-k}
        float4 *o = t + u1 + u2;
        o[e] = make_float4((float)cw, (float)sw, (float)(s1 * ca), (float)(s1 * cb));
        reinterpret_cast<float2 *>(o + L / 2)[e] = make_float2((float)(s1 * sa), (float)(s1 * sb));
    }
}

// |w| - 1 of w = exp(2 pi i m / d) with both parts rounded to FP32.
double root_error(long long m, long long d)
{
    const double a = 2.0 * 3.14159265358979323846 * (double)(m % d) / (double)d;
    const double c = (float)std::cos(a), s = (float)std::sin(a);
    return 0.5 * (c * c + s * s - 1.0);
}

// Mean gain error of an R-point FFT's rounded roots over its inputs and
// outputs (radix 2 and 3, decimation in time: one or two thirds of the terms
// of a stage are multiplied).
double fft_error(int R)
{
    double g = 0.0;
    if (R % 3 == 0) {
        const int M = R / 3;
        for (int k = 0; k < M; ++k) g += (root_error(k, R) + root_error(2 * k, R)) / (3.0 * M);
        const double h = 0.5 * std::sqrt(3.0);
        g += ((float)h / h - 1.0) / 3.0;  // the imaginary parts of the 3-point DFT: a third of its energy
        R = M;
    }
    for (; R > 1; R /= 2)
        for (int k = 0; k < R / 2; ++k) g += root_error(k, R) / R;
    return g;
}

// Mean gain error of a step's twiddles: column cc and its mirror, k signed in
// the step before the last (as k_gen_line_tw).
double step_error(int R, int mc, bool signed_k)
{
    double g = 0.0;
    for (int k = 0; k < R; ++k)
        for (int cc = 0; cc < mc / 2; ++cc) {
            const long long kk = signed_k && k >= R / 2 ? k - R : k, d = (long long)R * mc;
            g += root_error(cc * kk, d) + root_error((cc + 1) * kk, d);
        }
    return g / ((double)R * mc);
}

// Mean gain error of the whole line but for the split's last factor.  Rounded
// roots are shorter than 1 on average (1/sqrt 2, in every short FFT, by 1.7e-8),
// so it is -1.5e-8 to -4e-8, the same for every input, and a fifth to a third
// of the squared error of a round trip; the last factor takes it back.
double line_error(const TableShape &q)
{
    const int L = q.n / 2;
    double g = fft_error(q.r1) + fft_error(q.r2) + fft_error(q.r3) + step_error(q.r1, L / q.r1, q.r2 == 1);
    if (q.r2 > 1) g += step_error(q.r2, q.r3, true);
    double p = 0.0;
    for (int k = 0; k < L; ++k) p += root_error(k, q.n) / L;
    return g + 0.5 * p;
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
    if constexpr (has_few(N))
        if (set == 2) *q = shape_of<N, 2>();
    if (set != 2) *q = set == 0 ? shape_of<N, 0>() : shape_of<N, 1>();
    return set != 2 || has_few(N);
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
    // by log2 of the length, or of its third, and set; once per process
    static std::mutex mu;
    static double known[2][16][3];
    TableJobs jobs{};
    int most = 0;
    for (int i = 0; i < count; ++i) {
        const TableShape &q = jobs.shape[i];
        if (!table_shape(tables[i].n, tables[i].set, &jobs.shape[i])) return cudaErrorInvalidValue;
        jobs.dst[i] = tables[i].dst;
        {
            std::lock_guard<std::mutex> lock(mu);
            const bool three = q.n % 3 == 0;
            int e = 0;
            while ((three ? 3 : 1) << e < q.n) ++e;
            double &g = known[three][e][tables[i].set];
            if (g == 0.0) g = line_error(q);
            jobs.s1[i] = tables[i].s1 / (1.0 + g);
        }
        const int e = (int)lines_table_elems(tables[i].n, tables[i].set);
        if (e > most) most = e;
    }
    // one warp per block: FP64 runs at two lanes a cycle, so the warps are spread over the SMs
    k_gen_line_tw<<<dim3((most + 31) / 32, count), 32, 0, s>>>(jobs);
    return cudaGetLastError();
}

cudaError_t lines_pass(const LinesCall &c, int n, LinesMode mode, cudaStream_t stream)
{
    switch (n) {
        case 64: return lines_run<64>(mode, c, stream);
        case 128: return lines_run<128>(mode, c, stream);
        case 192: return lines_run<192>(mode, c, stream);
        case 256: return lines_run<256>(mode, c, stream);
        case 384: return lines_run<384>(mode, c, stream);
        case 512: return lines_run<512>(mode, c, stream);
        case 768: return lines_run<768>(mode, c, stream);
        default: return lines_long_pass(n, mode, c, stream);
    }
}

}  // namespace bdct
