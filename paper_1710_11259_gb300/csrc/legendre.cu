// Legendre coefficients in and out of the square solve (Sec. 3.4, Table 3.1 steps
// 1 and 4), as two banded 2D maps.  With C~_k = s_k C^(3/2)_k, s_k =
// sqrt((k + 3/2)/((k+1)(k+2))), and the identities
//   (2k+1) P_k = C^(3/2)_k - C^(3/2)_{k-2},
//   (1 - x^2) C^(3/2)_j = (j+1)(j+2)/(2j+3) (P_j - P_{j+2}),
// the input map is F = B G B^T with B[j][j] = 1/((2j+1) s_j), B[j][j+2] =
// -1/((2j+5) s_j), and the output map, the Legendre coefficients of
// u = (1-x^2)(1-y^2) sum X_ij C~_i(y) C~_j(x), is U = L X L^T with L ((n+2) x n)
// L[j][j] = c_j, L[j+2][j] = -c_j, c_j = s_j (j+1)(j+2)/(2j+3): the product
// B^{-1} M of the C~ -> Legendre conversion and the multiplication (3.7) by
// (1 - x^2) collapses to two terms.
//
// Both maps and their transposes are one kernel: every row a is combined along the
// columns,  q_a[k] = x_k in[a][k] + y_k in[a][k +- 2],  and two rows are combined,
// out = X q_a + Y q_{a +- 2}.  A thread walks down LEN rows of one parity in one column
// and forms every q once: four FP64 operations per element, the bound on GB300 (0.64 ms
// at n = 10^4; one read and one write of HBM would take 0.24 ms).
#include "legendre.cuh"

namespace fps {

namespace {

enum Map { kIn, kOut, kInT, kOutT };

constexpr int kCols = 32;  // a warp: 32 columns; two parities x kWarps / 2 column groups per CTA

// sqrt((j+1)(j+2)/(j+3/2)) / d, i.e. 1/(s_j d)
__device__ __forceinline__ double inv_snorm(int64_t j, double d)
{
    const double J = (double)j, A = (J + 1.0) * (J + 2.0);
    return A * rsqrt(A * (J + 1.5) * (d * d));
}
__device__ __forceinline__ double b_diag(int64_t j) { return inv_snorm(j, 2.0 * (double)j + 1.0); }
__device__ __forceinline__ double b_off(int64_t j) { return -inv_snorm(j, 2.0 * (double)j + 5.0); }
// c_j = s_j (j+1)(j+2)/(2j+3) = (j+1)(j+2)/2 / sqrt((j+1)(j+2)(j+3/2)); 0 outside [0, n)
__device__ __forceinline__ double c_val(int64_t j, int64_t n)
{
    if (j < 0 || j >= n) return 0.0;
    const double J = (double)j, A = (J + 1.0) * (J + 2.0);
    return 0.5 * A * rsqrt(A * (J + 1.5));
}

// Coefficients of position i of the output: x on the near index, y on the one two away
// (kIn, kOutT: i and i + 2; kOut, kInT: i and i - 2), zero where that one is outside.
template <int MAP>
__device__ __forceinline__ double2 coefficients(int64_t i, int64_t n)
{
    if (MAP == kIn) return make_double2(b_diag(i), i + 2 < n ? b_off(i) : 0.0);
    if (MAP == kOut) return make_double2(c_val(i, n), -c_val(i - 2, n));
    if (MAP == kInT) return make_double2(b_diag(i), i >= 2 ? b_off(i - 2) : 0.0);
    const double c = c_val(i, n);
    return make_double2(c, -c);
}

template <int MAP, int LEN, int kWarps>
__global__ void __launch_bounds__(kCols *kWarps) legendre_kernel(const double *__restrict__ in, double *__restrict__ out,
                                                                 int64_t n)
{
    constexpr bool kForward = MAP == kIn || MAP == kOutT;
    constexpr int kChunk = LEN < 8 ? LEN : 8;
    __shared__ double2 rc[2 * LEN];  // row coefficients of the tile's rows
    const int64_t m = n + 2;
    const int64_t rows_in = MAP == kOutT ? m : n, rows_out = MAP == kOut ? m : n;  // square matrices
    const int64_t i0 = (int64_t)blockIdx.y * (2 * LEN);
    for (int t = threadIdx.x; t < 2 * LEN; t += kCols * kWarps)
        if (i0 + t < rows_out) rc[t] = coefficients<MAP>(i0 + t, n);
    const int warp = threadIdx.x >> 5, par = warp & 1;
    const int64_t k = (int64_t)blockIdx.x * (kCols * kWarps / 2) + (warp >> 1) * kCols + (threadIdx.x & 31);
    const bool on = k < rows_out;
    const double2 cx = on ? coefficients<MAP>(k, n) : make_double2(0.0, 0.0);
    const int64_t k2 = kForward ? k + 2 : k - 2;
    const bool near_in = on && k < rows_in, far_in = on && k2 >= 0 && k2 < rows_in;
    __syncthreads();
    // q of row a; rows outside the input are zero
    auto combine = [&](double u, double v) { return fma(cx.y, v, fma(cx.x, u, 0.0)); };
    auto load = [&](int64_t a, double &u, double &v) {
        const bool ok = a >= 0 && a < rows_in;
        const double *row = in + a * rows_in;
        u = ok && near_in ? row[k] : 0.0;
        v = ok && far_in ? row[k2] : 0.0;
    };
    const int64_t first = i0 + par - (kForward ? 0 : 2);
    double u, v;
    load(first, u, v);
    double q = combine(u, v);
    for (int t0 = 0; t0 < LEN; t0 += kChunk) {
        double us[kChunk], vs[kChunk];
#pragma unroll
        for (int t = 0; t < kChunk; ++t) load(first + 2 * (t0 + t + 1), us[t], vs[t]);
#pragma unroll
        for (int t = 0; t < kChunk; ++t) {
            const int r = par + 2 * (t0 + t);
            const double nxt = combine(us[t], vs[t]);
            if (on && i0 + r < rows_out) {
                const double2 c = rc[r];
                out[(i0 + r) * rows_out + k] = kForward ? fma(c.x, q, fma(c.y, nxt, 0.0)) : fma(c.x, nxt, fma(c.y, q, 0.0));
            }
            q = nxt;
        }
    }
}

// Long walks amortise the coefficients (a reciprocal square root costs as much as four
// elements); short ones give a small matrix enough CTAs.  Both maps together, walks of
// 64 / 16 / 8 rows against one output element per thread with 6 and 4 operations:
// n = 10^4 1.75 ms (3.93 ms), n = 2048 109 us (179 us), n = 777 31 us (42 us).
template <int MAP, int LEN, int kWarps>
void launch_len(const double *in, double *out, int64_t n, cudaStream_t st)
{
    const int64_t rows = MAP == kOut ? n + 2 : n, cols = kCols * kWarps / 2;
    const dim3 grid((unsigned)((rows + cols - 1) / cols), (unsigned)((rows + 2 * LEN - 1) / (2 * LEN)));
    legendre_kernel<MAP, LEN, kWarps><<<grid, kCols * kWarps, 0, st>>>(in, out, n);
}

template <int MAP>
cudaError_t launch_map(const double *in, double *out, int64_t n, cudaStream_t st)
{
    if (n >= 3072) launch_len<MAP, 64, 8>(in, out, n, st);
    else if (n >= 900) launch_len<MAP, 16, 8>(in, out, n, st);
    else launch_len<MAP, 8, 4>(in, out, n, st);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_legendre_to_ctilde(const double *G, double *F, int64_t n, cudaStream_t st)
{
    return launch_map<kIn>(G, F, n, st);
}

cudaError_t launch_solution_to_legendre(const double *X, double *U, int64_t n, cudaStream_t st)
{
    return launch_map<kOut>(X, U, n, st);
}

// Transpose of the input map, Gbar = B^T Fbar B.
cudaError_t launch_legendre_to_ctilde_adjoint(const double *Fbar, double *Gbar, int64_t n, cudaStream_t st)
{
    return launch_map<kInT>(Fbar, Gbar, n, st);
}

// Transpose of the output map, Xbar = L^T Ubar L.
cudaError_t launch_solution_to_legendre_adjoint(const double *Ubar, double *Xbar, int64_t n, cudaStream_t st)
{
    return launch_map<kOutT>(Ubar, Xbar, n, st);
}

}  // namespace fps
