// Cylinder Fourier modes |k| >= 2 (Sec. 4.1, Case 1): see cylinder.h for the
// equations.  Host: band entries from closed forms, eigenvalue intervals, shifts and
// factor tables in FP64.
//
// The two half-steps are run without forming their banded products with W and with
// Q - p P.  With R = (Q - p_j P) X_j - G (R = -G before the first iteration, X_0 = 0),
//     N = M D^{-1} + p_j I,   w = R N^{-1},        S = R + (q_j - p_j) w,
//     (Q - q_j P) X = S + G,                       R <- S + (q_j - p_{j+1}) P X
// (from (M + q D) D^{-1} = N + (q - p) I and Q - p' P = (Q - q P) + (q - p') P): a
// tridiagonal solve along z, a pentadiagonal solve
// and a tridiagonal product along r, 11 FP64 operations per unknown and iteration
// instead of 25.  Pivots stay in the forward values and are folded into the next factor.
// Even and odd indices decouple in both directions: four quarters per (mode, rhs).
//
// n <= 256: one CTA per quarter runs all its iterations with R / S in shared memory
// (cyl_resident_kernel).  Larger n: two launches per iteration over 32 lines per CTA:
//   z kernel (32 rows, a row per lane pair):     R2 = S + G
//   r kernel (32 columns, a column per lane):    R1 = R2 - G + (q - p') P X   (or Y = X)
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>

#include "../../include/fps.h"
#include "cylinder.h"
#include "host_math.h"

namespace fps {

// ---------------------------------------------------------------- band entries
// s_j of C~_j = s_j C_j^(3/2)
static double ct_scale(int64_t j)
{
    const double x = (double)j;
    return std::sqrt((x + 1.5) / ((x + 1.0) * (x + 2.0)));
}

// (3.7) in the normalised basis: M = multiplication by (1 - x^2)
double cyl_M_diag(int64_t j)
{
    const double x = (double)j;
    return 2.0 * (x + 1.0) * (x + 2.0) / ((2.0 * x + 1.0) * (2.0 * x + 5.0));
}
double cyl_M_off(int64_t j)
{
    const double x = (double)j;
    const double prod4 = (x + 1.0) * (x + 2.0) * (x + 3.0) * (x + 4.0);
    return -std::sqrt(prod4 * (2.0 * x + 3.0) / (2.0 * x + 7.0)) / ((2.0 * x + 3.0) * (2.0 * x + 5.0));
}
static double Mentry(int64_t a, int64_t i)
{
    if (a < 0 || i < 0) return 0.0;
    if (a == i) return cyl_M_diag(a);
    if (a == i + 2) return cyl_M_off(i);
    if (i == a + 2) return cyl_M_off(a);
    return 0.0;
}

// x (1 - x^2) d/dx in the C^(3/2) basis, from (1 - x^2) C_m' = al_m C_{m-1} - be_m C_{m+1}
// and x C_j = ga_j C_{j+1} + de_j C_{j-1} (lambda = 3/2), then normalised.
static double X1entry(int64_t a, int64_t m)
{
    if (a < 0 || m < 0) return 0.0;
    const double M_ = (double)m;
    const double al = (M_ + 2.0) * (M_ + 3.0) / (2.0 * M_ + 3.0), be = M_ * (M_ + 1.0) / (2.0 * M_ + 3.0);
    auto ga = [](double j) { return (j + 1.0) / (2.0 * j + 3.0); };
    auto de = [](double j) { return (j + 2.0) / (2.0 * j + 3.0); };
    double v = 0.0;
    if (a == m) v = (m >= 1 ? al * ga(M_ - 1.0) : 0.0) - be * de(M_ + 1.0);
    else if (a == m - 2) v = al * de(M_ - 1.0);
    else if (a == m + 2) v = -be * ga(M_ + 1.0);
    else return 0.0;
    return v * ct_scale(m) / ct_scale(a);
}

// L1 = (I - M) D + 5 [x (1 - x^2) d/dx] + 14 M - 10 I, the matrix of
// r^2(1 - r^2) d^2/dr^2 + (5 - 9 r^2) r d/dr + 4 (1 - 4 r^2)
double cyl_L1(int64_t a, int64_t i)
{
    const double Dii = -((double)i + 1.0) * ((double)i + 2.0);
    return ((a == i ? 1.0 : 0.0) - Mentry(a, i)) * Dii + 5.0 * X1entry(a, i) + 14.0 * Mentry(a, i) -
           (a == i ? 10.0 : 0.0);
}

// Q = M - M^2 (the exact product: the inner index runs past n)
static double Qentry(int64_t a, int64_t i)
{
    double mm = 0.0;
    for (int64_t c = a - 2; c <= a + 2; c += 2) mm += Mentry(a, c) * Mentry(c, i);
    return Mentry(a, i) - mm;
}

namespace {

// Per-parity banded operators of one mode (index s <-> t = par + 2 s).
struct ParityOps {
    int m = 0;
    std::vector<double> pl, pd, pu;      // P[t][t-2], P[t][t], P[t][t+2]
    std::vector<double> q0, q2, q4;      // Q[t][t], Q[t][t+2], Q[t][t+4] (symmetric)
};

ParityOps parity_ops(int64_t n, int64_t k, int par)
{
    ParityOps o;
    o.m = (int)((n - par + 1) / 2);
    const double k2 = (double)k * (double)k;
    for (int s = 0; s < o.m; ++s) {
        const int64_t t = par + 2 * s;
        o.pl.push_back(t >= 2 ? cyl_L1(t, t - 2) - k2 * Mentry(t, t - 2) : 0.0);
        o.pd.push_back(cyl_L1(t, t) - k2 * Mentry(t, t));
        o.pu.push_back(t + 2 < n ? cyl_L1(t, t + 2) - k2 * Mentry(t, t + 2) : 0.0);
        o.q0.push_back(Qentry(t, t));
        o.q2.push_back(t + 2 < n ? Qentry(t, t + 2) : 0.0);
        o.q4.push_back(t + 4 < n ? Qentry(t, t + 4) : 0.0);
    }
    return o;
}

// y = P x, y = Q x (parity blocks)
void apply_P(const ParityOps &o, const std::vector<double> &x, std::vector<double> &y)
{
    for (int s = 0; s < o.m; ++s) {
        double v = o.pd[s] * x[s];
        if (s >= 1) v += o.pl[s] * x[s - 1];
        if (s + 1 < o.m) v += o.pu[s] * x[s + 1];
        y[s] = v;
    }
}
void apply_Q(const ParityOps &o, const std::vector<double> &x, std::vector<double> &y)
{
    for (int s = 0; s < o.m; ++s) {
        double v = o.q0[s] * x[s];
        if (s >= 1) v += o.q2[s - 1] * x[s - 1];
        if (s >= 2) v += o.q4[s - 2] * x[s - 2];
        if (s + 1 < o.m) v += o.q2[s] * x[s + 1];
        if (s + 2 < o.m) v += o.q4[s] * x[s + 2];
        y[s] = v;
    }
}
// x = P^{-1} b (tridiagonal, diagonally dominant: no pivoting)
void solve_P(const ParityOps &o, std::vector<double> b, std::vector<double> &x)
{
    std::vector<double> c(o.m), d(o.m);
    for (int s = 0; s < o.m; ++s) {
        double den = o.pd[s] - (s >= 1 ? o.pl[s] * c[s - 1] : 0.0);
        c[s] = o.pu[s] / den;
        d[s] = (b[s] - (s >= 1 ? o.pl[s] * d[s - 1] : 0.0)) / den;
    }
    for (int s = o.m - 1; s >= 0; --s) x[s] = d[s] - (s + 1 < o.m ? c[s] * x[s + 1] : 0.0);
}
// LU without pivoting of T = Q - q P (pentadiagonal per parity), as used on the device
struct LU5 {
    std::vector<double> l1, l2, iu0, u1, u2;
};
LU5 lu_QminusqP(const ParityOps &o, double q)
{
    LU5 f;
    const int m = o.m;
    f.l1.assign(m, 0.0);
    f.l2.assign(m, 0.0);
    f.iu0.assign(m, 0.0);
    f.u1.assign(m, 0.0);
    f.u2.assign(m, 0.0);
    std::vector<double> u0(m);
    for (int s = 0; s < m; ++s) {
        const double tm2 = s >= 2 ? o.q4[s - 2] : 0.0;                            // T[s][s-2]
        const double tm1 = s >= 1 ? o.q2[s - 1] - q * o.pl[s] : 0.0;              // T[s][s-1]
        const double t0 = o.q0[s] - q * o.pd[s];
        const double tp1 = s + 1 < m ? o.q2[s] - q * o.pu[s] : 0.0;
        const double tp2 = s + 2 < m ? o.q4[s] : 0.0;
        const double l2 = s >= 2 ? tm2 / u0[s - 2] : 0.0;
        const double l1 = s >= 1 ? (tm1 - (s >= 2 ? l2 * f.u1[s - 2] : 0.0)) / u0[s - 1] : 0.0;
        u0[s] = t0 - (s >= 1 ? l1 * f.u1[s - 1] : 0.0) - (s >= 2 ? l2 * f.u2[s - 2] : 0.0);
        f.u1[s] = tp1 - (s >= 1 ? l1 * f.u2[s - 1] : 0.0);
        f.u2[s] = tp2;
        f.l1[s] = l1;
        f.l2[s] = l2;
        f.iu0[s] = 1.0 / u0[s];
    }
    return f;
}
void solve_Q(const ParityOps &o, const std::vector<double> &b, std::vector<double> &x)
{
    const LU5 f = lu_QminusqP(o, 0.0);
    std::vector<double> y(o.m);
    for (int s = 0; s < o.m; ++s)
        y[s] = b[s] - (s >= 1 ? f.l1[s] * y[s - 1] : 0.0) - (s >= 2 ? f.l2[s] * y[s - 2] : 0.0);
    for (int s = o.m - 1; s >= 0; --s)
        x[s] = (y[s] - (s + 1 < o.m ? f.u1[s] * x[s + 1] : 0.0) - (s + 2 < o.m ? f.u2[s] * x[s + 2] : 0.0)) *
               f.iu0[s];
}

// Dominant eigenvalue of x -> op(x) by power iteration with a Rayleigh quotient.
template <class Op>
double power_eig(int m, Op op)
{
    std::vector<double> x(m), y(m);
    for (int s = 0; s < m; ++s) x[s] = 1.0 + 0.25 * std::sin(1.0 + 0.7 * s);
    double lam = 0.0;
    for (int it = 0; it < 3000; ++it) {
        double nx = 0.0;
        for (double v : x) nx += v * v;
        nx = std::sqrt(nx);
        for (double &v : x) v /= nx;
        op(x, y);
        double num = 0.0;
        for (int s = 0; s < m; ++s) num += x[s] * y[s];
        if (it > 20 && std::fabs(num - lam) <= 1e-12 * std::fabs(num)) return num;
        lam = num;
        x.swap(y);
    }
    return lam;
}

}  // namespace

int cyl_mode_interval(int64_t n, int64_t k, double &a, double &b)
{
    double most = 0.0, least = -1e300;
    for (int par = 0; par < 2 && par < n; ++par) {
        const ParityOps o = parity_ops(n, k, par);
        if (o.m == 0) continue;
        std::vector<double> tmp(o.m);
        const double big = power_eig(o.m, [&](const std::vector<double> &x, std::vector<double> &y) {
            apply_Q(o, x, tmp);
            solve_P(o, tmp, y);
        });
        const double inv = power_eig(o.m, [&](const std::vector<double> &x, std::vector<double> &y) {
            apply_P(o, x, tmp);
            solve_Q(o, tmp, y);
        });
        most = std::min(most, big);
        least = std::max(least, 1.0 / inv);
    }
    if (!(most < 0.0) || !(least < 0.0) || !std::isfinite(most) || !std::isfinite(least)) return FPS_ERR_UNSUPPORTED;
    a = 1.03 * most;
    b = 0.97 * least;
    return FPS_OK;
}

// ---------------------------------------------------------------- device side
namespace {

__device__ __forceinline__ double times(double a, double b) { return fma(a, b, 0.0); }  // cheaper than a product

// ---- n <= 256: a quarter per CTA ----
constexpr int kResMaxN = 256;

// Tables of one (mode, iteration, parity) for lines of 2 H unknowns; half h walks s = 0 ..
// H-1 from its outer end to the middle (unknown s or 2H-1-s), entries [2][H]:
//   z: l, m, g (= (q - p)/pivot), then per half the 2 coefficients of the middle solve;
//   r: l1, l2, n1, n2, a, b, c ((q - p') P with the outer, own and inner unknown, over
//      their pivots), 1/pivot, then per half the 3 x 4 coefficients of the middle solve.
__host__ __device__ constexpr int z_table(int H) { return 3 * 2 * H + 4; }
__host__ __device__ constexpr int r_table(int H) { return 8 * 2 * H + 24; }

struct CylUnit {
    int64_t off;     // caller layout: offset of the (mode, rhs) matrix
    int joff, J;     // first table set and iterations of the mode
    int rp, cp;
};
struct CylResArgs {
    int n;
    const CylUnit *units;
    const double *ztab, *rtab;  // [sum J][2][z_table], [sum J][2][r_table]
    const double *G;            // [unit][2 H][2 H]
    double *Y;
};

// Unknown at place t of a line of 2 H: both halves are stored from their outer end.
__host__ __device__ __forceinline__ int place_of(int t, int H) { return t < H ? t : 3 * H - 1 - t; }

template <int H>
struct CylGeo {
    static constexpr int N = 2 * H, pitch = N + 1;  // odd: threads on consecutive rows hit different banks
    static constexpr int kThreads = (N + 15) / 16 * 32;
    static constexpr size_t bytes = sizeof(double) * (size_t)(N * pitch + z_table(H) + r_table(H));
};

__device__ __forceinline__ void copy16_async(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Half-warp 0 / 1 = outer-to-middle walks from the two ends of the same 16 lines; each
// thread keeps the forward values of its half line in registers, so the quarter in shared
// memory is read twice and written once per solve.  The walks meet in the middle: two
// values (z) or four (r) are exchanged by shuffles and a precomputed 2 x 2 or 4 x 4
// inverse gives the unknowns next to the middle.  Bound: the FP64 pipe (11 operations per
// unknown and iteration, two warps per SM quadrant at n = 256); G is the only stream from
// HBM or L2, read 8 rows ahead.  n = 256, 127 modes x 4 right-hand sides: 27.6 ms a solve,
// 107 ms with two launches per iteration that formed the banded products.
template <int H>
__global__ void __launch_bounds__(CylGeo<H>::kThreads) cyl_resident_kernel(CylResArgs A)
{
    using C = CylGeo<H>;
    constexpr int N = C::N, kB = H < 8 ? H : 8;
    extern __shared__ __align__(16) double cyl_smem[];
    double *R = cyl_smem, *zt = R + N * C::pitch, *rt = zt + z_table(H);
    const int tid = threadIdx.x, lane = tid & 31, h = lane >> 4;
    const int ln = min((tid >> 5) * 16 + (lane & 15), N - 1);  // threads beyond the last line repeat it
    const bool on = (tid >> 5) * 16 + (lane & 15) < N;
    const CylUnit un = A.units[blockIdx.x];
    const double *G = A.G + (int64_t)blockIdx.x * N * N;
    auto load = [&](double *dst, const double *src, int count) {  // count even
        for (int q = 2 * tid; q < count; q += 2 * C::kThreads) copy16_async(dst + q, src + q);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    load(zt, A.ztab + ((int64_t)un.joff * 2 + un.cp) * z_table(H), z_table(H));
    for (int q = tid; q < N * N; q += C::kThreads) R[(q / N) * C::pitch + q % N] = -G[q];
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    // this thread's half row and half column, from the outer end (see place_of)
    double *zr = R + ln * C::pitch + h * H;
    double *rr = R + h * H * C::pitch + ln;
    const double *gr = G + h * H * N + ln;
    constexpr int rd = C::pitch, gd = N;
    const double *zl = zt + h * H, *zm = zl + N, *zg = zm + N, *zmid = zt + 3 * N + 2 * h;
    const double *l1 = rt + h * H, *l2 = l1 + N, *n1 = l2 + N, *n2 = n1 + N, *ca = n2 + N, *cb = ca + N, *cc = cb + N,
                 *iu = cc + N, *mid = rt + 8 * N + 12 * h;
    for (int j = 0; j < un.J; ++j) {
        const bool last = j + 1 == un.J;
        double v[H];
        load(rt, A.rtab + ((int64_t)(un.joff + j) * 2 + un.rp) * r_table(H), r_table(H));
        {
            double z = 0.0;
#pragma unroll
            for (int s = 0; s < H; ++s) {
                z = fma(-zl[s], z, zr[s]);
                v[s] = z;
            }
            double y = fma(zmid[1], __shfl_xor_sync(0xffffffffu, z, 16), times(zmid[0], z));
            asm volatile("" ::: "memory");  // R is read again, not kept in registers
#pragma unroll
            for (int s = H - 1; s >= 0; --s) {
                if (s < H - 1) y = fma(-zm[s], y, v[s]);
                const double out = fma(zg[s], y, zr[s]);
                if (on) zr[s] = out;
            }
        }
        double g[2][kB];
#pragma unroll
        for (int u = 0; u < kB; ++u) g[0][u] = gr[u * gd];
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
        if (!last) load(zt, A.ztab + ((int64_t)(un.joff + j + 1) * 2 + un.cp) * z_table(H), z_table(H));
        {
            double y1 = 0.0, y2 = 0.0;
#pragma unroll
            for (int s0 = 0; s0 < H; s0 += kB) {
#pragma unroll
                for (int u = 0; u < kB; ++u)
                    if (s0 + kB + u < H) g[(s0 / kB + 1) & 1][u] = gr[(s0 + kB + u) * gd];
#pragma unroll
                for (int u = 0; u < kB; ++u)
                    if (s0 + u < H) {
                        const int s = s0 + u;
                        const double b = fma(-l2[s], y2, fma(1.0, rr[s * rd], g[(s0 / kB) & 1][u]));
                        y2 = y1;
                        y1 = fma(-l1[s], y1, b);
                        v[s] = y1;
                    }
            }
            // middle: own H-2, own H-1, other H-1, other H-2
            const double o1 = __shfl_xor_sync(0xffffffffu, y1, 16), o2 = __shfl_xor_sync(0xffffffffu, y2, 16);
            double x[3];  // own H-2, own H-1, other H-1
#pragma unroll
            for (int q = 0; q < 3; ++q)
                x[q] = fma(mid[4 * q], y2, fma(mid[4 * q + 1], y1, fma(mid[4 * q + 2], o1, times(mid[4 * q + 3], o2))));
            double xi = x[2], xs = x[1], xo = x[0];  // inner, own, outer unknown of position s
            asm volatile("" ::: "memory");
            const int mr = (A.n - un.rp + 1) / 2, mc = (A.n - un.cp + 1) / 2, k = place_of(ln, H);
            double *yk = A.Y + un.off + (int64_t)un.rp * A.n + 2 * k + un.cp;
#pragma unroll
            for (int s = H - 1; s >= 0; --s) {
                if (s < H - 1) {
                    xi = xs;
                    xs = xo;
                    xo = s > 0 ? fma(-n1[s - 1], xs, fma(-n2[s - 1], xi, v[s - 1])) : 0.0;
                }
                if (last) {
                    const int i = h ? N - 1 - s : s;
                    const double out = times(iu[s], xs);
                    if (on && i < mr && k < mc) yk[(int64_t)2 * i * A.n] = out;
                } else {
                    const double out = fma(ca[s], xo, fma(cb[s], xs, fma(cc[s], xi, rr[s * rd])));
                    if (on) rr[s * rd] = out;
                }
            }
        }
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
    }
}

// G = F D^{-1} of every unit, [unit][N][N] in the order of place_of, zero beyond the quarter.
// Units are on grid.x: there are four per (mode, rhs) pair, up to 262140, and grid.y ends at 65535.
__global__ void __launch_bounds__(256) cyl_quarter_kernel(const double *__restrict__ F, double *__restrict__ G,
                                                          const CylUnit *__restrict__ units, int n, int N)
{
    const CylUnit un = units[blockIdx.x];
    const int64_t total = (int64_t)N * N;
    for (int64_t q = blockIdx.y * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.y * blockDim.x) {
        const int i = 2 * place_of((int)(q / N), N / 2) + un.rp, k = 2 * place_of((int)(q % N), N / 2) + un.cp;
        double v = 0.0;
        if (i < n && k < n) v = -F[un.off + (int64_t)i * n + k] / (((double)k + 1.0) * ((double)k + 2.0));
        G[blockIdx.x * total + q] = v;
    }
}

// ---- n > 256: 32 lines per CTA, two launches per iteration ----
constexpr int kCL = 32;        // lines per CTA
constexpr int kCylThreads = 256;  // threads per CTA: all move the tile, the first 2 kCL sweep
constexpr int kZ = 3, kR = 8;  // table entries per position: z l, m, g; r l1, l2, n1, n2, a, b, c, 1/pivot

struct CylArgs {
    int n, nrhs, j;
    const double *zfac, *rfac;  // [sum J][n][kZ], [sum J][n][kR]
    const int *joff, *jcount;
    const double *G;       // [modes][nrhs][n][n]
    const double *Rin;
    double *Rout, *Y;
    bool first;            // j == 0: the z kernel reads R1 = -G
};

__host__ __device__ inline int pitch_of(int n) { return (n % 2 == 0) ? n + 1 : n; }

constexpr int kC = 8;  // read-ahead chunk of the sweeps

// z kernel: blockIdx.x = block of 32 rows, blockIdx.y = (mode, rhs).  Shared memory: the
// tile [32][P], then the table set [n][kZ].
__global__ void __launch_bounds__(kCylThreads) cyl_z_kernel(CylArgs A)
{
    const int n = A.n, P = pitch_of(n);
    const int mode = blockIdx.y / A.nrhs;
    const int J = A.jcount[mode];
    if (A.j >= J) return;
    extern __shared__ __align__(16) double cyl_smem[];
    double *tile = cyl_smem, *fz = tile + kCL * P;
    const int64_t pair = blockIdx.y;
    const int i0 = blockIdx.x * kCL, nl = min(kCL, n - i0);
    const double *Rin = A.first ? A.G : A.Rin;
    const double sgn = A.first ? -1.0 : 1.0;
    const int64_t base = pair * (int64_t)n * n + (int64_t)i0 * n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int li = warp; li < nl; li += kCylThreads / 32) {
        const double *src = Rin + base + (int64_t)li * n;
#pragma unroll 4
        for (int t = lane; t < n; t += 32) tile[li * P + t] = A.first ? -src[t] : src[t];
    }
    const double *fzg = A.zfac + (int64_t)(A.joff[mode] + A.j) * n * kZ;
    for (int t = threadIdx.x; t < n * kZ; t += blockDim.x) fz[t] = fzg[t];
    __syncthreads();
    const int li = threadIdx.x & (kCL - 1), par = threadIdx.x / kCL;
    if (threadIdx.x < 2 * kCL && li < nl) {
        double *row = tile + li * P;
        const int m = (n - par + 1) / 2;
        double z = 0.0;
        for (int s0 = 0; s0 < m; s0 += kC) {
            double in[kC], l[kC];
#pragma unroll
            for (int u = 0; u < kC; ++u) {
                const int t = par + 2 * min(s0 + u, m - 1);
                in[u] = row[t];
                l[u] = fz[t * kZ];
            }
#pragma unroll
            for (int u = 0; u < kC; ++u)
                if (s0 + u < m) {
                    z = fma(-l[u], z, in[u]);
                    row[par + 2 * (s0 + u)] = z;
                }
        }
        double y = 0.0;
        for (int s0 = m - 1; s0 >= 0; s0 -= kC) {
            double zz[kC], mm[kC], g[kC];
#pragma unroll
            for (int u = 0; u < kC; ++u) {
                const int t = par + 2 * max(s0 - u, 0);
                zz[u] = row[t];
                mm[u] = fz[t * kZ + 1];
                g[u] = fz[t * kZ + 2];
            }
#pragma unroll
            for (int u = 0; u < kC; ++u)
                if (s0 - u >= 0) {
                    y = fma(-mm[u], y, zz[u]);
                    row[par + 2 * (s0 - u)] = times(g[u], y);
                }
        }
    }
    __syncthreads();
    for (int l = warp; l < nl; l += kCylThreads / 32) {
        const int64_t g0 = base + (int64_t)l * n;
#pragma unroll 4
        for (int t = lane; t < n; t += 32) {  // S + G = R + (q - p) w + G
            const double G = A.G[g0 + t];
            A.Rout[g0 + t] = fma(sgn, A.first ? G : Rin[g0 + t], tile[l * P + t]) + G;
        }
    }
}

// r kernel: blockIdx.x = block of 32 columns, blockIdx.y = (mode, rhs).  Shared memory: the
// tile [n][32], then the table set [n][kR].
__global__ void __launch_bounds__(kCylThreads) cyl_r_kernel(CylArgs A)
{
    const int n = A.n;
    const int mode = blockIdx.y / A.nrhs;
    const int J = A.jcount[mode];
    if (A.j >= J) return;
    const bool last = A.j + 1 == J;
    extern __shared__ __align__(16) double cyl_smem[];
    double *tile = cyl_smem, *fr = tile + (int64_t)n * kCL;
    const int64_t pair = blockIdx.y;
    const int c0 = blockIdx.x * kCL, nc = min(kCL, n - c0);
    const int64_t base = pair * (int64_t)n * n + c0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane < nc) {
#pragma unroll 4
        for (int t = warp; t < n; t += kCylThreads / 32) tile[t * kCL + lane] = A.Rin[base + (int64_t)t * n + lane];
    }
    const double *frg = A.rfac + (int64_t)(A.joff[mode] + A.j) * n * kR;
    for (int q = threadIdx.x; q < kR * n; q += blockDim.x) fr[q] = frg[q];
    __syncthreads();
    const int cj = threadIdx.x & (kCL - 1), par = threadIdx.x / kCL;
    if (threadIdx.x < 2 * kCL && cj < nc) {
        double *col = tile + cj;
        const int m = (n - par + 1) / 2;
        double y1 = 0.0, y2 = 0.0;  // y at s - 1, s - 2
        for (int s0 = 0; s0 < m; s0 += kC) {
            double bb[kC], l1[kC], l2[kC];
#pragma unroll
            for (int u = 0; u < kC; ++u) {
                const int t = par + 2 * min(s0 + u, m - 1);
                bb[u] = col[t * kCL];
                l1[u] = fr[t * kR + 0];
                l2[u] = fr[t * kR + 1];
            }
#pragma unroll
            for (int u = 0; u < kC; ++u)
                if (s0 + u < m) {
                    const double y = fma(-l1[u], y1, fma(-l2[u], y2, bb[u]));
                    col[(par + 2 * (s0 + u)) * kCL] = y;
                    y2 = y1;
                    y1 = y;
                }
        }
        // x (pivot left in) at s, s + 1, s + 2; position s + 1 is finished when x at s is known
        double x0 = 0.0, x1 = 0.0, x2 = 0.0;
        for (int s0 = m - 1; s0 >= -1; s0 -= kC) {
            double yy[kC], n1[kC], n2[kC], a[kC], b[kC], c[kC];
#pragma unroll
            for (int u = 0; u < kC; ++u) {
                const int t = par + 2 * max(s0 - u, 0);
                yy[u] = s0 - u >= 0 ? col[t * kCL] : 0.0;
                n1[u] = fr[t * kR + 2];
                n2[u] = fr[t * kR + 3];
                const int t1 = par + 2 * min(max(s0 - u + 1, 0), m - 1);
                a[u] = fr[t1 * kR + (last ? 7 : 4)];
                b[u] = fr[t1 * kR + 5];
                c[u] = fr[t1 * kR + 6];
            }
#pragma unroll
            for (int u = 0; u < kC; ++u) {
                const int s = s0 - u;
                if (s >= -1) {
                    x2 = x1;
                    x1 = x0;
                    x0 = s >= 0 ? fma(-n1[u], x1, fma(-n2[u], x2, yy[u])) : 0.0;
                    if (s + 1 < m)
                        col[(par + 2 * (s + 1)) * kCL] =
                            last ? times(a[u], x1) : fma(a[u], x0, fma(b[u], x1, times(c[u], x2)));
                }
            }
        }
    }
    __syncthreads();
    if (lane < nc) {
#pragma unroll 4
        for (int t = warp; t < n; t += kCylThreads / 32) {
            const int64_t g = base + (int64_t)t * n + lane;
            if (last) A.Y[g] = tile[t * kCL + lane];
            else A.Rout[g] = (A.Rin[g] - A.G[g]) + tile[t * kCL + lane];
        }
    }
}

int z_smem(int n) { return (int)sizeof(double) * (kCL * pitch_of(n) + kZ * n); }
int r_smem(int n) { return (int)sizeof(double) * (kCL * n + kR * n); }
// The refusal of sizes that do not fit stays where it has been: a shared memory of 12 n
// doubles beside the tile.
int smem_needed(int n) { return (int)sizeof(double) * (kCL * pitch_of(n) + 12 * n); }

// G = F D^{-1} (column j scaled by 1 / D_jj)
__global__ void cyl_scale_kernel(const double *F, double *G, int n, int64_t total)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(q % n);
        G[q] = -F[q] / (((double)j + 1.0) * ((double)j + 2.0));
    }
}

// ---------------------------------------------------------------- host tables
// Tridiagonal N^T = D^{-1} M + p of one parity (along z) and, along r, the bands of
// Q - q P and P; unknowns beyond m are decoupled (identity, P = 0).
struct ZBands {
    std::vector<double> d, c, e;  // diagonal, coupling to i - 1, coupling to i + 1
};
ZBands z_bands(int64_t n, int par, double p, int size)
{
    ZBands b;
    b.d.assign(size, 1.0);
    b.c.assign(size, 0.0);
    b.e.assign(size, 0.0);
    const int m = (int)((n - par + 1) / 2);
    for (int s = 0; s < m; ++s) {
        const int64_t t = par + 2 * s;
        const double iD = -1.0 / (((double)t + 1.0) * ((double)t + 2.0));
        b.d[s] = cyl_M_diag(t) * iD + p;
        if (s >= 1) b.c[s] = cyl_M_off(t - 2) * iD;
        if (s + 1 < m) b.e[s] = cyl_M_off(t) * iD;
    }
    return b;
}

bool finite_all(const double *v, int count)
{
    for (int i = 0; i < count; ++i)
        if (!std::isfinite(v[i])) return false;
    return true;
}

// z_table of the twisted elimination; alpha = q - p.
bool twisted_z(const ZBands &B, int H, double alpha, double *out)
{
    const int N = 2 * H;
    double *l = out, *m = l + N, *g = m + N, *mid = g + N;
    std::vector<double> piv(N);
    auto idx = [&](int h, int s) { return h ? N - 1 - s : s; };
    auto outer = [&](int h, int s) { return h ? B.e[idx(h, s)] : B.c[idx(h, s)]; };
    auto inner = [&](int h, int s) { return h ? B.c[idx(h, s)] : B.e[idx(h, s)]; };
    for (int h = 0; h < 2; ++h)
        for (int s = 0; s < H; ++s) {
            const double lv = s ? outer(h, s) / piv[h * H + s - 1] : 0.0;
            l[h * H + s] = lv;
            piv[h * H + s] = B.d[idx(h, s)] - (s ? lv * inner(h, s - 1) : 0.0);
            g[h * H + s] = alpha / piv[h * H + s];
        }
    for (int h = 0; h < 2; ++h)
        for (int s = 0; s < H; ++s) m[h * H + s] = s + 1 < H ? inner(h, s) / piv[h * H + s + 1] : 0.0;
    const double d0 = piv[H - 1], d1 = piv[N - 1], e0 = inner(0, H - 1), c1 = inner(1, H - 1), det = d0 * d1 - e0 * c1;
    mid[0] = d0 * d1 / det;
    mid[1] = -e0 * d0 / det;
    mid[2] = d0 * d1 / det;
    mid[3] = -c1 * d1 / det;
    return finite_all(out, z_table(H));
}

// Inverse of a 4 x 4 matrix by Gauss-Jordan elimination with partial pivoting.
bool invert4(double a[4][4], double inv[4][4])
{
    for (int i = 0; i < 4; ++i)
        for (int k = 0; k < 4; ++k) inv[i][k] = i == k ? 1.0 : 0.0;
    for (int c = 0; c < 4; ++c) {
        int p = c;
        for (int r = c + 1; r < 4; ++r)
            if (std::fabs(a[r][c]) > std::fabs(a[p][c])) p = r;
        if (a[p][c] == 0.0) return false;
        for (int k = 0; k < 4; ++k) {
            std::swap(a[c][k], a[p][k]);
            std::swap(inv[c][k], inv[p][k]);
        }
        const double s = 1.0 / a[c][c];
        for (int k = 0; k < 4; ++k) {
            a[c][k] *= s;
            inv[c][k] *= s;
        }
        for (int r = 0; r < 4; ++r) {
            if (r == c) continue;
            const double f = a[r][c];
            for (int k = 0; k < 4; ++k) {
                a[r][k] -= f * a[c][k];
                inv[r][k] -= f * inv[c][k];
            }
        }
    }
    return true;
}

// r_table of the twisted elimination of Q - q P (H >= 2); beta = q - p' (0 in the last iteration).
bool twisted_r(const ParityOps &o, double q, double beta, int H, double *out)
{
    const int N = 2 * H;
    double *l1 = out, *l2 = l1 + N, *n1 = l2 + N, *n2 = n1 + N, *ca = n2 + N, *cb = ca + N, *cc = cb + N, *iu = cc + N,
           *mid = iu + N;
    auto P = [&](int i, int k) {
        if (i < 0 || k < 0 || i >= o.m || k >= o.m) return 0.0;
        return k == i ? o.pd[i] : (k == i - 1 ? o.pl[i] : (k == i + 1 ? o.pu[i] : 0.0));
    };
    auto Q = [&](int i, int k) {
        const int a = std::min(i, k), d = std::abs(i - k);
        if (a < 0 || std::max(i, k) >= o.m || d > 2) return 0.0;
        return d == 0 ? o.q0[a] : (d == 1 ? o.q2[a] : o.q4[a]);
    };
    auto T = [&](int i, int k) { return i == k && i >= o.m ? 1.0 : Q(i, k) - q * P(i, k); };
    auto idx = [&](int h, int s) { return h ? N - 1 - s : s; };
    std::vector<double> u0(N), u1(N), u2(N);
    for (int h = 0; h < 2; ++h)
        for (int s = 0; s < H; ++s) {
            const int i = idx(h, s), b = h * H;
            const double a2 = s >= 2 ? T(i, idx(h, s - 2)) / u0[b + s - 2] : 0.0;
            const double a1 = s >= 1 ? (T(i, idx(h, s - 1)) - (s >= 2 ? a2 * u1[b + s - 2] : 0.0)) / u0[b + s - 1] : 0.0;
            u0[b + s] = T(i, i) - (s >= 1 ? a1 * u1[b + s - 1] : 0.0) - (s >= 2 ? a2 * u2[b + s - 2] : 0.0);
            u1[b + s] = T(i, idx(h, s + 1)) - (s >= 1 ? a1 * u2[b + s - 1] : 0.0);
            u2[b + s] = T(i, idx(h, s + 2));
            l1[b + s] = a1;
            l2[b + s] = a2;
            iu[b + s] = 1.0 / u0[b + s];
        }
    for (int h = 0; h < 2; ++h)
        for (int s = 0; s < H; ++s) {
            const int i = idx(h, s), b = h * H;
            n1[b + s] = s + 2 < H ? u1[b + s] / u0[b + s + 1] : 0.0;
            n2[b + s] = s + 2 < H ? u2[b + s] / u0[b + s + 2] : 0.0;
            ca[b + s] = s >= 1 ? beta * P(i, idx(h, s - 1)) / u0[b + s - 1] : 0.0;
            cb[b + s] = beta * P(i, i) / u0[b + s];
            cc[b + s] = beta * P(i, idx(h, s + 1)) / (s + 1 < H ? u0[b + s + 1] : u0[(1 - h) * H + H - 1]);
        }
    // unknowns 0: H-2, 0: H-1, 1: H-1, 1: H-2 from the four forward values in this order
    double K[4][4] = {{u0[H - 2], u1[H - 2], u2[H - 2], 0.0},
                      {0.0, u0[H - 1], u1[H - 1], u2[H - 1]},
                      {u2[N - 1], u1[N - 1], u0[N - 1], 0.0},
                      {0.0, u2[N - 2], u1[N - 2], u0[N - 2]}};
    double inv[4][4];
    if (!invert4(K, inv)) return false;
    const double piv[4] = {u0[H - 2], u0[H - 1], u0[N - 1], u0[N - 2]};
    for (int h = 0; h < 2; ++h)
        for (int x = 0; x < 3; ++x)  // own H-2, own H-1, other H-1
            for (int k = 0; k < 4; ++k) {
                const int row = h ? 3 - x : x, col = h ? 3 - k : k;
                mid[12 * h + 4 * x + k] = piv[row] * inv[row][col];
            }
    return finite_all(out, r_table(H));
}

// Table sets of the streaming kernels: plain elimination from the first unknown.
bool stream_z(const ZBands &B, int m, int par, double alpha, double *out)
{
    double piv = 0.0, e = 0.0;
    for (int s = 0; s < m; ++s) {
        double *o = out + (int64_t)(par + 2 * s) * kZ;
        o[0] = s ? B.c[s] / piv : 0.0;
        const double np = B.d[s] - (s ? o[0] * e : 0.0);
        if (s) out[(int64_t)(par + 2 * (s - 1)) * kZ + 1] = e / np;
        o[1] = 0.0;
        o[2] = alpha / np;
        piv = np;
        e = B.e[s];
        if (!std::isfinite(o[0]) || !std::isfinite(o[2])) return false;
    }
    return true;
}
bool stream_r(const ParityOps &o, double q, double beta, int par, double *out)
{
    const LU5 f = lu_QminusqP(o, q);
    for (int s = 0; s < o.m; ++s) {
        double *e = out + (int64_t)(par + 2 * s) * kR;
        e[0] = f.l1[s];
        e[1] = f.l2[s];
        e[2] = s + 1 < o.m ? f.u1[s] * f.iu0[s + 1] : 0.0;
        e[3] = s + 2 < o.m ? f.u2[s] * f.iu0[s + 2] : 0.0;
        e[4] = s >= 1 ? beta * o.pl[s] * f.iu0[s - 1] : 0.0;
        e[5] = beta * o.pd[s] * f.iu0[s];
        e[6] = s + 1 < o.m ? beta * o.pu[s] * f.iu0[s + 1] : 0.0;
        e[7] = f.iu0[s];
        if (!finite_all(e, kR)) return false;
    }
    return true;
}

// Half lengths with a compiled resident kernel.
#define CYL_SIZES(X) X(2) X(4) X(8) X(12) X(16) X(20) X(24) X(32) X(40) X(48) X(56) X(64)
int half_of(int64_t n)
{
    const int m = (int)((n + 1) / 2);
#define TRY(h) if (m <= 2 * h) return h;
    CYL_SIZES(TRY)
#undef TRY
    return 0;
}
template <int H>
cudaError_t setup_half()
{
    return cudaFuncSetAttribute(cyl_resident_kernel<H>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CylGeo<H>::bytes);
}
template <int H>
cudaError_t launch_half(const CylResArgs &a, int units, cudaStream_t st)
{
    cyl_resident_kernel<H><<<(unsigned)units, CylGeo<H>::kThreads, CylGeo<H>::bytes, st>>>(a);
    return cudaGetLastError();
}

}  // namespace

template <typename U>
cudaError_t CylinderEngine::dalloc(U **p, size_t count)
{
    cudaError_t e = cudaMalloc((void **)p, sizeof(U) * std::max<size_t>(count, 1));
    if (e == cudaSuccess) {
        allocs_.push_back(*p);
        bytes += (int64_t)(sizeof(U) * count);
    }
    return e;
}

#define CYL_CK(call)                                                                                      \
    do {                                                                                                  \
        cudaError_t e_ = (call);                                                                          \
        if (e_ != cudaSuccess) {                                                                          \
            err = std::string(#call) + ": " + cudaGetErrorString(e_);                                     \
            return FPS_ERR_CUDA;                                                                          \
        }                                                                                                 \
    } while (0)

int CylinderEngine::create(int64_t n_, int64_t kmin_, int64_t kmax_, double tol, int nrhs_, std::string &err)
{
    n = n_;
    kmin = kmin_;
    kmax = kmax_;
    nrhs = nrhs_;
    const int modes = (int)(kmax - kmin + 1);
    // The streaming kernels hold whole lines of 32 (mode, rhs) rows or columns in shared
    // memory: about 352 n bytes per CTA, n <= 659 at 227 KB.
    int dev = 0, optin = 0;
    CYL_CK(cudaGetDevice(&dev));
    CYL_CK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    const int need = smem_needed((int)n);
    if (need > optin) {
        err = "n = " + std::to_string(n) + " needs " + std::to_string(need) +
              " bytes of shared memory per CTA (device limit " + std::to_string(optin) + ")";
        return FPS_ERR_UNSUPPORTED;
    }
    // sigma(B) = sigma(-M D^{-1}) = sigma(-A~): the tight interval of A~
    lo = square_eps(n);
    hi = 1.0;
    square_tight_interval(n, lo, hi);
    J.assign(modes, 0);
    a.assign(modes, 0.0);
    b.assign(modes, 0.0);
    std::vector<std::vector<double>> P(modes), Qs(modes);
    Jmax = 0;
    for (int md = 0; md < modes; ++md) {
        const int64_t k = kmin + md;
        if (cyl_mode_interval(n, k, a[md], b[md]) != FPS_OK) {
            err = "mode " + std::to_string(k) + ": eigenvalue interval of A_k not found";
            return FPS_ERR_UNSUPPORTED;
        }
        J[md] = adi_iterations(a[md], b[md], lo, hi, tol);
        zolotarev_shifts(a[md], b[md], lo, hi, J[md], P[md], Qs[md]);
        if (!shifts_valid(Qs[md], lo, hi)) {
            err = "shift list failed validation (a shift is not finite or lies outside the spectral interval)";
            return FPS_ERR_INVALID_ARG;
        }
        for (double &v : P[md]) v = -v;
        const bool ok = shifts_valid(P[md], -b[md], -a[md]);
        for (double &v : P[md]) v = -v;
        if (!ok) {
            err = "shift list failed validation (a shift is not finite or lies outside the spectral interval)";
            return FPS_ERR_INVALID_ARG;
        }
        Jmax = std::max(Jmax, J[md]);
    }
    // tables
    std::vector<int> joff(modes), jc(modes);
    int sumJ = 0;
    for (int md = 0; md < modes; ++md) {
        joff[md] = sumJ;
        jc[md] = J[md];
        sumJ += J[md];
    }
    half_ = n <= kResMaxN ? half_of(n) : 0;
    const int H = half_, size = H ? 2 * H : (int)((n + 1) / 2);
    const size_t zsz = H ? 2 * (size_t)z_table(H) : (size_t)n * kZ, rsz = H ? 2 * (size_t)r_table(H) : (size_t)n * kR;
    // every entry is written below
    const std::unique_ptr<double[]> zf(new double[(size_t)sumJ * zsz]), rf(new double[(size_t)sumJ * rsz]);
    for (int md = 0; md < modes; ++md) {
        const int64_t k = kmin + md;
        const ParityOps ops[2] = {parity_ops(n, k, 0), parity_ops(n, k, 1)};
        for (int j = 0; j < J[md]; ++j) {
            const double p = P[md][j], q = Qs[md][j], alpha = q - p, beta = j + 1 < J[md] ? q - P[md][j + 1] : 0.0;
            double *z = zf.get() + (size_t)(joff[md] + j) * zsz, *r = rf.get() + (size_t)(joff[md] + j) * rsz;
            for (int par = 0; par < 2; ++par) {
                const ZBands B = z_bands(n, par, p, size);
                const bool ok = H ? twisted_z(B, H, alpha, z + par * z_table(H)) &&
                                        twisted_r(ops[par], q, beta, H, r + par * r_table(H))
                                  : stream_z(B, ops[par].m, par, alpha, z) && stream_r(ops[par], q, beta, par, r);
                if (!ok) {
                    err = "mode " + std::to_string(k) + ": pivot breakdown in the factors";
                    return FPS_ERR_UNSUPPORTED;
                }
            }
        }
    }
    // quarters, most iterations first
    std::vector<CylUnit> units;
    if (H) {
        std::vector<int> order(modes);
        for (int md = 0; md < modes; ++md) order[md] = md;
        std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return J[x] > J[y]; });
        for (int md : order)
            for (int r = 0; r < nrhs; ++r)
                for (int q = 0; q < 4; ++q) {
                    CylUnit u;
                    u.off = ((int64_t)md * nrhs + r) * n * n;
                    u.joff = joff[md];
                    u.J = J[md];
                    u.rp = q >> 1;
                    u.cp = q & 1;
                    units.push_back(u);
                }
    }
    const size_t total = (size_t)modes * nrhs * n * n;
    nunits_ = (int)units.size();
    CYL_CK(dalloc(&G_, H ? units.size() * (size_t)size * size : total));
    if (!H) {
        CYL_CK(dalloc(&R1_, total));
        CYL_CK(dalloc(&R2_, total));
    }
    CYL_CK(dalloc(&zfac_, (size_t)sumJ * zsz));
    CYL_CK(dalloc(&rfac_, (size_t)sumJ * rsz));
    CYL_CK(dalloc(&joff_, (size_t)modes));
    CYL_CK(dalloc(&jcount_, (size_t)modes));
    CYL_CK(dalloc((char **)&units_, sizeof(CylUnit) * units.size()));
    CYL_CK(cudaMemcpy(zfac_, zf.get(), sizeof(double) * (size_t)sumJ * zsz, cudaMemcpyHostToDevice));
    CYL_CK(cudaMemcpy(rfac_, rf.get(), sizeof(double) * (size_t)sumJ * rsz, cudaMemcpyHostToDevice));
    CYL_CK(cudaMemcpy(joff_, joff.data(), sizeof(int) * modes, cudaMemcpyHostToDevice));
    CYL_CK(cudaMemcpy(jcount_, jc.data(), sizeof(int) * modes, cudaMemcpyHostToDevice));
    if (H) {
        CYL_CK(cudaMemcpy(units_, units.data(), sizeof(CylUnit) * units.size(), cudaMemcpyHostToDevice));
        switch (H) {
#define CASE_SETUP(h) case h: CYL_CK(setup_half<h>()); break;
            CYL_SIZES(CASE_SETUP)
#undef CASE_SETUP
        }
    } else {
        CYL_CK(cudaFuncSetAttribute(cyl_z_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, z_smem((int)n)));
        CYL_CK(cudaFuncSetAttribute(cyl_r_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, r_smem((int)n)));
    }
    return FPS_OK;
}

void CylinderEngine::release()
{
    for (void *p : allocs_) cudaFree(p);
    allocs_.clear();
}

int CylinderEngine::solve(const double *F, double *Y, cudaStream_t st, std::string &err)
{
    const int modes = (int)(kmax - kmin + 1);
    const int64_t total = (int64_t)modes * nrhs * n * n;
    launches_last = 0;
    if (half_) {
        const int N = 2 * half_;
        const unsigned by = (unsigned)std::max(1, std::min(N * N / 1024, 16));
        cyl_quarter_kernel<<<dim3((unsigned)nunits_, by), 256, 0, st>>>(F, G_, (const CylUnit *)units_, (int)n, N);
        CYL_CK(cudaGetLastError());
        const CylResArgs a{(int)n, (const CylUnit *)units_, zfac_, rfac_, G_, Y};
        switch (half_) {
#define CASE_LAUNCH(h) case h: CYL_CK(launch_half<h>(a, nunits_, st)); break;
            CYL_SIZES(CASE_LAUNCH)
#undef CASE_LAUNCH
        }
        launches_last = 2;
        return FPS_OK;
    }
    cyl_scale_kernel<<<(unsigned)std::min<int64_t>((total + 255) / 256, 4096), 256, 0, st>>>(F, G_, (int)n, total);
    ++launches_last;
    CYL_CK(cudaGetLastError());
    CylArgs A;
    A.n = (int)n;
    A.nrhs = nrhs;
    A.zfac = zfac_;
    A.rfac = rfac_;
    A.joff = joff_;
    A.jcount = jcount_;
    A.G = G_;
    A.Y = Y;
    const dim3 grid((unsigned)((n + kCL - 1) / kCL), (unsigned)(modes * nrhs));
    const int zs = z_smem((int)n), rs = r_smem((int)n);
    for (int j = 0; j < Jmax; ++j) {
        A.j = j;
        A.first = j == 0;
        A.Rin = R1_;
        A.Rout = R2_;
        cyl_z_kernel<<<grid, kCylThreads, zs, st>>>(A);
        A.first = false;
        A.Rin = R2_;
        A.Rout = R1_;
        cyl_r_kernel<<<grid, kCylThreads, rs, st>>>(A);
        launches_last += 2;
        CYL_CK(cudaGetLastError());
    }
    return FPS_OK;
}

}  // namespace fps
