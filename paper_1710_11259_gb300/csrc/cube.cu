// The cube (Sec. 5): nested ADI for (T_01 + T_02 + T_12) Y = G on n x n x n
// tensors (row-major, mode 0 = i, mode 1 = j, mode 2 = k), T_ab applying A~ on
// modes a and b, G = -F / sqrt(E_i E_j E_k), X = Y / sqrt(E_i E_j E_k).
//   outer  (5.3)-(5.4): H = T_01 + T_02, V = T_12,
//          (V + p) Y_h = G - (H - p) Y,   (H - q) Y+ = G - (V + q) Y_h
//   middle (5.5)-(5.6): H + s = (T_01 + s/2) + (T_02 + s/2),
//          (B' + a) W_h = R - (A' - a) W,  (A' + a) W+ = R - (B' - a) W_h
//   inner  (5.7)-(5.9): A~_a Z A~_b + c Z = R per slice, as A~_a Z - Z(-c A~_b^{-1}) = R A~_b^{-1}:
//          Z_h = [R - (A~_a - p) Z A~_b] (c + p A~_b)^{-1}
//          (A~_a - q) Z+ = (R - c Z_h) A~_b^{-1} - q Z_h
// FP64: every operation is a banded product or a banded (even/odd decoupled, App. B)
// solve along one mode of the whole tensor: all slices of a level are solved at
// once.  The solves run one thread per (line, parity) over 32 lines per CTA with
// coalesced global traffic.
//
// FP32 + refinement: the nested ADI (every level in residual-propagating form, see
// CubeRounds::run and hsolve_res; the inner level runs all its iterations in one launch,
// one CTA per parity quarter of a slice, cube_unit.cuh; every level's shifts on the tight
// Sturm-bisection interval of A~, 2.5x fewer inner iterations than on Lemma B.2's
// at n = 256) runs in FP32 at loose level tolerances on
// the normalised residual rho = R / max|R|, R = G - (T_01 + T_02 + T_12) Y computed
// in FP64 (a 27-point product), and Y += max|R| * delta accumulates in FP64, until
// max|R| / max|G| meets the plan's tolerance.  The defect correction only needs
// each round's correction to reduce the residual, so the loose inner levels make a
// round several times cheaper than one solve at the paper's 1e-15 inner levels.
//
// Index arithmetic inside the kernels is 32-bit where it divides: plans cap n at
// 320, so n^3 < 2^31.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/fps.h"
#include "cube.h"
#include "cube_unit.cuh"
#include "device_info.h"
#include "host_math.h"
#include "trace.h"

namespace fps {

namespace {

constexpr int kLines = 32;  // lines per CTA of the solve kernels
constexpr int kLineThreads = 128;  // threads per CTA: all move the tiles, the first 2 kLines sweep

// Y = sop * ((alpha A~ + beta) X along `mode`) + sr * R   (R may be null; Y may alias R)
__global__ void cube_band_kernel(const double *__restrict__ X, const double *R, double *Y, const double *__restrict__ d,
                                 const double *__restrict__ e, int n, int mode, double alpha, double beta,
                                 double sop, double sr)
{
    const int N = n * n * n;
    const int st = (mode == 0) ? n * n : ((mode == 1) ? n : 1);
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += gridDim.x * blockDim.x) {
        const int t = (mode == 0) ? idx / (n * n) : ((mode == 1) ? (idx / n) % n : idx % n);
        double v = (alpha * d[t] + beta) * X[idx];
        if (t >= 2) v = fma(alpha * e[t - 2], X[idx - 2 * st], v);
        if (t + 2 < n) v = fma(alpha * e[t], X[idx + 2 * st], v);
        v *= sop;
        if (R) v = fma(sr, R[idx], v);
        Y[idx] = v;
    }
}

// Z = a X + b Y (element-wise; Z may alias X or Y)
__global__ void cube_axpby_kernel(const double *X, const double *Y, double *Z, int N, double a, double b)
{
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += gridDim.x * blockDim.x)
        Z[idx] = fma(a, X[idx], b * Y[idx]);
}

// Thomas factors of (alpha A~ + beta I) for a list of (alpha, beta) pairs, one
// thread per (set, parity); fac[set * n + t] =
// {1/den_t, alpha e_t / den_t}.
__global__ void cube_factor_kernel(const double *__restrict__ d, const double *__restrict__ e, int n,
                                   const double2 *__restrict__ ab, int nsets, double2 *__restrict__ fac)
{
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= 2 * nsets) return;
    const int set = tid >> 1, par = tid & 1;
    const double alpha = ab[set].x, beta = ab[set].y;
    double u_prev = 0.0;
    for (int t = par; t < n; t += 2) {
        double den = alpha * d[t] + beta;
        if (t >= 2) den -= alpha * e[t - 2] * u_prev;
        const double ip = 1.0 / den;
        const double u = alpha * e[t] * ip;
        fac[(int64_t)set * n + t] = make_double2(ip, u);
        u_prev = u;
    }
}

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// Asynchronous copy of one element from global to shared memory.
__device__ __forceinline__ void cp_async8(double *dst, const double *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// Shared-memory row pitch of a contiguous-mode tile: odd, so that the 32 lanes of a
// warp (one line each, same t) hit distinct banks.
__host__ __device__ __forceinline__ int contig_pitch(int n) { return (n % 2 == 0) ? n + 1 : n + 2; }

// Elements of one shared-memory tile of the line solve.
__host__ __device__ __forceinline__ int line_tile_elems(int n, bool contig)
{
    return contig ? kLines * contig_pitch(n) : kLines * n;
}

// Dynamic shared memory of the line solve: the factor set and one or two tiles.
int line_smem_bytes(int n, bool contig, int ntiles)
{
    return n * (int)sizeof(double2) + ntiles * line_tile_elems(n, contig) * (int)sizeof(double);
}

// 16-byte asynchronous copy (both addresses 16-byte aligned).
__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// Banded solves along one mode for kLines lines per CTA:
//   X = (alpha A~ + beta)^{-1} (R1 + s2 R2)      (R2 may be null)
// The whole tile of R1 (and R2) is fetched with asynchronous copies (16-byte ones
// when the rows are aligned), so one CTA has all its bytes in flight at once.  The
// forward sweep forms the right-hand side as it goes; both Thomas sweeps (App. B parity
// decoupling: warp = parity, lane = line) run in shared memory in chunks whose operands
// are read ahead of the dependent FMAs, and the solution is written back coalesced.  X
// may alias R1 or R2.  Tile A holds R1, then z and x; tile B holds R2.
// CONTIG (mode 2): kLines consecutive lines, tile [line][t].  Otherwise (modes 0,
// 1): kLines lines adjacent in mode 2, one CTA per (index of the other strided mode,
// block of kLines), tile [t][line].
template <bool CONTIG>
__global__ void __launch_bounds__(kLineThreads) cube_line_kernel(const double2 *__restrict__ fac, const double *R1,
                                                                 const double *R2, double s2, double *X, int n,
                                                                 int mode)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tsz = line_tile_elems(n, CONTIG);
    double2 *fs = reinterpret_cast<double2 *>(smem_raw);  // the factor set, n entries
    double *A = reinterpret_cast<double *>(fs + n);
    double *B = A + tsz;
    for (int t = threadIdx.x; t < n; t += blockDim.x) fs[t] = fac[t];
    const int pitch = CONTIG ? contig_pitch(n) : 0;
    // geometry: element (li, t) of the tile <-> global offset gbase + li * gl + t * gt
    int nl;
    int64_t gbase, gl, gt;
    if (CONTIG) {
        const int L0 = blockIdx.x * kLines;
        nl = min(kLines, n * n - L0);
        gbase = (int64_t)L0 * n;
        gl = n;
        gt = 1;
    } else {
        const int nkb = (n + kLines - 1) / kLines;
        const int other = blockIdx.x / nkb, k0 = (blockIdx.x % nkb) * kLines;
        const int64_t nn = (int64_t)n * n;
        nl = min(kLines, n - k0);
        gbase = ((mode == 0) ? (int64_t)other * n : (int64_t)other * nn) + k0;
        gl = 1;
        gt = (mode == 0) ? nn : (int64_t)n;
    }
    auto sidx = [&](int li, int t) { return CONTIG ? li * pitch + t : t * kLines + li; };
    // element q of the tile in load/store order (consecutive threads -> consecutive addresses)
    auto qmap = [&](int q, int &li, int &t) {
        if (CONTIG) {
            li = q / n;
            t = q - li * n;
        } else {
            t = q >> 5;
            li = q & 31;
        }
    };
    const bool has_r2 = R2 != nullptr;
    // strided tiles whose rows are whole, 16-byte aligned rows of the tensor move in
    // 16-byte pieces (V elements)
    constexpr int V = 2;
    const bool vec = !CONTIG && nl == kLines && gt % V == 0 && gbase % V == 0 && ((uintptr_t)R1 & 15) == 0 &&
                     (!has_r2 || ((uintptr_t)R2 & 15) == 0) && ((uintptr_t)X & 15) == 0;
    const int total = kLines * n;
    if (vec) {
        for (int q = threadIdx.x * V; q < total; q += blockDim.x * V) {
            const int t = q >> 5, li = q & 31;
            const int64_t g = gbase + li + t * gt;
            cp_async16(&A[t * kLines + li], R1 + g);
            if (has_r2) cp_async16(&B[t * kLines + li], R2 + g);
        }
    } else {
        for (int q = threadIdx.x; q < total; q += blockDim.x) {
            int li, t;
            qmap(q, li, t);
            if (li < nl) {
                const int64_t g = gbase + li * gl + t * gt;
                cp_async8(&A[sidx(li, t)], R1 + g);
                if (has_r2) cp_async8(&B[sidx(li, t)], R2 + g);
            }
        }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    const int lane = threadIdx.x & 31, par = threadIdx.x >> 5;
    const int m = (n - par + 1) / 2;  // unknowns of this parity: t = par + 2 i, i < m
    if (threadIdx.x < 2 * kLines && lane < nl) {
        // Both sweeps in chunks of kC steps: the chunk's operands are read from shared
        // memory first, so only the kC dependent FMAs remain on the critical path.
        constexpr int kC = 8;
        double z = 0, u_prev = 0;
        for (int i0 = 0; i0 < m; i0 += kC) {
            double in[kC], uf[kC];
#pragma unroll
            for (int u = 0; u < kC; ++u) {
                const int t = par + 2 * min(i0 + u, m - 1);
                double v = A[sidx(lane, t)];
                if (has_r2) v = fma(s2, B[sidx(lane, t)], v);
                in[u] = v;
                uf[u] = fs[t].y;
            }
#pragma unroll
            for (int u = 0; u < kC; ++u)
                if (i0 + u < m) {
                    z = fma(-u_prev, z, in[u]);
                    A[sidx(lane, par + 2 * (i0 + u))] = z;
                    u_prev = uf[u];
                }
        }
        double x = 0;
        for (int i0 = m - 1; i0 >= 0; i0 -= kC) {
            double zz[kC];
            double2 ff[kC];
#pragma unroll
            for (int u = 0; u < kC; ++u) {
                const int t = par + 2 * max(i0 - u, 0);
                zz[u] = A[sidx(lane, t)];
                ff[u] = fs[t];
            }
#pragma unroll
            for (int u = 0; u < kC; ++u)
                if (i0 - u >= 0) {
                    x = fma(-ff[u].y, x, ff[u].x * zz[u]);
                    A[sidx(lane, par + 2 * (i0 - u))] = x;
                }
        }
    }
    __syncthreads();
    if (vec) {
        for (int q = threadIdx.x * V; q < total; q += blockDim.x * V) {
            const int t = q >> 5, li = q & 31;
            *reinterpret_cast<double2 *>(X + gbase + li + t * gt) = *reinterpret_cast<double2 *>(&A[t * kLines + li]);
        }
    } else {
        for (int q = threadIdx.x; q < total; q += blockDim.x) {
            int li, t;
            qmap(q, li, t);
            if (li < nl) X[gbase + li * gl + t * gt] = A[sidx(li, t)];
        }
    }
}

// G = -F s_i s_j s_k (scale-in) or X = Y s_i s_j s_k (scale-out, sign = +1)
__global__ void cube_scale_kernel(const double *__restrict__ A, double *__restrict__ B, const double *__restrict__ s,
                                  int n, double sign)
{
    const int N = n * n * n;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += gridDim.x * blockDim.x) {
        const int row = idx / n, k = idx - row * n, i = row / n, j = row - i * n;
        B[idx] = sign * A[idx] * s[i] * s[j] * s[k];
    }
}

// ---- FP64 defect correction ----

// A~[t, t + dt] for dt in {-2, 0, 2} (the caller keeps t + dt inside [0, n))
__device__ __forceinline__ double band_coef(const double *d, const double *e, int t, int dt)
{
    return dt == 0 ? d[t] : (dt > 0 ? e[t] : e[t - 2]);
}

__device__ __forceinline__ void block_max_bits(double local, unsigned long long *out)
{
    for (int off = 16; off > 0; off >>= 1) local = fmax(local, __shfl_xor_sync(0xffffffffu, local, off));
    __shared__ double wmax[32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) wmax[w] = local;
    __syncthreads();
    if (threadIdx.x == 0) {
        double bm = 0.0;
        for (int t = 0; t < (int)(blockDim.x >> 5); ++t) bm = fmax(bm, wmax[t]);
        atomicMax(out, (unsigned long long)__double_as_longlong(bm));
    }
}

// R = G - (T_01 + T_02 + T_12) Y in FP64 (Y read as zero if y_zero); *rmax = max |R|
// as a bit pattern (must start at 0; NaN and Inf are reported as +Inf).
__global__ void __launch_bounds__(256) cube_residual_kernel(const double *__restrict__ G, const double *__restrict__ Y,
                                                            const double *__restrict__ d, const double *__restrict__ e,
                                                            int n, double *__restrict__ R, bool y_zero,
                                                            unsigned long long *rmax)
{
    const int N = n * n * n;
    const int nn = n * n;
    double local = 0.0;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += gridDim.x * blockDim.x) {
        double r = G[idx];
        if (!y_zero) {
            const int row = idx / n, k = idx - row * n, i = row / n, j = row - i * n;
            const int idx3[3] = {i, j, k};
            const int st[3] = {nn, n, 1};
            double acc = 0.0;
            // pairs (0,1), (0,2), (1,2): offsets {0, +-2} on both modes of the pair
#pragma unroll
            for (int pr = 0; pr < 3; ++pr) {
                const int ma = pr == 2 ? 1 : 0, mb = pr == 0 ? 1 : 2;
                const int ta = idx3[ma], tb = idx3[mb];
#pragma unroll
                for (int da = -2; da <= 2; da += 2) {
                    if (ta + da < 0 || ta + da >= n) continue;
                    const double ca = band_coef(d, e, ta, da);
#pragma unroll
                    for (int db = -2; db <= 2; db += 2) {
                        if (tb + db < 0 || tb + db >= n) continue;
                        acc = fma(ca * band_coef(d, e, tb, db), Y[idx + da * st[ma] + db * st[mb]], acc);
                    }
                }
            }
            r -= acc;
        }
        R[idx] = r;
        const double a = fabs(r);
        local = (a <= 1.7976931348623157e308) ? fmax(local, a) : __longlong_as_double(0x7ff0000000000000LL);
    }
    block_max_bits(local, rmax);
}

// The FP32 tensors have mode 0 fastest, (i, j, k) at (j n + k) n + i; the FP64 ones mode 2.
// Tiles of 32 x 32 over (i, k) at fixed j go through shared memory.
__device__ __forceinline__ bool cube_tile(int n, int &j, int &i0, int &k0)
{
    const int nt = (n + 31) / 32;
    const int b = blockIdx.x;
    j = b / (nt * nt);
    i0 = (b / nt) % nt * 32;
    k0 = b % nt * 32;
    return j < n;
}

// rho = R / max|R| in FP32
__global__ void __launch_bounds__(256) cube_to32_kernel(const double *__restrict__ R, float *__restrict__ rho, int n,
                                                        const unsigned long long *__restrict__ rmax)
{
    __shared__ float t[32][33];
    const double inv = 1.0 / __longlong_as_double((long long)*rmax);
    int j, i0, k0;
    if (!cube_tile(n, j, i0, k0)) return;
    const int x = threadIdx.x & 31;
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (i0 + y < n && k0 + x < n) t[y][x] = (float)(R[((int64_t)(i0 + y) * n + j) * n + k0 + x] * inv);
    __syncthreads();
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (k0 + y < n && i0 + x < n) rho[((int64_t)j * n + k0 + y) * n + i0 + x] = t[x][y];
}

// Y = (first ? 0 : Y) + max|R| delta  in FP64
__global__ void __launch_bounds__(256) cube_update_kernel(double *__restrict__ Y, const float *__restrict__ delta, int n,
                                                          const unsigned long long *__restrict__ rmax, bool first)
{
    __shared__ float t[32][33];
    const double sc = __longlong_as_double((long long)*rmax);
    int j, i0, k0;
    if (!cube_tile(n, j, i0, k0)) return;
    const int x = threadIdx.x & 31;
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (k0 + y < n && i0 + x < n) t[y][x] = delta[((int64_t)j * n + k0 + y) * n + i0 + x];
    __syncthreads();
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (i0 + y < n && k0 + x < n) {
            double *p = Y + ((int64_t)(i0 + y) * n + j) * n + k0 + x;
            *p = fma(sc, (double)t[x][y], first ? 0.0 : *p);
        }
}

unsigned tiles_for(int n)
{
    const int nt = (n + 31) / 32;
    return (unsigned)(n * nt * nt);
}

int grid_for(int64_t N) { return (int)std::min<int64_t>((N + 255) / 256, 16 * (int64_t)current_sm_count()); }

}  // namespace

#define CUBE_CK(call)                                                                                    \
    do {                                                                                                 \
        cudaError_t ce_ = (call);                                                                        \
        if (ce_ != cudaSuccess) {                                                                        \
            err = std::string(#call) + ": " + cudaGetErrorString(ce_);                                   \
            return FPS_ERR_CUDA;                                                                         \
        }                                                                                                \
    } while (0)

// ===========================================================================
// CubeSchedule
// ===========================================================================

int CubeSchedule::add_stein(double c)
{
    // A~_a Z - Z B = C with sigma(A~_a) in [-hi, -lo] and sigma(B) = sigma(-c A~_b^{-1})
    // in [c/hi, c/lo]
    Stein s;
    s.c = c;
    const double a = -hi_, b = -lo_, cl = c / hi_, d = c / lo_;
    s.J = adi_iterations(a, b, cl, d, tol_in_);
    zolotarev_shifts(a, b, cl, d, s.J, s.p, s.q);
    steins_.push_back(std::move(s));
    return (int)steins_.size() - 1;
}

void CubeSchedule::schedule(int64_t n, double tol, double tol_mid, double tol_in, bool residual, bool tight)
{
    n_ = n;
    tol_in_ = tol_in;
    lo_ = square_eps(n);
    hi_ = 1.0;
    if (tight) square_tight_interval(n, lo_, hi_);
    // the schedule of every level, fixed for the plan: T_ab (A~ on two modes) has its
    // spectrum in [lo^2, hi^2], so sigma(H) is in [2 lo^2, 2 hi^2] and sigma(-V) in
    // [-hi^2, -lo^2]
    const double e2 = lo_ * lo_, h2 = hi_ * hi_;
    J_outer = adi_iterations(-h2, -e2, 2 * e2, 2 * h2, tol);
    std::vector<double> pp, qq;
    zolotarev_shifts(-h2, -e2, 2 * e2, 2 * h2, J_outer, pp, qq);
    inner_per_run = 0;
    for (int j = 0; j < J_outer; ++j) {
        Outer o;
        o.p = qq[j];  // in sigma(H)'s interval [2 lo^2, 2 hi^2]
        o.q = pp[j];  // in sigma(-V)'s interval [-hi^2, -lo^2]
        o.stein_v = add_stein(o.p);
        inner_per_run += (residual && j + 1 < J_outer ? 2 : 1) * steins_[o.stein_v].J;
        const double s = -o.q, lo = e2 + s / 2, hi = h2 + s / 2;
        const int Jm = adi_iterations(-hi, -lo, lo, hi, tol_mid);
        std::vector<double> am;
        zolotarev_shifts_symmetric(lo, hi, Jm, am);
        for (int m = 0; m < Jm; ++m) {
            Middle mid;
            mid.a = am[m];
            mid.stein = add_stein(s / 2 + am[m]);
            inner_per_run += (residual && m + 1 < Jm ? 3 : 2) * steins_[mid.stein].J;
            o.mid.push_back(mid);
        }
        outer_.push_back(std::move(o));
    }
}

cudaError_t CubeSchedule::alloc(void **p, size_t b)
{
    cudaError_t r = cudaMalloc(p, b ? b : 1);
    if (r == cudaSuccess) {
        allocs_.push_back(*p);
        bytes += (int64_t)b;
    }
    return r;
}

cudaError_t CubeSchedule::copy(void **p, const void *src, size_t b)
{
    const cudaError_t r = alloc(p, b);
    return r == cudaSuccess ? cudaMemcpy(*p, src, b, cudaMemcpyHostToDevice) : r;
}

void CubeSchedule::release()
{
    for (void *p : allocs_) cudaFree(p);
    allocs_.clear();
}

// ===========================================================================
// CubeNested
// ===========================================================================

int CubeNested::create(int64_t n, double tol, double tol_level, std::string &err)
{
    schedule(n, tol, tol_level, tol_level, false, false);
    std::vector<double2> ab;
    int64_t sets = 0;
    for (Stein &s : steins_) {
        s.off = (int64_t)ab.size();
        sets = std::max(sets, 2 * (int64_t)s.J + 1);
        ab.push_back(make_double2(1.0, 0.0));
        for (int l = 0; l < s.J; ++l) {
            ab.push_back(make_double2(s.p[l], s.c));
            ab.push_back(make_double2(1.0, -s.q[l]));
        }
    }
    std::vector<double> d, e;
    square_bands(n, d, e);
    const size_t N = (size_t)n * n * n;
    CUBE_CK(copy((void **)&bd_, d.data(), sizeof(double) * n));
    CUBE_CK(copy((void **)&be_, e.data(), sizeof(double) * n));
    for (double *&w : work_) CUBE_CK(alloc((void **)&w, sizeof(double) * N));
    CUBE_CK(alloc((void **)&fac_, sizeof(double2) * (size_t)sets * n));
    CUBE_CK(copy((void **)&ab_, ab.data(), sizeof(double2) * ab.size()));
    CUBE_CK(cudaFuncSetAttribute(cube_line_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 line_smem_bytes((int)n, true, 2)));
    CUBE_CK(cudaFuncSetAttribute(cube_line_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 line_smem_bytes((int)n, false, 2)));
    entry_ = -1;
    return FPS_OK;
}

cudaError_t CubeNested::band(const double *X, const double *R, double *Y, int mode, double alpha, double beta,
                             double sop, double sr)
{
    const int64_t N = n_ * n_ * n_;
    cube_band_kernel<<<grid_for(N), 256, 0, st_>>>(X, R, Y, bd_, be_, (int)n_, mode, alpha, beta, sop, sr);
    ++launches;
    return cudaGetLastError();
}

cudaError_t CubeNested::axpby(const double *X, const double *Y, double *Z, double a, double b)
{
    const int64_t N = n_ * n_ * n_;
    cube_axpby_kernel<<<grid_for(N), 256, 0, st_>>>(X, Y, Z, (int)N, a, b);
    ++launches;
    return cudaGetLastError();
}

cudaError_t CubeNested::solve(int set, const double *R1, const double *R2, double s2, double *X, int mode)
{
    const double2 *fac = fac_ + (int64_t)set * n_;
    const int n = (int)n_;
    const int smem = line_smem_bytes(n, mode == 2, R2 ? 2 : 1);
    if (mode == 2)
        cube_line_kernel<true><<<(n * n + kLines - 1) / kLines, kLineThreads, smem, st_>>>(fac, R1, R2, s2, X, n, mode);
    else
        cube_line_kernel<false>
            <<<n * ((n + kLines - 1) / kLines), kLineThreads, smem, st_>>>(fac, R1, R2, s2, X, n, mode);
    ++launches;
    return cudaGetLastError();
}

int CubeNested::load_factors(int entry, std::string &err)
{
    if (entry_ == entry) return FPS_OK;
    const Stein &S = steins_[entry];
    const int nsets = 2 * S.J + 1;
    // factor sets: 0 = A~; 1 + 2l = c + p_l A~; 2 + 2l = A~ - q_l
    cube_factor_kernel<<<(2 * nsets + 127) / 128, 128, 0, st_>>>(bd_, be_, (int)n_, ab_ + S.off, nsets, fac_);
    ++launches;
    CUBE_CK(cudaGetLastError());
    entry_ = entry;
    return FPS_OK;
}

// Z = (T_ab + c)^{-1} R, the inner level in the paper's form (entry = schedule
// index).  Uses work_[0], work_[1].
int CubeNested::stein(int ma, int mb, int entry, const double *R, double *Z, std::string &err)
{
    int st = load_factors(entry, err);
    if (st != FPS_OK) return st;
    const Stein &S = steins_[entry];
    double *W1 = work_[0], *W2 = work_[1];
    const double c = S.c;
    for (int l = 0; l < S.J; ++l) {
        const double *U = R;
        if (l > 0) {
            CUBE_CK(band(Z, nullptr, W1, mb, 1.0, 0.0, 1.0, 0.0));                // Z A~_b
            CUBE_CK(band(W1, R, W2, ma, 1.0, -S.p[l], -1.0, 1.0));                // R - (A~_a - p) ( . )
            U = W2;
        }
        CUBE_CK(solve(1 + 2 * l, U, nullptr, 0.0, W1, mb));    // Z_h = ( . ) (c + p A~_b)^{-1}
        CUBE_CK(solve(0, R, W1, -c, W2, mb));              // (R - c Z_h) A~_b^{-1}
        CUBE_CK(solve(2 + 2 * l, W2, W1, -S.q[l], Z, ma));  // (A~_a - q)^{-1} ( . - q Z_h)
    }
    return FPS_OK;
}

// Y = (T_01 + T_02 + s)^{-1} R with s = -o.q, the middle level in the paper's
// form.  Uses work_[2..4].
int CubeNested::hsolve(const Outer &o, const double *R, double *Y, std::string &err)
{
    const double s = -o.q;
    double *Wh = work_[2], *T1 = work_[3], *T2 = work_[4];
    for (size_t m = 0; m < o.mid.size(); ++m) {
        const double a = o.mid[m].a;
        const double *U = R;  // R - (T_01 + s/2 - a) Y, with Y = 0 at m = 0
        if (m > 0) {
            CUBE_CK(band(Y, nullptr, T1, 0, 1.0, 0.0, 1.0, 0.0));
            CUBE_CK(band(T1, R, T2, 1, 1.0, 0.0, -1.0, 1.0));
            CUBE_CK(axpby(T2, Y, T1, 1.0, -(s / 2 - a)));
            U = T1;
        }
        int st = stein(0, 2, o.mid[m].stein, U, Wh, err);
        if (st != FPS_OK) return st;
        // T1 = R - (T_02 + s/2 - a) Wh
        CUBE_CK(band(Wh, nullptr, T1, 0, 1.0, 0.0, 1.0, 0.0));
        CUBE_CK(band(T1, R, T2, 2, 1.0, 0.0, -1.0, 1.0));
        CUBE_CK(axpby(T2, Wh, T1, 1.0, -(s / 2 - a)));
        st = stein(0, 1, o.mid[m].stein, T1, Y, err);
        if (st != FPS_OK) return st;
    }
    return FPS_OK;
}

int CubeNested::run(const double *G, double *Y, cudaStream_t st, std::string &err)
{
    st_ = st;
    launches = 0;
    double *Yh = work_[5], *T1 = work_[6], *T2 = work_[7];
    for (int j = 0; j < J_outer; ++j) {
        const Outer &o = outer_[j];
        const double *U = G;  // G - (H - p) Y, with Y = 0 at j = 0
        if (j > 0) {
            CUBE_CK(band(Y, nullptr, T2, 0, 1.0, 0.0, 1.0, 0.0));      // A~_0 Y
            CUBE_CK(band(T2, G, T1, 1, 1.0, 0.0, -1.0, 1.0));          // G - T_01 Y
            CUBE_CK(band(T2, T1, T1, 2, 1.0, 0.0, -1.0, 1.0));         // ... - T_02 Y (element-wise in place)
            CUBE_CK(axpby(T1, Y, T1, 1.0, o.p));
            U = T1;
        }
        int s = stein(1, 2, o.stein_v, U, Yh, err);
        if (s != FPS_OK) return s;
        // T1 = G - (V + q) Y_h = G - T_12 Y_h - q Y_h
        CUBE_CK(band(Yh, nullptr, T2, 1, 1.0, 0.0, 1.0, 0.0));
        CUBE_CK(band(T2, G, T1, 2, 1.0, 0.0, -1.0, 1.0));
        CUBE_CK(axpby(T1, Yh, T1, 1.0, -o.q));
        s = hsolve(o, T1, Y, err);
        if (s != FPS_OK) return s;
    }
    return FPS_OK;
}

// ===========================================================================
// CubeRounds
// ===========================================================================

int CubeRounds::create(int64_t n, double tol, double tol_mid, double tol_in, std::string &err)
{
    schedule(n, tol, tol_mid, tol_in, true, true);
    unit_ = unit_half(n);
    if (!unit_) {
        err = "the cube supports n <= 320";
        return FPS_ERR_UNSUPPORTED;
    }
    std::vector<double> d, e;
    square_bands(n, d, e);
    const size_t N = (size_t)n * n * n;
    CUBE_CK(copy((void **)&bd_, d.data(), sizeof(double) * n));
    CUBE_CK(copy((void **)&be_, e.data(), sizeof(double) * n));
    for (float *&w : work_) CUBE_CK(alloc((void **)&w, sizeof(float) * N));
    CUBE_CK(unit_setup(unit_));
    // tables of every entry of the schedule
    int64_t total = 0;
    std::vector<UnitEntry> entries;
    std::vector<double2> pq;
    for (Stein &s : steins_) {
        s.off = total;
        entries.push_back(UnitEntry{s.c, total, (int)pq.size(), s.J});
        for (int l = 0; l < s.J; ++l) pq.push_back(make_double2(s.p[l], s.q[l]));
        total += (int64_t)s.J * 4 * unit_table(unit_);
    }
    CUBE_CK(alloc((void **)&tab_, sizeof(float) * (size_t)total));
    CUBE_CK(alloc((void **)&bands_, sizeof(float) * 2 * unit_bands(unit_)));
    CUBE_CK(copy((void **)&entries_, entries.data(), sizeof(UnitEntry) * entries.size()));
    CUBE_CK(copy((void **)&pq_, pq.data(), sizeof(double2) * pq.size()));
    CUBE_CK(launch_unit_bands(bd_, be_, (int)n, unit_, bands_, nullptr));
    CUBE_CK(launch_unit_tables(entries_, (int)entries.size(), (int)pq.size(), pq_, bd_, be_, (int)n, unit_, tab_,
                               nullptr));
    CUBE_CK(cudaStreamSynchronize(nullptr));
    return FPS_OK;
}

// One launch of the inner level: every job's out = kR R + kZ (T_ab + c)^{-1} R + kacc out
// (R = r1 R1 + r2 R2), the jobs sharing the schedule entry.
int CubeRounds::stein(int ma, int mb, int entry, const UnitJob *jobs, int njobs, std::string &err)
{
    const Stein &S = steins_[entry];
    // mode 0 fastest: both slice kinds of the middle level contain it, so their elements are
    // read and written in runs
    const int64_t st[3] = {1, n_ * n_, n_};
    UnitArgs a;
    a.tab = tab_ + S.off;
    a.bands = bands_;
    a.J = S.J;
    a.n = (int)n_;
    a.njobs = njobs;
    a.sa = st[ma];
    a.sb = st[mb];
    a.sc = st[3 - ma - mb];
    for (int q = 0; q < njobs; ++q) a.job[q] = jobs[q];
    CUBE_CK(launch_stein_units(a, unit_, st_));
    ++launches;
    return FPS_OK;
}

// The middle level with its residual carried: for A' W + B' W = R (A' = T_01 + s/2,
// B' = T_02 + s/2) and shifts +-a,
//   rho+ = [I - 2a (A' + a)^{-1}] [I - 2a (B' + a)^{-1}] rho,
//   W+   = W + (A' + a)^{-1} 2a (B' + a)^{-1} rho,
// with v = (B' + a)^{-1} rho in one launch and (A' + a)^{-1} of rho - 2a v (giving rho+)
// and of 2a v (added to W) in a second.  Uses work_[0..1].
int CubeRounds::hsolve_res(const Outer &o, const float *R, float *W, std::string &err)
{
    float *rho = work_[0], *v = work_[1];
    const size_t J = o.mid.size();
    for (size_t m = 0; m < J; ++m) {
        const float a2 = (float)(2.0 * o.mid[m].a);
        const int entry = o.mid[m].stein;
        const float *r = (m == 0) ? R : rho;
        const UnitJob first{r, nullptr, v, 1.0f, 0.0f, 0.0f, 1.0f, 0.0f};
        int st = stein(0, 2, entry, &first, 1, err);
        if (st != FPS_OK) return st;
        const UnitJob jobs[2] = {{v, nullptr, W, a2, 0.0f, 0.0f, 1.0f, m > 0 ? 1.0f : 0.0f},
                                 {r, v, rho, 1.0f, -a2, 1.0f, -a2, 0.0f}};
        st = stein(0, 1, entry, jobs, m + 1 < J ? 2 : 1, err);
        if (st != FPS_OK) return st;
    }
    return FPS_OK;
}

// The outer level with the residual rho = G - (H + V) Y carried instead of Y's
// right-hand sides.  The two half-steps of (5.3)-(5.4) are Y_h = Y + (V + p)^{-1} rho
// and Y+ = Y_h + (H - q)^{-1} rho_h, so that, the operators commuting,
//   rho+ = [I + (q - p)(V + p)^{-1}] [I + (q - p)(H - q)^{-1}] rho,
//   Y+   = Y + (V + p)^{-1} (p - q) (H - q)^{-1} rho:
// only residuals are solved with and no product with H or V of a growing iterate
// is formed, which keeps FP32 rounding relative to the residual (the paper's form
// loses it to cancellation at small shifts).  Uses work_[2..3].
int CubeRounds::run(const float *G, float *Y, cudaStream_t st, std::string &err)
{
    st_ = st;
    launches = 0;
    float *rho = work_[2], *w = work_[3];
    for (int j = 0; j < J_outer; ++j) {
        const Outer &o = outer_[j];
        const float *r = (j == 0) ? G : rho;
        int s = hsolve_res(o, r, w, err);  // w = (H - q)^{-1} rho
        if (s != FPS_OK) return s;
        // Y += (V + p)^{-1} (p - q) w and, with c = rho + (q - p) w, rho+ = c + (q - p) (V + p)^{-1} c.
        // The scalar p - q enters with the right-hand side: w ~ rho / eps^2 and
        // (V + p)^{-1} w ~ rho / eps^4 would leave the FP32 range for n >~ 100
        const float qp = (float)(o.q - o.p);
        const UnitJob jobs[2] = {{w, nullptr, Y, -qp, 0.0f, 0.0f, 1.0f, j > 0 ? 1.0f : 0.0f},
                                 {r, w, rho, 1.0f, qp, 1.0f, qp, 0.0f}};
        s = stein(1, 2, o.stein_v, jobs, j + 1 < J_outer ? 2 : 1, err);
        if (s != FPS_OK) return s;
    }
    return FPS_OK;
}

// ===========================================================================
// CubeEngine
// ===========================================================================

// Outer tolerance t of the FP32 rounds.  A round reduces max|R| by about t/2
// (measured 0.52 t at n = 256 with the middle and inner levels at 1e-6 and 1e-7), so
// reaching `tol` takes R(t) = ceil(log(tol) / log(0.55 t)) rounds of J_outer(t) outer
// iterations each; the candidate with the least R(t) J_outer(t) wins.  A round that
// falls short only adds a round: the stopping test is the measured residual.
double refinement_outer_tol(int64_t n, double tol)
{
    double lo = square_eps(n), hi = 1.0;
    square_tight_interval(n, lo, hi);
    const double e2 = lo * lo, h2 = hi * hi;
    double best = CubeEngine::kRefTolOuter[0], best_cost = 1e300;
    for (double t : CubeEngine::kRefTolOuter) {
        const int R = std::max(1, (int)std::ceil(std::log(tol) / std::log(0.55 * t) - 1e-9));
        const double cost = (double)R * adi_iterations(-h2, -e2, 2 * e2, 2 * h2, t);
        if (cost < best_cost) {
            best_cost = cost;
            best = t;
        }
    }
    return best;
}

int CubeEngine::create(int64_t n, double tol, int precision, std::string &err)
{
    n_ = n;
    tol_ = tol;
    precision_ = precision;
    if (const char *mr = std::getenv("FPS_MAX_REFINE_ROUNDS")) {  // cap on refinement rounds (>= 1)
        const int v = std::atoi(mr);
        if (v >= 1) max_rounds = v;
    }
    std::vector<double> d, e, s;
    square_bands(n, d, e);
    inv_sqrt_E(n, s);
    const size_t N = (size_t)n * n * n;
    auto alloc = [&](void **p, size_t b) -> cudaError_t {
        cudaError_t r = cudaMalloc(p, b ? b : 1);
        if (r == cudaSuccess) {
            allocs_.push_back(*p);
            bytes += (int64_t)b;
        }
        return r;
    };
    CUBE_CK(alloc((void **)&bd_, sizeof(double) * n));
    CUBE_CK(alloc((void **)&be_, sizeof(double) * n));
    CUBE_CK(alloc((void **)&bs_, sizeof(double) * n));
    CUBE_CK(alloc((void **)&G_, sizeof(double) * N));
    CUBE_CK(alloc((void **)&Y_, sizeof(double) * N));
    CUBE_CK(cudaMemcpy(bd_, d.data(), sizeof(double) * n, cudaMemcpyHostToDevice));
    CUBE_CK(cudaMemcpy(be_, e.data(), sizeof(double) * n, cudaMemcpyHostToDevice));
    CUBE_CK(cudaMemcpy(bs_, s.data(), sizeof(double) * n, cudaMemcpyHostToDevice));
    int st;
    if (precision == FPS_FP64) {
        n64_ = new CubeNested();
        st = n64_->create(n, tol, 1e-15, err);
        if (st != FPS_OK) return st;
        J_outer = n64_->J_outer;
        bytes += n64_->bytes;
    } else {
        CUBE_CK(alloc((void **)&R_, sizeof(double) * N));
        CUBE_CK(alloc((void **)&rho_, sizeof(float) * N));
        CUBE_CK(alloc((void **)&delta_, sizeof(float) * N));
        CUBE_CK(alloc((void **)&d_max_, sizeof(unsigned long long)));
        CUBE_CK(cudaMallocHost((void **)&h_max_, sizeof(unsigned long long)));
        n32_ = new CubeRounds();
        ref_tol_outer = refinement_outer_tol(n, tol);
        st = n32_->create(n, ref_tol_outer, kRefTolMid, kRefTolIn, err);
        if (st != FPS_OK) return st;
        J_outer = J_outer_inner = n32_->J_outer;
        bytes += n32_->bytes;
    }
    return FPS_OK;
}

void CubeEngine::release()
{
    if (n64_) {
        n64_->release();
        delete n64_;
        n64_ = nullptr;
    }
    if (n32_) {
        n32_->release();
        delete n32_;
        n32_ = nullptr;
    }
    for (void *p : allocs_) cudaFree(p);
    allocs_.clear();
    if (h_max_) cudaFreeHost(h_max_);
    h_max_ = nullptr;
}

int CubeEngine::solve_cube(const double *F, double *X, cudaStream_t st, std::string &err)
{
    inner_iters = 0;
    launches_last = 0;
    rounds_last = 0;
    resid_last = 0.0;
    const int64_t N = n_ * n_ * n_;
    cube_scale_kernel<<<grid_for(N), 256, 0, st>>>(F, G_, bs_, (int)n_, -1.0);
    ++launches_last;
    CUBE_CK(cudaGetLastError());
    if (precision_ == FPS_FP64) {
        const int s = n64_->run(G_, Y_, st, err);
        launches_last += n64_->launches;
        if (s != FPS_OK) return s;
        inner_iters = n64_->inner_per_run;
    } else {
        double gmax = 0.0;
        int status = FPS_ERR_NOT_CONVERGED;
        for (int r = 0; r <= max_rounds; ++r) {
            TraceRange tr("fps cube refinement round");
            CUBE_CK(cudaMemsetAsync(d_max_, 0, sizeof(unsigned long long), st));
            cube_residual_kernel<<<grid_for(N), 256, 0, st>>>(G_, Y_, bd_, be_, (int)n_, R_, r == 0, d_max_);
            ++launches_last;
            CUBE_CK(cudaGetLastError());
            CUBE_CK(cudaMemcpyAsync(h_max_, d_max_, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
            CUBE_CK(cudaStreamSynchronize(st));
            const unsigned long long bits = *h_max_;
            double rmax;
            std::memcpy(&rmax, &bits, sizeof(double));
            if (!std::isfinite(rmax)) {
                err = "non-finite right-hand side or residual";
                return FPS_ERR_NONFINITE;
            }
            if (r == 0) {
                gmax = rmax;
                if (gmax == 0.0) {
                    CUBE_CK(cudaMemsetAsync(Y_, 0, sizeof(double) * N, st));
                    status = FPS_OK;
                    break;
                }
            }
            resid_last = rmax / gmax;
            if (r > 0 && resid_last <= tol_) {
                status = FPS_OK;
                break;
            }
            if (r == max_rounds) break;
            cube_to32_kernel<<<tiles_for((int)n_), 256, 0, st>>>(R_, rho_, (int)n_, d_max_);
            ++launches_last;
            CUBE_CK(cudaGetLastError());
            const int s = n32_->run(rho_, delta_, st, err);
            launches_last += n32_->launches;
            if (s != FPS_OK) return s;
            cube_update_kernel<<<tiles_for((int)n_), 256, 0, st>>>(Y_, delta_, (int)n_, d_max_, r == 0);
            ++launches_last;
            CUBE_CK(cudaGetLastError());
            inner_iters += n32_->inner_per_run;
            rounds_last = r + 1;
        }
        if (status != FPS_OK) {
            cube_scale_kernel<<<grid_for(N), 256, 0, st>>>(Y_, X, bs_, (int)n_, 1.0);
            ++launches_last;
            err = "refinement did not reach the tolerance";
            return status;
        }
    }
    cube_scale_kernel<<<grid_for(N), 256, 0, st>>>(Y_, X, bs_, (int)n_, 1.0);
    ++launches_last;
    CUBE_CK(cudaGetLastError());
    return FPS_OK;
}

}  // namespace fps
