// All ADI iterations of a small square in one launch (see resident.cuh).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "bulk.cuh"
#include "resident.cuh"
#include "sweep.cuh"

namespace cg = cooperative_groups;

namespace fps {

namespace {

constexpr int kG = kResSeg;

template <typename T>
__device__ __forceinline__ typename Vec2<T>::type pair_of(T x, T y);
template <>
__device__ __forceinline__ float2 pair_of<float>(float x, float y)
{
    return make_float2(x, y);
}
template <>
__device__ __forceinline__ double2 pair_of<double>(double x, double y)
{
    return make_double2(x, y);
}

// Shared memory of a CTA (elements of T, in this order; every part starts on 16 bytes).
template <typename T, int S>
struct ResGeo {
    static constexpr int A = 16 / (int)sizeof(T);
    __host__ __device__ static constexpr int up(int n) { return (n + A - 1) / A * A; }
    // Lines (rows, then columns) per thread.  FP32 is bound by shared memory, half of it table
    // entries that serve every line: with two lines a thread reads them once for both.  FP64
    // wants all its warps.
    static constexpr int kR = sizeof(T) == 4 && S >= 20 ? 2 : 1;
    static constexpr int kThreads = (kG * S / kR + 31) / 32 * 32;
    // a segment takes an odd number of elements and a row 16 of them, so that the 32 lanes
    // of the row solve (16 segments of two rows) hit different banks
    static constexpr int SS = S | 1, pitch = kG * SS;
    static constexpr int cpitch = kG + 1;
    static constexpr int off_x = 0;
    static constexpr int off_cs = off_x + up(S * pitch);       // column summaries of the owned columns
    static constexpr int off_bd = off_cs + up(2 * S * cpitch);  // zin, yout of this CTA's column segments
    static constexpr int off_tab = off_bd + up(2 * kG * S);
    // tables of one iteration: row record, column scan coefficients, column slice [5][SP]
    static constexpr int SP = up(S);
    static constexpr int tab = res_record(S) + kScan + kTabs * SP;
    static constexpr int off_bar = off_tab + 2 * tab;  // two mbarriers
    static constexpr size_t bytes = sizeof(T) * (size_t)off_bar + 16;
};

__device__ __forceinline__ void copy16_async(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
template <typename T>
__device__ __forceinline__ void copy_async(T *dst, const T *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(sizeof(T))
                 : "memory");
}

// A 16-byte word of a table.
__device__ __forceinline__ void read16(float (&o)[4], const float *p)
{
    const float4 f = *reinterpret_cast<const float4 *>(p);
    o[0] = f.x, o[1] = f.y, o[2] = f.z, o[3] = f.w;
}
__device__ __forceinline__ void read16(double (&o)[2], const double *p)
{
    const double2 f = *reinterpret_cast<const double2 *>(p);
    o[0] = f.x, o[1] = f.y;
}

// zin and yout of segment g (lane g of a half-warp) of a line from the summaries that the
// half-warp's lanes hold.
template <typename T>
__device__ __forceinline__ void scan_segments(T wl, T yl, const T *k, int g, T &zin, T &yout)
{
    T W = wl;
#pragma unroll
    for (int t = 0; t < 4; ++t) W = fma(k[t * kG + g], __shfl_up_sync(0xffffffffu, W, 1 << t, kG), W);
    zin = __shfl_up_sync(0xffffffffu, W, 1, kG);
    if (g == 0) zin = T(0);
    T Y = fma(k[4 * kG + g], zin, yl);
#pragma unroll
    for (int t = 0; t < 4; ++t) Y = fma(k[(5 + t) * kG + g], __shfl_down_sync(0xffffffffu, Y, 1 << t, kG), Y);
    yout = __shfl_down_sync(0xffffffffu, Y, 1, kG);
    if (g == kG - 1) yout = T(0);
}

template <typename T, int S>
__global__ void __launch_bounds__(ResGeo<T, S>::kThreads) resident_kernel(ResArgs<T> a)
{
    using G = ResGeo<T, S>;
    using T2 = typename Vec2<T>::type;
    constexpr int M = kG * S, kR = G::kR;
    // partial sums of a summary: an FP64 instruction of a warp occupies its issue for as long as
    // its latency, so a second chain only costs its addition; two lines are two chains
    constexpr int kAcc = sizeof(T) == 8 || kR == 2 ? 1 : 2;
    auto total = [](const T(&x)[kAcc]) { return kAcc == 1 ? x[0] : x[0] + x[kAcc - 1]; };
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cl = cg::this_cluster();
    const int C = a.C, rank = (int)cl.block_rank(), tid = threadIdx.x;
    const ResItem<T> &it = a.items[blockIdx.x / C];
    if (*a.masked && !a.active[it.prob]) return;  // the whole cluster
    const int n = it.n, J = it.J, i0 = rank * S;
    const int mr = (n - it.rp + 1) / 2, mc = (n - it.cp + 1) / 2;
    T *X = reinterpret_cast<T *>(smem) + G::off_x;
    T2 *cs = reinterpret_cast<T2 *>(reinterpret_cast<T *>(smem) + G::off_cs);
    T2 *bd = reinterpret_cast<T2 *>(reinterpret_cast<T *>(smem) + G::off_bd);
    T *tab = reinterpret_cast<T *>(smem) + G::off_tab;
    uint64_t *bar = reinterpret_cast<uint64_t *>(reinterpret_cast<T *>(smem) + G::off_bar);
    // global position of element (i, k) of the quarter
    auto qpos = [&](int i, int k) {
        return it.xoff + (((int64_t)(i >> 5) * it.lnb + (k >> 5)) << 10) + block_pos<T>(i & 31, k & 31, 32);
    };
    auto npos = [&](int i, int k) { return it.foff + (int64_t)(2 * i + it.rp) * n + (2 * k + it.cp); };
    const int64_t rec = 2 * res_record(S);  // records of the two parities per iteration
    auto load_tables = [&](int j) {
        T *t = tab + (j & 1) * G::tab;
        const T *tR = it.tabR + j * rec, *tC = it.tabC + j * rec;
        for (int q = tid * G::A; q < res_record(S); q += G::kThreads * G::A) copy16_async(t + q, tR + q);
        t += res_record(S);
        for (int q = tid * G::A; q < kScan; q += G::kThreads * G::A) copy16_async(t + q, tC + res_scan_col(S) + q);
        t += kScan;
        if (tid < S)
#pragma unroll
            for (int q = 0; q < kTabs; ++q) copy_async(t + q * G::SP + tid, tC + q * M + i0 + tid);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    load_tables(0);
    if (tid == 0) {
        bulk::mbar_init(bar, 1);
        bulk::mbar_init(bar + 1, 1);
        bulk::fence_mbar_init();
    }
    for (int q = tid; q < S * M; q += G::kThreads) {  // the slab: rows i0 .. i0 + S
        const int r = q / M, k = q - r * M, i = i0 + r;
        T v = 0;
        if (i < mr && k < mc)
            v = a.F ? (T)(a.F[npos(i, k)] * it.s[2 * i + it.rp] * it.s[2 * k + it.cp]) : a.X[qpos(i, k)];
        X[r * G::pitch + (k / S) * G::SS + k % S] = v;
    }
    for (int q = tid; q < S * G::cpitch; q += G::kThreads) cs[q] = pair_of<T>(T(0), T(0));
    T D[kR][S];
#pragma unroll
    for (int i = 0; i < S; ++i)
#pragma unroll
        for (int h = 0; h < kR; ++h) D[h][i] = 0;
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    cl.sync();  // the slab is complete and every CTA of the cluster runs

    // row solve: rows r0 and r0 + S / 2, segment g; column solve: columns col and col + M / 2.
    // Threads beyond the last row or column (16 S is no multiple of 32, or fewer segments in
    // use) compute on zeros that nobody reads.
    const int g = tid & (kG - 1), r0 = min(tid >> 4, S / kR - 1);
    const bool row_on = (tid >> 4) < S / kR;
    T *xr = X + r0 * G::pitch + g * G::SS;
    constexpr int rstep = S / kR, cstep = M / kR;
    // Exchange: each of the C S pairs of a step is an asynchronous store that the receiver's
    // barrier counts.  A CTA sends a step's pairs only after it has received all of the step
    // before, which its peers send after reading what the new pairs overwrite.
    const unsigned bytes = (unsigned)(C * S * sizeof(T2));
    const int pr = min(g, C - 1);  // peer that wants its segment of the owned columns
    const unsigned to_bd = bulk::peer_smem(bd + i0 + r0, pr), bar_bd = bulk::peer_smem(bar + 1, pr);
    int col[kR];
    bool col_on[kR];
    T *xc[kR];
    unsigned to_cs[kR], bar_cs[kR];  // at the peer that owns the column
#pragma unroll
    for (int h = 0; h < kR; ++h) {
        col[h] = min(tid + h * cstep, M - 1);
        const int gc = col[h] / S, cc = col[h] % S;
        col_on[h] = tid < cstep && gc < C;  // a column has one thread: its summaries are counted once
        xc[h] = X + gc * G::SS + cc;
        to_cs[h] = bulk::peer_smem(cs + cc * G::cpitch + rank, min(gc, C - 1));
        bar_cs[h] = bulk::peer_smem(bar, min(gc, C - 1));
    }
    bool ok = true;  // false: a wait gave up; the thread runs on without waiting, sending or arming
    const int give_up = rank == 0 ? a.give_up : -1;
    auto wait = [&](uint64_t *b, int j) {
        if (ok && (j == give_up || !bulk::mbar_wait_cluster(b, j & 1))) {
            ok = false;
            *(volatile int *)a.err = 1;
        }
    };
    for (int j = 0; j < J; ++j) {
        const T *tr = tab + (j & 1) * G::tab;
        const T2 *sums = reinterpret_cast<const T2 *>(tr) + g, *back = reinterpret_cast<const T2 *>(tr + 2 * M) + g;
        const T2 *fwd = reinterpret_cast<const T2 *>(tr + 4 * M) + g;
        const T *kr = tr + res_scan_row(S), *kc = tr + res_record(S), *tc = kc + kScan;
        // while its waits succeed thread 0 knows that both phases before are complete; a phase
        // that is not has had its one arrival
        if (tid == 0 && ok) {
            bulk::mbar_arrive_expect_tx(bar, bytes);
            bulk::mbar_arrive_expect_tx(bar + 1, bytes);
        }
        if (j + 1 < J) load_tables(j + 1);
        T v[kR][S], w[kR][S];
        {
            T wl[kR][kAcc] = {}, yl[kR][kAcc] = {};
#pragma unroll
            for (int i = 0; i < S; ++i) {
                const T2 p = sums[i * kG];
#pragma unroll
                for (int h = 0; h < kR; ++h) {
                    v[h][i] = xr[h * rstep * G::pitch + i];
                    wl[h][i % kAcc] = fma(p.x, v[h][i], wl[h][i % kAcc]);
                    yl[h][i % kAcc] = fma(p.y, v[h][i], yl[h][i % kAcc]);
                }
            }
            T z[kR], y[kR];
#pragma unroll
            for (int h = 0; h < kR; ++h) scan_segments<T>(total(wl[h]), total(yl[h]), kr, g, z[h], y[h]);
#pragma unroll
            for (int i = 0; i < S; i += 2) {
                const T2 l = fwd[i / 2 * kG];
#pragma unroll
                for (int h = 0; h < kR; ++h) {
                    z[h] = fma(-l.x, z[h], v[h][i]);
                    w[h][i] = z[h];
                    if (i + 1 < S) {
                        z[h] = fma(-l.y, z[h], v[h][i + 1]);
                        w[h][i + 1] = z[h];
                    }
                }
            }
            const bool first = j == 0;
#pragma unroll
            for (int i = S - 1; i >= 0; --i) {
                const T2 p = back[i * kG];
#pragma unroll
                for (int h = 0; h < kR; ++h) {
                    y[h] = fma(-p.x, y[h], w[h][i]);
                    v[h][i] = fma(p.y, y[h], first ? T(0) : v[h][i]);
                }
            }
            if (row_on)
#pragma unroll
                for (int i = 0; i < S; ++i)
#pragma unroll
                    for (int h = 0; h < kR; ++h) xr[h * rstep * G::pitch + i] = v[h][i];
        }
        __syncthreads();
        {
            T wl[kR][kAcc] = {}, yl[kR][kAcc] = {};
#pragma unroll
            for (int c = 0; c < S; c += G::A) {
                T psi[G::A], chi[G::A];
                read16(psi, tc + 3 * G::SP + c);
                read16(chi, tc + 4 * G::SP + c);
#pragma unroll
                for (int i = c; i < min(c + G::A, S); ++i)
#pragma unroll
                    for (int h = 0; h < kR; ++h) {
                        v[h][i] = xc[h][i * G::pitch];
                        wl[h][i % kAcc] = fma(psi[i - c], v[h][i], wl[h][i % kAcc]);
                        yl[h][i % kAcc] = fma(chi[i - c], v[h][i], yl[h][i % kAcc]);
                    }
            }
#pragma unroll
            for (int h = 0; h < kR; ++h)
                if (col_on[h] && ok) bulk::send_pair(to_cs[h], bar_cs[h], pair_of<T>(total(wl[h]), total(yl[h])));
        }
        wait(bar, j);
#pragma unroll
        for (int h = 0; h < kR; ++h) {  // the columns this CTA owns, rank * S + r0 (+ S / 2), all their segments
            const T2 s = cs[(r0 + h * rstep) * G::cpitch + g];
            T z, y;
            scan_segments<T>(s.x, s.y, kc, g, z, y);
            if (row_on && g < C && ok)
                bulk::send_pair(to_bd + h * rstep * (unsigned)sizeof(T2), bar_bd, pair_of<T>(z, y));
        }
        wait(bar + 1, j);
        if (col_on[0]) {
            T z[kR], y[kR];
#pragma unroll
            for (int h = 0; h < kR; ++h) {
                const T2 b = bd[col[h]];
                z[h] = b.x;
                y[h] = b.y;
            }
#pragma unroll
            for (int c = 0; c < S; c += G::A) {
                T l[G::A];
                read16(l, tc + c);
#pragma unroll
                for (int i = c; i < min(c + G::A, S); ++i)
#pragma unroll
                    for (int h = 0; h < kR; ++h) {
                        z[h] = fma(-l[i - c], z[h], v[h][i]);
                        w[h][i] = z[h];
                    }
            }
#pragma unroll
            for (int c = G::SP - G::A; c >= 0; c -= G::A) {
                T mm[G::A], gg[G::A];
                read16(mm, tc + G::SP + c);
                read16(gg, tc + 2 * G::SP + c);
#pragma unroll
                for (int i = min(c + G::A, S) - 1; i >= c; --i)
#pragma unroll
                    for (int h = 0; h < kR; ++h) {
                        y[h] = fma(-mm[i - c], y[h], w[h][i]);
                        if (col_on[h]) xc[h][i * G::pitch] = fma(gg[i - c], y[h], v[h][i]);
                        D[h][i] = fma(gg[i - c], y[h], D[h][i]);
                    }
            }
        }
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
    }
    // no CTA leaves while a peer may still have stores under way to it: a CTA whose waits
    // succeeded has received all of its own
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");
#pragma unroll
    for (int h = 0; h < kR; ++h) {
        if (!col_on[h] || col[h] >= mc) continue;
#pragma unroll
        for (int r = 0; r < S; ++r) {
            const int i = i0 + r, k = col[h];
            const T d = ok ? D[h][r] : (T)NAN;
            if (i < mr) {
                if (a.F) a.out[npos(i, k)] = it.out_scale * (double)d * it.s[2 * i + it.rp] * it.s[2 * k + it.cp];
                else a.D[qpos(i, k)] = d;
            }
        }
    }
    asm volatile("barrier.cluster.wait.aligned;\n" ::: "memory");
    // every store is issued by now, but one whose wait gave up has not seen the last ones arrive
    if (!ok)
        for (int t = 0; t < 1000; ++t) __nanosleep(1000);
}

// One thread per (job, parity), FP64 arithmetic; the recurrences of fac_tables_kernel.
template <typename T>
__global__ void resident_tables_kernel(const ResTabJob<T> *__restrict__ jobs, int njobs)
{
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= 2 * njobs) return;
    const ResTabJob<T> &jb = jobs[tid >> 1];
    const int p = tid & 1, S = jb.S, M = kG * S, m = (jb.n - p + 1) / 2;
    T *row = jb.row ? jb.row + (int64_t)p * res_record(S) : nullptr;
    T *col = jb.col ? jb.col + (int64_t)p * res_record(S) : nullptr;
    T *row_scan = row ? row + res_scan_row(S) : nullptr, *col_scan = col ? col + res_scan_col(S) : nullptr;
    const double *d = jb.d + p, *e = jb.e + p;  // position i of this parity: index 2 i
    double ip = 0.0, ip_next = m > 0 ? 1.0 / (d[0] - jb.q) : 0.0, l_next = 0.0;
    double lv[32], mv[32], v[32], phi[kG], bv[kG], ps[kG];
    for (int g = 0; g < kG; ++g) {
        for (int u = 0; u < S; ++u) {
            const int i = g * S + u;
            double l = 0.0, mm = 0.0;
            ip = 0.0;
            if (i < m) {
                ip = ip_next;
                l = l_next;
                if (i + 1 < m) {
                    const double ei = e[2 * i];
                    l_next = ei * ip;
                    ip_next = 1.0 / (d[2 * (i + 1)] - jb.q - ei * l_next);
                    mm = ei * ip_next;
                }
            }
            lv[u] = l;
            mv[u] = mm;
            v[u] = u == 0 ? 1.0 : v[u - 1] * -mv[u - 1];
            if (row) {
                row[2 * M + 2 * (u * kG + g)] = (T)mm;
                row[2 * M + 2 * (u * kG + g) + 1] = (T)(jb.sc_row * ip);
                row[4 * M + (u / 2 * kG + g) * 2 + u % 2] = (T)l;
            }
            if (col) {
                col[i] = (T)l;
                col[M + i] = (T)mm;
                col[2 * M + i] = (T)(jb.sc_col * ip);
            }
        }
        double psi = 1.0, chi = 0.0;
        for (int u = S - 1; u >= 0; --u) {
            const int i = g * S + u;
            if (u + 1 < S) psi *= -lv[u + 1];
            chi = u + 1 < S ? v[u] - lv[u + 1] * chi : v[u];
            const bool live = i < m;
            if (row) {
                row[2 * (u * kG + g)] = live ? (T)psi : T(0);
                row[2 * (u * kG + g) + 1] = live ? (T)chi : T(0);
            }
            if (col) {
                col[3 * M + i] = live ? (T)psi : T(0);
                col[4 * M + i] = live ? (T)chi : T(0);
            }
        }
        phi[g] = -lv[0] * psi;
        bv[g] = -lv[0] * chi;
        ps[g] = v[S - 1] * -mv[S - 1];
    }
    for (int s = 0; s < kG; ++s) {
        for (int t = 0; t < 4; ++t) {
            double kf = 0.0, kb = 0.0;
            if (s >= (1 << t)) {
                kf = 1.0;
                for (int u = s - (1 << t) + 1; u <= s; ++u) kf *= phi[u];
            }
            if (s + (1 << t) < kG) {
                kb = 1.0;
                for (int u = s; u < s + (1 << t); ++u) kb *= ps[u];
            }
            for (T *o : {row_scan, col_scan})
                if (o) {
                    o[t * kG + s] = (T)kf;
                    o[(5 + t) * kG + s] = (T)kb;
                }
        }
        for (T *o : {row_scan, col_scan})
            if (o) o[4 * kG + s] = (T)bv[s];
    }
}

template <typename T, int S>
cudaLaunchConfig_t config_of(int64_t nitems, int C, cudaLaunchAttribute *at, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nitems * C));
    cfg.blockDim = dim3((unsigned)ResGeo<T, S>::kThreads);
    cfg.dynamicSmemBytes = ResGeo<T, S>::bytes;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

template <typename T, int S>
cudaError_t setup_S(int C, int *side_by_side)
{
    *side_by_side = 0;
    cudaError_t e = cudaFuncSetAttribute(resident_kernel<T, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)ResGeo<T, S>::bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(resident_kernel<T, S>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = config_of<T, S>(1, C, at, nullptr);
    if (cudaOccupancyMaxActiveClusters(side_by_side, resident_kernel<T, S>, &cfg) != cudaSuccess) {
        cudaGetLastError();  // no such cluster on this device: the passes stream the problem
        *side_by_side = 0;
    }
    return cudaSuccess;
}

template <typename T, int S>
cudaError_t launch_S(const ResArgs<T> &a, cudaStream_t st)
{
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = config_of<T, S>(a.nitems, a.C, at, st);
    return cudaLaunchKernelEx(&cfg, resident_kernel<T, S>, a);
}

}  // namespace

// Compiled segment lengths; FP64 stops at 24 (three arrays of S doubles per thread are
// registers: 168 a thread there, spills beyond).
#define RES_SIZES_64(X) X(1) X(2) X(3) X(4) X(5) X(6) X(8) X(10) X(12) X(14) X(16) X(20) X(24)
#define RES_SIZES_32(X) RES_SIZES_64(X) X(28) X(32)

int resident_segment(bool fp64, int m)
{
#define TRY(s) if (m <= kG * s && !(fp64 && s > 24)) return s;
    RES_SIZES_32(TRY)
#undef TRY
    return 0;
}

#define CASE_SETUP(s) case s: return setup_S<T, s>(C, side_by_side);
#define CASE_LAUNCH(s) case s: return launch_S<T, s>(a, st);

template <typename T>
cudaError_t resident_setup(int S, int C, int *side_by_side)
{
    if constexpr (sizeof(T) == 4) {
        switch (S) { RES_SIZES_32(CASE_SETUP) }
    } else {
        switch (S) { RES_SIZES_64(CASE_SETUP) }
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_resident(const ResArgs<T> &a, cudaStream_t st)
{
    if constexpr (sizeof(T) == 4) {
        switch (a.S) { RES_SIZES_32(CASE_LAUNCH) }
    } else {
        switch (a.S) { RES_SIZES_64(CASE_LAUNCH) }
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_resident_tables(const ResTabJob<T> *jobs, int njobs, cudaStream_t st)
{
    resident_tables_kernel<T><<<(unsigned)((2 * njobs + 31) / 32), 32, 0, st>>>(jobs, njobs);
    return cudaGetLastError();
}

template cudaError_t resident_setup<float>(int, int, int *);
template cudaError_t resident_setup<double>(int, int, int *);

bool resident_pays(bool fp64, int S, int nrhs, int side_by_side)
{
    return side_by_side >= 1 && (!fp64 || S <= 16 || 4 * nrhs <= side_by_side);
}
template cudaError_t launch_resident<float>(const ResArgs<float> &, cudaStream_t);
template cudaError_t launch_resident<double>(const ResArgs<double> &, cudaStream_t);
template cudaError_t launch_resident_tables<float>(const ResTabJob<float> *, int, cudaStream_t);
template cudaError_t launch_resident_tables<double>(const ResTabJob<double> *, int, cudaStream_t);

}  // namespace fps
