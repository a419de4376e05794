// Inner level of the cube, one CTA per parity quarter of a slice (see cube_unit.cuh).
#include <cuda_runtime.h>

#include "cube_unit.cuh"

namespace fps {

namespace {

// Unknown at place t of a line of 2 H: both halves are stored from their outer end.
__host__ __device__ __forceinline__ int unit_place(int t, int H) { return t < H ? t : 3 * H - 1 - t; }

template <int H>
struct UnitGeo {
    static constexpr int N = 2 * H;
    static constexpr int A = 4;  // elements of a 16-byte copy
    static constexpr int kThreads = (N + 15) / 16 * 32;
    static constexpr int stages = 4;  // iterations whose tables are in shared memory or on their way
    // Steps of a sweep whose operands are read together, ahead of the dependent FMAs (a
    // store between them would keep every later read behind it).
    static constexpr int kC = H <= 12 ? H : (H == 20 ? 10 : (H <= 64 ? 8 : 4));
    // what a thread keeps in registers beside its half of a line and of Z: the line's
    // right-hand side (read twice otherwise) and the bands (the same in every iteration)
    static constexpr bool keep_row = H <= 32, keep_bands = H <= 16;
    // 16 lanes on consecutive rows (columns) of one half, 16 of the other: an odd pitch
    // separates the first, a distance of 16 banks between the halves the two groups
    static constexpr int half = H + ((16 - H % 32) + 32) % 32;
    static constexpr int pitch = (half + H) | 1;
    static constexpr int row_gap = ((16 - (H * pitch) % 32) + 32) % 32;
    static constexpr int square = (N * pitch + row_gap + A - 1) / A * A;
    static constexpr int table = unit_table(H), stage = 2 * table, LS = unit_half_pitch(H);
    static constexpr size_t bytes = sizeof(float) * (size_t)(square + stages * stage + unit_bands(H));
    __device__ static __forceinline__ int at(int a, int b)
    {
        return a * pitch + (a < H ? 0 : row_gap) + b + (b < H ? 0 : half - H);
    }
};

// K consecutive elements of a table (8-byte aligned; 16-byte if K is a multiple of 4)
template <int K>
__device__ __forceinline__ void read_run(float (&o)[K], const float *p)
{
    if constexpr (K % 4 == 0) {
#pragma unroll
        for (int i = 0; i < K; i += 4) {
            const float4 f = *reinterpret_cast<const float4 *>(p + i);
            o[i] = f.x, o[i + 1] = f.y, o[i + 2] = f.z, o[i + 3] = f.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < K; i += 2) {
            const float2 f = *reinterpret_cast<const float2 *>(p + i);
            o[i] = f.x, o[i + 1] = f.y;
        }
    }
}

__device__ __forceinline__ void copy16_async(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

template <int H>
__global__ void __launch_bounds__(UnitGeo<H>::kThreads) stein_unit_kernel(UnitArgs A)
{
    using G = UnitGeo<H>;
    constexpr int N = G::N, P = G::pitch, tab = G::table, kStages = G::stages, LS = G::LS, kC = G::kC, nC = H / kC;
    constexpr int kB = 8;  // global loads in flight per thread
    extern __shared__ __align__(16) unsigned char unit_smem[];
    float *U = reinterpret_cast<float *>(unit_smem), *ring = U + G::square, *bd = ring + kStages * G::stage;
    const int tid = threadIdx.x, lane = tid & 31, h = lane >> 4;
    const int raw = (tid >> 5) * 16 + (lane & 15), ln = min(raw, N - 1);  // threads beyond the last line repeat it
    const bool on = raw < N;
    const int n = A.n, J = A.J;
    // slices fastest: neighbouring CTAs read neighbouring elements where the slice index is contiguous
    const int q = blockIdx.x / n, k = blockIdx.x - q * n, rp = q >> 1, cp = q & 1;
    const UnitJob job = A.job[blockIdx.y];
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    auto load_tables = [&](int j) {
        if (j < J) {
            float *dst = ring + (j % kStages) * G::stage;
            const float *src = A.tab + (int64_t)j * 4 * tab;
            for (int x = tid * G::A; x < tab; x += G::kThreads * G::A) {
                copy16_async(dst + x, src + cp * tab + x);
                copy16_async(dst + tab + x, src + (2 + rp) * tab + x);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    for (int x = tid * G::A; x < unit_bands(H); x += G::kThreads * G::A)
        copy16_async(bd + x, A.bands + cp * unit_bands(H) + x);
    for (int j = 0; j < kStages - 1; ++j) load_tables(j);
    // bands and tables are the plan's; everything below may come from the launch before
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    const int mr = (n - rp + 1) / 2, mc = (n - cp + 1) / 2;
    const int64_t base = (int64_t)k * A.sc + rp * A.sa + cp * A.sb;
    const bool a_fast = A.sa < A.sb;  // consecutive threads along the mode with the smaller stride
    // element x of the quarter: its place in U and its offset, negative beyond the last unknown
    auto element = [&](int x, int &u, int64_t &g) {
        const int x0 = x / N, x1 = x - x0 * N, a = a_fast ? x1 : x0, b = a_fast ? x0 : x1;
        const int i = unit_place(a, H), l = unit_place(b, H);
        u = G::at(a, b);
        g = x < N * N && i < mr && l < mc ? base + 2 * i * A.sa + 2 * l * A.sb : -1;
    };
    for (int x0 = tid; x0 < N * N; x0 += kB * G::kThreads) {
        float v[kB];
        int u[kB];
#pragma unroll
        for (int t = 0; t < kB; ++t) {
            int64_t g;
            element(x0 + t * G::kThreads, u[t], g);
            v[t] = 0;
            if (g >= 0) {
                v[t] = job.r1 * job.R1[g];
                if (job.R2) v[t] = fmaf(job.r2, job.R2[g], v[t]);
            }
        }
#pragma unroll
        for (int t = 0; t < kB; ++t)
            if (x0 + t * G::kThreads < N * N) U[u[t]] = v[t];
    }
    float *row = U + G::at(ln, h * H);                         // this thread's half row ...
    const float *across = U + G::at(ln, (1 - h) * H + H - 1);  // ... and the unknown across the middle
    float *col = U + G::at(h * H, ln);
    float zc[H], dg[G::keep_bands ? H : 1], eo[G::keep_bands ? H : 1];
#pragma unroll
    for (int s = 0; s < H; ++s) zc[s] = 0;
    for (int j = 0; j < J; ++j) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kStages - 2) : "memory");
        __syncthreads();
        load_tables(j + kStages - 1);
        const float *lb = ring + (j % kStages) * G::stage + h * LS, *la = lb + tab;
        const float *gb = lb + 2 * LS + h * LS, *ga = gb + tab;  // {m, scale}
        const float *mb = ring + (j % kStages) * G::stage + 6 * LS + 2 * h, *ma = mb + tab;
        const float *be = bd + 2 * h * LS;
        if (G::keep_bands && j == 0)
#pragma unroll
            for (int s = 0; s < (G::keep_bands ? H : 1); ++s) dg[s] = be[2 * s], eo[s] = be[2 * s + 1];
        float v[H], uk[G::keep_row ? H : 1];
        {  // along b: a = u - (p - q') (u A~_b) K^{-1}; the factor -(p - q') is part of the scale
            float z = 0, um = 0, u0 = row[0];
#pragma unroll
            for (int c = 0; c < nC; ++c) {
                float l[kC], up[kC], bb[2 * kC];
                read_run(l, lb + c * kC);
                if constexpr (!G::keep_bands) read_run(bb, be + 2 * c * kC);
                float en = 0;
                if constexpr (!G::keep_bands) en = c + 1 < nC ? be[2 * (c + 1) * kC + 1] : 0.0f;
#pragma unroll
                for (int t = 0; t < kC; ++t) up[t] = c * kC + t + 1 < H ? row[c * kC + t + 1] : *across;
#pragma unroll
                for (int t = 0; t < kC; ++t) {
                    const int s = c * kC + t;
                    float r = u0;
                    if (j > 0) {
                        float d0, e0, e1;
                        if constexpr (G::keep_bands) d0 = dg[s], e0 = eo[s], e1 = s + 1 < H ? eo[s + 1] : 0.0f;
                        else d0 = bb[2 * t], e0 = bb[2 * t + 1], e1 = t + 1 < kC ? bb[2 * t + 3] : en;
                        if (s + 1 == H) e1 = bd[4 * LS];
                        r = fmaf(d0, u0, fmaf(e0, um, e1 * up[t]));
                    }
                    if constexpr (G::keep_row) uk[s] = u0;
                    z = fmaf(-l[t], z, r);
                    v[s] = z;
                    um = u0;
                    u0 = up[t];
                }
            }
            float y = fmaf(mb[1], __shfl_xor_sync(0xffffffffu, z, 16), mb[0] * z);
            if constexpr (!G::keep_row) asm volatile("" ::: "memory");  // u is read again, not kept in registers
#pragma unroll
            for (int c = nC - 1; c >= 0; --c) {
                float mg[2 * kC], u[kC];
                read_run(mg, gb + 2 * c * kC);
#pragma unroll
                for (int t = 0; t < kC; ++t) u[t] = G::keep_row ? uk[G::keep_row ? c * kC + t : 0] : row[c * kC + t];
#pragma unroll
                for (int t = kC - 1; t >= 0; --t) {
                    const int s = c * kC + t;
                    if (s < H - 1) y = fmaf(-mg[2 * t], y, v[s]);
                    const float out = fmaf(mg[2 * t + 1], y, j == 0 ? 0.0f : u[t]);
                    if (on) row[s] = out;
                }
            }
        }
        __syncthreads();
        {  // along a: t = (q - p) (A~_a - q)^{-1} a
            float z = 0;
#pragma unroll
            for (int c = 0; c < nC; ++c) {
                float l[kC];
                read_run(l, la + c * kC);
#pragma unroll
                for (int t = 0; t < kC; ++t) {
                    const int s = c * kC + t;
                    const float a = col[s * P];
                    if constexpr (G::keep_row) uk[s] = a;
                    z = fmaf(-l[t], z, a);
                    v[s] = z;
                }
            }
            float y = fmaf(ma[1], __shfl_xor_sync(0xffffffffu, z, 16), ma[0] * z);
            if constexpr (!G::keep_row) asm volatile("" ::: "memory");
#pragma unroll
            for (int c = nC - 1; c >= 0; --c) {
                float mg[2 * kC], u[kC];
                read_run(mg, ga + 2 * c * kC);
#pragma unroll
                for (int t = 0; t < kC; ++t) u[t] = G::keep_row ? uk[G::keep_row ? c * kC + t : 0] : col[(c * kC + t) * P];
#pragma unroll
                for (int t = kC - 1; t >= 0; --t) {
                    const int s = c * kC + t;
                    if (s < H - 1) y = fmaf(-mg[2 * t], y, v[s]);
                    const float w = fmaf(mg[2 * t + 1], y, u[t]);
                    zc[s] = fmaf(mg[2 * t + 1], y, zc[s]);
                    if (on) col[s * P] = w;
                }
            }
        }
    }
    if (on)
#pragma unroll
        for (int s = 0; s < H; ++s) col[s * P] = zc[s];  // u is not needed any more
    __syncthreads();
    for (int x0 = tid; x0 < N * N; x0 += kB * G::kThreads) {
        float v[kB], acc[kB];
        int u[kB];
        int64_t g[kB];
#pragma unroll
        for (int t = 0; t < kB; ++t) {
            element(x0 + t * G::kThreads, u[t], g[t]);
            v[t] = acc[t] = 0;
            if (g[t] >= 0) {
                if (job.kR != 0.0f) {
                    v[t] = job.r1 * job.R1[g[t]];
                    if (job.R2) v[t] = fmaf(job.r2, job.R2[g[t]], v[t]);
                }
                if (job.kacc != 0.0f) acc[t] = job.out[g[t]];
            }
        }
#pragma unroll
        for (int t = 0; t < kB; ++t)
            if (g[t] >= 0) {
                float o = job.kZ * U[u[t]];
                if (job.kR != 0.0f) o = fmaf(job.kR, v[t], o);
                if (job.kacc != 0.0f) o = fmaf(job.kacc, acc[t], o);
                job.out[g[t]] = o;
            }
    }
}

// A~ of one parity in the order of a line of 2 H unknowns, zero beyond its m unknowns.
struct LineBands {
    const double *d, *e;
    int n, H, par;
    __device__ int at(int h, int s) const { return h ? 2 * H - 1 - s : s; }
    __device__ double diag(int i) const { return 2 * i + par < n ? d[2 * i + par] : 0.0; }
    __device__ double off(int i) const { return i >= 0 && 2 * (i + 1) + par < n ? e[2 * i + par] : 0.0; }  // i to i + 1
    __device__ double outer(int h, int s) const { return s ? off(h ? at(h, s) : at(h, s) - 1) : 0.0; }
};

// One thread per (shift, direction, parity, half), FP64 arithmetic; the two halves of a
// line are neighbouring lanes.
__global__ void __launch_bounds__(64) unit_tables_kernel(const UnitEntry *__restrict__ entries, int count,
                                                         int shifts, const double2 *__restrict__ pq,
                                                         const double *__restrict__ d, const double *__restrict__ e,
                                                         int n, int H, float *__restrict__ tabs)
{
    const int raw = blockIdx.x * blockDim.x + threadIdx.x;
    const int id = unit_table_thread(raw, shifts), h = id & 1, LS = unit_half_pitch(H);
    const bool live = raw < 8 * shifts;
    const int x = (id >> 1) & 3, sh = id >> 3, tab = unit_table(H);
    int lo = 0, hi = count - 1;  // the entry of shift sh
    while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (entries[mid].first <= sh) lo = mid;
        else hi = mid - 1;
    }
    const UnitEntry en = entries[lo];
    const int l0 = sh - en.first;
    const bool along_a = x >= 2;
    const LineBands B{d, e, n, H, x & 1};
    const int m = (n - B.par + 1) / 2;
    const double p = pq[sh].x, q = pq[sh].y, qp = l0 > 0 ? pq[sh - 1].y : 0.0;
    // the tridiagonal alpha A~ + beta (along b c + p A~, along a A~ - q) and the solution's scale
    const double alpha = along_a ? 1.0 : p, beta = along_a ? -q : en.c;
    const double scale = along_a ? q - p : (l0 == 0 ? -1.0 : qp - p);
    float *l = tabs + en.tab_off + ((int64_t)l0 * 4 + x) * tab, *mg = l + 2 * LS, *mid = l + 6 * LS;
    double prev = 1.0;  // pivot of the outer neighbour
    for (int s = 0; s < H; ++s) {
        const int i = B.at(h, s);
        const double eo = B.outer(h, s), c = alpha * eo, ip = 1.0 / prev, lv = c * ip;
        const double own = i < m ? alpha * B.diag(i) + beta : 1.0, piv = own - lv * c;
        const double iv = 1.0 / piv;
        if (live) {
            l[h * LS + s] = (float)lv;
            if (s) mg[2 * (h * LS + s - 1)] = (float)(c * iv);
            mg[2 * (h * LS + s) + 1] = (float)(i < m ? scale * iv : 0.0);
        }
        prev = piv;
    }
    const double other = __shfl_xor_sync(0xffffffffu, prev, 1), em = B.off(H - 1), c = alpha * em;
    const double det = prev * other - c * c;
    if (!live) return;
    mg[2 * (h * LS + H - 1)] = 0.0f;
    mid[2 * h] = (float)(prev * other / det);
    mid[2 * h + 1] = (float)(-c * prev / det);
}

__global__ void unit_bands_kernel(const double *__restrict__ d, const double *__restrict__ e, int n, int H,
                                  float *__restrict__ bands)
{
    const int par = blockIdx.x, LS = unit_half_pitch(H);
    const LineBands B{d, e, n, H, par};
    float *o = bands + par * unit_bands(H);
    for (int t = threadIdx.x; t < unit_bands(H) / 2; t += blockDim.x) {
        const int h = t / LS, s = t % LS;
        o[2 * t] = t == 2 * LS ? (float)B.off(H - 1) : (h < 2 && s < H ? (float)B.diag(B.at(h, s)) : 0.0f);
        o[2 * t + 1] = h < 2 && s < H ? (float)B.outer(h, s) : 0.0f;
    }
}

template <int H>
cudaError_t setup_H()
{
    return cudaFuncSetAttribute(stein_unit_kernel<H>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)UnitGeo<H>::bytes);
}

template <int H>
cudaError_t launch_H(const UnitArgs &a, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(4 * a.n), (unsigned)a.njobs);
    cfg.blockDim = dim3((unsigned)UnitGeo<H>::kThreads);
    cfg.dynamicSmemBytes = UnitGeo<H>::bytes;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, stein_unit_kernel<H>, a);
}

}  // namespace

// Half lengths with a compiled kernel.
#define UNIT_SIZES(X) \
    X(2) X(4) X(6) X(8) X(12) X(16) X(20) X(24) X(32) X(40) X(48) X(56) X(64) X(72) X(80)

int unit_half(int64_t n)
{
    const int m = (int)((n + 1) / 2);
#define TRY(h) if (m <= 2 * h) return h;
    UNIT_SIZES(TRY)
#undef TRY
    return 0;
}

#define CASE_SETUP(h) case h: return setup_H<h>();
#define CASE_LAUNCH(h) case h: return launch_H<h>(a, st);

cudaError_t unit_setup(int H)
{
    switch (H) { UNIT_SIZES(CASE_SETUP) }
    return cudaErrorInvalidValue;
}

cudaError_t launch_stein_units(const UnitArgs &a, int H, cudaStream_t st)
{
    switch (H) { UNIT_SIZES(CASE_LAUNCH) }
    return cudaErrorInvalidValue;
}

cudaError_t launch_unit_tables(const UnitEntry *entries, int count, int shifts, const double2 *pq, const double *d,
                               const double *e, int n, int H, float *tab, cudaStream_t st)
{
    const int64_t threads = 8 * (int64_t)shifts;
    unit_tables_kernel<<<(unsigned)((threads + 63) / 64), 64, 0, st>>>(entries, count, shifts, pq, d, e, n, H, tab);
    return cudaGetLastError();
}

cudaError_t launch_unit_bands(const double *d, const double *e, int n, int H, float *bands, cudaStream_t st)
{
    unit_bands_kernel<<<2, 128, 0, st>>>(d, e, n, H, bands);
    return cudaGetLastError();
}

}  // namespace fps
