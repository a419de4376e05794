// ADI pass kernels of the square solve (see sweep.cuh for the scheme and layout).
//
// Tiles travel through shared memory by bulk asynchronous copies (cp.async.bulk, one
// copy per S x S block, completion on an mbarrier; results leave by bulk stores), so no
// thread spends registers or issue slots on address streams.  Inside a tile every
// thread owns one line (a row in the row pass, a column in the column pass) and keeps
// the forward values of its segment in registers.
#include <cuda_runtime.h>

#include "bulk.cuh"
#include "device_info.h"
#include "sweep.cuh"

namespace fps {

namespace {

constexpr int kL = kPassLines;  // lines of a tile = threads of a pass CTA

// 16-byte chunks of T
template <typename T>
__device__ __forceinline__ void ld16(const T *p, T (&v)[16 / sizeof(T)]);
template <>
__device__ __forceinline__ void ld16<float>(const float *p, float (&v)[4])
{
    const float4 f = *reinterpret_cast<const float4 *>(p);
    v[0] = f.x;
    v[1] = f.y;
    v[2] = f.z;
    v[3] = f.w;
}
template <>
__device__ __forceinline__ void ld16<double>(const double *p, double (&v)[2])
{
    const double2 f = *reinterpret_cast<const double2 *>(p);
    v[0] = f.x;
    v[1] = f.y;
}
template <typename T>
__device__ __forceinline__ void st16(T *p, const T (&v)[16 / sizeof(T)]);
template <>
__device__ __forceinline__ void st16<float>(float *p, const float (&v)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
template <>
__device__ __forceinline__ void st16<double>(double *p, const double (&v)[2])
{
    *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
}

template <typename T>
__device__ __forceinline__ typename Vec2<T>::type mk2(T x, T y);
template <>
__device__ __forceinline__ float2 mk2<float>(float x, float y)
{
    return make_float2(x, y);
}
template <>
__device__ __forceinline__ double2 mk2<double>(double x, double y)
{
    return make_double2(x, y);
}

// Segments per thread of the recurrences that the passes run.
__host__ __device__ constexpr int chain_segments(bool fp64) { return fp64 ? 4 : 8; }

__host__ __device__ __forceinline__ int round4(int n) { return (n + 3) & ~3; }

// Shared memory of a pass CTA: tile (and the tile of D), the solve tables of the tile's
// positions, the summary tables of one segment, and the exchange of the segment recurrence
// (zin and yout of the kL threads, partial values of the thread groups).
template <typename T, int S>
struct Geo {
    static constexpr int V = 16 / (int)sizeof(T);
    static constexpr int B = S * S;       // elements of a block
    static constexpr int CH = S / V;      // chunks of a row
    static constexpr size_t off_tile = 128;
    static constexpr size_t tile_bytes = sizeof(T) * kL * S;
    static constexpr int G = kL / S;      // blocks of a tile, thread groups of the segment recurrence
    static constexpr size_t tab_elems = 3 * kL + 2 * S + 2 * kL + 2 * kL + 2 * G;
    static constexpr size_t row_bytes = off_tile + tile_bytes + sizeof(T) * tab_elems;
    static constexpr size_t col_bytes = off_tile + 2 * tile_bytes + sizeof(T) * tab_elems;
    static constexpr size_t sum_bytes = row_bytes;
    // Resident CTAs per SM that the registers are limited for.  Blocks of 32 in FP32 serve
    // n = 1025 .. 2048, about one wave of tiles: 7 per SM hold the 1024 tiles of n = 2048 of the
    // row pass at once, 6 (what shared memory admits) those of the column pass up to n = 1792;
    // above, up to 112 of its tiles are a second wave.  Without the limits (6 and 5) n = 2048
    // took 5 % longer.
    static constexpr int row_ctas = sizeof(T) == 8 ? 3 : (S == 32 ? 7 : 4);
    static constexpr int col_ctas = sizeof(T) == 4 && S == 32 ? 6 : 3;
    static_assert(CH >= 8, "the XOR permutation needs eight chunks per row");
};

// ---------------------------------------------------------------------------
// Shift tables: one thread per (job, parity), FP64 arithmetic.
// ---------------------------------------------------------------------------
constexpr int kMaxS = 64;

template <typename T>
__global__ void fac_tables_kernel(const FacJob<T> *__restrict__ jobs, int njobs)
{
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= 2 * njobs) return;
    const FacJob<T> &jb = jobs[tid >> 1];
    const int p = tid & 1;
    const int S = jb.S, nb = jb.nb, Mp = nb * S, m = (jb.n - p + 1) / 2, nbp = round4(nb);
    const int64_t to = (int64_t)p * kTabs * Mp;
    const double *d = jb.d + p, *e = jb.e + p;  // position i of this parity: index 2 i
    // l_i = e_{i-1} ip_{i-1} and m_i = e_i ip_{i+1}; ip runs one position ahead
    double ip = 0.0, ip_next = m > 0 ? 1.0 / (d[0] - jb.q) : 0.0;
    double l_next = 0.0;
    double lv[kMaxS], mv[kMaxS], v[kMaxS];
    for (int s = 0; s < nb; ++s) {
        for (int u = 0; u < S; ++u) {
            const int i = s * S + u;
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
            v[u] = u == 0 ? 1.0 : v[u - 1] * -mv[u - 1];  // weight of w_i in y at the segment's start
            for (int t = 0; t < 2; ++t) {
                T *out = t == 0 ? jb.out1 : jb.out2;
                if (!out) continue;
                out[to + i] = (T)l;
                out[to + Mp + i] = (T)mm;
                out[to + 2 * Mp + i] = (T)((t == 0 ? jb.sc1 : jb.sc2) * ip);
            }
        }
        double psi = 1.0, chi = 0.0;
        for (int u = S - 1; u >= 0; --u) {
            const int i = s * S + u;
            if (u + 1 < S) psi *= -lv[u + 1];
            chi = u + 1 < S ? v[u] - lv[u + 1] * chi : v[u];
            const bool live = i < m;
            for (int t = 0; t < 2; ++t) {
                T *out = t == 0 ? jb.out1 : jb.out2;
                if (!out) continue;
                out[to + 3 * Mp + i] = live ? (T)psi : T(0);
                out[to + 4 * Mp + i] = live ? (T)chi : T(0);
            }
        }
        for (int t = 0; t < 2; ++t) {
            T *ch = t == 0 ? jb.ch1 : jb.ch2;
            if (!ch) continue;
            ch += (int64_t)p * 3 * nbp;
            ch[s] = (T)(-lv[0] * psi);
            ch[nbp + s] = (T)(-lv[0] * chi);
            ch[2 * nbp + s] = (T)(v[S - 1] * -mv[S - 1]);
        }
    }
}

// Bounded wait on the tile barrier; on a timeout flag the error word and give the
// copies in flight one more bounded wait before the CTA leaves.
__device__ __forceinline__ bool tile_ready(uint64_t *bar, int *err)
{
    if (bulk::mbar_wait_bounded(bar, 0)) return true;
    if (threadIdx.x == 0) atomicOr(err, 1);
    bulk::mbar_wait_bounded(bar, 0);
    return false;
}

// The launches of a solve form one dependent chain; programmatic dependent launch lets
// the next kernel's CTAs start while the last CTAs of this one run.  pdl_wait() returns
// when every earlier kernel has completed; nothing that those write is read before it.
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// Start of a pass CTA: the item, and whether there is work (mask of active problems, J,
// an error anywhere).  Initialises `nbar` barriers; ends with a CTA barrier.
template <typename T>
__device__ __forceinline__ bool pass_begin(const SwArgs<T> &a, const SwItem<T> &it, int j, uint64_t *bar, int nbar)
{
    const bool in_range = j < it.J;
    pdl_wait();
    const int masked = *a.masked;
    const bool act = in_range && (!masked || a.active[it.prob]);
    if (threadIdx.x == 0) {
        for (int b = 0; b < nbar; ++b) bulk::mbar_init(bar + b, 1);
        bulk::fence_mbar_init();
    }
    // after a timeout anywhere, leave at once (one read, agreed on by the whole CTA)
    const int stop = __syncthreads_or(threadIdx.x == 0 ? *(volatile int *)a.err : 0);
    return act && !stop;
}

// Segment recurrence of the S lines of a tile by the pass itself: the G groups of S
// threads (lane = line) own LEN consecutive segments each; a group composes the affine maps
// W -> alpha W + beta of its segments, the groups' maps are composed through shared memory
// and the true values follow from one more walk; then the same backwards.  The result
// {zin, yout} of the tile's segments is left in zx[block][line].  Runs while the tile is in
// flight.  (A tile across the lines, every thread walking all segments of its own line, read
// the summaries once per segment of the line and ended at 16 segments.)
template <typename T, int S>
struct LineChain {
    using T2 = typename Vec2<T>::type;
    static constexpr int LEN = chain_segments(sizeof(T) == 8);
    static constexpr int G = kL / S;
    T phi[LEN], bv[LEN], ps[LEN];
    T2 v[LEN];
    int s0, li, g;

    // tables of the plan: may be read before the kernels before have finished
    __device__ __forceinline__ void tables(const T *__restrict__ co, int P)
    {
        li = threadIdx.x % S;
        g = threadIdx.x / S;
        s0 = g * LEN;
        const int nbp = round4(P);
#pragma unroll
        for (int b = 0; b < LEN; ++b) {
            const bool ok = s0 + b < P;
            phi[b] = ok ? co[s0 + b] : T(0);
            bv[b] = ok ? co[nbp + s0 + b] : T(0);
            ps[b] = ok ? co[2 * nbp + s0 + b] : T(0);
        }
    }
    // sum: segment 0 of the tile's first line, segments `step` apart
    __device__ __forceinline__ void load(const T2 *__restrict__ sum, int64_t step, int P)
    {
#pragma unroll
        for (int b = 0; b < LEN; ++b) v[b] = s0 + b < P ? sum[li + (s0 + b) * step] : mk2<T>(T(0), T(0));
    }
    // part: 2 kL + 2 G elements; first, count: the tile's segments.  Ends with a CTA barrier.
    __device__ __forceinline__ void run(T2 *zx, T *part, int first, int count)
    {
        T *beta = part, *alpha = part + 2 * kL;
        T al = phi[0], be = v[0].x;
#pragma unroll
        for (int b = 1; b < LEN; ++b) {
            be = fma(phi[b], be, v[b].x);
            al *= phi[b];
        }
        beta[threadIdx.x] = be;
        if (li == 0) alpha[g] = al;
        __syncthreads();
        T W = 0;
        for (int h = 0; h < g; ++h) W = fma(alpha[h], W, beta[h * S + li]);
        T z[LEN];
#pragma unroll
        for (int b = 0; b < LEN; ++b) {
            z[b] = W;
            if (b + 1 < LEN) W = fma(phi[b], W, v[b].x);
            v[b].y = fma(bv[b], z[b], v[b].y);
        }
        // segments past the last have zero maps: what a group composes starts at its last segment
        al = ps[LEN - 1];
        be = v[LEN - 1].y;
#pragma unroll
        for (int b = LEN - 2; b >= 0; --b) {
            be = fma(ps[b], be, v[b].y);
            al *= ps[b];
        }
        beta[kL + threadIdx.x] = be;
        if (li == 0) alpha[G + g] = al;
        __syncthreads();
        T Y = 0;
        for (int h = G - 1; h > g; --h) Y = fma(alpha[G + h], Y, beta[kL + h * S + li]);
#pragma unroll
        for (int b = LEN - 1; b >= 0; --b) {
            const int t = s0 + b - first;
            if (t >= 0 && t < count) zx[t * S + li] = mk2<T>(z[b], Y);
            if (b > 0) Y = fma(ps[b], Y, v[b].y);
        }
        __syncthreads();
    }
};

// ---------------------------------------------------------------------------
// Row pass.  A tile is n_blk blocks of one block row: S rows x up to 128 columns, so that
// its threads can share the segment recurrence of its S rows.  FIRST: j = 0 (a = v).
// FUSED: the recurrence runs here; otherwise its own launch has left zin and yout.
// ---------------------------------------------------------------------------
template <typename T, int S, bool FIRST, bool FUSED>
__global__ void __launch_bounds__(kL, Geo<T, S>::row_ctas) row_pass_kernel(SwArgs<T> A, int j)
{
    using G = Geo<T, S>;
    using T2 = typename Vec2<T>::type;
    constexpr int V = G::V;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem);
    T *tile = reinterpret_cast<T *>(smem + G::off_tile);
    T *tl = tile + kL * S, *tm = tl + kL, *ts = tm + kL, *psi = ts + kL, *chi = psi + S;
    T2 *zx = reinterpret_cast<T2 *>(chi + S);
    T *part = reinterpret_cast<T *>(zx + kL);
    const int tid = threadIdx.x;
    pdl_launch();
    const SwItem<T> it = A.items[blockIdx.x];
    const int nb = it.nb, bi = it.b0, bk0 = it.b1, nblk = it.n_blk, Mp = nb * S;
    LineChain<T, S> chain;
    if (FUSED && j < it.J) chain.tables(it.chR + (int64_t)j * 6 * round4(nb), nb);
    if (!pass_begin(A, it, j, bar, 1)) return;
    T *X = A.X + it.xoff;
    const unsigned xb = (unsigned)(nblk * G::B * sizeof(T));  // the blocks of the tile are adjacent
    if (tid == 0) {
        const T *tR = it.tabR + (int64_t)j * (2 * kTabs) * Mp + bk0 * S;
        const T *tC = it.tabC + (int64_t)j * (2 * kTabs) * Mp + bi * S;
        const unsigned tb = (unsigned)(nblk * S * sizeof(T)), pb = (unsigned)(S * sizeof(T));
        bulk::mbar_arrive_expect_tx(bar, xb + 3 * tb + 2 * pb);
        bulk::g2s(tile, X, xb, bar);
        bulk::g2s(tl, tR, tb, bar);
        bulk::g2s(tm, tR + Mp, tb, bar);
        bulk::g2s(ts, tR + 2 * Mp, tb, bar);
        bulk::g2s(psi, tC + 3 * Mp, pb, bar);
        bulk::g2s(chi, tC + 4 * Mp, pb, bar);
    }
    const int b = tid / S, r = tid % S;
    const bool on = b < nblk;
    T2 zy = mk2<T>(T(0), T(0));
    if (FUSED) {
        chain.load(A.sumR + it.soff + bi * S, Mp, nb);
        chain.run(zx, part, bk0, nblk);
        if (on) zy = zx[tid];
    } else if (on) {
        zy = A.zxR[it.soff + bi * S + r + (int64_t)(bk0 + b) * Mp];
    }
    if (!tile_ready(bar, A.err)) return;
    if (on) {
        T *row = tile + b * G::B + r * S;
        int sw[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) sw[q] = (q ^ (r & 7)) * V;
        T w[S];
        T z = zy.x;
#pragma unroll
        for (int c = 0; c < G::CH; ++c) {
            T u[V], l[V];
            ld16(row + (c / 8) * 8 * V + sw[c % 8], u);
            ld16(tl + b * S + c * V, l);
#pragma unroll
            for (int e = 0; e < V; ++e) {
                z = fma(-l[e], z, u[e]);
                w[c * V + e] = z;
            }
        }
        T y = zy.y;
#pragma unroll
        for (int c = G::CH - 1; c >= 0; --c) {
            T u[V], m[V], s[V];
            T *pc = row + (c / 8) * 8 * V + sw[c % 8];
            if (!FIRST) ld16(pc, u);
            ld16(tm + b * S + c * V, m);
            ld16(ts + b * S + c * V, s);
#pragma unroll
            for (int e = V - 1; e >= 0; --e) {
                y = fma(-m[e], y, w[c * V + e]);
                u[e] = FIRST ? s[e] * y : fma(s[e], y, u[e]);
            }
            st16(pc, u);
        }
    }
    bulk::fence_proxy_async_shared();
    __syncthreads();
    if (tid == 0) {
        bulk::s2g(X, tile, xb);
        bulk::commit();
    }
    // summaries of the column solve: thread = (column c, block g)
    {
        const int g = tid / S, c = tid % S;
        if (g < nblk) {
            const T *col = tile + g * G::B + c % V;
            int sw[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) sw[q] = ((c / V) ^ q) * V + q * S;
            T wl[2] = {0, 0}, yl[2] = {0, 0};
#pragma unroll
            for (int r0 = 0; r0 < S; r0 += V) {
                T ps[V], ch[V];
                ld16(psi + r0, ps);
                ld16(chi + r0, ch);
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    const int rr = r0 + e;
                    const T x = col[(rr / 8) * 8 * S + sw[rr % 8]];
                    wl[e & 1] = fma(ps[e], x, wl[e & 1]);
                    yl[e & 1] = fma(ch[e], x, yl[e & 1]);
                }
            }
            A.sumC[it.soff + (int64_t)bi * Mp + (bk0 + g) * S + c] = mk2<T>(wl[0] + wl[1], yl[0] + yl[1]);
        }
    }
    if (tid == 0) bulk::wait_read_all();
}

// Summaries of the row solve (psi, chi staged in shared memory for the tile's columns):
// thread = (row r, block g) of a column-pass tile.
template <typename T, int S>
__device__ __forceinline__ void row_summaries(const SwArgs<T> &A, const SwItem<T> &it, const T *tile, const T *psi,
                                              const T *chi)
{
    using G = Geo<T, S>;
    constexpr int V = G::V;
    const int g = threadIdx.x / S, r = threadIdx.x % S;
    if (g >= it.n_blk) return;
    const T *row = tile + g * G::B + r * S;
    int sw[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) sw[q] = (q ^ (r & 7)) * V;
    T wl[2] = {0, 0}, yl[2] = {0, 0};
#pragma unroll
    for (int c = 0; c < G::CH; ++c) {
        T x[V], ps[V], ch[V];
        ld16(row + (c / 8) * 8 * V + sw[c % 8], x);
        ld16(psi + c * V, ps);
        ld16(chi + c * V, ch);
#pragma unroll
        for (int e = 0; e < V; ++e) {
            wl[e & 1] = fma(ps[e], x[e], wl[e & 1]);
            yl[e & 1] = fma(ch[e], x[e], yl[e & 1]);
        }
    }
    const int Mp = it.nb * S;
    A.sumR[it.soff + (int64_t)it.b1 * Mp + (it.b0 + g) * S + r] = mk2<T>(wl[0] + wl[1], yl[0] + yl[1]);
}

// ---------------------------------------------------------------------------
// Column pass.  A tile is n_blk blocks of one block column: up to 128 rows x S columns.
// FIRST: j = 0 (D written, not read).  In the last iteration of a problem u and the
// summaries are not needed.
// ---------------------------------------------------------------------------
template <typename T, int S, bool FIRST, bool FUSED>
__global__ void __launch_bounds__(kL, Geo<T, S>::col_ctas) col_pass_kernel(SwArgs<T> A, int j)
{
    using G = Geo<T, S>;
    using T2 = typename Vec2<T>::type;
    constexpr int V = G::V;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem);
    T *tile = reinterpret_cast<T *>(smem + G::off_tile), *dt = tile + kL * S;
    T *tl = dt + kL * S, *tm = tl + kL, *ts = tm + kL, *psi = ts + kL, *chi = psi + S;
    T2 *zx = reinterpret_cast<T2 *>(chi + S);
    T *part = reinterpret_cast<T *>(zx + kL);
    const int tid = threadIdx.x;
    pdl_launch();
    // tiles in the reverse order of the row pass: those it wrote last are still in L2
    const SwItem<T> it = A.items[gridDim.x - 1 - blockIdx.x];
    const int nb = it.nb, bi0 = it.b0, bk = it.b1, nblk = it.n_blk, Mp = nb * S;
    LineChain<T, S> chain;
    if (FUSED && j < it.J) chain.tables(it.chC + (int64_t)j * 6 * round4(nb), nb);
    if (!pass_begin(A, it, j, bar, 2)) return;
    const bool last = j + 1 == it.J;
    T *X = A.X + it.xoff, *D = A.D + it.xoff;
    const int64_t bstride = (int64_t)nb * G::B;  // blocks of the tile are one block row apart
    constexpr unsigned bb = (unsigned)(G::B * sizeof(T));
    if (tid == 0) {
        const T *tC = it.tabC + (int64_t)j * (2 * kTabs) * Mp + bi0 * S;
        const unsigned tb = (unsigned)(nblk * S * sizeof(T)), pb = (unsigned)(S * sizeof(T));
        bulk::mbar_arrive_expect_tx(bar, nblk * bb + 3 * tb);
        for (int q = 0; q < nblk; ++q) bulk::g2s(tile + q * G::B, X + q * bstride, bb, bar);
        bulk::g2s(tl, tC, tb, bar);
        bulk::g2s(tm, tC + Mp, tb, bar);
        bulk::g2s(ts, tC + 2 * Mp, tb, bar);
        const unsigned second = (FIRST ? 0u : nblk * bb) + (last ? 0u : 2 * pb);
        if (second) bulk::mbar_arrive_expect_tx(bar + 1, second);
        if (!FIRST)
            for (int q = 0; q < nblk; ++q) bulk::g2s(dt + q * G::B, D + q * bstride, bb, bar + 1);
        if (!last) {
            const T *tR = it.tabR + (int64_t)(j + 1) * (2 * kTabs) * Mp + bk * S;
            bulk::g2s(psi, tR + 3 * Mp, pb, bar + 1);
            bulk::g2s(chi, tR + 4 * Mp, pb, bar + 1);
        }
    }
    const int b = tid / S, c = tid % S;
    const bool on = b < nblk;
    T2 zy = mk2<T>(T(0), T(0));
    if (FUSED) {
        chain.load(A.sumC + it.soff + bk * S, Mp, nb);
        chain.run(zx, part, bi0, nblk);
        if (on) zy = zx[tid];
    } else if (on) {
        zy = A.zxC[it.soff + bk * S + c + (int64_t)(bi0 + b) * Mp];
    }
    if (!tile_ready(bar, A.err)) {
        if (!FIRST || !last) bulk::mbar_wait_bounded(bar + 1, 0);
        return;
    }
    int sw[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) sw[q] = ((c / V) ^ q) * V + q * S + c % V;
    T w[S];
    if (on) {
        const T *col = tile + b * G::B;
        T z = zy.x;
#pragma unroll
        for (int r0 = 0; r0 < S; r0 += V) {
            T l[V];
            ld16(tl + b * S + r0, l);
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const int r = r0 + e;
                z = fma(-l[e], z, col[(r / 8) * 8 * S + sw[r % 8]]);
                w[r] = z;
            }
        }
    }
    if (!FIRST || !last) {
        if (!tile_ready(bar + 1, A.err)) return;
    }
    if (on) {
        T *col = tile + b * G::B, *dcol = dt + b * G::B;
        T y = zy.y;
#pragma unroll
        for (int r0 = S - V; r0 >= 0; r0 -= V) {
            T m[V], s[V];
            ld16(tm + b * S + r0, m);
            ld16(ts + b * S + r0, s);
#pragma unroll
            for (int e = V - 1; e >= 0; --e) {
                const int r = r0 + e, o = (r / 8) * 8 * S + sw[r % 8];
                y = fma(-m[e], y, w[r]);
                col[o] = fma(s[e], y, col[o]);
                dcol[o] = FIRST ? s[e] * y : fma(s[e], y, dcol[o]);
            }
        }
    }
    bulk::fence_proxy_async_shared();
    __syncthreads();
    if (tid == 0) {
        for (int q = 0; q < nblk; ++q) {
            if (!last) bulk::s2g(X + q * bstride, tile + q * G::B, bb);
            bulk::s2g(D + q * bstride, dt + q * G::B, bb);
        }
        bulk::commit();
    }
    if (!last) row_summaries<T, S>(A, it, tile, psi, chi);
    if (tid == 0) bulk::wait_read_all();
}

// Summaries of the row solve of iteration 0 (items of the column pass).
template <typename T, int S>
__global__ void __launch_bounds__(kL) row_sums_kernel(SwArgs<T> A)
{
    using G = Geo<T, S>;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem);
    T *tile = reinterpret_cast<T *>(smem + G::off_tile);
    T *psi = tile + kL * S, *chi = psi + S;
    pdl_launch();
    const SwItem<T> it = A.items[blockIdx.x];
    if (!pass_begin(A, it, 0, bar, 1)) return;
    const int Mp = it.nb * S;
    if (threadIdx.x == 0) {
        const T *tR = it.tabR + it.b1 * S;
        const unsigned bb = (unsigned)(G::B * sizeof(T)), pb = (unsigned)(S * sizeof(T));
        bulk::mbar_arrive_expect_tx(bar, it.n_blk * bb + 2 * pb);
        for (int q = 0; q < it.n_blk; ++q)
            bulk::g2s(tile + q * G::B, A.X + it.xoff + (int64_t)q * it.nb * G::B, bb, bar);
        bulk::g2s(psi, tR + 3 * Mp, pb, bar);
        bulk::g2s(chi, tR + 4 * Mp, pb, bar);
    }
    if (!tile_ready(bar, A.err)) return;
    row_summaries<T, S>(A, it, tile, psi, chi);
}

// ---------------------------------------------------------------------------
// Segment recurrences of 32 lines, latency bound.  Warp g owns LEN consecutive segments of every line
// (lane = line): it composes their affine maps W -> alpha W + beta from the summaries in
// registers, the warps' maps are composed through shared memory, and the true values
// follow from one more walk; then the same backwards.  The summaries are read once
// (n = 10^4, FP32: 10 us a launch; one thread walking all segments of a line took 16).
// Lines of few segments have no launch at all (LineChain).
// ---------------------------------------------------------------------------
template <typename T, int LEN>
__global__ void chain_kernel(SwArgs<T> A, int dir, int j)
{
    using T2 = typename Vec2<T>::type;
    __shared__ T beta[2][32][32];
    __shared__ T alpha[2][32];
    pdl_launch();
    const SwItem<T> it = A.items[blockIdx.x];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, G = blockDim.x >> 5;
    const int P = it.nb, nbp = round4(P), Mp = P * A.S;
    const T *co = (dir == 0 ? it.chR : it.chC) + (int64_t)j * 6 * nbp;
    const int s0 = g * LEN;
    const bool in_range = j < it.J;
    T phi[LEN], bv[LEN], ps[LEN];
#pragma unroll
    for (int b = 0; b < LEN; ++b) {  // tables of the plan: no launch of this solve writes them
        const bool ok = in_range && s0 + b < P;
        phi[b] = ok ? co[s0 + b] : T(0);
        bv[b] = ok ? co[nbp + s0 + b] : T(0);
        ps[b] = ok ? co[2 * nbp + s0 + b] : T(0);
    }
    pdl_wait();
    if (!in_range || (*A.masked && !A.active[it.prob])) return;
    const int64_t line = it.soff + it.b1 * 32 + lane;
    const T2 *__restrict__ sum = (dir == 0 ? A.sumR : A.sumC) + line;
    T2 *__restrict__ zx = (dir == 0 ? A.zxR : A.zxC) + line;
    T2 v[LEN];
#pragma unroll
    for (int b = 0; b < LEN; ++b) v[b] = s0 + b < P ? sum[(int64_t)(s0 + b) * Mp] : mk2<T>(T(0), T(0));
    T al = 1, be = 0;
#pragma unroll
    for (int b = 0; b < LEN; ++b) {
        be = fma(phi[b], be, v[b].x);
        al *= phi[b];
    }
    beta[0][g][lane] = be;
    if (lane == 0) alpha[0][g] = al;
    __syncthreads();
    T W = 0;
    for (int h = 0; h < g; ++h) W = fma(alpha[0][h], W, beta[0][h][lane]);
    T z[LEN];
#pragma unroll
    for (int b = 0; b < LEN; ++b) {
        z[b] = W;
        W = fma(phi[b], W, v[b].x);
        v[b].y = fma(bv[b], z[b], v[b].y);
    }
    al = 1;
    be = 0;
#pragma unroll
    for (int b = LEN - 1; b >= 0; --b)
        if (s0 + b < P) {
            be = fma(ps[b], be, v[b].y);
            al *= ps[b];
        }
    beta[1][g][lane] = be;
    if (lane == 0) alpha[1][g] = al;
    __syncthreads();
    T Y = 0;
    for (int h = G - 1; h > g; --h) Y = fma(alpha[1][h], Y, beta[1][h][lane]);
#pragma unroll
    for (int b = LEN - 1; b >= 0; --b)
        if (s0 + b < P) {
            zx[(int64_t)(s0 + b) * Mp] = mk2<T>(z[b], Y);
            Y = fma(ps[b], Y, v[b].y);
        }
}

// The same for lines of more segments than a CTA's registers hold: kWalkWarps warps, each
// walking its share of the line in steps of kC segments, whose operands are read together.  The summaries
// are read once more than by chain_kernel, and {zin, y from zin} is left in the results'
// place between the walk forwards, which also composes the maps of the walk backwards, and
// that one.  Latency bound as chain_kernel; a solve of n = 16500 in FP64 takes 736 ms and of
// n = 40000 4.58 s (2.76 times n = 10^4 of chain_kernel for 2.72 times the unknowns, and
// 17.2 times for 16), FP32 with refinement n = 33000 0.49 s (12.0 times for 10.9).
template <typename T>
__global__ void __launch_bounds__(32 * kWalkWarps) chain_walk_kernel(SwArgs<T> A, int dir, int j)
{
    using T2 = typename Vec2<T>::type;
    constexpr int kWarps = kWalkWarps, kC = sizeof(T) == 8 ? 4 : 8;
    __shared__ T beta[2][kWarps][32];
    __shared__ T alpha[2][kWarps];
    pdl_launch();
    const SwItem<T> it = A.items[blockIdx.x];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int P = it.nb, nbp = round4(P), Mp = P * A.S, run = (P + kWarps - 1) / kWarps;
    const bool in_range = j < it.J;
    pdl_wait();
    if (!in_range || (*A.masked && !A.active[it.prob])) return;
    const T *co = (dir == 0 ? it.chR : it.chC) + (int64_t)j * 6 * nbp;
    const int64_t line = it.soff + it.b1 * 32 + lane;
    const T2 *__restrict__ sum = (dir == 0 ? A.sumR : A.sumC) + line;
    T2 *zx = (dir == 0 ? A.zxR : A.zxC) + line;
    const int s0 = min(g * run, P), s1 = min(s0 + run, P);
    T al = 1, be = 0;
    for (int s = s0; s < s1; s += kC) {
        T phi[kC], w[kC];
#pragma unroll
        for (int b = 0; b < kC; ++b) {
            const bool ok = s + b < s1;
            phi[b] = ok ? co[s + b] : T(1);
            w[b] = ok ? sum[(int64_t)(s + b) * Mp].x : T(0);
        }
#pragma unroll
        for (int b = 0; b < kC; ++b) {
            be = fma(phi[b], be, w[b]);
            al *= phi[b];
        }
    }
    beta[0][g][lane] = be;
    if (lane == 0) alpha[0][g] = al;
    __syncthreads();
    T W = 0;
    for (int h = 0; h < g; ++h) W = fma(alpha[0][h], W, beta[0][h][lane]);
    al = 1;
    be = 0;
    for (int s = s0; s < s1; s += kC) {
        T phi[kC], bv[kC], ps[kC];
        T2 v[kC];
#pragma unroll
        for (int b = 0; b < kC; ++b)
            if (s + b < s1) {
                phi[b] = co[s + b];
                bv[b] = co[nbp + s + b];
                ps[b] = co[2 * nbp + s + b];
                v[b] = sum[(int64_t)(s + b) * Mp];
            }
#pragma unroll
        for (int b = 0; b < kC; ++b)
            if (s + b < s1) {
                const T y = fma(bv[b], W, v[b].y);
                zx[(int64_t)(s + b) * Mp] = mk2<T>(W, y);
                be = fma(al, y, be);
                al *= ps[b];
                W = fma(phi[b], W, v[b].x);
            }
    }
    beta[1][g][lane] = be;
    if (lane == 0) alpha[1][g] = al;
    __syncthreads();
    T Y = 0;
    for (int h = kWarps - 1; h > g; --h) Y = fma(alpha[1][h], Y, beta[1][h][lane]);
    for (int s = s1 - 1; s >= s0; s -= kC) {
        T ps[kC];
        T2 v[kC];
#pragma unroll
        for (int b = 0; b < kC; ++b)
            if (s - b >= s0) {
                ps[b] = co[2 * nbp + s - b];
                v[b] = zx[(int64_t)(s - b) * Mp];
            }
#pragma unroll
        for (int b = 0; b < kC; ++b)
            if (s - b >= s0) {
                zx[(int64_t)(s - b) * Mp] = mk2<T>(v[b].x, Y);
                Y = fma(ps[b], Y, v[b].y);
            }
    }
}

// ---------------------------------------------------------------------------
// Elementwise kernels.  GB300's FP64 pipe takes 64 cycles of an SM quadrant per warp
// instruction, conversions and comparisons included (and 64-bit integer comparisons
// measured the same), so these kernels convert between float and double, scale by powers
// of two and compare magnitudes with 32-bit integer instructions, and keep the FP64
// operations to the multiply-adds of the formulas.  A product alone is written as a
// multiply-add with zero: multiplications measured 76 cycles.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double times(double a, double b) { return fma(a, b, 0.0); }

// Largest magnitude as the bit pattern of |x| (NaN and Inf are above every finite value).
struct MaxBits {
    unsigned hi = 0, lo = 0;
    __device__ __forceinline__ void add(unsigned h, unsigned l)
    {
        const bool gt = h > hi || (h == hi && l > lo);
        hi = gt ? h : hi;
        lo = gt ? l : lo;
    }
    __device__ __forceinline__ void add(double x)
    {
        add((unsigned)__double2hiint(x) & 0x7fffffffu, (unsigned)__double2loint(x));
    }
    __device__ __forceinline__ double value() const { return __hiloint2double((int)hi, (int)lo); }
};

// Conversions of subnormal floats are rare and left to the FP64 pipe, out of line.
__device__ __noinline__ double widen_subnormal(float f) { return (double)f; }
__device__ __noinline__ float narrow_subnormal(double x, int k) { return (float)scalbn(x, -k); }

// (double)f
__device__ __forceinline__ double widen(float f)
{
    const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
    if (a - 1u < 0x007fffffu) return widen_subnormal(f);
    unsigned hi = (a >> 3) + 0x38000000u;
    if (a >= 0x7f800000u) hi |= 0x7ff00000u;  // Inf, NaN
    if (a == 0u) hi = 0u;
    return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}

// x 2^54 where the scale is so small that subnormal doubles count (k is raised to match);
// kept out of line, so that the product is not executed speculatively.
__device__ __noinline__ double lift_subnormal(double x) { return x * 18014398509481984.0; }

// (float)(x 2^-k), rounded to nearest even, -896 <= k; above the range Inf.
__device__ __forceinline__ float narrow_scaled(double x, int k)
{
    const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu, lo = (unsigned)__double2loint(x);
    const unsigned sign = (unsigned)__double2hiint(x) & 0x80000000u;
    const int e = (int)(h >> 20) - 896 - k;  // exponent field of the float
    if (e <= 0 && (h | lo)) return narrow_subnormal(x, k);
    unsigned f = ((h - ((unsigned)(896 + k) << 20)) << 3) | (lo >> 29);
    const unsigned rest = lo << 3;
    f += rest > 0x80000000u || (rest == 0x80000000u && (f & 1u)) ? 1u : 0u;
    if (e <= 0) f = 0u;
    if (e >= 255) f = h >= 0x7ff00000u ? 0x7fc00000u : 0x7f800000u;  // the residual's NaN or Inf reaches the host
    return __uint_as_float(sign | f);
}

// Scale of a pair's FP32 iteration: 2^k <= smax < 2^(k+1) (k >= -1022).
__device__ __forceinline__ int scale_exponent(unsigned long long smax_bits)
{
    const int e = (int)(smax_bits >> 52);
    return (e > 0 ? e : 1) - 1023;
}
__device__ __forceinline__ double power_of_two(int k)
{
    return __hiloint2double((k + 1023) << 20, 0);
}

// Tiles: q.x >> 8 problem, q.x & 255 right-hand side.
struct TileView {
    const TileProb *p;
    int n, nb, ls, pair, by, bx;
    int64_t off64, off;
};
__device__ __forceinline__ TileView tile_view(const TileArgs &t, int64_t idx)
{
    const int4 q = t.tiles[idx];
    TileView v;
    v.p = t.probs + (q.x >> 8);
    const int rhs = q.x & 255;
    v.n = v.p->n;
    v.nb = v.p->nb;
    v.ls = v.p->log_s;
    v.pair = v.p->pair0 + rhs;
    v.off64 = v.p->off64 + (int64_t)rhs * v.n * v.n;
    v.off = v.p->off + (int64_t)rhs * v.p->rhs;
    v.bx = q.y;
    v.by = q.z;
    return v;
}
// Offset of element (a, b) of quarter q in the passes' arrays, and in the FP64 arrays of
// the refinement (the same blocks, rows in natural order), from the pair's offset v.off:
// below 2^31, n <= 40000.
__device__ __forceinline__ unsigned block_base(const TileView &v, int q, int a, int b)
{
    return ((unsigned)(q * v.nb + (a >> v.ls)) * v.nb + (b >> v.ls)) << (2 * v.ls);
}
template <typename T>
__device__ __forceinline__ unsigned quarter_pos(const TileView &v, int q, int a, int b)
{
    const int S = 1 << v.ls;
    return block_base(v, q, a, b) + block_pos<T>(a & (S - 1), b & (S - 1), S);
}
__device__ __forceinline__ unsigned plain_pos(const TileView &v, int q, int a, int b)
{
    const int S = 1 << v.ls;
    return block_base(v, q, a, b) + ((a & (S - 1)) << v.ls) + (b & (S - 1));
}

// The contiguous run of tiles of this CTA, for the reduction kernels (tiles are
// ordered pair by pair, so a run meets each (problem, rhs) pair once: one atomic per
// pair and CTA instead of one per tile).
__device__ __forceinline__ void tile_run(int64_t ntiles, int64_t &t0, int64_t &t1)
{
    const int64_t per = (ntiles + gridDim.x - 1) / gridDim.x;
    t0 = (int64_t)blockIdx.x * per;
    t1 = t0 + per < ntiles ? t0 + per : ntiles;
}

// Largest magnitude of the CTA.
__device__ __forceinline__ void block_max_to(const MaxBits &m, unsigned long long *out)
{
    unsigned long long local = ((unsigned long long)m.hi << 32) | m.lo;
    for (int off = 16; off > 0; off >>= 1) local = max(local, __shfl_xor_sync(0xffffffffu, local, off));
    __shared__ unsigned long long wmax[8];
    if (threadIdx.x == 0) wmax[threadIdx.y] = local;
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        unsigned long long bm = 0;
        for (int q = 0; q < (int)blockDim.y; ++q) bm = max(bm, wmax[q]);
        atomicMax(out, bm);
    }
    __syncthreads();  // wmax is reused by the next reduction
}

// Natural 64 x 64 tiles: one multiplication per element (|F| s_i, largest over the
// thread's rows, then times s_k).
__global__ void __launch_bounds__(256) absmax_kernel(TileArgs t, const double *__restrict__ F,
                                                     unsigned long long *__restrict__ smax)
{
    int64_t t0, t1;
    tile_run(t.ntiles, t0, t1);
    MaxBits local;
    int cur = -1;
    for (int64_t tt = t0; tt < t1; ++tt) {
        const TileView v = tile_view(t, tt);
        if (v.pair != cur) {
            if (cur >= 0) block_max_to(local, smax + cur);
            local = MaxBits();
            cur = v.pair;
        }
        const double *s = v.p->s;
        double f[8][2], si[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int i = v.by * 64 + threadIdx.y + 8 * q;
            const double *row = F + v.off64 + (int64_t)i * v.n;
            si[q] = i < v.n ? s[i] : 0.0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = v.bx * 64 + 32 * h + threadIdx.x;
                f[q][h] = i < v.n && k < v.n ? row[k] : 0.0;
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            MaxBits m;
#pragma unroll
            for (int q = 0; q < 8; ++q) m.add(times(f[q][h], si[q]));
            const int k = v.bx * 64 + 32 * h + threadIdx.x;
            if (k < v.n) local.add(times(m.value(), s[k]));
        }
    }
    if (cur >= 0) block_max_to(local, smax + cur);
}

// Pairs and problems with something to solve: 0 < smax < Inf (masked: any problem without).
__global__ void init_masks_kernel(const unsigned long long *__restrict__ smax, int np, int nrhs,
                                  int *__restrict__ pair_active, int *__restrict__ active, int *__restrict__ masked)
{
    for (int p = threadIdx.x; p < np; p += blockDim.x) {
        int any = 0;
        for (int r = 0; r < nrhs; ++r) {
            const unsigned long long b = smax[p * nrhs + r];
            const int on = b > 0 && b < 0x7ff0000000000000ULL;
            pair_active[p * nrhs + r] = on;
            any |= on;
        }
        active[p] = any;
        if (!any) *masked = 1;
    }
}

// Tiles of 32 x 32 positions of all four quarters (64 x 64 natural), padded region: F~ in
// the FP64 blocks (if Ft), rho0 = F~ 2^-k (float) or F~ (double) in the passes' blocks,
// zero at unused positions.
template <typename T>
__global__ void __launch_bounds__(256) scale_in_kernel(TileArgs t, const double *__restrict__ F, double *__restrict__ Ft,
                                                       T *__restrict__ rho0, const unsigned long long *__restrict__ smax)
{
    const TileView v = tile_view(t, blockIdx.x);
    const double *s = v.p->s;
    const int k = smax ? scale_exponent(smax[v.pair]) : 0;
    const int b = v.bx * 32 + threadIdx.x;
    double sk[2], f[8][2], si[8];
#pragma unroll
    for (int cp = 0; cp < 2; ++cp) sk[cp] = 2 * b + cp < v.n ? s[2 * b + cp] : 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int i = v.by * 64 + threadIdx.y + 8 * q;
        si[q] = i < v.n ? s[i] : 0.0;
#pragma unroll
        for (int cp = 0; cp < 2; ++cp)
            f[q][cp] = i < v.n && 2 * b + cp < v.n ? F[v.off64 + (int64_t)i * v.n + 2 * b + cp] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int i = v.by * 64 + threadIdx.y + 8 * q, a = i >> 1, rp = i & 1;
#pragma unroll
        for (int cp = 0; cp < 2; ++cp) {
            const int qd = rp * 2 + cp;
            const double val = times(times(f[q][cp], si[q]), sk[cp]);
            if (Ft && i < v.n && 2 * b + cp < v.n) Ft[v.off + plain_pos(v, qd, a, b)] = val;
            T *out = rho0 + v.off + quarter_pos<T>(v, qd, a, b);
            if constexpr (sizeof(T) == 4) *out = k < -896 ? narrow_scaled(lift_subnormal(val), k + 54) : narrow_scaled(val, k);
            else *out = val;
        }
    }
}

// X[i][k] = sc Z s_i s_k, Z in the passes' blocks (FP64 solve) or in the FP64 blocks
// (PLAIN, refinement).  Tiles as in scale_in_kernel; even and odd columns are put in
// natural order by shuffles, so that every store is contiguous.
template <bool PLAIN>
__global__ void __launch_bounds__(256) scale_out_kernel(TileArgs t, const double *__restrict__ Z, double *__restrict__ X)
{
    const TileView v = tile_view(t, blockIdx.x);
    const double *s = v.p->s;
    const double sc = PLAIN ? 1.0 : -v.p->inv_ky;
    const int lane = threadIdx.x, b = v.bx * 32 + lane, m0 = (v.n + 1) / 2;
    double sk[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int kk = v.bx * 64 + 32 * h + lane;
        sk[h] = kk < v.n ? (PLAIN ? s[kk] : sc * s[kk]) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int rr = threadIdx.y + 8 * q, a = v.by * 32 + (rr >> 1), rp = rr & 1, i = 2 * a + rp;
        if (i >= v.n) continue;  // the whole warp
        double z[2];
#pragma unroll
        for (int cp = 0; cp < 2; ++cp) {
            const unsigned pos = PLAIN ? plain_pos(v, rp * 2 + cp, a, b) : quarter_pos<double>(v, rp * 2 + cp, a, b);
            z[cp] = b < m0 - (cp & v.n) ? Z[v.off + pos] : 0.0;
        }
        const double si = s[i];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int src = 16 * h + (lane >> 1);
            const double e = __shfl_sync(0xffffffffu, z[0], src), o = __shfl_sync(0xffffffffu, z[1], src);
            const int kk = v.bx * 64 + 32 * h + lane;
            if (kk < v.n) X[v.off64 + (int64_t)i * v.n + kk] = times(times(lane & 1 ? o : e, si), sk[h]);
        }
    }
}

// Yout = Y - s D / ky; R = F~ - A~ Yout - Yout A~; rho0 = R / s; rmax = max |R|, with s the
// power of two of the pair's scale.  In a quarter the products with A~ are 3-point
// stencils with neighbours at distance one.  Tiles of 64 rows x 32 columns of a quarter;
// Y and Yout are distinct buffers, so every CTA sees the same not-yet-updated halo.
// Bound: the FP64 pipe, 7.1 operations per element (the update 1.1 with the halo, the
// stencils 6).  n = 4096: 250 us (78 % of the pipe; 24 to 32 B per element of HBM would
// take 80 us), 370 us with conversions left to the FP64 pipe and 64-bit comparisons;
// n = 10^4: 1.5 ms, 3.5 ms on interleaved parities with a halo of two.
constexpr int kResR = 64;
__global__ void __launch_bounds__(256, 3) residual_kernel(TileArgs t, const double *__restrict__ Y,
                                                       double *__restrict__ Yout, const float *__restrict__ D,
                                                       const double *__restrict__ Ft, float *__restrict__ rho0,
                                                       const unsigned long long *__restrict__ smax,
                                                       unsigned long long *__restrict__ rmax,
                                                       const int *__restrict__ pair_active, int y_zero)
{
    __shared__ double Ys[kResR + 2][35];
    // stencil coefficients of the tile's rows and columns: -kx {d_i, e_{i-1}, e_i} and -ky
    __shared__ double cr[3][kResR], cc[3][32];
    int64_t t0, t1;
    tile_run(t.ntiles, t0, t1);
    MaxBits local;
    int cur = -1;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * 32 + tx;
    for (int64_t tt = t0; tt < t1; ++tt) {
        const TileView v = tile_view(t, tt);
        const int qd = v.bx & 3, bx = (v.bx >> 2) * 32, by = v.by * kResR, rp = qd >> 1, cp = qd & 1;
        const int mr = (v.n - rp + 1) / 2, mc = (v.n - cp + 1) / 2;
        if (v.pair != cur) {
            if (cur >= 0) block_max_to(local, rmax + cur);
            local = MaxBits();
            cur = v.pair;
        }
        if (!pair_active[v.pair]) {  // converged pair: carry its iterate over unchanged
            for (int r = ty; r < kResR; r += 8)
                if (by + r < mr && bx + tx < mc) {
                    const int64_t pos = v.off + plain_pos(v, qd, by + r, bx + tx);
                    Yout[pos] = y_zero ? 0.0 : Y[pos];
                }
            continue;
        }
        const double *Yp = Y + v.off, *Fp = Ft + v.off;
        double *Yo = Yout + v.off;
        const float *Dp = D + v.off;
        float *rho = rho0 + v.off;
        const int k = scale_exponent(smax[v.pair]);
        const double sD = -power_of_two(k) * v.p->inv_ky;
        // all of the tile's loads in flight before the first is used
        constexpr int kHalo = (kResR + 2) * 34, kIt = (kHalo + 255) / 256;
        double yv[kIt], fv[kResR / 8];
        float dv[kIt];
#pragma unroll
        for (int q = 0; q < kIt; ++q) {
            const int idx = tid + 256 * q, r = idx / 34, c = idx - r * 34, a = by - 1 + r, b = bx - 1 + c;
            const bool ok = a >= 0 && a < mr && b >= 0 && b < mc && idx < kHalo;
            dv[q] = ok ? Dp[quarter_pos<float>(v, qd, a, b)] : 0.f;
            yv[q] = ok && !y_zero ? Yp[plain_pos(v, qd, a, b)] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < kResR / 8; ++q) {
            const int a = by + ty + 8 * q, b = bx + tx;
            fv[q] = a < mr && b < mc ? Fp[plain_pos(v, qd, a, b)] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < kIt; ++q) {
            const int idx = tid + 256 * q, r = idx / 34, c = idx - r * 34;
            if (idx < kHalo) Ys[r][c] = fma(sD, widen(dv[q]), yv[q]);
        }
        {
            const double *nd = v.p->nd, *ne = v.p->ne;  // -kx d, -kx e (rows), then -ky d, -ky e
            for (int q = tid; q < 3 * (kResR + 32); q += 256) {
                const bool row = q < 3 * kResR;
                const int set = row ? q / kResR : (q - 3 * kResR) / 32, w = row ? q % kResR : (q - 3 * kResR) % 32;
                const int a = (row ? by : bx) + w, full = 2 * a + (row ? rp : cp);
                const double *dd = row ? nd : nd + v.n, *ee = row ? ne : ne + v.n;
                double c = 0.0;
                if (full < v.n) c = set == 0 ? dd[full] : (set == 1 ? (a >= 1 ? ee[full - 2] : 0.0) : ee[full]);
                (row ? cr[set] : cc[set])[w] = c;  // e is zero where full + 2 >= n
            }
        }
        __syncthreads();
        const int b = bx + tx;
        const double c0 = cc[0][tx], c1 = cc[1][tx], c2 = cc[2][tx];
#pragma unroll
        for (int q = 0; q < kResR / 8; ++q) {
            const int r = ty + 8 * q, a = by + r;
            if (a < mr && b < mc) {
                const double y = Ys[r + 1][tx + 1];
                const unsigned pos = plain_pos(v, qd, a, b);
                double acc = fv[q];
                acc = fma(cr[0][r], y, acc);
                acc = fma(c0, y, acc);
                acc = fma(cr[1][r], Ys[r][tx + 1], acc);
                acc = fma(cr[2][r], Ys[r + 2][tx + 1], acc);
                acc = fma(c1, Ys[r + 1][tx], acc);
                acc = fma(c2, Ys[r + 1][tx + 2], acc);
                Yo[pos] = y;
                local.add(acc);
                rho[quarter_pos<float>(v, qd, a, b)] =
                    k < -896 ? narrow_scaled(lift_subnormal(acc), k + 54) : narrow_scaled(acc, k);
            }
        }
        __syncthreads();  // Ys is refilled by the next tile
    }
    if (cur >= 0) block_max_to(local, rmax + cur);
}

// Launch on `st` as a dependent of the launch before it (see pdl_wait).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*k)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

template <typename T, int S>
cudaError_t row_pass_S(const SwArgs<T> &a, int j, cudaStream_t st)
{
    const size_t sm = Geo<T, S>::row_bytes;
    const unsigned grid = (unsigned)a.nitems;
    if (a.fused) {
        if (j == 0) return launch_pdl(row_pass_kernel<T, S, true, true>, grid, kL, sm, st, a, j);
        return launch_pdl(row_pass_kernel<T, S, false, true>, grid, kL, sm, st, a, j);
    }
    if (j == 0) return launch_pdl(row_pass_kernel<T, S, true, false>, grid, kL, sm, st, a, j);
    return launch_pdl(row_pass_kernel<T, S, false, false>, grid, kL, sm, st, a, j);
}
template <typename T, int S>
cudaError_t col_pass_S(const SwArgs<T> &a, int j, cudaStream_t st)
{
    const size_t sm = Geo<T, S>::col_bytes;
    const unsigned grid = (unsigned)a.nitems;
    if (a.fused) {
        if (j == 0) return launch_pdl(col_pass_kernel<T, S, true, true>, grid, kL, sm, st, a, j);
        return launch_pdl(col_pass_kernel<T, S, false, true>, grid, kL, sm, st, a, j);
    }
    if (j == 0) return launch_pdl(col_pass_kernel<T, S, true, false>, grid, kL, sm, st, a, j);
    return launch_pdl(col_pass_kernel<T, S, false, false>, grid, kL, sm, st, a, j);
}

// CTAs of a reduction kernel: 8 per SM, at most one per tile.  The registers admit 4 (maximum)
// and 3 (residual) of them at a time.
unsigned reduction_grid(int64_t ntiles)
{
    const int64_t g = 8 * (int64_t)current_sm_count();
    return (unsigned)(ntiles < g ? (ntiles > 0 ? ntiles : 1) : g);
}

template <typename T, int S>
cudaError_t setup_S()
{
    cudaError_t e = cudaSuccess;
    auto set = [&](auto *k, size_t bytes) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    set(row_pass_kernel<T, S, true, true>, Geo<T, S>::row_bytes);
    set(row_pass_kernel<T, S, true, false>, Geo<T, S>::row_bytes);
    set(row_pass_kernel<T, S, false, true>, Geo<T, S>::row_bytes);
    set(row_pass_kernel<T, S, false, false>, Geo<T, S>::row_bytes);
    set(col_pass_kernel<T, S, true, true>, Geo<T, S>::col_bytes);
    set(col_pass_kernel<T, S, true, false>, Geo<T, S>::col_bytes);
    set(col_pass_kernel<T, S, false, true>, Geo<T, S>::col_bytes);
    set(col_pass_kernel<T, S, false, false>, Geo<T, S>::col_bytes);
    set(row_sums_kernel<T, S>, Geo<T, S>::sum_bytes);
    return e;
}

}  // namespace

bool sweep_fused(bool fp64, int S, int nb) { return nb <= chain_segments(fp64) * (kL / S); }

bool sweep_segment_supported(bool fp64, int seg) { return seg == 64 || (!fp64 && seg == 128); }

cudaError_t sweep_setup_kernels()
{
    cudaError_t e = setup_S<float, 32>();
    if (e == cudaSuccess) e = setup_S<float, 64>();
    if (e == cudaSuccess) e = setup_S<double, 32>();
    // the registers of the chain kernels admit the launches of chain_length
    auto admits = [&](auto *k, int warps) {
        cudaFuncAttributes at;
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, k);
        if (e == cudaSuccess && at.maxThreadsPerBlock < 32 * warps) e = cudaErrorInvalidConfiguration;
    };
    admits(chain_kernel<float, 8>, chain_warps(false, 8));
    admits(chain_kernel<float, 16>, chain_warps(false, 16));
    admits(chain_kernel<double, 8>, chain_warps(true, 8));
    return e;
}

template <typename T>
cudaError_t launch_fac_tables(const FacJob<T> *jobs, int njobs, cudaStream_t st)
{
    const int threads = 2 * njobs;
    fac_tables_kernel<T><<<(threads + 31) / 32, 32, 0, st>>>(jobs, njobs);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_row_sums(const SwArgs<T> &a, cudaStream_t st)
{
    // the first kernel of a graph: an ordinary launch
    if constexpr (sizeof(T) == 4) {
        if (a.S == 64) {
            row_sums_kernel<T, 64><<<(unsigned)a.nitems, kL, Geo<T, 64>::sum_bytes, st>>>(a);
            return cudaGetLastError();
        }
    }
    if (a.S != 32) return cudaErrorInvalidValue;
    row_sums_kernel<T, 32><<<(unsigned)a.nitems, kL, Geo<T, 32>::sum_bytes, st>>>(a);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_row_pass(const SwArgs<T> &a, int j, cudaStream_t st)
{
    if constexpr (sizeof(T) == 4) {
        if (a.S == 64) return row_pass_S<T, 64>(a, j, st);
    }
    if (a.S == 32) return row_pass_S<T, 32>(a, j, st);
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_col_pass(const SwArgs<T> &a, int j, cudaStream_t st)
{
    if constexpr (sizeof(T) == 4) {
        if (a.S == 64) return col_pass_S<T, 64>(a, j, st);
    }
    if (a.S == 32) return col_pass_S<T, 32>(a, j, st);
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_chain(const SwArgs<T> &a, int dir, int j, cudaStream_t st)
{
    constexpr bool kFP64 = sizeof(T) == 8;
    const unsigned grid = (unsigned)a.nitems;
    if (a.chain_len == 0) return launch_pdl(chain_walk_kernel<T>, grid, 32 * kWalkWarps, 0, st, a, dir, j);
    const int warps = (a.max_nb + a.chain_len - 1) / a.chain_len;
    if (warps > chain_warps(kFP64, a.chain_len)) return cudaErrorInvalidValue;
    if (a.chain_len == 8) return launch_pdl(chain_kernel<T, 8>, grid, 32 * warps, 0, st, a, dir, j);
    if constexpr (!kFP64) {
        if (a.chain_len == 16) return launch_pdl(chain_kernel<T, 16>, grid, 32 * warps, 0, st, a, dir, j);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_absmax(const TileArgs &t, const double *F, unsigned long long *smax, cudaStream_t st)
{
    absmax_kernel<<<reduction_grid(t.ntiles), dim3(32, 8), 0, st>>>(t, F, smax);
    return cudaGetLastError();
}

cudaError_t launch_init_masks(const unsigned long long *smax, int np, int nrhs, int *pair_active, int *active,
                              int *masked, cudaStream_t st)
{
    const cudaError_t e = cudaMemsetAsync(masked, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    init_masks_kernel<<<1, 256, 0, st>>>(smax, np, nrhs, pair_active, active, masked);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_scale_in(const TileArgs &t, const double *F, double *Ft, T *rho0, const unsigned long long *smax,
                            cudaStream_t st)
{
    scale_in_kernel<T><<<(unsigned)t.ntiles, dim3(32, 8), 0, st>>>(t, F, Ft, rho0, smax);
    return cudaGetLastError();
}

cudaError_t launch_residual(const TileArgs &t, const double *Y, double *Yout, const float *D, const double *Ft,
                            float *rho0, const unsigned long long *smax, unsigned long long *rmax,
                            const int *pair_active, bool y_zero, cudaStream_t st)
{
    residual_kernel<<<reduction_grid(t.ntiles), dim3(32, 8), 0, st>>>(t, Y, Yout, D, Ft, rho0, smax, rmax, pair_active,
                                                               y_zero ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_scale_out(const TileArgs &t, const double *Z, bool plain, double *X, cudaStream_t st)
{
    if (plain) scale_out_kernel<true><<<(unsigned)t.ntiles, dim3(32, 8), 0, st>>>(t, Z, X);
    else scale_out_kernel<false><<<(unsigned)t.ntiles, dim3(32, 8), 0, st>>>(t, Z, X);
    return cudaGetLastError();
}

template cudaError_t launch_fac_tables<float>(const FacJob<float> *, int, cudaStream_t);
template cudaError_t launch_fac_tables<double>(const FacJob<double> *, int, cudaStream_t);
template cudaError_t launch_row_sums<float>(const SwArgs<float> &, cudaStream_t);
template cudaError_t launch_row_sums<double>(const SwArgs<double> &, cudaStream_t);
template cudaError_t launch_row_pass<float>(const SwArgs<float> &, int, cudaStream_t);
template cudaError_t launch_row_pass<double>(const SwArgs<double> &, int, cudaStream_t);
template cudaError_t launch_col_pass<float>(const SwArgs<float> &, int, cudaStream_t);
template cudaError_t launch_col_pass<double>(const SwArgs<double> &, int, cudaStream_t);
template cudaError_t launch_chain<float>(const SwArgs<float> &, int, int, cudaStream_t);
template cudaError_t launch_chain<double>(const SwArgs<double> &, int, int, cudaStream_t);
template cudaError_t launch_scale_in<float>(const TileArgs &, const double *, double *, float *,
                                            const unsigned long long *, cudaStream_t);
template cudaError_t launch_scale_in<double>(const TileArgs &, const double *, double *, double *,
                                             const unsigned long long *, cudaStream_t);

}  // namespace fps
