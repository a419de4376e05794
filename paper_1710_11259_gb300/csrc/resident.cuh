// All ADI iterations of a small square in one launch (internal header; the scheme and
// the notation are those of sweep.cuh).
//
// A quarter of at most 16 S unknowns per side stays in the shared memory of one cluster
// of ceil(m / S) <= 16 CTAs: CTA q holds S rows of u / a, D lives in registers, and every
// line is cut into 16 segments of S.  An iteration is
//   row solve     thread (row, segment), the 16 segments of a row on neighbouring lanes:
//                 two summaries per thread, the recurrence over the segments as warp
//                 scans, then the sweeps of the segment in registers (long FP32 segments:
//                 two rows, then two columns, per thread);
//   column solve  thread = column, the CTA's S rows are one segment: its summaries go to
//                 the CTA that owns the column, which runs the same scans and returns zin
//                 and yout to every CTA, then the sweeps.  Both ways each pair is an
//                 asynchronous store into the receiver's shared memory, counted by the
//                 receiver's mbarrier.
// Scans: with kf[t][s] = prod_{s-2^t < u <= s} phi(u) and kb[t][s] = prod_{s <= u < s+2^t}
// Psi(u), four steps W_s += kf[t][s] W_{s-2^t} and four backwards.
//
// Bound: the FP64 pipe in FP64 (a warp-wide FP64 instruction takes 64 cycles of an SM
// quadrant, so threads are laid out to do few of them: 16 segments per line, scans
// instead of one long recurrence), latency of the two exchanges and the sweeps in FP32.
// Measured on GB300 per solve: n = 64 FP64, two right-hand sides, 192 us (801 us with one
// cluster of 8 CTAs per right-hand side solving every line by cyclic reduction and
// exchanging whole iterates; 250 us with remote stores between cluster barriers, whose
// fences alone were a fifth of the time), n = 301 FP64 0.60 ms (2.5 ms streamed by the
// passes, 0.69 with cluster barriers), n = 1000 FP32+refine 0.50 ms (1.18 streamed, 0.56
// with cluster barriers, 0.53 with one line per thread).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace fps {

constexpr int kResSeg = 16;                    // segments per line, and the largest cluster
constexpr int kScan = 9 * kResSeg;             // kf[4], Bv, kb[4] of the segments

// Tables of one (shift, parity), elements of T.
// Row record: {psi, chi}[S][16], {m, scale}[S][16], l[(S + 1) / 2][16][2] (position i of
// segment g at [i][g], l at [i / 2][g][i % 2]), then the scan coefficients.  Column record:
// l, m, scale, psi, chi [5][16 S] in natural order, then the scan coefficients.
__host__ __device__ constexpr int res_scan_row(int S) { return kResSeg * (5 * S + S % 2); }
__host__ __device__ constexpr int res_scan_col(int S) { return kResSeg * 5 * S; }
__host__ __device__ constexpr int res_record(int S) { return res_scan_row(S) + kScan; }

// One quarter of one (problem, right-hand side).
template <typename T>
struct alignas(16) ResItem {
    int64_t xoff;            // quarter-block arrays: offset of the quarter (blocks of 32)
    int64_t foff;            // caller arrays: offset of the (problem, rhs) matrix
    const T *tabR, *tabC;    // [J][2][res_record(S)], offset to this quarter's parities
    const double *s;         // 1/sqrt(E), n entries
    double out_scale;        // X = out_scale D D_s (x) D_s
    int prob, J, n, lnb;     // lnb: blocks of 32 per side of the quarter-block arrays
    int rp, cp, pad[2];
};

template <typename T>
struct ResArgs {
    const ResItem<T> *items;
    int64_t nitems;
    int S, C;                // segment length, cluster size (segments in use)
    const int *active, *masked;
    T *X, *D;                // quarter-block arrays (F == nullptr)
    const double *F;         // caller's right-hand sides and solution: scale-in and -out in the launch
    double *out;
    int *err;                // set if a bounded wait gave up (device or pinned host memory)
    int give_up;             // fault injection: iteration in which the waits of CTA 0 give up (-1: none)
};

template <typename T>
struct ResTabJob {
    double q, sc_row, sc_col;  // shift; factors of ip in the two solution scales
    int n, S;
    const double *d, *e;       // FP64 bands, e zero-padded to length n
    T *row, *col;              // [2][res_record(S)] (parities); either may be null
};

// Segment length for quarters of m unknowns per side (0: too large for a cluster).
int resident_segment(bool fp64, int m);
inline int resident_cluster(int m, int S) { return (m + S - 1) / S; }
// Prepares the kernel; *side_by_side: clusters of it that the device runs at a time.
template <typename T>
cudaError_t resident_setup(int S, int C, int *side_by_side);
// Whether a problem of nrhs right-hand sides, four clusters each, runs in one launch rather than
// by the passes.  FP64 beyond n = 512 (S > 16) only while its clusters run at once (7 on GB300:
// one right-hand side): n = 513 1.93 ms (4.16 by the passes), 640 2.05 (4.58), 641 2.69 (4.57), 768
// 2.85 (4.67), but 5.36 against 4.72 for two right-hand sides at n = 641.
bool resident_pays(bool fp64, int S, int nrhs, int side_by_side);
template <typename T>
cudaError_t launch_resident_tables(const ResTabJob<T> *jobs, int njobs, cudaStream_t st);
template <typename T>
cudaError_t launch_resident(const ResArgs<T> &a, cudaStream_t st);

}  // namespace fps
