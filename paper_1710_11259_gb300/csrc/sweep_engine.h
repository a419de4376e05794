// Host side of the square solve on the ADI pass kernels of sweep.cu, for one
// problem or a batch of squares of different sizes (internal header).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "resident.cuh"
#include "sweep.cuh"

namespace fps {

// T = float: FP32 sweeps inside an FP64 iterative refinement (tolerance levels,
//            residual R~ = F~ - A~Y - YA~ in FP64, Y -= s D / ky with s a power of two).
// T = double: the plain FP64 method, J iterations of (2.9) at the plan's tolerance.
template <typename T>
class SweepEngine {
public:
    // `ns`: problem sizes (caller packing: problem after problem, each problem's nrhs
    // n x n matrices back to back).  `tight`: shifts from the Sturm-bisection interval
    // of A~ instead of Lemma B.2's.  `seg`: segment length of the partitioned sweeps,
    // counted in unknowns of both parities
    // (64 or 128 for FP32, 64 for FP64); seg <= 0 lets the autotuner pick it (FP32).
    // Returns an fps_status; on error `err` holds a message.
    // kx, ky: scales of the second derivatives along x and y (a kx^{-1/2} x ky^{-1/2}
    // rectangle of half-widths; 1, 1 on [-1,1]^2).
    int create(const std::vector<int64_t> &ns, int nrhs, double tol, bool tight, cudaStream_t setup_stream,
               std::string &err, int seg = 0, double kx = 1.0, double ky = 1.0);
    void release();

    // Solve for device pointers F, X (packed as above) on stream st.  FP32: returns
    // FPS_ERR_NOT_CONVERGED with the last iterate in X when the refinement misses tol.
    int solve(const double *F, double *X, cudaStream_t st, std::string &err);

    // Whether a bounded device wait of a finished solve gave up.  Nothing clears it: the
    // plan's later solves return FPS_ERR_TIMEOUT.
    bool timed_out() const { return h_stat_ && (unsigned)*(volatile unsigned long long *)(h_stat_ + 2 * npairs_) != 0; }

    int set_instrument(bool on, std::string &err);
    // ADI pass kernels (row and column passes) of the last solve: launches, summed
    // duration, and the bytes they must move (6 words per element and iteration: u, a and
    // D read and written once; 5 in the first and the last).  Resident problems have none.
    int kernel_times(int *count, double *total_ms, double *alg_bytes, double *row_ms, double *col_ms,
                     std::string &err);

    int64_t bytes = 0;
    int J_first = 0;             // iterations of the finest level for the largest problem
    int rounds_last = 0;
    double resid_last = 0.0;     // largest max|R~|/max|F~| after the last solve (FP32)
    int64_t launches_last = 0;
    int max_rounds = 8;
    std::vector<std::vector<double>> shifts;  // level-0 shifts per problem
    int seg_len = 0;                          // segment length in use
    int chain_mode = 0;                       // segments per thread of the chain kernel (chain_length)
    std::vector<float> tune_ms;               // autotuner timings per candidate (ms), if it ran
    int64_t total_elems() const { return tot64_; }

private:
    using T2 = typename Vec2<T>::type;
    // Problems whose quarters stay in one cluster's shared memory (resident.cuh), by
    // segment length and cluster size: one launch of all their iterations.
    struct ResClass {
        int S, C;
        ResItem<T> *items = nullptr;
        int64_t nitems = 0;
    };
    struct Level {
        double tol = 0;
        int Jstream = 0;  // largest J of the streamed problems
        std::vector<int> J;
        T *tab = nullptr, *ch = nullptr;  // solve and summary tables, segment coefficients: rows, then columns
        T *res_tab = nullptr;             // records of the resident problems, likewise
        SwItem<T> *items[3] = {nullptr, nullptr, nullptr};  // row passes, column passes, recurrences
        int64_t nitems[3] = {0, 0, 0};
        std::vector<ResClass> res;
        int64_t launches = 0;             // kernels of the graph
        cudaGraphExec_t graph = nullptr;
        std::vector<cudaEvent_t> ev;  // when instrumented: 4 per iteration of the passes
    };
    int build_graph(Level &L, std::string &err);
    int autotune(const std::vector<int64_t> &ns, int nrhs, double tol, bool tight, std::string &err);
    int time_level(size_t li, int reps, float &ms, std::string &err);
    int time_chain(int mode, float &ms, std::string &err);
    SwArgs<T> args(const Level &L, int which) const;
    ResArgs<T> res_args(const ResClass &c, const double *F, double *X) const;
    struct TableJobs {
        std::vector<FacJob<T>> fac;
        std::vector<ResTabJob<T>> res;
    };
    int build_tables(Level &L, int level, const std::vector<double> &lo, const std::vector<double> &hi,
                     TableJobs &tables, std::string &err);
    int run_table_jobs(const TableJobs &jobs, std::string &err);
    cudaError_t run_resident(const Level &L, const double *F, double *X, cudaStream_t st, bool busy, int64_t &launches);
    cudaError_t join_resident(cudaStream_t st);
    // branches of the resident launches (streams of this engine, joined by every solve)
    static constexpr int kSide = 8;
    struct Side {
        cudaStream_t st = nullptr;
        cudaEvent_t done = nullptr;
    };
    std::vector<Side> side_;
    cudaEvent_t fork_ = nullptr;
    int side_used_ = 0;
    enum { kLive, kPadded, kResidual };  // tile lists (sweep.cuh)
    TileArgs tiles(int which) const;
    void set_active();
    int solve_refine(const double *F, double *X, cudaStream_t st, std::string &err);
    int solve_plain(const double *F, double *X, cudaStream_t st, std::string &err);

    std::vector<int64_t> ns_;
    int nrhs_ = 1;
    double tol_ = 0;
    double kx_ = 1.0, ky_ = 1.0;
    cudaStream_t cap_ = nullptr;
    std::vector<int> nb_;      // blocks per side of a quarter (of 32 for resident problems)
    std::vector<int> res_s_;   // resident problems: segment length; 0: streamed by the passes
    bool streams_ = false;     // any problem is streamed
    bool graphs() const { return sizeof(T) == 4 || streams_; }  // otherwise one launch per class, outside a graph
    int max_nb_ = 0;
    bool fused_ = false;   // the passes run the segment recurrences
    std::vector<int64_t> off64_, offT_, offS_;
    int64_t tot64_ = 0, totT_ = 0, totS_ = 0;
    int npairs_ = 0;
    double *Ft_ = nullptr, *Y0_ = nullptr, *Y1_ = nullptr, *bands64_ = nullptr;
    T *X_ = nullptr, *D_ = nullptr;
    T2 *sumR_ = nullptr, *sumC_ = nullptr, *zxR_ = nullptr, *zxC_ = nullptr;
    int *err_ = nullptr;
    TileProb *d_tp_ = nullptr;
    int4 *d_tiles_[3] = {nullptr, nullptr, nullptr};
    int64_t ntiles_[3] = {0, 0, 0};
    int *d_active_ = nullptr, *d_pair_active_ = nullptr;
    int *h_active_ = nullptr, *h_pair_active_ = nullptr;
    unsigned long long *d_stat_ = nullptr, *h_stat_ = nullptr;  // rmax, smax [npairs], error word
    std::vector<Level> levels_;
    std::vector<int64_t> ob64_;  // offset of each problem's bands in bands64_
    std::vector<int> order_;     // problems, largest first
    std::vector<int> levels_used_;
    bool instrument_ = false;
    bool wait_fault_ = false;  // fault injection (host_math.h)
    std::vector<void *> allocs_;

    template <typename U>
    cudaError_t dalloc(U **p, size_t count);
};

}  // namespace fps
