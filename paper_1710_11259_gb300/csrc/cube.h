// Nested ADI for the cube (Sec. 5) (internal header).
//
// The nested ADI runs the three levels of Sec. 5 on the symmetrised tensor equation
// (T_01 + T_02 + T_12) Y = G; its schedule (every shift of every level) is fixed at plan
// time.  CubeEngine is the plan object: FP64 runs the nested ADI once at the requested
// tolerance in the paper's form (CubeNested, inner and middle levels to 1e-15); FP32 +
// refinement runs it in FP32 at loose tolerances, every level in residual-propagating form
// (CubeRounds), inside an FP64 defect-correction loop on the residual
// G - (T_01 + T_02 + T_12) Y.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "cube_unit.cuh"

namespace fps {

// Shifts of every level and the device memory of a nested ADI.
class CubeSchedule {
public:
    void release();

    int J_outer = 0;
    int64_t inner_per_run = 0;   // inner (slice Stein) iterations over full tensors per run
    int64_t launches = 0;        // kernel launches of the last run
    int64_t bytes = 0;

protected:
    struct Stein {
        double c = 0;
        int J = 0;
        int64_t off = 0;         // of this entry in its class's device tables
        std::vector<double> p, q;
    };
    struct Middle {
        double a = 0;
        int stein = 0;
    };
    struct Outer {
        double p = 0, q = 0;
        int stein_v = 0;
        std::vector<Middle> mid;
    };
    // tol: outer tolerance of (2.9); tol_mid / tol_in: middle and inner levels; residual:
    // inner iterations counted for the residual-propagating form; tight: every level's
    // intervals from the Sturm-bisection interval of A~ instead of Lemma B.2's
    // [-1, -1/(30 n^4)].
    void schedule(int64_t n, double tol, double tol_mid, double tol_in, bool residual, bool tight);
    int add_stein(double c);
    cudaError_t alloc(void **p, size_t b);
    cudaError_t copy(void **p, const void *src, size_t b);  // alloc and upload

    int64_t n_ = 0;
    double tol_in_ = 0;
    double lo_ = 0, hi_ = 1;     // sigma(A~) in [-hi_, -lo_]
    cudaStream_t st_ = nullptr;
    double *bd_ = nullptr, *be_ = nullptr;
    std::vector<Stein> steins_;
    std::vector<Outer> outer_;
    std::vector<void *> allocs_;
};

// FP64, the paper's form: an error of one iteration is part of the next one's residual, so
// the solution keeps FP64 accuracy without refinement.
class CubeNested : public CubeSchedule {
public:
    int create(int64_t n, double tol, double tol_level, std::string &err);
    // Y = the nested-ADI approximation of (T_01 + T_02 + T_12)^{-1} G (device tensors).
    int run(const double *G, double *Y, cudaStream_t st, std::string &err);

private:
    cudaError_t band(const double *X, const double *R, double *Y, int mode, double alpha, double beta, double sop,
                     double sr);
    cudaError_t axpby(const double *X, const double *Y, double *Z, double a, double b);
    // X = (alpha A~ + beta)^{-1} (R1 + s2 R2) along `mode` (R2 may be null)
    cudaError_t solve(int set, const double *R1, const double *R2, double s2, double *X, int mode);
    int load_factors(int entry, std::string &err);
    int stein(int ma, int mb, int entry, const double *R, double *Z, std::string &err);
    int hsolve(const Outer &o, const double *R, double *Y, std::string &err);

    double *work_[8] = {nullptr};
    double2 *fac_ = nullptr;     // factor sets of the current Stein entry ({1/den, u})
    double2 *ab_ = nullptr;      // (alpha, beta) of every factor set of every Stein entry
    int entry_ = -1;             // entry whose factors fac_ holds (stream order makes reuse safe)
};

// FP32, every level in residual-propagating form; tensors have mode 0 fastest, (i, j, k) at
// (j n + k) n + i.
class CubeRounds : public CubeSchedule {
public:
    int create(int64_t n, double tol, double tol_mid, double tol_in, std::string &err);
    int run(const float *G, float *Y, cudaStream_t st, std::string &err);

private:
    int stein(int ma, int mb, int entry, const UnitJob *jobs, int njobs, std::string &err);
    int hsolve_res(const Outer &o, const float *R, float *W, std::string &err);

    float *work_[4] = {nullptr};
    int unit_ = 0;               // half line length of the inner level's kernel
    float *tab_ = nullptr, *bands_ = nullptr;  // its tables, every Stein entry
    UnitEntry *entries_ = nullptr;
    double2 *pq_ = nullptr;
};

class CubeEngine {
public:
    // precision: FPS_FP64 or FPS_FP32_REFINE (fps.h).
    int create(int64_t n, double tol, int precision, std::string &err);
    void release();
    // X = solution of (5.2) for F (device pointers, n^3 row-major) on stream st.
    int solve_cube(const double *F, double *X, cudaStream_t st, std::string &err);

    int64_t bytes = 0;
    int J_outer = 0;
    int J_outer_inner = 0;       // FP32 + refinement: J of the outer level inside a round
    int64_t inner_iters = 0;     // inner iterations over full tensors in the last solve
    int64_t launches_last = 0;
    int rounds_last = 0;
    double resid_last = 0.0;     // max|G - T Y| / max|G| after the last solve (FP32 + refinement)
    int max_rounds = 12;

    // Level tolerances of the FP32 rounds: middle and inner fixed; the outer one is
    // picked per plan from kRefTolOuter (refinement_outer_tol).
    static constexpr double kRefTolMid = 1e-6, kRefTolIn = 1e-7;
    static constexpr double kRefTolOuter[] = {1e-3, 7e-4, 5e-4, 3e-4, 2e-4, 1e-4};
    double ref_tol_outer = 1e-3;  // outer tolerance of the FP32 rounds in use

private:
    int64_t n_ = 0;
    double tol_ = 0;
    int precision_ = 0;
    CubeNested *n64_ = nullptr;
    CubeRounds *n32_ = nullptr;
    double *bd_ = nullptr, *be_ = nullptr, *bs_ = nullptr;
    double *G_ = nullptr, *Y_ = nullptr, *R_ = nullptr;
    float *rho_ = nullptr, *delta_ = nullptr;
    unsigned long long *d_max_ = nullptr, *h_max_ = nullptr;
    std::vector<void *> allocs_;
};

}  // namespace fps
