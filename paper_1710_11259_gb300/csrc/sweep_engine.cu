// Host side of the square solve on the ADI pass kernels (sweep.cu), one problem or
// a batch.
//
// FP32 (refinement), per solve:
//   smax = max |F~| per (problem, rhs) pair; F~ = D_s F D_s; s = 2^floor(log2 smax);
//   rho_0 = F~ / s
//   round r: inner ADI in FP32 (one CUDA graph per tolerance level: every pass
//            launch covers every problem) gives the correction -D/ky; the FP64
//            residual kernel applies Y -= s D/ky, forms
//            R~ = F~ - A~Y - YA~ and the next rho_0; pairs with max|R~| <= tol smax
//            stop (their iterate is carried unchanged).
//   X = D_s Y D_s.
// The inner tolerance of a round is the coarsest level that still gains ten times
// what the worst active pair is missing; the first round stops at the coarsest
// level not above sqrt(0.1 tol), so that two rounds of equal gain reach tol (the
// finest level, 1e-7, is about what one FP32 inner solve can deliver).  Inner shifts come from the
// tight spectral interval of A~ (the refinement is judged by the FP64 residual).
// Problems small enough for one cluster per quarter run all their iterations in one
// launch (resident.cuh); the others are streamed by the passes.
// FP64 (plain method): rho_0 = F~, one graph of J iterations of (2.9), then
// X = D_s Y_J D_s.
#include "sweep_engine.h"
#include "trace.h"

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <fstream>
#include <sstream>

#include <sys/stat.h>

#include "../../include/fps.h"
#include "host_math.h"

namespace fps {

namespace {
double bits_to_double(unsigned long long b)
{
    double d;
    std::memcpy(&d, &b, sizeof(d));
    return d;
}
const double kLevelTols[] = {1e-7, 1e-6, 1e-5, 1e-4, 1e-3, 1e-2};
const char kGaveUp[] = "a bounded device wait gave up (data not arrived)";
}  // namespace

template <typename T>
template <typename U>
cudaError_t SweepEngine<T>::dalloc(U **p, size_t count)
{
    *p = nullptr;
    if (!count) return cudaSuccess;
    cudaError_t e = cudaMalloc((void **)p, sizeof(U) * count);
    if (e == cudaSuccess) {
        bytes += (int64_t)(sizeof(U) * count);
        allocs_.push_back((void *)*p);
    }
    return e;
}

template <typename T>
void SweepEngine<T>::release()
{
    for (auto &L : levels_) {
        for (cudaEvent_t e : L.ev) cudaEventDestroy(e);
        if (L.graph) cudaGraphExecDestroy(L.graph);
    }
    levels_.clear();
    for (void *p : allocs_) cudaFree(p);
    allocs_.clear();
    for (Side &x : side_) {
        if (x.st) cudaStreamDestroy(x.st);
        cudaEventDestroy(x.done);
    }
    side_.clear();
    if (fork_) cudaEventDestroy(fork_);
    fork_ = nullptr;
    if (h_stat_) cudaFreeHost(h_stat_);
    h_active_ = h_pair_active_ = nullptr;
    h_stat_ = nullptr;
}

#define ENG_CK(call)                                                                                     \
    do {                                                                                                 \
        cudaError_t e_ = (call);                                                                         \
        if (e_ != cudaSuccess) {                                                                         \
            err = std::string(#call) + ": " + cudaGetErrorString(e_);                                    \
            return FPS_ERR_CUDA;                                                                         \
        }                                                                                                \
    } while (0)

// ---------------------------------------------------------------------------
// Autotuner of the segment length (unknowns of both parities: twice the block size of
// sweep.cuh; it also fixes the number of segments a recurrence walks).  Every
// candidate gets a complete engine of its own on the same sizes; the graph of the
// coarsest tolerance level is timed with CUDA events and the fastest candidate
// kept.  Results are cached per (GPU name, nrhs, size list) in $FPS_AUTOTUNE_CACHE
// (default ~/.cache/fps_gb300_autotune.txt); FPS_AUTOTUNE=0 skips tuning (128).
// ---------------------------------------------------------------------------
namespace {
std::string tune_key(const std::vector<int64_t> &ns, int nrhs)
{
    cudaDeviceProp prop;
    int dev = 0;
    cudaGetDevice(&dev);
    std::string name = "gpu";
    if (cudaGetDeviceProperties(&prop, dev) == cudaSuccess) name = prop.name;
    for (char &c : name)
        if (c == ' ') c = '_';
    uint64_t h = 1469598103934665603ULL;  // FNV-1a over the sizes
    for (int64_t n : ns) {
        for (int b = 0; b < 8; ++b) {
            h ^= (uint64_t)((n >> (8 * b)) & 0xff);
            h *= 1099511628211ULL;
        }
    }
    std::ostringstream os;
    os << "blk|" << name << "|" << nrhs << "|" << ns.size() << "|" << std::hex << h;
    return os.str();
}

std::string tune_cache_path()
{
    const char *p = std::getenv("FPS_AUTOTUNE_CACHE");
    if (p && *p) return p;
    const char *home = std::getenv("HOME");
    return std::string(home ? home : "/tmp") + "/.cache/fps_gb300_autotune.txt";
}
}  // namespace

// Entries per segment-coefficient array: 16-byte multiples for the bulk copies.
static int nbp_of(int nb) { return (nb + 3) & ~3; }

template <typename T>
TileArgs SweepEngine<T>::tiles(int which) const
{
    TileArgs t;
    t.probs = d_tp_;
    t.tiles = d_tiles_[which];
    t.ntiles = ntiles_[which];
    return t;
}

// Problems with an active pair, and whether any problem is inactive.
template <typename T>
void SweepEngine<T>::set_active()
{
    const int np = (int)ns_.size();
    h_active_[np] = 0;
    for (int p = 0; p < np; ++p) {
        h_active_[p] = 0;
        for (int r = 0; r < nrhs_; ++r) h_active_[p] |= h_pair_active_[p * nrhs_ + r];
        if (!h_active_[p]) h_active_[np] = 1;
    }
}

template <typename T>
int SweepEngine<T>::time_level(size_t li, int reps, float &ms, std::string &err)
{
    cudaEvent_t e0, e1;
    ENG_CK(cudaEventCreate(&e0));
    ENG_CK(cudaEventCreate(&e1));
    ENG_CK(cudaGraphLaunch(levels_[li].graph, cap_));  // warm-up
    ENG_CK(cudaEventRecord(e0, cap_));
    for (int r = 0; r < reps; ++r) ENG_CK(cudaGraphLaunch(levels_[li].graph, cap_));
    ENG_CK(cudaEventRecord(e1, cap_));
    ENG_CK(cudaEventSynchronize(e1));
    ENG_CK(cudaEventElapsedTime(&ms, e0, e1));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    ms /= (float)reps;
    return FPS_OK;
}

// Mean time of a chain launch (both directions alternately) with the given load
// batching, on this engine's arrays (the values do not change the time); 0 where the
// passes run the recurrences themselves.
template <typename T>
int SweepEngine<T>::time_chain(int mode, float &ms, std::string &err)
{
    SwArgs<T> a = args(levels_.back(), 2);
    ms = 0.f;
    if (a.fused) return FPS_OK;
    a.chain_len = chain_length(sizeof(T) == 8, mode, max_nb_);
    cudaEvent_t e0, e1;
    ENG_CK(cudaEventCreate(&e0));
    ENG_CK(cudaEventCreate(&e1));
    ENG_CK(launch_chain(a, 0, 0, cap_));  // warm-up
    ENG_CK(cudaEventRecord(e0, cap_));
    constexpr int kReps = 20;
    for (int r = 0; r < kReps; ++r) ENG_CK(launch_chain(a, r & 1, 0, cap_));
    ENG_CK(cudaEventRecord(e1, cap_));
    ENG_CK(cudaEventSynchronize(e1));
    ENG_CK(cudaEventElapsedTime(&ms, e0, e1));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    ms /= (float)kReps;
    return FPS_OK;
}

template <typename T>
int SweepEngine<T>::autotune(const std::vector<int64_t> &ns, int nrhs, double tol, bool tight, std::string &err)
{
    seg_len = 128;
    const char *env = std::getenv("FPS_AUTOTUNE");
    if (env && std::string(env) == "0") return FPS_OK;
    const std::string key = tune_key(ns, nrhs);
    const std::string path = tune_cache_path();
    {
        std::ifstream in(path);
        std::string line;
        while (std::getline(in, line)) {
            std::istringstream ls(line);
            std::string k;
            int v = 0, cm = 0;
            if (!(ls >> k >> v)) continue;
            if (!(ls >> cm) || cm < 0 || cm > 2) cm = 0;  // entries without a chain mode: by grid size
            if (k == key && sweep_segment_supported(false, v)) {
                seg_len = v;
                chain_mode = cm;
                return FPS_OK;
            }
        }
    }
    auto remember = [&]() {
        const size_t slash = path.find_last_of('/');
        if (slash != std::string::npos && slash > 0) mkdir(path.substr(0, slash).c_str(), 0755);  // may exist
        std::ofstream out(path, std::ios::app);
        if (out) out << key << " " << seg_len << " " << chain_mode << "\n";
    };
    if (!streams_) {  // no pass runs: nothing to time
        chain_mode = 1;
        remember();
        return FPS_OK;
    }
    // tile shape: the segment length of the passes (a whole graph level timed per
    // candidate); then the chain kernel's load batching, timed on the winner's arrays
    const int cand[] = {64, 128};
    float best = 3.4e38f;
    tune_ms.clear();
    for (int S : cand) {
        SweepEngine<T> t;
        std::string e2;
        int st = t.create(ns, nrhs, tol, tight, cap_, e2, S, kx_, ky_);
        float ms = 0.f, c1 = 0.f, c2 = 0.f;
        if (st == FPS_OK) st = t.time_level(t.levels_.size() - 1, 2, ms, e2);
        if (st == FPS_OK) st = t.time_chain(1, c1, e2);
        if (st == FPS_OK) st = t.time_chain(2, c2, e2);
        t.release();
        if (st != FPS_OK) {
            err = "autotune: " + e2;
            return st;
        }
        tune_ms.push_back(ms);
        if (ms < best) {
            best = ms;
            seg_len = S;
            chain_mode = c2 < c1 ? 2 : 1;
        }
    }
    remember();
    return FPS_OK;
}

template <typename T>
int SweepEngine<T>::create(const std::vector<int64_t> &ns, int nrhs, double tol, bool tight,
                           cudaStream_t setup_stream, std::string &err, int seg, double kx, double ky)
{
    kx_ = kx;
    ky_ = ky;
    constexpr bool kFP64 = sizeof(T) == 8;
    ns_ = ns;
    nrhs_ = nrhs;
    tol_ = tol;
    cap_ = setup_stream;
    const int np = (int)ns.size();
    if (const char *mr = std::getenv("FPS_MAX_REFINE_ROUNDS")) {  // cap on refinement rounds (>= 1)
        const int v = std::atoi(mr);
        if (v >= 1) max_rounds = v;
    }
    wait_fault_ = inject_wait_fault();
    res_s_.assign(np, 0);
    streams_ = false;
    for (int p = 0; p < np; ++p) {
        const int m = (int)((ns[p] + 1) / 2), rs = resident_segment(kFP64, m);
        int side_by_side = 0;
        if (rs > 0) ENG_CK(resident_setup<T>(rs, resident_cluster(m, rs), &side_by_side));
        if (resident_pays(kFP64, rs, nrhs, side_by_side)) res_s_[p] = rs;
        else streams_ = true;
    }
    if (seg <= 0) {
        if (kFP64) {
            seg_len = 64;
        } else {
            const int st = autotune(ns, nrhs, tol, tight, err);
            if (st != FPS_OK) return st;
        }
    } else {
        if (!sweep_segment_supported(kFP64, seg)) {
            err = "unsupported segment length";
            return FPS_ERR_INVALID_ARG;
        }
        seg_len = seg;
    }
    const int S = seg_len / 2;  // block size: unknowns of one parity
    nb_.resize(np);
    off64_.resize(np);
    offT_.resize(np);
    offS_.resize(np);
    tot64_ = totT_ = totS_ = 0;
    max_nb_ = 0;
    int64_t totB64 = 0;
    for (int p = 0; p < np; ++p) {
        const int64_t n = ns[p];
        const int Sp = res_s_[p] ? 32 : S;
        const int64_t nb = ((n + 1) / 2 + Sp - 1) / Sp;
        nb_[p] = (int)nb;
        off64_[p] = tot64_;
        offT_[p] = totT_;
        offS_[p] = totS_;
        tot64_ += (int64_t)nrhs * n * n;
        totT_ += (int64_t)nrhs * 4 * nb * nb * Sp * Sp;
        if (!res_s_[p]) {
            max_nb_ = std::max(max_nb_, (int)nb);
            totS_ += (int64_t)nrhs * 4 * nb * nb * S;
        }
        totB64 += 7 * n;
    }
    fused_ = sweep_fused(kFP64, S, max_nb_);
    npairs_ = np * nrhs;

    if (streams_) ENG_CK(sweep_setup_kernels());
    if (!kFP64) {
        ENG_CK(dalloc(&Ft_, (size_t)totT_));  // quarter blocks, as X and D
        ENG_CK(dalloc(&Y0_, (size_t)totT_));
        ENG_CK(dalloc(&Y1_, (size_t)totT_));
    }
    ENG_CK(dalloc(&bands64_, (size_t)totB64));
    // FP64 plans that stream nothing work on the caller's arrays (solve_plain): no X, D, graph
    const size_t elems = graphs() ? (size_t)totT_ : 0;
    ENG_CK(dalloc(&X_, elems));
    ENG_CK(dalloc(&D_, elems));
    ENG_CK(dalloc(&sumR_, (size_t)totS_));
    ENG_CK(dalloc(&sumC_, (size_t)totS_));
    if (!fused_) {
        ENG_CK(dalloc(&zxR_, (size_t)totS_));
        ENG_CK(dalloc(&zxC_, (size_t)totS_));
    }
    ENG_CK(dalloc(&d_active_, (size_t)np + 1));
    ENG_CK(dalloc(&d_pair_active_, (size_t)npairs_));
    // what a round reports, read back in one copy: rmax and smax per pair, the error word
    ENG_CK(dalloc(&d_stat_, 2 * (size_t)npairs_ + 1));
    err_ = (int *)(d_stat_ + 2 * npairs_);
    // one pinned block: statistics, then the masks (of the problems: last, any problem inactive)
    const size_t stat_words = 2 * (size_t)npairs_ + 1;
    ENG_CK(cudaMallocHost((void **)&h_stat_, sizeof(unsigned long long) * stat_words + sizeof(int) * (np + 1 + npairs_)));
    h_active_ = (int *)(h_stat_ + stat_words);
    h_pair_active_ = h_active_ + np + 1;
    h_stat_[2 * npairs_] = 0;
    // unused positions must be zero and stay zero
    auto zero = [&](void *p, size_t b) { return b ? cudaMemsetAsync(p, 0, b, cap_) : cudaSuccess; };
    ENG_CK(zero(X_, sizeof(T) * elems));
    ENG_CK(zero(D_, sizeof(T) * elems));
    ENG_CK(zero(sumR_, sizeof(T2) * (size_t)totS_));
    ENG_CK(zero(sumC_, sizeof(T2) * (size_t)totS_));
    ENG_CK(cudaMemsetAsync(d_stat_, 0, sizeof(unsigned long long) * (2 * (size_t)npairs_ + 1), cap_));
    if (wait_fault_ && streams_) ENG_CK(cudaMemsetAsync(err_, 1, 1, cap_));  // as if a pass had given up

    // bands: FP64 (d, e zero-padded, 1/sqrt(E), then {-kx d, -ky d} and {-kx e, -ky e})
    std::vector<double> hb64((size_t)totB64);
    std::vector<TileProb> tp(np);
    std::vector<int4> tiles[3];  // live region, padded region, residual
    ob64_.resize(np);
    {
        int64_t o64 = 0;
        std::vector<double> d, e, s;
        for (int p = 0; p < np; ++p) {
            const int64_t n = ns[p];
            square_bands(n, d, e);
            inv_sqrt_E(n, s);
            std::copy(d.begin(), d.end(), hb64.begin() + o64);
            std::copy(e.begin(), e.end(), hb64.begin() + o64 + n);
            std::copy(s.begin(), s.end(), hb64.begin() + o64 + 2 * n);
            for (int64_t i = 0; i < n; ++i) {
                hb64[o64 + 3 * n + i] = -kx_ * d[i];
                hb64[o64 + 4 * n + i] = -ky_ * d[i];
                hb64[o64 + 5 * n + i] = -kx_ * e[i];
                hb64[o64 + 6 * n + i] = -ky_ * e[i];
            }
            ob64_[p] = o64;
            TileProb &t = tp[p];
            t.n = (int)n;
            t.nb = nb_[p];
            t.log_s = res_s_[p] || S == 32 ? 5 : 6;
            t.off64 = off64_[p];
            t.off = offT_[p];
            t.rhs = 4 * (int64_t)nb_[p] * nb_[p] << (2 * t.log_s);
            t.s = bands64_ + o64 + 2 * n;
            t.nd = bands64_ + o64 + 3 * n;
            t.ne = bands64_ + o64 + 5 * n;
            t.pair0 = p * nrhs;
            t.inv_ky = 1.0 / ky_;
            o64 += 7 * n;
            const int m = (int)((n + 1) / 2), nt = (m + 31) / 32, ntp = (nb_[p] << t.log_s) / 32;
            for (int r = 0; r < nrhs && graphs(); ++r) {
                const int id = p * 256 + r;
                for (int ty = 0; ty < nt; ++ty)
                    for (int tx = 0; tx < nt; ++tx) tiles[0].push_back(make_int4(id, tx, ty, 0));
                for (int ty = 0; ty < ntp; ++ty)
                    for (int tx = 0; tx < ntp; ++tx) tiles[1].push_back(make_int4(id, tx, ty, 0));
                if (!kFP64)
                    for (int q = 0; q < 4; ++q)
                        for (int ty = 0; ty < (m + 63) / 64; ++ty)
                            for (int tx = 0; tx < nt; ++tx) tiles[2].push_back(make_int4(id, tx * 4 + q, ty, 0));
            }
        }
    }
    ENG_CK(dalloc(&d_tp_, (size_t)np));
    for (int w = 0; w < 3; ++w) {
        ntiles_[w] = (int64_t)tiles[w].size();
        if (tiles[w].empty()) continue;
        ENG_CK(dalloc(&d_tiles_[w], tiles[w].size()));
        ENG_CK(cudaMemcpyAsync(d_tiles_[w], tiles[w].data(), sizeof(int4) * tiles[w].size(), cudaMemcpyHostToDevice, cap_));
    }
    ENG_CK(cudaMemcpyAsync(bands64_, hb64.data(), sizeof(double) * totB64, cudaMemcpyHostToDevice, cap_));
    ENG_CK(cudaMemcpyAsync(d_tp_, tp.data(), sizeof(TileProb) * np, cudaMemcpyHostToDevice, cap_));

    order_.resize(np);
    for (int p = 0; p < np; ++p) order_[p] = p;
    std::stable_sort(order_.begin(), order_.end(), [&](int x, int y) { return ns[x] > ns[y]; });
    for (int p = 0; p < np; ++p) h_active_[p] = 1;
    h_active_[np] = 0;
    for (int k = 0; k < npairs_; ++k) h_pair_active_[k] = 1;
    ENG_CK(cudaMemcpyAsync(d_active_, h_active_, sizeof(int) * (np + 1), cudaMemcpyHostToDevice, cap_));
    ENG_CK(cudaMemcpyAsync(d_pair_active_, h_pair_active_, sizeof(int) * npairs_, cudaMemcpyHostToDevice, cap_));

    // tolerance levels: shifts, per-shift tables (FP64 arithmetic on the device)
    std::vector<double> lo(np), hi(np);
    for (int p = 0; p < np; ++p) {
        if (tight) square_tight_interval(ns[p], lo[p], hi[p]);
        else {
            lo[p] = square_eps(ns[p]);
            hi[p] = 1.0;
        }
    }
    std::vector<double> tols;
    if (kFP64) tols.push_back(tol);
    else tols.assign(std::begin(kLevelTols), std::end(kLevelTols));
    shifts.assign(np, {});
    TableJobs jobs;
    for (size_t li = 0; li < tols.size(); ++li) {
        levels_.emplace_back();
        levels_.back().tol = tols[li];
        const int st = build_tables(levels_.back(), (int)li, lo, hi, jobs, err);
        if (st != FPS_OK) return st;
    }
    {
        const int st = run_table_jobs(jobs, err);
        if (st != FPS_OK) return st;
    }
    {
        int big = 0;
        for (int p = 0; p < np; ++p)
            if (ns[p] > ns[big]) big = p;
        J_first = levels_[0].J[big];
    }
    for (auto &L : levels_) {
        int st = build_graph(L, err);
        if (st != FPS_OK) return st;
    }
    return FPS_OK;
}

// The tables of all levels: a thread walks a whole line, so one launch of every level's jobs
// takes as long as the longest line, where a launch per level took that six times over
// (n = 1000 3.5 ms of the plan, n = 2048 6 ms).
template <typename T>
int SweepEngine<T>::run_table_jobs(const TableJobs &jobs, std::string &err)
{
    struct Scratch {  // device copies of the job lists
        void *p[2] = {nullptr, nullptr};
        ~Scratch()
        {
            for (void *q : p)
                if (q) cudaFree(q);
        }
    } scratch;
    cudaError_t e1 = cudaSuccess;
    auto upload = [&](int slot, const void *src, size_t bytes) -> void * {
        if (e1 == cudaSuccess) e1 = cudaMalloc(&scratch.p[slot], bytes);
        if (e1 == cudaSuccess) e1 = cudaMemcpyAsync(scratch.p[slot], src, bytes, cudaMemcpyHostToDevice, cap_);
        return scratch.p[slot];
    };
    if (!jobs.fac.empty()) {
        const FacJob<T> *d = (const FacJob<T> *)upload(0, jobs.fac.data(), sizeof(FacJob<T>) * jobs.fac.size());
        if (e1 == cudaSuccess) e1 = launch_fac_tables<T>(d, (int)jobs.fac.size(), cap_);
    }
    if (!jobs.res.empty()) {
        const ResTabJob<T> *d = (const ResTabJob<T> *)upload(1, jobs.res.data(), sizeof(ResTabJob<T>) * jobs.res.size());
        if (e1 == cudaSuccess) e1 = launch_resident_tables<T>(d, (int)jobs.res.size(), cap_);
    }
    // the scratch must outlive the asynchronous work
    const cudaError_t e2 = cudaStreamSynchronize(cap_);
    ENG_CK(e1);
    ENG_CK(e2);
    return FPS_OK;
}

// Shifts and work items of one tolerance level; its tables go on the job lists.
template <typename T>
int SweepEngine<T>::build_tables(Level &L, int level, const std::vector<double> &lo, const std::vector<double> &hi,
                                 TableJobs &tables, std::string &err)
{
    const int np = (int)ns_.size(), S = seg_len / 2;
    // intervals of kx A~ (row side) and -ky A~ (column side): [a, b] = -kx [hi, lo],
    // [c, d] = ky [lo, hi]; on a square (kx = ky) the symmetric route gives p = -q and one
    // set of factors serves rows and columns
    const bool sym = kx_ == ky_;
    L.J.resize(np);
    int64_t nfac = 0, nch = 0, nres = 0;  // elements of one direction's tables, coefficients, records
    int nq = 0, nq_res = 0;               // shifts of the streamed and of the resident problems
    for (int p = 0; p < np; ++p) {
        L.J[p] = adi_iterations(-kx_ * hi[p], -kx_ * lo[p], ky_ * lo[p], ky_ * hi[p], L.tol);
        if (res_s_[p]) {
            nres += (int64_t)L.J[p] * 2 * res_record(res_s_[p]);
            nq_res += L.J[p];
        } else {
            L.Jstream = std::max(L.Jstream, L.J[p]);
            nfac += (int64_t)L.J[p] * 2 * kTabs * nb_[p] * S;
            nch += (int64_t)L.J[p] * 2 * 3 * nbp_of(nb_[p]);
            nq += L.J[p];
        }
    }
    ENG_CK(dalloc(&L.tab, (size_t)(2 * nfac)));
    ENG_CK(dalloc(&L.ch, (size_t)(2 * nch)));
    ENG_CK(dalloc(&L.res_tab, (size_t)(2 * nres)));
    std::vector<FacJob<T>> &jobs = tables.fac;
    std::vector<ResTabJob<T>> &rjobs = tables.res;
    jobs.reserve(jobs.size() + (size_t)nq * 2);
    rjobs.reserve(rjobs.size() + (size_t)nq_res * 2);
    std::vector<int64_t> otab(np), och(np);  // offsets of a problem's tables (records) and coefficients
    int64_t of = 0, oc = 0, ores = 0;
    std::vector<double> q, pp;
    for (int p = 0; p < np; ++p) {
        const int64_t n = ns_[p];
        const double a = -kx_ * hi[p], b = -kx_ * lo[p], c = ky_ * lo[p], d = ky_ * hi[p];
        if (sym) {
            zolotarev_shifts_symmetric(lo[p], hi[p], L.J[p], q);
            pp.resize(q.size());
            for (size_t u = 0; u < q.size(); ++u) {
                q[u] *= kx_;
                pp[u] = -q[u];
            }
        } else {
            zolotarev_shifts(a, b, c, d, L.J[p], pp, q);
        }
        inject_shift_fault(q);
        std::vector<double> mp(pp.size());
        for (size_t u = 0; u < pp.size(); ++u) mp[u] = -pp[u];
        if (!shifts_valid(q, c, d) || !shifts_valid(mp, -b, -a)) {
            err = "shift list failed validation (a shift is not finite or lies outside the spectral interval)";
            return FPS_ERR_INVALID_ARG;
        }
        if (level == 0) shifts[p] = q;
        otab[p] = res_s_[p] ? ores : of;
        och[p] = oc;
        const double *bd = bands64_ + ob64_[p], *be = bd + n;
        for (int j = 0; j < L.J[p]; ++j) {
            // row solve, shift -p_j/ky: a = u + (q_{j-1} - p_j)/ky v;
            // column solve, shift q_j/kx: t = (q_j - p_j)/kx c
            const double q_row = -pp[j] / ky_, sc_row = j == 0 ? 1.0 : (q[j - 1] - pp[j]) / ky_;
            const double q_col = q[j] / kx_, sc_col = (q[j] - pp[j]) / kx_;
            if (res_s_[p]) {
                const int64_t ts = 2 * (int64_t)res_record(res_s_[p]);
                T *row = L.res_tab + ores + j * ts, *col = row + nres;
                ResTabJob<T> jb{q_row, sc_row, sc_col, (int)n, res_s_[p], bd, be, row, sym ? col : nullptr};
                rjobs.push_back(jb);
                if (!sym) {
                    jb.q = q_col;
                    jb.row = nullptr;
                    jb.col = col;
                    rjobs.push_back(jb);
                }
                continue;
            }
            const int nb = nb_[p];
            const int64_t ts = 2 * (int64_t)kTabs * nb * S, cs = 2 * 3 * (int64_t)nbp_of(nb);
            T *row = L.tab + of + j * ts, *col = row + nfac, *ch_row = L.ch + oc + j * cs, *ch_col = ch_row + nch;
            FacJob<T> jb{q_row, sc_row, sc_col, (int)n, nb, S, bd, be, row, sym ? col : nullptr,
                         ch_row, sym ? ch_col : nullptr};
            jobs.push_back(jb);
            if (!sym) {
                jb.q = q_col;
                jb.sc1 = sc_col;
                jb.out1 = col;
                jb.ch1 = ch_col;
                jobs.push_back(jb);
            }
        }
        if (res_s_[p]) {
            ores += L.J[p] * 2 * (int64_t)res_record(res_s_[p]);
        } else {
            of += L.J[p] * 2 * (int64_t)kTabs * nb_[p] * S;
            oc += L.J[p] * 2 * 3 * (int64_t)nbp_of(nb_[p]);
        }
    }
    // work items of the row passes, the column passes and the recurrences; resident items
    std::vector<SwItem<T>> it[3];
    std::vector<std::vector<ResItem<T>>> rit;
    const int R = kPassLines / S;
    for (int p : order_) {
        const int nb = nb_[p], rs = res_s_[p], Sp = rs ? 32 : S;
        const int64_t quarter = (int64_t)nb * nb * Sp * Sp, squarter = (int64_t)nb * nb * S;
        size_t rc = 0;
        if (rs) {
            const int C = resident_cluster((int)((ns_[p] + 1) / 2), rs);
            while (rc < L.res.size() && (L.res[rc].S != rs || L.res[rc].C != C)) ++rc;
            if (rc == L.res.size()) {
                ResClass c;
                c.S = rs;
                c.C = C;
                L.res.push_back(c);
                rit.emplace_back();
            }
        }
        for (int r = 0; r < nrhs_; ++r)
            for (int qd = 0; qd < 4; ++qd) {
                const int rp = qd >> 1, cp = qd & 1;
                if (ns_[p] <= std::max(rp, cp)) continue;  // n = 1: one quarter only
                const int64_t x0 = offT_[p] + ((int64_t)r * 4 + qd) * quarter;
                if (rs) {
                    ResItem<T> x;
                    x.xoff = x0;
                    x.foff = off64_[p] + (int64_t)r * ns_[p] * ns_[p];
                    x.tabR = L.res_tab + otab[p] + cp * res_record(rs);
                    x.tabC = L.res_tab + nres + otab[p] + rp * res_record(rs);
                    x.s = bands64_ + ob64_[p] + 2 * ns_[p];
                    x.out_scale = -1.0 / ky_;
                    x.prob = p;
                    x.J = L.J[p];
                    x.n = (int)ns_[p];
                    x.lnb = nb;
                    x.rp = rp;
                    x.cp = cp;
                    rit[rc].push_back(x);
                    continue;
                }
                SwItem<T> x;
                x.soff = offS_[p] + ((int64_t)r * 4 + qd) * squarter;
                x.tabR = L.tab + otab[p] + (int64_t)cp * kTabs * nb * S;
                x.tabC = L.tab + nfac + otab[p] + (int64_t)rp * kTabs * nb * S;
                x.chR = L.ch + och[p] + cp * 3 * nbp_of(nb);
                x.chC = L.ch + nch + och[p] + rp * 3 * nbp_of(nb);
                x.prob = p;
                x.J = L.J[p];
                x.nb = (unsigned short)nb;
                for (int b0 = 0; b0 < nb; ++b0)
                    for (int b1 = 0; b1 < nb; b1 += R) {
                        x.b0 = (unsigned short)b0;
                        x.b1 = (unsigned short)b1;
                        x.n_blk = (unsigned short)std::min(R, nb - b1);
                        x.xoff = x0 + ((int64_t)b0 * nb + b1) * S * S;
                        it[0].push_back(x);
                    }
                for (int b0 = 0; b0 < nb; b0 += R)
                    for (int b1 = 0; b1 < nb; ++b1) {
                        x.b0 = (unsigned short)b0;
                        x.b1 = (unsigned short)b1;
                        x.n_blk = (unsigned short)std::min(R, nb - b0);
                        x.xoff = x0 + ((int64_t)b0 * nb + b1) * S * S;
                        it[1].push_back(x);
                    }
                if (!fused_)
                    for (int b1 = 0; b1 < nb * S / 32; ++b1) {
                        x.b0 = 0;
                        x.b1 = (unsigned short)b1;
                        x.n_blk = 0;
                        x.xoff = x0;
                        it[2].push_back(x);
                    }
            }
    }
    cudaError_t e1 = cudaSuccess;
    for (int w = 0; w < 3 && e1 == cudaSuccess; ++w) {
        L.nitems[w] = (int64_t)it[w].size();
        e1 = dalloc(&L.items[w], it[w].size());
        if (e1 == cudaSuccess && !it[w].empty())
            e1 = cudaMemcpyAsync(L.items[w], it[w].data(), sizeof(SwItem<T>) * it[w].size(), cudaMemcpyHostToDevice, cap_);
    }
    for (size_t c = 0; c < L.res.size() && e1 == cudaSuccess; ++c) {
        L.res[c].nitems = (int64_t)rit[c].size();
        e1 = dalloc(&L.res[c].items, rit[c].size());
        if (e1 == cudaSuccess)
            e1 = cudaMemcpyAsync(L.res[c].items, rit[c].data(), sizeof(ResItem<T>) * rit[c].size(), cudaMemcpyHostToDevice,
                                 cap_);
    }
    // the host vectors must outlive the asynchronous work
    const cudaError_t e2 = cudaStreamSynchronize(cap_);
    ENG_CK(e1);
    ENG_CK(e2);
    return FPS_OK;
}

template <typename T>
ResArgs<T> SweepEngine<T>::res_args(const ResClass &c, const double *F, double *X) const
{
    ResArgs<T> a;
    a.items = c.items;
    a.nitems = c.nitems;
    a.S = c.S;
    a.C = c.C;
    a.active = d_active_;
    a.masked = d_active_ + ns_.size();
    a.X = X_;
    a.D = D_;
    a.F = F;
    a.out = X;
    // a launch outside the solve that copies err_ back reports to the host's copy itself
    a.err = F ? (int *)(h_stat_ + 2 * npairs_) : err_;
    a.give_up = wait_fault_ ? 0 : -1;
    return a;
}

template <typename T>
SwArgs<T> SweepEngine<T>::args(const Level &L, int which) const
{
    SwArgs<T> a;
    a.items = L.items[which];
    a.nitems = L.nitems[which];
    a.active = d_active_;
    a.masked = d_active_ + ns_.size();
    a.X = X_;
    a.D = D_;
    a.sumR = sumR_;
    a.sumC = sumC_;
    a.zxR = zxR_;
    a.zxC = zxC_;
    a.err = err_;
    a.S = seg_len / 2;
    a.fused = fused_ ? 1 : 0;
    a.chain_len = chain_length(sizeof(T) == 8, chain_mode, max_nb_);
    a.max_nb = max_nb_;
    return a;
}

// The resident launches of a level, one per class, side by side: a launch of a few clusters
// is bound by the latency of its iterations and leaves most of the GPU idle.  Branches of at
// most kSide streams from `st`; the first class stays on `st` unless other work follows there.
// join_resident() makes `st` wait for the branches.  One after the other a batch of 8 problems
// in as many classes took 1.2 times as long as the passes over all of them; side by side
// 0.59 ms against 1.70 (8 problems of n = 38 .. 457, two right-hand sides each).
template <typename T>
cudaError_t SweepEngine<T>::run_resident(const Level &L, const double *F, double *X, cudaStream_t st, bool busy,
                                         int64_t &launches)
{
    cudaError_t e = cudaSuccess;
    const int n = (int)L.res.size(), here = busy ? 0 : 1, nside = std::min((int)side_.size(), n - here);
    side_used_ = std::max(nside, 0);
    if (nside > 0) {
        e = cudaEventRecord(fork_, st);
        for (int k = 0; k < nside && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(side_[k].st, fork_, 0);
    }
    for (int c = 0; c < n && e == cudaSuccess; ++c) {
        e = launch_resident<T>(res_args(L.res[c], F, X), c < here || nside <= 0 ? st : side_[(c - here) % nside].st);
        ++launches;
    }
    return e;
}

template <typename T>
cudaError_t SweepEngine<T>::join_resident(cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < side_used_ && e == cudaSuccess; ++k) {
        e = cudaEventRecord(side_[k].done, side_[k].st);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(st, side_[k].done, 0);
    }
    side_used_ = 0;
    return e;
}

template <typename T>
int SweepEngine<T>::build_graph(Level &L, std::string &err)
{
    if (L.graph) {
        cudaGraphExecDestroy(L.graph);
        L.graph = nullptr;
    }
    const SwArgs<T> ar = args(L, 0), ac = args(L, 1), ach = args(L, 2);
    // branches of the resident launches, created outside the capture
    for (int k = (int)side_.size(), want = std::min<int>(kSide, (int)L.res.size() - (streams_ ? 0 : 1)); k < want; ++k) {
        Side x;
        ENG_CK(cudaEventCreateWithFlags(&x.done, cudaEventDisableTiming));
        side_.push_back(x);
        ENG_CK(cudaStreamCreateWithFlags(&side_.back().st, cudaStreamNonBlocking));
    }
    if (!side_.empty() && !fork_) ENG_CK(cudaEventCreateWithFlags(&fork_, cudaEventDisableTiming));
    if (!graphs()) return FPS_OK;
    ENG_CK(cudaStreamBeginCapture(cap_, cudaStreamCaptureModeThreadLocal));
    cudaError_t e = cudaSuccess;
    const bool ins = instrument_ && (int)L.ev.size() == 4 * L.Jstream;
    auto rec = [&](int k) {
        if (ins && e == cudaSuccess) e = cudaEventRecordWithFlags(L.ev[k], cap_, cudaEventRecordExternal);
    };
    L.launches = 0;
    auto run = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
        ++L.launches;
    };
    e = run_resident(L, nullptr, nullptr, cap_, streams_, L.launches);
    if (streams_) run(launch_row_sums<T>(ac, cap_));
    for (int j = 0; j < L.Jstream && e == cudaSuccess; ++j) {
        if (!fused_) run(launch_chain<T>(ach, 0, j, cap_));
        rec(4 * j);
        run(launch_row_pass<T>(ar, j, cap_));
        rec(4 * j + 1);
        if (!fused_) run(launch_chain<T>(ach, 1, j, cap_));
        rec(4 * j + 2);
        run(launch_col_pass<T>(ac, j, cap_));
        rec(4 * j + 3);
    }
    if (e == cudaSuccess) e = join_resident(cap_);
    cudaGraph_t g = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(cap_, &g);
    if (e != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        err = std::string("sweep graph capture: ") + cudaGetErrorString(e);
        return FPS_ERR_CUDA;
    }
    ENG_CK(e2);
    e = cudaGraphInstantiate(&L.graph, g, 0);
    cudaGraphDestroy(g);
    ENG_CK(e);
    return FPS_OK;
}

template <typename T>
int SweepEngine<T>::solve(const double *F, double *X, cudaStream_t st, std::string &err)
{
    launches_last = 0;
    levels_used_.clear();
    if (timed_out()) {  // an FP64 solve on device buffers returned before its waits ended
        err = kGaveUp;
        return FPS_ERR_TIMEOUT;
    }
    return sizeof(T) == 8 ? solve_plain(F, X, st, err) : solve_refine(F, X, st, err);
}

template <typename T>
int SweepEngine<T>::solve_plain(const double *F, double *X, cudaStream_t st, std::string &err)
{
    if constexpr (sizeof(T) == 8) {
        if (!graphs()) {  // scale-in, all iterations and scale-out in one launch per class
            ENG_CK(run_resident(levels_[0], F, X, st, false, launches_last));
            ENG_CK(join_resident(st));
            levels_used_.push_back(0);
            rounds_last = 1;
            return FPS_OK;
        }
        ENG_CK(launch_scale_in<double>(tiles(kPadded), F, nullptr, X_, nullptr, st));
        ENG_CK(cudaGraphLaunch(levels_[0].graph, st));
        ENG_CK(launch_scale_out(tiles(kLive), D_, false, X, st));
        ENG_CK(cudaMemcpyAsync(h_stat_ + 2 * npairs_, err_, sizeof(int), cudaMemcpyDeviceToHost, st));
        levels_used_.push_back(0);
        launches_last = 2 + levels_[0].launches;
        rounds_last = 1;
        return FPS_OK;
    } else {
        (void)F;
        (void)X;
        (void)st;
        err = "plain solve needs FP64 sweeps";
        return FPS_ERR_UNSUPPORTED;
    }
}

template <typename T>
int SweepEngine<T>::solve_refine(const double *F, double *X, cudaStream_t st, std::string &err)
{
    if constexpr (sizeof(T) == 4) {
        const int np = (int)ns_.size();

        // The first round is launched without waiting for smax: the device masks what has
        // nothing to solve, and the host looks at smax together with the round's residuals.
        unsigned long long *d_rmax = d_stat_, *d_smax = d_stat_ + npairs_;
        const unsigned long long *h_rmax = h_stat_, *h_smax = h_stat_ + npairs_;
        ENG_CK(cudaMemsetAsync(d_stat_, 0, sizeof(unsigned long long) * 2 * npairs_, st));
        ENG_CK(launch_absmax(tiles(kLive), F, d_smax, st));
        ENG_CK(launch_init_masks(d_smax, np, nrhs_, d_pair_active_, d_active_, d_active_ + np, st));
        ENG_CK(launch_scale_in<float>(tiles(kPadded), F, Ft_, X_, d_smax, st));
        launches_last += 3;

        std::vector<double> rel(npairs_, 0.0), sF(npairs_, 0.0);
        double *Ycur = Y0_, *Ynext = Y1_;
        bool any_active = true;
        int round = 0;
        bool converged = false;
        for (; round < max_rounds && !converged; ++round) {
            TraceRange tr("fps refinement round");
            // two balanced rounds: the first stops near sqrt(0.1 tol), which leaves the
            // second a gain of the same size (1e-6 then 1e-5 for tol = 1e-10)
            double want = std::sqrt(0.1 * tol_);
            if (round > 0) {
                double worst = 0.0;
                for (int k = 0; k < npairs_; ++k)
                    if (h_pair_active_[k]) worst = std::max(worst, rel[k]);
                want = 0.1 * tol_ / worst;
            }
            size_t li = 0;
            for (size_t l = 0; l < levels_.size(); ++l)
                if (levels_[l].tol <= want) li = l;
            ENG_CK(cudaGraphLaunch(levels_[li].graph, st));
            levels_used_.push_back((int)li);
            launches_last += levels_[li].launches;
            if (round > 0) ENG_CK(cudaMemsetAsync(d_rmax, 0, sizeof(unsigned long long) * npairs_, st));
            ENG_CK(launch_residual(tiles(kResidual), Ycur, Ynext, D_, Ft_, X_, d_smax, d_rmax, d_pair_active_, round == 0,
                                   st));
            launches_last += 1;
            ENG_CK(cudaMemcpyAsync(h_stat_, d_stat_, sizeof(unsigned long long) * (2 * (size_t)npairs_ + 1),
                                   cudaMemcpyDeviceToHost, st));
            ENG_CK(cudaStreamSynchronize(st));
            if (timed_out()) {
                err = kGaveUp;
                return FPS_ERR_TIMEOUT;
            }
            if (round == 0) {
                any_active = false;
                for (int k = 0; k < npairs_; ++k) {
                    sF[k] = bits_to_double(h_smax[k]);
                    if (!std::isfinite(sF[k])) {
                        err = "F holds NaN or Inf";
                        return FPS_ERR_NONFINITE;
                    }
                    h_pair_active_[k] = sF[k] > 0.0 ? 1 : 0;  // an all-zero right-hand side is already solved (X = 0)
                    any_active = any_active || h_pair_active_[k];
                }
                if (!any_active) break;
            }
            std::swap(Ycur, Ynext);
            converged = true;
            for (int k = 0; k < npairs_; ++k) {
                if (!h_pair_active_[k]) continue;
                const double r = bits_to_double(h_rmax[k]) / sF[k];
                if (!std::isfinite(r)) {
                    err = "non-finite residual";
                    return FPS_ERR_NONFINITE;
                }
                rel[k] = r;
                if (r <= tol_) h_pair_active_[k] = 0;
                else converged = false;
            }
            if (converged) continue;
            set_active();
            ENG_CK(cudaMemcpyAsync(d_active_, h_active_, sizeof(int) * (np + 1), cudaMemcpyHostToDevice, st));
            ENG_CK(cudaMemcpyAsync(d_pair_active_, h_pair_active_, sizeof(int) * npairs_, cudaMemcpyHostToDevice, st));
        }
        rounds_last = round;
        resid_last = 0.0;
        for (int k = 0; k < npairs_; ++k) resid_last = std::max(resid_last, rel[k]);
        if (!any_active) {
            ENG_CK(cudaMemsetAsync(X, 0, sizeof(double) * tot64_, st));  // every right-hand side was zero
            return FPS_OK;
        }
        ENG_CK(launch_scale_out(tiles(kLive), Ycur, true, X, st));
        launches_last += 1;
        if (!converged) {
            err = "refinement did not reach tol";
            return FPS_ERR_NOT_CONVERGED;
        }
        return FPS_OK;
    } else {
        (void)F;
        (void)X;
        (void)st;
        err = "refinement needs FP32 sweeps";
        return FPS_ERR_UNSUPPORTED;
    }
}

template <typename T>
int SweepEngine<T>::set_instrument(bool on, std::string &err)
{
    instrument_ = on;
    for (auto &L : levels_) {
        for (cudaEvent_t e : L.ev) cudaEventDestroy(e);
        L.ev.clear();
        if (on) {
            L.ev.resize(4 * (size_t)L.Jstream);
            for (auto &e : L.ev) ENG_CK(cudaEventCreate(&e));
        }
        int st = build_graph(L, err);
        if (st != FPS_OK) return st;
    }
    return FPS_OK;
}

template <typename T>
int SweepEngine<T>::kernel_times(int *count, double *total_ms, double *alg_bytes, double *row_ms, double *col_ms,
                                 std::string &err)
{
    if (timed_out()) {
        err = kGaveUp;
        return FPS_ERR_TIMEOUT;
    }
    int c = 0;
    double rms = 0.0, cms = 0.0, by = 0.0;
    std::vector<int> seen;
    for (int li : levels_used_) {
        if (std::find(seen.begin(), seen.end(), li) != seen.end()) continue;
        seen.push_back(li);
        const Level &L = levels_[li];
        if ((int)L.ev.size() != 4 * L.Jstream) continue;
        for (int j = 0; j < L.Jstream; ++j) {
            float t0 = 0.f, t1 = 0.f;
            ENG_CK(cudaEventElapsedTime(&t0, L.ev[4 * j], L.ev[4 * j + 1]));
            ENG_CK(cudaEventElapsedTime(&t1, L.ev[4 * j + 2], L.ev[4 * j + 3]));
            rms += t0;
            cms += t1;
            c += 2;
            // row pass: u read, a written; column pass: a read, u written (but for the last
            // iteration of a problem), D written and, after the first iteration, read
            for (size_t p = 0; p < ns_.size(); ++p)
                if (!res_s_[p] && j < L.J[p])
                    by += (4.0 + (j > 0 ? 1.0 : 0.0) + (j + 1 < L.J[p] ? 1.0 : 0.0)) * sizeof(T) * (double)nrhs_ *
                          (double)ns_[p] * (double)ns_[p];
        }
    }
    *count = c;
    *total_ms = rms + cms;
    *alg_bytes = by;
    if (row_ms) *row_ms = rms;
    if (col_ms) *col_ms = cms;
    return FPS_OK;
}

template class SweepEngine<float>;
template class SweepEngine<double>;

}  // namespace fps
