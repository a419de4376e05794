// ADI pass kernels of the square solve, for one problem or a batch (internal header).
//
// Every ADI iteration j of Algorithm 2 (on the symmetric equation (3.9), shifts
// q_j > 0) is run in residual-propagating form,
//     c_j = (L - q_j)^{-1} (R - q_j)^{-1} rho_j,
//     D  <- D - 2 q_j c_j,                  rho_{j+1} = (L + q_j)(R + q_j) c_j,
// with L(Y) = A~ Y (along columns) and R(Y) = Y A~ (along rows); D after J
// iterations is the ADI iterate Y_J of the paper's form started from Y_0 = 0 with
// right-hand side rho_0 (the two forms agree term by term in exact arithmetic).
// The products with A~ + q are never formed.  With a_j = (R - q_j)^{-1} rho_j and
// u_j = (L + q_j) c_j,
//     u_j = a_j + 2 q_j c_j                                (L + q = (L - q) + 2q),
//     a_{j+1} = (R - q_{j+1})^{-1} (R + q_j) u_j
//             = u_j + (q_j + q_{j+1}) (R - q_{j+1})^{-1} u_j,
// so an iteration is two solves, two multiply-adds per element and the update of D:
//     row pass:     a = u + s v,  v = (R - q_j)^{-1} u,  s = q_{j-1} + q_j  (a = v at j = 0)
//     column pass:  t = 2 q_j c,  c = (L - q_j)^{-1} a,  u = a + t,  D <- D + t
// and Y_J = -D.  The shifts fall with j, so neither sum cancels: on an eigenvector
// with R -> 0 the row factor 1 - s/q_j is -q_{j-1}/q_j, the column factor -1.
// On a rectangle the equation is kx A~ Y + ky Y A~ = F~ with shifts p_j (row side)
// and q_j (column side) of App. A's general intervals; the row solves then have the
// shift -p_j/ky and s = (q_{j-1} - p_j)/ky, the column solves q_j/kx and
// t = (q_j - p_j)/kx c, and Y_J = -D/ky.
//
// Even and odd indices decouple in both directions (App. B), so the n x n problem is
// four independent problems ("quarters": row parity x column parity) of tridiagonal
// systems of about n/2 unknowns, stored apart.
//
// A tridiagonal A~ - qI of one parity, pivots piv_i, ip_i = 1/piv_i, is solved as
//     w_i = r_i - l_i w_{i-1},     l_i = e_{i-1} ip_{i-1},
//     y_i = w_i - m_i y_{i+1},     m_i = e_i ip_{i+1},       x_i = ip_i y_i
// (the pivot of w is left in place and ip_i is folded into the scalars s and 2q that
// x is multiplied with: one multiply-add per sweep and element).  Systems are cut into
// segments of S unknowns.  A pass needs, per segment and line, w just before (zin) and
// y just after it (yout); they follow from a recurrence over the segments of the two
// segment summaries that the pass before left:
//     wl = sum_i psi_i r_i  (w at the segment's end started from zero),
//     yl = sum_i chi_i r_i  (y at its start, started from and ended at zero),
//     W_s = wl(s) + phi(s) W_{s-1},                    zin(s)  = W_{s-1},
//     Y_s = yl(s) + Bv(s) zin(s) + Psi(s) Y_{s+1},     yout(s) = Y_{s+1}
// (psi, chi, phi, Bv, Psi depend on the shift only and are tabulated in FP64
// arithmetic).  So every pass reads true values, writes true values, and forms on the
// finished tile the summaries of the next solve, which runs across it:
//   row pass j     reads u, writes a in place;  summaries of column solve j
//   column pass j  reads a, D, writes u, D in place;  summaries of row solve j + 1
// Every element is read and written once per pass by the same CTA: no halo, no second
// array, 8 + 16 bytes per element and iteration in FP32, 11 FP64 operations in FP64.
// Bound: HBM in FP32 where the arrays exceed L2, the FP64 rate in FP64.  Measured on
// GB300: FP32 n = 10^4 row pass 128 us, column pass 237 us (6.1 and 6.7 TB/s of DRAM
// traffic; a copy reaches 6.7), FP64 n = 4096 154 and 183 us; passes that formed the
// products with A~ + q on tiles with halos and rebuilt the solve before them while
// loading took 341 + 158 us and 393 + 174 us.
//
// Storage (type T = float or double) of a (problem, rhs): four quarters of nb x nb
// blocks of S x S elements, nb = ceil(ceil(n/2)/S), block (bi, bk) of a quarter at
// ((quarter * nb + bi) * nb + bk) * S * S, rows of S elements.  A tile is whole blocks,
// so one bulk copy per block moves it.  The 16-byte chunks of row r are permuted by
// XOR with r mod 8, which makes the row-wise 16-byte accesses of the sweeps along rows
// free of bank conflicts.  Unused positions (>= the parity's size) are zero.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace fps {

template <typename T>
struct Vec2;
template <>
struct Vec2<float> {
    using type = float2;
};
template <>
struct Vec2<double> {
    using type = double2;
};

constexpr int kPassLines = 128;  // columns of a row-pass tile, rows of a column-pass tile (whole blocks)
constexpr int kTabs = 5;         // per position and shift: l, m, solution scale, psi, chi

// Offset of element (r, c) inside an S x S block (V elements per 16-byte chunk).
template <typename T>
__host__ __device__ __forceinline__ int block_pos(int r, int c, int S)
{
    constexpr int V = 16 / (int)sizeof(T);
    return r * S + (((c / V) ^ (r & 7)) * V) + c % V;
}

// One work item of a pass or chain launch at one tolerance level: everything a CTA
// needs before it can issue its copies, in one 64-byte record (one round trip).
template <typename T>
struct alignas(16) SwItem {
    int64_t xoff;          // passes: element offset of the tile's first block in X and D
    int64_t soff;          // offset of the quarter in the segment arrays
    const T *tabR, *tabC;  // [J][2][kTabs][nb * S] tables of the row / column solves of this quarter's parities
                           // (offset to the parity: iteration j at + j * 2 * kTabs * nb * S)
    const T *chR, *chC;    // [J][2][3][nbp] segment coefficients phi, Bv, Psi (nbp = nb rounded up to 4), likewise
    int prob;              // problem index (mask of active problems)
    int J;                 // iterations of the problem at this level
    unsigned short nb, b0; // blocks per side; passes: block row of the tile's first block
    unsigned short b1, n_blk;  // passes: its block column; blocks of the tile.  Chains: first line / 32, -
};
static_assert(sizeof(SwItem<float>) == 64, "one 64-byte record per item");

template <typename T>
struct SwArgs {
    using T2 = typename Vec2<T>::type;
    const SwItem<T> *items;
    int64_t nitems;
    const int *active;     // per problem
    const int *masked;     // != 0 if any problem is inactive
    T *X, *D;              // X: u / a in place; D: sum of t
    T2 *sumR, *sumC;       // segment summaries {wl, yl}: [quarter][segment][line]
    T2 *zxR, *zxC;         // recurrence results {zin, yout}, same layout (plans that run it in its own kernel)
    int *err;              // device error word: bit 0 = a bounded wait gave up
    int S;                 // block and segment size of every problem (sweep_segment_supported(., 2 S))
    int fused;             // passes run the segment recurrence themselves (sweep_fused)
    int chain_len;         // chain kernel: segments per thread (chain_length)
    int max_nb;
};

// Elementwise tile kernels of the solve around the ADI loop.  A tile item is
// {problem * 256 + rhs, x, y, 0}: x, y in tiles of 64 x 64 elements (32 x 32 of every
// quarter) of the live or of the padded region, or, for the residual, x = tile column * 4 +
// quarter and y = tile row in tiles of 64 rows x 32 columns of a quarter.
struct TileProb {
    int n, nb, log_s;       // nb: blocks of 2^log_s per side of a quarter
    int64_t off64;          // FP64 packing of the caller's arrays: offset of rhs 0 (rhs stride n*n)
    int64_t off, rhs;       // quarter-block arrays: offset of rhs 0, stride between right-hand sides
    const double *s;        // 1/sqrt(E), n entries
    const double *nd, *ne;  // {-kx d, -ky d} and {-kx e, -ky e}, n entries each (e zero-padded)
    int pair0;              // index of (problem, rhs 0) among all pairs
    double inv_ky;          // 1 / scale of the second derivative along y
};

struct TileArgs {
    const TileProb *probs;
    const int4 *tiles;
    int64_t ntiles;
};

// Shift tables of a list of (problem, shift) jobs, computed in FP64.
template <typename T>
struct FacJob {
    double q;
    double sc1, sc2;       // factors of ip in the solution scales of out1 and out2
    int n, nb, S;
    const double *d, *e;   // FP64 bands, e zero-padded to length n
    T *out1, *out2;        // [2][kTabs][nb * S]; out2 may be null
    T *ch1, *ch2;          // [2][3][nbp]; ch2 null with out2
};

cudaError_t sweep_setup_kernels();
// Whether the passes run the segment recurrences of lines of up to nb segments of S
// themselves, while their tiles are in flight (otherwise launch_chain does).  A thread group
// of a tile takes 8 segments in FP32 (n <= 2048 with both block sizes: each chain launch took
// 5.7 us of about 20 per pass; Dirichlet solve and adjoint at n = 2048 4.43 -> 4.21 ms, 3.95
// with fuller waves) and 4 in FP64 (n <= 1024), where the operations come on top of a bound
// FP64 pipe.
bool sweep_fused(bool fp64, int S, int nb);
// Warps that a chain launch with `len` segments per thread can have: the segments are in
// registers, 64 a thread (len 8) and 96 (len 16) in FP32, 96 (len 8) in FP64
// (sweep_setup_kernels checks it).
constexpr int chain_warps(bool fp64, int len)
{
    return fp64 ? (len == 8 ? 20 : 0) : (len == 8 ? 32 : (len == 16 ? 20 : 0));
}
// Segments per thread of the chain launches over lines of up to `nb` segments, in registers:
// 8, or 16 where FP32 prefers it (mode 2) or needs it; 0 where no such launch covers a line
// (FP64 n > 10240, FP32 n > 20480 in blocks of 32): its threads walk over as many as it takes.
constexpr int chain_length(bool fp64, int mode, int nb)
{
    if (mode != 2 && nb <= 8 * chain_warps(fp64, 8)) return 8;
    if (nb <= 16 * chain_warps(fp64, 16)) return 16;
    return nb <= 8 * chain_warps(fp64, 8) ? 8 : 0;
}
constexpr int kWalkWarps = 16;
// Segment lengths (unknowns of both parities) with compiled pass kernels: 64 (FP32, FP64)
// and 128 (FP32), i.e. blocks of 32 and 64.
bool sweep_segment_supported(bool fp64, int seg);

template <typename T>
cudaError_t launch_fac_tables(const FacJob<T> *jobs, int njobs, cudaStream_t st);

// Summaries of the row solve of iteration 0 of the right-hand sides in X (items of the
// column pass).
template <typename T>
cudaError_t launch_row_sums(const SwArgs<T> &a, cudaStream_t st);
template <typename T>
cudaError_t launch_row_pass(const SwArgs<T> &a, int j, cudaStream_t st);
template <typename T>
cudaError_t launch_col_pass(const SwArgs<T> &a, int j, cudaStream_t st);
// Segment recurrences of the row (dir 0) or column (dir 1) solve of iteration j.
template <typename T>
cudaError_t launch_chain(const SwArgs<T> &a, int dir, int j, cudaStream_t st);

// Per (problem, rhs): smax = max |D_s F D_s| (bit patterns; must start at 0).
cudaError_t launch_absmax(const TileArgs &t, const double *F, unsigned long long *smax, cudaStream_t st);
// Masks of the pairs and problems with 0 < smax < Inf; *masked = any problem without one.
cudaError_t launch_init_masks(const unsigned long long *smax, int np, int nrhs, int *pair_active, int *active,
                              int *masked, cudaStream_t st);
// F~ = D_s F D_s (FP64 blocks, if Ft != nullptr) and rho0 = F~ / s (passes' blocks, unused
// positions set to zero), s the power of two below smax (smax == nullptr: s = 1).  Tiles
// cover the padded region.
template <typename T>
cudaError_t launch_scale_in(const TileArgs &t, const double *F, double *Ft, T *rho0, const unsigned long long *smax,
                            cudaStream_t st);
// Yout = Y - s D / ky (Y read as zero if y_zero), R = F~ - A~ Yout - Yout A~, rho0 = R / s,
// rmax = max |R| per pair (bit patterns; must start at 0); inactive pairs copy Y.
cudaError_t launch_residual(const TileArgs &t, const double *Y, double *Yout, const float *D, const double *Ft,
                            float *rho0, const unsigned long long *smax, unsigned long long *rmax,
                            const int *pair_active, bool y_zero, cudaStream_t st);
// Caller layout: X = D_s Z D_s of the FP64 blocks (plain), or X = -D_s Z D_s / ky of the
// passes' blocks.
cudaError_t launch_scale_out(const TileArgs &t, const double *Z, bool plain, double *X, cudaStream_t st);

}  // namespace fps
