// Inner level of the cube's nested ADI: all iterations of every slice equation
//     A~_a Z A~_b + c Z = R
// in one launch (internal header).
//
// As a Sylvester equation A Z - Z B = C (A = A~_a, B = -c A~_b^{-1}, C = R A~_b^{-1}) with
// shifts p_j, q_j the ADI in residual-propagating form is, with c_j the solve of the
// residual on both sides and u_j = (A - p_j) c_j,
//     a_j = u_{j-1} (B - q_{j-1}) (B - p_j)^{-1} = u_{j-1} - (p_j - q_{j-1}) (u_{j-1} A~_b) K_j^{-1},
//     t_j = (q_j - p_j) (A - q_j)^{-1} a_j,     u_j = a_j + t_j,     Z <- Z + t_j,
// K_j = c + p_j A~_b, and a_0 = -R K_0^{-1}: two tridiagonal solves and one banded product
// per iteration, no product with A~_a and no second solve along a.  Where p and q differ
// by orders of magnitude the two sums cancel: every slice is solved to rounding relative to
// its right-hand side but, unlike the paper's form, an error made in one iteration is not
// part of the next residual.  The FP32 rounds measure their residual in FP64 outside and
// correct it; the FP64 cube, which has no such loop, keeps the paper's form (its error with
// a flat right-hand side at n = 32 would grow from 6e-11 to 7e-8).
//
// Slices are independent, and so are the four parity quarters of a slice: one CTA per
// quarter keeps u in shared memory and Z in registers for all iterations.  A line of 2 H
// unknowns is eliminated from both ends by two threads (half-warps) that keep the forward
// values of their half in registers and meet in the middle.  Tables are read 16 bytes at a
// time and in groups ahead of the dependent FMAs.
//
// What bounds it: at small n the latency of the 260 instructions of an iteration on the one
// or two warps of a CTA (n = 32: 0.4 us) and the launches that depend on one another; at
// large n the shared-memory accesses.  Against one launch per line solve and banded product
// (5 per iteration), and against this kernel with u and Z in shared memory and tables read
// word by word: n = 32 635 -> 31 -> 21 ms, n = 64 2.44 s -> 222 -> 88 ms, n = 256 44.4 ->
// 10.3 -> 7.0 s.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace fps {

// Distance between the two halves of a table: whole 16-byte words, and not a multiple of 8
// so that the two half-warps read from different banks.
__host__ __device__ constexpr int unit_half_pitch(int H)
{
    return (H + 3) / 4 * 4 % 8 ? (H + 3) / 4 * 4 : (H + 3) / 4 * 4 + 4;
}
// Tables of one tridiagonal of N = 2 H unknowns, both halves from their outer end: l [2][H],
// {m, the solution scale} [2][H], then the two coefficients per half of the middle solve.
__host__ __device__ constexpr int unit_table(int H) { return 6 * unit_half_pitch(H) + 4; }
// Bands of A~ of one parity: {diagonal, coupling to the outer neighbour} [2][H], then the
// coupling across the middle, padded.
__host__ __device__ constexpr int unit_bands(int H) { return 4 * unit_half_pitch(H) + 4; }

// out = kR R + kZ Z + kacc out, Z = (T_ab + c)^{-1} R, R = r1 R1 + r2 R2 (R2 may be null; out
// may be R1 or R2).
struct UnitJob {
    const float *R1, *R2;
    float *out;
    float r1, r2, kR, kZ, kacc;
};

struct UnitArgs {
    const float *tab;    // [J][b parity 0, b parity 1, a parity 0, a parity 1][unit_table]
    const float *bands;  // [2][unit_bands]
    int J, n, njobs;
    int64_t sa, sb, sc;  // strides of modes a, b and of the slice index
    UnitJob job[2];      // solves with the same tables in one launch
};

// One schedule entry: shifts first .. first + J - 1 of the shift list, tables at tab_off.
struct UnitEntry {
    double c;
    int64_t tab_off;
    int first, J;
};

// Thread `raw` of the table kernel over `shifts` shifts computes half (id & 1) of the line
// id >> 1 of (shift, direction, parity), id as returned; the halves of a line are a lane pair.
// Threads past the end repeat the last pair (each its own half: they take part in the
// exchange of the pivots) and store nothing.
__host__ __device__ constexpr int unit_table_thread(int raw, int shifts)
{
    return raw < 8 * shifts ? raw : 8 * shifts - 2 + (raw & 1);
}

int unit_half(int64_t n);  // H of the compiled kernel (n <= 320; 0 beyond)
cudaError_t unit_setup(int H);
// Tables of `count` entries (device list, ascending `first`) with `shifts` shifts {p, q}
// altogether; d, e: FP64 bands of A~.
cudaError_t launch_unit_tables(const UnitEntry *entries, int count, int shifts, const double2 *pq, const double *d,
                               const double *e, int n, int H, float *tab, cudaStream_t st);
cudaError_t launch_unit_bands(const double *d, const double *e, int n, int H, float *bands, cudaStream_t st);
cudaError_t launch_stein_units(const UnitArgs &a, int H, cudaStream_t st);

}  // namespace fps
