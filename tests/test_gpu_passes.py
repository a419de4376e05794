"""Square solves at the edges of their kernels' blocks, tiles and segment counts, against
the CPU oracle through the C ABI.

One launch (resident kernel): quarters of m = ceil(n/2) <= 16 S unknowns for the compiled
segment lengths S, FP64 up to n = 512, FP32 up to n = 1024.  Streamed: blocks of 32 (FP64,
FP32 segment length 64) or 64 (FP32 segment length 128) unknowns, tiles of 128 x one block;
the passes run the segment recurrence themselves up to n = 1024 (FP64) and 2048 (FP32), the
chain kernel does beyond.  Bars: the FP64 and
refinement bars of the workload definition."""
import numpy as np
import pytest

import oracle
from paper_1710_11259_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_FP64 = 1e-12
TOL_REFINE = 1e-10


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_11259_gb300 import api as _api
    from paper_1710_11259_gb300 import build_ext

    build_ext.build()
    _api.lib()
    return _api


def _relmax(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def _check_fp64(api, n):
    F = np.stack([inputs.square_rhs(n, 40 + n), inputs.square_rhs(n, 41 + n, power=1)])
    plan = api.plan_create(n, 2, 1e-13, "fp64", nrhs=2)
    X = api.poisson_square_solve(plan, torch.from_numpy(F).cuda()).cpu().numpy()
    launches = api.plan_info(plan)["kernel_launches"]
    api.plan_destroy(plan)
    for r in range(2):
        assert _relmax(X[r], oracle.poisson_square(F[r], 1e-13)) <= TOL_FP64, r
    return launches


# full and just overfull segments of every compiled length: n = 32 S and 32 S + 1
@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 6, 8, 10, 12, 14])
def test_fp64_resident_edges(api, S):
    for n in (32 * S - 1, 32 * S, 32 * S + 1):
        assert _check_fp64(api, n) == 1, n


# the last resident size; a last block of one unknown (513, 577, 1025, 1089); full blocks;
# the last size without and the first with the chain kernel (1024, 1025)
@pytest.mark.parametrize("n", [511, 512, 513, 514, 576, 577, 640, 1024, 1025, 1089])
def test_fp64_block_edges(api, n):
    assert (_check_fp64(api, n) == 1) == (n <= 512)


@pytest.mark.parametrize("n", [512, 513, 640, 641, 768, 769, 896, 897, 1023, 1024, 1025])
def test_refine_resident_edges(api, n):
    F = inputs.square_rhs(n, 60 + n)
    plan = api.plan_create(n, 2, 1e-10, "fp32_refine")
    X = api.poisson_square_solve(plan, torch.from_numpy(F).cuda()).cpu().numpy()
    api.plan_destroy(plan)
    assert _relmax(X, oracle.poisson_square(F, 1e-13)) <= TOL_REFINE


@pytest.mark.parametrize("seg,chain", [(64, 1), (64, 2), (128, 1), (128, 2)])
def test_refine_segment_counts(api, tmp_path, monkeypatch, seg, chain):
    """Both block sizes and both run lengths of the chain kernel, on a batch whose largest
    problem has more than 16 segments per line and whose others have one or few."""
    ns = [2113, 1024, 130, 31, 1]
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("FPS_AUTOTUNE_CACHE", str(cache))
    monkeypatch.delenv("FPS_AUTOTUNE", raising=False)
    api.plan_destroy(api.plan_create_batched(ns, nrhs=1, tol=1e-10, precision="fp32_refine"))
    cache.write_text(f"{cache.read_text().split()[0]} {seg} {chain}\n")
    plan = api.plan_create_batched(ns, nrhs=1, tol=1e-10, precision="fp32_refine")
    assert (api.plan_info(plan)["seg_len"], api.plan_info(plan)["chain_mode"]) == (seg, chain)
    rhs = [inputs.square_rhs(n, 90 + n) for n in ns]
    X = api.poisson_square_solve(plan, torch.from_numpy(np.concatenate([f.ravel() for f in rhs])).cuda()).cpu().numpy()
    api.plan_destroy(plan)
    o = 0
    for n, f in zip(ns, rhs):
        assert _relmax(X[o:o + n * n].reshape(n, n), oracle.poisson_square(f, 1e-13)) <= TOL_REFINE, n
        o += n * n


# lines of 17, 32 and 33 segments of 32 and of 9, 16 and 17 segments of 64: the passes run the
# segment recurrence up to 32 and 16, the chain kernel beyond
@pytest.mark.parametrize("seg", [64, 128])
@pytest.mark.parametrize("n", [1025, 2047, 2048, 2049])
def test_refine_recurrence_edges(api, tmp_path, monkeypatch, seg, n):
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("FPS_AUTOTUNE_CACHE", str(cache))
    monkeypatch.delenv("FPS_AUTOTUNE", raising=False)
    api.plan_destroy(api.plan_create(n, 2, 1e-10, "fp32_refine"))
    cache.write_text(f"{cache.read_text().split()[0]} {seg} 1\n")
    F = inputs.square_rhs(n, 70 + n)
    plan = api.plan_create(n, 2, 1e-10, "fp32_refine")
    X = api.poisson_square_solve(plan, torch.from_numpy(F).cuda()).cpu().numpy()
    assert api.plan_info(plan)["seg_len"] == seg
    api.plan_destroy(plan)
    assert _relmax(X, oracle.poisson_square(F, 1e-13)) <= TOL_REFINE


@pytest.mark.parametrize("n", [101, 601])
def test_nonfinite_input_leaves_no_trace(api, n):
    """The kernels work in place: a right-hand side with NaN and Inf must not reach the next
    solve of the plan through the unused positions of the blocks."""
    F = torch.from_numpy(inputs.square_rhs(n, 5)).cuda()
    plan = api.plan_create(n, 2, 1e-13, "fp64")
    X = api.poisson_square_solve(plan, F).clone()
    bad = F.clone()
    bad[3, 4], bad[50, 99] = float("nan"), float("inf")
    api.poisson_square_solve(plan, bad)
    again = api.poisson_square_solve(plan, F)
    torch.cuda.synchronize()
    api.plan_destroy(plan)
    assert torch.equal(X, again)


@pytest.mark.parametrize("n", [65, 1100])
@pytest.mark.parametrize("k", [900, -600, -1000])
def test_refine_scales_with_powers_of_two(api, n, k):
    """The FP32 iteration runs on the residual scaled by a power of two, converted with
    integer instructions: right-hand sides near the ends of the FP64 range (at k = -1000
    part of the scaled right-hand side is subnormal) give the scaled solution."""
    F = inputs.square_rhs(n, 3)
    plan = api.plan_create(n, 2, 1e-10, "fp32_refine")
    X = api.poisson_square_solve(plan, torch.from_numpy(np.ldexp(F, k)).cuda()).cpu().numpy()
    info = api.plan_info(plan)
    api.plan_destroy(plan)
    assert info["last_residual"] <= 1e-10
    assert _relmax(np.ldexp(X, -k), oracle.poisson_square(F, 1e-13)) <= TOL_REFINE


@pytest.mark.parametrize("n", [15, 17, 65, 127, 129, 899, 900, 3071, 3072, 3073])
def test_legendre_walk_edges(api, n):
    """Legendre maps at the edges of their tiles (16 rows x 64 columns, 32 and 128 x 128) and on
    both sides of the sizes where the walk length changes."""
    G, X = inputs.gaussian(n, (n, n)), inputs.square_rhs(n, n + 1)
    F = api.legendre_to_ctilde(torch.from_numpy(G).cuda()).cpu().numpy()
    U = api.solution_to_legendre(torch.from_numpy(X).cuda()).cpu().numpy()
    assert _relmax(F, oracle.legendre_to_ctilde(G)) <= 1e-14
    assert _relmax(U, oracle.solution_to_legendre(X)) <= 1e-13


# half lines of 2, 4, .., 64 unknowns per CTA, full and with unused places; 256 is the last
# size that stays on chip, 257 and 300 stream.  Against the oracle's ADI at tol 1e-15 with
# the bar of the n = 128 cylinder test, 10 tol kappa_k + 3e-11; its rounding floor grows
# with the entries of P, k^2 + n^2, hence the factor above n = 128.
@pytest.mark.parametrize("n,k", [(4, 2), (5, 3), (9, 2), (33, 2), (47, 5), (65, 17), (97, 2), (129, 3), (161, 2),
                                 (193, 40), (224, 2), (255, 5), (256, 2), (257, 2), (300, 12)])
def test_cylinder_line_lengths(api, n, k):
    from oracle import cylinder as cyl

    F = np.stack([inputs.square_rhs(n, n), inputs.square_rhs(n, n + 1)])
    plan = api.plan_create_cylinder(n, k, k, 1e-13, 2)
    Y = api.poisson_cylinder_solve(plan, torch.from_numpy(F[None].copy()).cuda()).cpu().numpy()[0]
    api.plan_destroy(plan)
    P, Q, _, _ = cyl.mode_operators(n, k)
    kappa = np.linalg.cond(np.linalg.eig(np.linalg.solve(P, Q))[1])
    bar = 10 * 1e-13 * kappa + 3e-11 * max(1.0, (n / 128.0) ** 2)
    for r in range(2):
        Yo, _ = cyl.mode_adi(F[r], k, 1e-15)
        assert _relmax(Y[r], Yo) <= bar, (r, bar)


def _along(T, B):  # B on all three modes
    for _ in range(3):
        T = np.tensordot(T, B, axes=([0], [1]))
    return T


# the slice kernel's line lengths (2 H unknowns per parity), full and with unused places
@pytest.mark.parametrize("n", [3, 4, 7, 9, 12, 13, 16, 24, 25, 33, 40, 41, 49, 65, 81, 97, 113, 129, 145, 161, 193, 257, 289])
def test_cube_refine_line_lengths(api, n):
    """Against the exact solution by diagonalisation, at the cube's refinement bar."""
    F = inputs.cube_rhs(n, n)
    plan = api.plan_create(n, 3, 1e-10, "fp32_refine")
    X = api.poisson_cube_solve(plan, torch.from_numpy(F).cuda()).cpu().numpy()
    api.plan_destroy(plan)
    d, e = oracle.square_bands(n)
    A = np.diag(d) + np.diag(e[: n - 2], 2) + np.diag(e[: n - 2], -2)
    lam, V = np.linalg.eigh(A)
    s = 1.0 / np.sqrt((np.arange(n) + 1.0) * (np.arange(n) + 2.0))
    S = s[:, None, None] * s[None, :, None] * s[None, None, :]
    L = lam[:, None, None] * lam[None, :, None] + lam[:, None, None] * lam[None, None, :] + \
        lam[None, :, None] * lam[None, None, :]
    Xd = _along(_along(-F * S, V.T) / L, V) * S
    assert _relmax(X, Xd) <= TOL_REFINE


# more than 65535 / 4 (mode, right-hand side) pairs, and the most a plan takes (65535)
@pytest.mark.parametrize("n,modes,nrhs", [(5, 65, 256), (4, 255, 257)])
def test_cylinder_many_pairs(api, n, modes, nrhs):
    """Every pair of a large plan equals the same right-hand side alone in its mode's plan, and
    the first and the last agree with the dense solve (bar of the small cylinder tests)."""
    from oracle import cylinder as cyl

    F = inputs.gaussian(n, (modes, nrhs, n, n))
    plan = api.plan_create_cylinder(n, 2, modes + 1, 1e-13, nrhs)
    Y = api.poisson_cylinder_solve(plan, torch.from_numpy(F).cuda()).cpu().numpy()
    api.plan_destroy(plan)
    one = api.plan_create_cylinder(n, 2, modes + 1, 1e-13, 1)
    for r in (0, 1, nrhs // 2, nrhs - 1):
        Fr = torch.from_numpy(np.ascontiguousarray(F[:, r:r + 1])).cuda()
        assert np.array_equal(api.poisson_cylinder_solve(one, Fr).cpu().numpy()[:, 0], Y[:, r]), r
    api.plan_destroy(one)
    for m, r in ((0, 0), (modes - 1, nrhs - 1)):
        P, Q, _, _ = cyl.mode_operators(n, m + 2)
        kappa = np.linalg.cond(np.linalg.eig(np.linalg.solve(P, Q))[1])
        assert _relmax(Y[m, r], cyl.mode_solve_dense(F[m, r], m + 2)) <= 10 * 1e-13 * kappa


@pytest.mark.parametrize("n", [65, 1100])
@pytest.mark.parametrize("k", [0, -1000])
def test_refine_keeps_subnormal_quarters(api, n, k):
    """Parity quarters do not couple, so one whose scaled right-hand side is below FP32's normal
    range still gets its own solution: to 1e-3, from values held to 2^-149 (22 bits at the
    largest, about 40 iterations) and one round at 1e-6 or finer."""
    F = inputs.square_rhs(n, 3)
    s = 1.0 / np.sqrt((np.arange(n) + 1.0) * (np.arange(n) + 2.0))
    scaled = np.abs(F * s[:, None] * s[None])
    own = scaled[1::2, 1::2].max()
    scaled[1::2, 1::2] = 0.0
    e = int(np.floor(np.log2(scaled.max())) - np.floor(np.log2(own))) - 128  # largest in [2^-128, 2^-127) units
    small = np.zeros_like(F)
    small[1::2, 1::2] = F[1::2, 1::2]
    G = F - small + np.ldexp(small, e)
    plan = api.plan_create(n, 2, 1e-10, "fp32_refine")
    X = api.poisson_square_solve(plan, torch.from_numpy(np.ldexp(G, k)).cuda()).cpu().numpy()
    api.plan_destroy(plan)
    got, want = np.ldexp(X, -k), oracle.poisson_square(small, 1e-13)
    if k == 0:
        assert _relmax(np.ldexp(got[1::2, 1::2], -e), want[1::2, 1::2]) <= 1e-3
    assert _relmax(got, oracle.poisson_square(G, 1e-13)) <= TOL_REFINE


# FP64 beyond n = 512: one right-hand side runs in one launch up to n = 768, more are streamed
@pytest.mark.parametrize("n", [513, 577, 639, 640, 641, 705, 767, 768, 769])
@pytest.mark.parametrize("nrhs", [1, 2])
def test_fp64_one_launch_of_few_clusters(api, n, nrhs):
    F = inputs.square_rhs(n, n) if nrhs == 1 else np.stack([inputs.square_rhs(n, n + r) for r in range(nrhs)])
    plan = api.plan_create(n, 2, 1e-13, "fp64", nrhs=nrhs)
    X = api.poisson_square_solve(plan, torch.from_numpy(F).cuda()).cpu().numpy()
    launches = api.plan_info(plan)["kernel_launches"]
    api.plan_destroy(plan)
    assert (launches == 1) == (nrhs == 1 and n <= 768)
    for f, x in zip(F.reshape(nrhs, n, n), X.reshape(nrhs, n, n)):
        assert _relmax(x, oracle.poisson_square(f, 1e-13)) <= TOL_FP64


def test_nonfinite_input_leaves_no_trace_streamed(api):
    test_nonfinite_input_leaves_no_trace(api, 801)
