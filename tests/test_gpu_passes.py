"""Pass kernels of the square solve at the edges of their blocks, tiles and segment
counts, against the CPU oracle through the C ABI.

A quarter (one parity per direction) has ceil(n/2) unknowns per side in blocks of 32
(FP64, FP32 segment length 64) or 64 (FP32 segment length 128) and tiles of 128 lines;
up to 16 segments per line the passes run the segment recurrence themselves, beyond that
the chain kernel does (FP64: n > 1024; FP32: n > 1024 or n > 2048).  Bars: the FP64 and
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


# one block and its neighbours, one tile of 128 lines, the last fused size and the first
# size with the chain kernel (1024 / 1025), a last block of one unknown (1089)
@pytest.mark.parametrize("n", [66, 127, 128, 129, 255, 256, 258, 1024, 1025, 1089])
def test_fp64_block_edges(api, n):
    F = np.stack([inputs.square_rhs(n, 40 + n), inputs.square_rhs(n, 41 + n, power=1)])
    plan = api.plan_create(n, 2, 1e-13, "fp64", nrhs=2)
    X = api.poisson_square_solve(plan, torch.from_numpy(F).cuda()).cpu().numpy()
    api.plan_destroy(plan)
    for r in range(2):
        assert _relmax(X[r], oracle.poisson_square(F[r], 1e-13)) <= TOL_FP64, r


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


def test_nonfinite_input_leaves_no_trace(api):
    """The passes work in place: a right-hand side with NaN and Inf must not reach the next
    solve of the plan through the unused positions of the blocks."""
    n = 101
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
