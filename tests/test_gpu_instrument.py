"""Pass timing of instrumented plans: the row and column passes of streamed problems and
nothing of problems that are solved in one launch, whose route it does not change."""
import numpy as np
import pytest

from paper_1710_11259_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_11259_gb300 import api as _api
    from paper_1710_11259_gb300 import build_ext

    build_ext.build()
    _api.lib()
    return _api


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-13), ("fp32_refine", 1e-10)])
def test_one_launch_problems_have_no_passes(api, precision, tol):
    F = torch.from_numpy(inputs.square_rhs(300, 8)).cuda()
    plan = api.plan_create(300, 2, tol, precision)
    X = api.poisson_square_solve(plan, F).clone()
    launches = api.plan_info(plan)["kernel_launches"]
    api.plan_set_instrument(plan, True)
    Xi = api.poisson_square_solve(plan, F)
    kt, li = api.plan_kernel_times(plan), api.plan_info(plan)["kernel_launches"]
    api.plan_destroy(plan)
    assert (kt["count"], kt["total_ms"], kt["alg_bytes"], kt["row_ms"], kt["col_ms"]) == (0, 0.0, 0.0, 0.0, 0.0)
    assert torch.equal(X, Xi) and li == launches


@pytest.mark.parametrize("ns", [[1100], [1100, 300, 40]])
def test_batch_counts_the_streamed_problem(api, ns):
    """With J_l iterations at each of the L tolerance levels used: 2 sum J_l launches, and
    sum (6 J_l - 2) FP32 words per element of the problem of n = 1100."""
    F = torch.cat([torch.from_numpy(inputs.square_rhs(n, n)).cuda().reshape(-1) for n in ns])
    plan = api.plan_create_batched(ns, nrhs=1, tol=1e-10, precision="fp32_refine")
    X = api.poisson_square_solve(plan, F).clone()
    api.plan_set_instrument(plan, True)
    Xi = api.poisson_square_solve(plan, F)
    kt, rounds = api.plan_kernel_times(plan), api.plan_info(plan)["refine_rounds"]
    api.plan_destroy(plan)
    assert torch.equal(X, Xi)
    assert kt["count"] > 0 and kt["row_ms"] > 0 and kt["col_ms"] > 0
    levels = (3 * kt["count"] - kt["alg_bytes"] / (4.0 * 1100 ** 2)) / 2
    assert levels == int(levels) and 1 <= levels <= rounds
