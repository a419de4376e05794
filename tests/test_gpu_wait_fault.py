"""A bounded device wait that gives up (injected: the waits of one CTA per cluster give up in
the first iteration, so that its peers' waits run out too; streamed plans find the error word
set): the solve reports FPS_ERR_TIMEOUT, the launch ends by itself and the device stays
usable."""
import numpy as np
import pytest

import oracle
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


# one CTA per cluster, 15, and 16 with two lines per thread
@pytest.mark.parametrize("n", [20, 300, 1000])
def test_resident_refinement_reports_timeout(api, monkeypatch, n):
    F = inputs.square_rhs(n, n)
    Fd = torch.from_numpy(F).cuda()
    monkeypatch.setenv("FPS_INJECT_WAIT_FAULT", "1")
    plan = api.plan_create(n, 2, 1e-10, "fp32_refine")
    monkeypatch.delenv("FPS_INJECT_WAIT_FAULT")
    with pytest.raises(api.FpsError) as e:
        api.poisson_square_solve(plan, Fd)
    assert e.value.status == -6
    api.plan_destroy(plan)
    plan = api.plan_create(n, 2, 1e-10, "fp32_refine")  # the same request without the fault
    X = api.poisson_square_solve(plan, Fd).cpu().numpy()
    api.plan_destroy(plan)
    Xo = oracle.poisson_square(F, 1e-13)
    assert np.abs(X - Xo).max() <= 1e-10 * np.abs(Xo).max()


# one launch and streamed
@pytest.mark.parametrize("n", [20, 300, 769])
def test_fp64_reports_timeout(api, monkeypatch, n):
    """A solve on device buffers returns before its kernels end: the next one reports what
    happened, and so does every later one.  With a host buffer the solve itself does."""
    F = inputs.square_rhs(n, n)
    Fd = torch.from_numpy(F).cuda()
    monkeypatch.setenv("FPS_INJECT_WAIT_FAULT", "1")
    plan, plan_host, plan_out = (api.plan_create(n, 2, 1e-13, "fp64") for _ in range(3))
    monkeypatch.delenv("FPS_INJECT_WAIT_FAULT")
    api.poisson_square_solve(plan, Fd)
    torch.cuda.synchronize()
    for _ in range(2):
        with pytest.raises(api.FpsError) as e:
            api.poisson_square_solve(plan, Fd)
        assert e.value.status == -6
    for p, f, x in ((plan_host, F, np.empty_like(F)), (plan_out, Fd, torch.empty(n, n, dtype=torch.float64).pin_memory())):
        with pytest.raises(api.FpsError) as e:
            api.poisson_square_solve(p, f, x)
        assert e.value.status == -6
    for p in (plan, plan_host, plan_out):
        api.plan_destroy(p)
    plan = api.plan_create(n, 2, 1e-13, "fp64")
    X = api.poisson_square_solve(plan, Fd).cpu().numpy()
    api.plan_destroy(plan)
    Xo = oracle.poisson_square(F, 1e-13)
    assert np.abs(X - Xo).max() <= 1e-12 * np.abs(Xo).max()
