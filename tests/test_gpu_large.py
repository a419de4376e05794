"""Large squares: lines of more segments than one CTA's registers hold, whose recurrences are
walked (FP64 from n = 10241, FP32 in blocks of 32 from n = 20481), the last sizes below and the
FP32 sizes that need 16 segments per thread.  The residual of kx A~ Y + ky Y A~ = F~ is formed
by PyTorch from the returned X; its bars are those of the workload definition, relative to
max |F~|.  Problems of few segments in the same plan are compared with the oracle."""
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


def _rhs(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = 1.0 / (1.0 + torch.arange(n, dtype=torch.float64, device="cuda"))
    return torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g).mul_(w[:, None]).mul_(w[None])


def _residual(F, X, kx=1.0, ky=1.0):
    n = F.shape[0]
    d, e = (torch.from_numpy(np.ascontiguousarray(b)).cuda() for b in oracle.square_bands(n))
    e = e[: n - 2]
    k = torch.arange(n, dtype=torch.float64, device="cuda")
    s = 1.0 / torch.sqrt((k + 1) * (k + 2))
    Y = X / s[:, None] / s[None]
    R = F * s[:, None] * s[None]
    scale = float(R.abs().max())
    R -= (kx * d)[:, None] * Y
    R[2:] -= (kx * e)[:, None] * Y[:-2]
    R[:-2] -= (kx * e)[:, None] * Y[2:]
    R -= Y * (ky * d)[None]
    R[:, 2:] -= Y[:, :-2] * (ky * e)[None]
    R[:, :-2] -= Y[:, 2:] * (ky * e)[None]
    return float(R.abs().max()) / scale


@pytest.mark.parametrize("n,w,h", [(10240, 2.0, 2.0), (10241, 2.0, 2.0), (10300, 4.0, 1.0), (16449, 2.0, 2.0)])
def test_fp64_large(api, n, w, h):
    F = _rhs(n, n)
    plan = api.plan_create_rect(n, w, h, 1e-13, "fp64")
    X = api.poisson_square_solve(plan, F)
    torch.cuda.synchronize()
    api.plan_destroy(plan)
    assert _residual(F, X, (2.0 / w) ** 2, (2.0 / h) ** 2) <= TOL_FP64


@pytest.mark.parametrize("n,seg,chain", [(16449, 64, 1), (20480, 64, 2), (20481, 64, 1), (20481, 64, 2), (22001, 128, 1)])
def test_refine_large_with_small(api, tmp_path, monkeypatch, n, seg, chain):
    ns = [1100, n, 300, 2113]
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("FPS_AUTOTUNE_CACHE", str(cache))
    monkeypatch.delenv("FPS_AUTOTUNE", raising=False)
    api.plan_destroy(api.plan_create_batched(ns, nrhs=1, tol=1e-10, precision="fp32_refine"))  # tunes both block sizes
    cache.write_text(f"{cache.read_text().split()[0]} {seg} {chain}\n")
    plan = api.plan_create_batched(ns, nrhs=1, tol=1e-10, precision="fp32_refine")
    assert (api.plan_info(plan)["seg_len"], api.plan_info(plan)["chain_mode"]) == (seg, chain)
    F = [_rhs(n, m) if m == n else torch.from_numpy(inputs.square_rhs(m, m)).cuda() for m in ns]
    X = api.poisson_square_solve(plan, torch.cat([f.reshape(-1) for f in F]))
    torch.cuda.synchronize()
    api.plan_destroy(plan)
    o = 0
    for m, f in zip(ns, F):
        x = X[o:o + m * m].reshape(m, m)
        o += m * m
        if m == n:
            assert _residual(f, x) <= TOL_REFINE
        else:
            xo = oracle.poisson_square(f.cpu().numpy(), 1e-13)
            assert np.abs(x.cpu().numpy() - xo).max() <= TOL_REFINE * np.abs(xo).max(), m
