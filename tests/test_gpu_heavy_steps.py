"""Inner steps on MaxCut graphs with rows that are summed beforehand (more than 256 entries, several segments
of 512) against the oracle's steps.  Bars as for the steps in test_gpu_rows.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from gpu_common import as_np, rel_err  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2505_15775_gb300 import alm  # noqa: E402
from test_gpu_rows import _hubs  # noqa: E402


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("r", [2, 9, 32])
@pytest.mark.parametrize("degrees,n", [((257, 300, 2), 700), ((600, 1100), 1500), ((2049, 513, 17), 2500)])
def test_steps(degrees, n, r, prec):
    inst = _hubs(degrees, n)
    P = O.OracleProblem(inst)
    rng = np.random.default_rng(r)
    R = rng.standard_normal((n, r))
    R /= np.linalg.norm(R, axis=1, keepdims=True)
    y = np.full(n, -8.0)
    h = alm.alm_create(inst, precision=prec, r_max=r, max_outer=1, max_inner=3, inner_start=1e-9, inner_precond=0)
    try:
        Rg, _, yg, st = alm.alm_solve(h, R, y)
    finally:
        alm.alm_destroy(h)
    assert st["inner_total"] == 3
    X = R.astype(np.float32).astype(np.float64) if prec else R
    Z, Dd, zg_prev = np.zeros_like(X), np.zeros_like(X), 0.0
    for _ in range(3):
        G = O.gradient(P, X, y, 1.0)
        zg, go = float((G * G).sum()), float((G * Z).sum())
        beta = max(0.0, (zg - go) / zg_prev) if zg_prev > 0 else 0.0
        if -zg + beta * float((G * Dd).sum()) >= 0:
            beta = 0.0
        Dd, Z, zg_prev = -G + beta * Dd, G, zg
        X = X + O.exact_step(O.quartic_coeffs(P, X, Dd, y, 1.0)) * Dd
    assert rel_err(as_np(Rg), X) <= (2e-4 if prec else 1e-10)
    assert rel_err(as_np(yg), O.dual_candidate(P, X, y, 1.0)) <= (2e-4 if prec else 1e-10)
