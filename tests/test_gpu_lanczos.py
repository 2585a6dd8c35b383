"""The eigensolve at the sizes where its kernels can go wrong: bases of 1 to 64 vectors
(tridiagonal matrices down to one row), vectors around the sizes of tiles and groups, both
precisions, and starts whose Krylov space is exhausted early."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
import sdp_instances as si  # noqa: E402
from gpu_common import as_np  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2505_15775_gb300 import alm  # noqa: E402

# relative to the norm of S: the eigenvalue error is at most the residual, which the solver takes
# to 1e-10 (FP64) or 1e-5 (FP32, the least it accepts) of its norm estimate, and the estimate is
# at most the largest row of the tridiagonal, three times the norm
TOL = {0: 3e-10, 1: 3e-5}


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,k", [(1, 2), (2, 2), (3, 3), (5, 8), (33, 2), (33, 32), (65, 33), (255, 64), (257, 32),
                                 (800, 32), (1023, 64), (1025, 31), (4099, 32)])
def test_lambda_min_sizes(n, k, prec):
    inst = si.maxcut(n, *(si.er_edges(n, min(1.0, 6.0 / max(n - 1, 1)), (n, k)) if n > 1 else (np.zeros(0), np.zeros(0))),
                     w=np.ones(si.er_edges(n, min(1.0, 6.0 / max(n - 1, 1)), (n, k))[0].size if n > 1 else 0))
    rng = np.random.default_rng(n + k)
    y = rng.uniform(-1.0, 1.0, n)
    h = alm.alm_create(inst, precision=prec, lanczos_k=k)
    try:
        lam, v, res = alm.alm_lambda_min(h, None, 0, y, 0.0)
    finally:
        alm.alm_destroy(h)
    P = O.OracleProblem(inst)
    S = O.slack_dense(P, y)
    ev = np.linalg.eigvalsh(S)
    norm = max(abs(ev[0]), abs(ev[-1]), 1e-3)
    vv = as_np(v)
    assert abs(np.linalg.norm(vv) - 1.0) <= (1e-5 if prec else 1e-12)
    assert np.linalg.norm(S @ vv - lam * vv) <= TOL[prec] * norm
    assert lam >= ev[0] - (1e-6 if prec else 1e-12) * norm
    assert min(abs(ev - lam)) <= TOL[prec] * norm


@pytest.mark.parametrize("prec", [0, 1])
def test_lambda_min_exhausted_krylov_space(prec):
    """S = C_ii I on the even rows and another multiple on the odd ones: two distinct
    eigenvalues, so the second step of a cycle meets an invariant subspace."""
    n = 1000
    diag = np.arange(n, dtype=np.int64)
    inst = si.maxcut(n, np.zeros(0), np.zeros(0), np.zeros(0))
    inst.c_v = np.where(diag % 2 == 0, 1.0, -0.75)
    h = alm.alm_create(inst, precision=prec)
    try:
        lam, v, res = alm.alm_lambda_min(h, None, 0, np.zeros(n), 0.0)
    finally:
        alm.alm_destroy(h)
    assert lam == pytest.approx(-0.75, abs=1e-6 if prec else 1e-12)
    assert np.linalg.norm(as_np(v)[::2]) <= (1e-4 if prec else 1e-10)
