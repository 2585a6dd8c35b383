"""The eigensolve around the longest vectors of its one-launch form (6000 in FP64, 8192 in FP32 and for
dense rows) and beyond: the launches with the normalisation fused into the next step, one row and
four rows a thread, bases that are no multiple of eight vectors, an exhausted Krylov space and a
low-rank part.  S has one eigenvalue far below the others, so that the pair found is known to be the
smallest; bars as in test_gpu_lanczos.py."""
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

TOL = {0: 3e-10, 1: 3e-5}


def _check(P, y, lam, v, prec):
    S = O.slack_sparse(P, y)
    norm = float(abs(S).sum(axis=1).max()) + float(np.abs(P.lr_s) @ (P.lr_u ** 2).sum(axis=1))
    assert abs(np.linalg.norm(v) - 1.0) <= (1e-5 if prec else 1e-12)
    assert np.linalg.norm(O.slack_matvec(P, S, v) - lam * v) <= TOL[prec] * norm
    return norm


def _lambda(inst, y, prec, k):
    h = alm.alm_create(inst, precision=prec, lanczos_k=k)
    try:
        lam, v, _ = alm.alm_lambda_min(h, None, 0, y, 0.0)
    finally:
        alm.alm_destroy(h)
    return lam, as_np(v)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,deg,k", [(6000, 6.0, 32), (6001, 6.0, 32), (8192, 6.0, 13), (8192, 260.0, 32), (8193, 6.0, 32),
                                     (8449, 6.0, 5), (9000, 6.0, 63), ("sms", 4.0, 9), ("sms+1", 4.0, 9)])
def test_lambda_min(n, deg, k, prec):
    if isinstance(n, str):  # the last length with one row a thread, the first with four
        n = torch.cuda.get_device_properties(0).multi_processor_count * 1024 - 1024 + (n == "sms+1")
    inst = si.er_maxcut(n, deg / (n - 1), seed=int(deg))
    y = np.random.default_rng(n).uniform(-1.0, 1.0, n)
    low = n // 3
    y[low] += 8.0 * np.sqrt(deg) + 30.0  # S_ii = C_ii - y_i far below the rest of the spectrum
    P = O.OracleProblem(inst)
    lam, v = _lambda(inst, y, prec, k)
    norm = _check(P, y, lam, v, prec)
    assert v[low] ** 2 > 0.5  # the pair of the low entry: every other eigenvalue is far above
    assert lam < -0.4 * norm


@pytest.mark.parametrize("prec", [0, 1])
def test_exhausted_krylov_space(prec):
    n = 9001
    diag = np.arange(n, dtype=np.int64)
    inst = si.maxcut(n, np.zeros(0), np.zeros(0), np.zeros(0))
    inst.c_v = np.where(diag % 2 == 0, 1.0, -0.75)
    lam, v = _lambda(inst, np.zeros(n), prec, 32)
    assert lam == pytest.approx(-0.75, abs=1e-6 if prec else 1e-12)
    assert np.linalg.norm(v[::2]) <= (1e-4 if prec else 1e-10)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [5000, 8300])
def test_low_rank_part(n, prec):
    inst = si.theta_er(n, 6.0, seed=2)  # C = -1 1^T
    y = np.random.default_rng(n).uniform(-1.0, 1.0, inst.m)
    lam, v = _lambda(inst, y, prec, 12)
    _check(O.OracleProblem(inst), y, lam, v, prec)
    assert lam < -0.9 * n and abs(v.sum()) > 0.9 * np.sqrt(n)
