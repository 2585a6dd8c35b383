"""Row lengths at which the CSR kernels change their form: rows shared by the subgroups of a
warp or not, rows cut into segments (128 upper entries), rows summed by a CTA each (more than
256 entries), general constraints cut into chunks (256 entries) -- and the inner loop's slack
update of off-diagonal selectors against the general path.  Bars as in the primitives' tests
(FP64 1e-12, FP32 1e-5 of the largest magnitude of the compared terms)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
import sdp_instances as si  # noqa: E402
from gpu_common import RTOL, as_np, rel_err  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2505_15775_gb300 import alm  # noqa: E402


def _hubs(degrees, n):
    """MaxCut on hubs 0, 1, .. of the given degrees towards random distinct other vertices."""
    rng = np.random.default_rng(len(degrees) + n)
    ei, ej = [], []
    for h, d in enumerate(degrees):
        ei.append(np.full(d, h, np.int64))
        ej.append(np.sort(rng.choice(np.arange(len(degrees), n), size=d, replace=False)))
    ei, ej = np.concatenate(ei), np.concatenate(ej)
    return si.maxcut(n, ei, ej, rng.uniform(-1, 1, ei.size))


def _check_primitives(inst, r, prec):
    P = O.OracleProblem(inst)
    rng = np.random.default_rng(r)
    R, D = rng.standard_normal((inst.n, r)) / np.sqrt(r), 0.1 * rng.standard_normal((inst.n, r))
    y = rng.uniform(-1, 1, inst.m)
    h = alm.alm_create(inst, precision=prec)
    try:
        Rd, Dd = alm.factor_tensor(h, R), alm.factor_tensor(h, D)
        Rq, Dq = as_np(Rd)[:, :r], as_np(Dd)[:, :r]
        L, AX, CX = alm.alm_eval(h, Rd, r, y, 0.7)
        G, g2 = alm.alm_grad(h, Rd, r, y, 0.7)
        q, _ = alm.alm_linesearch(h, Rd, Dd, r, y, 0.7)
    finally:
        alm.alm_destroy(h)
    w = O.dual_candidate(P, Rq, y, 0.7)
    big = max(1.0, float(np.max(np.abs(O.slack_sparse(P, w)).sum(axis=1))))
    ax = O.amap(P, Rq)
    assert rel_err(as_np(AX), ax) <= RTOL[prec]
    cost = max(1.0, float(np.abs(inst.c_v).sum()))
    assert abs(CX - O.cost(P, Rq)) <= RTOL[prec] * cost
    Go = O.gradient(P, Rq, y, 0.7)
    assert rel_err(as_np(G)[:, :r], Go, 2 * big * max(1.0, float(np.abs(Rq).max()))) <= RTOL[prec]
    a0, a1, a2 = ax - P.b, 2 * O.amap(P, Rq, Dq), O.amap(P, Dq)
    mag = max(1.0, cost, float(np.abs(y) @ (np.abs(a1) + np.abs(a2))), 0.7 * float(np.abs(a0) @ (np.abs(a1) + np.abs(a2))),
              0.7 * float(a1 @ a1 + a2 @ a2), float(np.abs(y) @ np.abs(a0)) + 0.35 * float(a0 @ a0))
    assert rel_err(q, O.quartic_coeffs(P, Rq, Dq, y, 0.7), mag) <= 4 * RTOL[prec]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("r", [1, 5, 13, 32])
@pytest.mark.parametrize("degrees,n", [((17, 1), 40), ((127, 128, 129), 400), ((255, 256, 257), 400),
                                       ((1, 600, 300, 2), 1001), ((900,) * 3, 1000)])
def test_row_lengths(degrees, n, r, prec):
    _check_primitives(_hubs(degrees, n), r, prec)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("r", [1, 5, 32])
@pytest.mark.parametrize("degrees,n", [((511, 512, 513), 700), ((1024, 1025, 257, 3), 1100), ((6000, 2049), 6500)])
def test_long_rows_in_segments(degrees, n, r, prec):
    """Rows summed by several CTAs (512 entries each)."""
    _check_primitives(_hubs(degrees, n), r, prec)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("r", [3, 32])
@pytest.mark.parametrize("count", [1, 255, 256, 257, 1000])
def test_general_constraint_lengths(count, r, prec):
    """A constraint over `count` diagonal entries, one over as many off-diagonal ones, and selectors."""
    n = 1100
    rng = np.random.default_rng(count)
    inst = si.maxcut(n, *si.cycle_edges(n), np.ones(n))
    i = np.arange(count)
    inst.a_k = np.concatenate([inst.a_k, np.full(count, n), np.full(count, n + 1)]).astype(np.int32)
    inst.a_i = np.concatenate([inst.a_i, i, i]).astype(np.int32)
    inst.a_j = np.concatenate([inst.a_j, i, i + 7]).astype(np.int32)
    inst.a_v = np.concatenate([inst.a_v, rng.uniform(-1, 1, 2 * count) / count])
    inst.b = np.concatenate([inst.b, [0.3, -0.2]])
    inst.m = n + 2
    _check_primitives(inst, r, prec)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("coef", [0.5, 0.3])
@pytest.mark.parametrize("r", [2, 9])
def test_off_diagonal_selector_steps(r, coef, prec):
    """Three inner steps of a problem with selectors on and off the diagonal, against the
    oracle's steps from the same start (coefficient 0.5 takes the FP32 form's slack update
    without FP64, 0.3 is no float and takes the general one)."""
    n = 150
    rng = np.random.default_rng(r)
    inst = si.er_maxcut(n, 0.1, seed=r)
    ei, ej, _ = inst.graph
    pick = rng.random(ei.size) < 0.6
    k = np.arange(int(pick.sum()))
    inst.a_k = np.concatenate([inst.a_k, n + k]).astype(np.int32)
    inst.a_i = np.concatenate([inst.a_i, ei[pick]]).astype(np.int32)
    inst.a_j = np.concatenate([inst.a_j, ej[pick]]).astype(np.int32)
    inst.a_v = np.concatenate([inst.a_v, np.full(k.size, coef)])
    inst.b = np.concatenate([inst.b, rng.uniform(-0.3, 0.3, k.size)])
    inst.m = n + k.size
    P = O.OracleProblem(inst)
    R = rng.standard_normal((n, r))
    R /= np.linalg.norm(R, axis=1, keepdims=True)
    y = np.concatenate([np.full(n, -3.0), rng.uniform(-0.1, 0.1, k.size)])
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
