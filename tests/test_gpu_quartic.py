"""The exact line-search step on quartics of every kind that its closed form tells apart: one or
three real stationary points, two of them close together, one far beyond the others (a small
leading coefficient), and scales far from 1.  A problem of two rows with X_ii = b_i gives any
quartic with q4 > 0: rows and direction fix q3 and q4, the multiplier fixes q1 and q2.  The step is
held against the quartic that the call returns."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import sdp_instances as si  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2505_15775_gb300 import alm  # noqa: E402


def _from_stationary_points(p, scale):
    """q1 .. q4 of the quartic with q4 = scale whose derivative vanishes at p."""
    c = np.poly(p)
    return scale * np.array([4 * c[3], 2 * c[2], 4 / 3 * c[1], 1.0])


def _quartics(kind, rng):
    if kind == "three":
        return _from_stationary_points(rng.uniform(-2, 4, 3), 1.0)
    if kind == "one":
        a, p = rng.uniform(-1, 1) * 10 ** rng.uniform(-3, 3), 10 ** rng.uniform(-3, 3)
        b = rng.uniform(-1, 1) * np.sqrt(p)
        c = np.polymul([1, -a], [1, -2 * b, b * b + p])
        return np.array([4 * c[3], 2 * c[2], 4 / 3 * c[1], 1.0])
    if kind == "close":
        a = rng.uniform(0.1, 3)
        return _from_stationary_points([rng.uniform(-3, 3), a, a * (1 + 10 ** rng.uniform(-10, -1))], 1.0)
    if kind == "far":  # a minimum near 1, a stationary point at -1e6 .. -1e9
        e = rng.uniform(0.3, 3.0, 2)
        return _from_stationary_points([e[0], -e[1], -(10 ** rng.uniform(6, 9))], 10 ** rng.uniform(-10, 0))
    p = 10 ** rng.uniform(-12, 12)  # scaled
    return _from_stationary_points(p * rng.uniform(-1, 2, 3), 10 ** rng.uniform(-8, 8) / p**2)


def problem_of(q, b=1.0):
    """(rows, direction, S_11 and S_22) of the two-row problem at sigma = 1 with these q1 .. q4."""
    d = q[3] ** 0.25
    s = q[2] / (2 * d**3)
    rho = np.array([0.63 * s, 0.37 * s]) if s else np.array([1.0, -1.0])
    # q1 = 2 d (S_1 rho_1 + S_2 rho_2), q2 = d^2 (S_1 + S_2) + 2 d^2 |rho|^2
    S = np.linalg.solve(np.array([2 * d * rho, [d**2, d**2]]), [q[0], q[1] - 2 * d**2 * (rho @ rho)])
    return rho, np.array([d, d]), S


@pytest.mark.parametrize("kind", ["three", "one", "close", "far", "scaled"])
def test_step_is_the_minimiser(kind):
    inst = si.maxcut(2, np.array([0]), np.array([1]), np.array([1e-30]))
    diag = np.bincount(inst.c_i[inst.c_i == inst.c_j], inst.c_v[inst.c_i == inst.c_j], 2)
    rng = np.random.default_rng(5)
    h = alm.alm_create(inst, precision=alm.ALM_FP64)
    try:
        for _ in range(200):
            rho, d, S = problem_of(_quartics(kind, rng))
            y = diag + (rho**2 - 1.0) - S
            q, alpha = alm.alm_linesearch(h, alm.factor_tensor(h, rho[:, None]), alm.factor_tensor(h, d[:, None]), 1, y, 1.0)

            def terms(a):
                return np.stack([q[1] * a, q[2] * a**2, q[3] * a**3, q[4] * a**4])

            assert alpha >= 0.0 and np.isfinite(alpha)
            at = terms(np.array([alpha]))
            # no lower point: on a grid of all magnitudes, and close to the step on both sides
            a = np.concatenate([10.0 ** np.linspace(-25, 25, 4001), alpha * (1 + np.array([-1e-2, -1e-4, 1e-4, 1e-2]))])
            t = terms(a)
            slack = 1e-12 * (np.abs(t).sum(0) + np.abs(at).sum())
            assert np.all(at.sum() <= t.sum(0) + slack), (kind, q.tolist(), alpha)
    finally:
        alm.alm_destroy(h)
