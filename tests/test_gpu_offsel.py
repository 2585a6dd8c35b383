"""The inner loop's slack update of off-diagonal selectors where S is a small difference of large
terms: residuals of 1e4, a multiplier close to sigma times the residual, and a sigma that is no
float.  The FP32 form's step is held against the FP64 form's from the same factor: its factor is
rounded to 2^-24, S to 2^-24 of itself, and the step length and the gradient come from FP32 sums of
a few hundred terms, each good to about 1e-6; 2e-5 of the largest displacement covers them, and S
rounded at the size of its terms (2^-24 x 1 against 1e-5) would be off by 6e-3."""
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

SIGMA = 1e-4


def cancelling_problem(n, density, r, seed):
    """Selectors on the diagonal (coefficient 1) and on 60% of the edges (0.5), b of size 1e4, and a
    multiplier for which w = y - sigma (A(RR^T) - b) is of size 1e-5."""
    rng = np.random.default_rng(seed)
    inst = si.er_maxcut(n, density, seed=seed)
    ei, ej, _ = inst.graph
    pick = rng.random(ei.size) < 0.6
    k = np.arange(int(pick.sum()))
    inst.a_k = np.concatenate([inst.a_k, n + k]).astype(np.int32)
    inst.a_i = np.concatenate([inst.a_i, ei[pick]]).astype(np.int32)
    inst.a_j = np.concatenate([inst.a_j, ej[pick]]).astype(np.int32)
    inst.a_v = np.concatenate([inst.a_v, np.full(k.size, 0.5)])
    inst.m = n + k.size
    inst.b = 1e4 * rng.uniform(0.5, 2.0, inst.m) * rng.choice([-1.0, 1.0], inst.m)
    inst.c_v = inst.c_v * 1e-5
    R = rng.standard_normal((n, r)).astype(np.float32).astype(np.float64)
    small = 1e-5 * rng.uniform(-1.0, 1.0, inst.m)
    small[:n] = -3e-5  # S_ii = C_ii - w_i positive
    P = O.OracleProblem(inst)
    y = SIGMA * (O.amap(P, R) - inst.b) + small
    return inst, R, y


@pytest.mark.parametrize("n,density,r", [(60, 0.2, 1), (150, 0.1, 5), (400, 0.7, 3)])
def test_small_slack_of_large_terms(n, density, r):
    inst, R, y = cancelling_problem(n, density, r, seed=n)
    out = []
    for prec in (alm.ALM_FP64, alm.ALM_FP32):
        h = alm.alm_create(inst, precision=prec, r_max=r, sigma0=SIGMA, max_outer=1, max_inner=1, inner_start=1e-12,
                           inner_precond=0)
        try:
            Rg, _, _, st = alm.alm_solve(h, R, y)
        finally:
            alm.alm_destroy(h)
        assert st["inner_total"] == 1
        out.append(as_np(Rg) - R)
    moved = np.abs(out[0]).max()
    assert moved > 1e-2  # large against the factor's rounding
    assert np.abs(out[1] - out[0]).max() <= 2e-5 * moved
