"""alm_eval where it walks the upper entries by rows (FP32 factors of 30 MB or more with at most two entries a
row) and just below, with a row of several segments among them, against the oracle.  Bars as in the
primitives' tests: 1e-5 of the compared terms' magnitude."""
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


@pytest.mark.parametrize("r,n", [(32, 240_001), (32, 234_000), (29, 240_001), (5, 1_000_003)])
def test_eval(r, n):
    prec = alm.ALM_FP32
    rng = np.random.default_rng(r)
    ei, ej = si.cycle_edges(n)
    hub = np.arange(2, 402)  # row 0: 400 more entries, all of them upper
    ei, ej = np.concatenate([ei, np.zeros(hub.size, np.int64)]), np.concatenate([ej, hub])
    inst = si.maxcut(n, ei, ej, rng.uniform(-1, 1, ei.size))
    P = O.OracleProblem(inst)
    R = (rng.standard_normal((n, r)) / np.sqrt(r)).astype(np.float32)
    y = rng.uniform(-1, 1, inst.m)
    h = alm.alm_create(inst, precision=prec)
    try:
        L, AX, CX = alm.alm_eval(h, alm.factor_tensor(h, R), r, y, 0.7)
    finally:
        alm.alm_destroy(h)
    Rq = R.astype(np.float64)
    ax = O.amap(P, Rq)
    assert rel_err(as_np(AX), ax) <= RTOL[prec]
    cost = float(np.abs(inst.c_v).sum())
    assert abs(CX - O.cost(P, Rq)) <= RTOL[prec] * cost
    a0 = ax - P.b
    assert abs(L - O.aug_lagrangian(P, Rq, y, 0.7)) <= RTOL[prec] * (cost + float(np.abs(y) @ np.abs(a0)) + 0.35 * float(a0 @ a0))
