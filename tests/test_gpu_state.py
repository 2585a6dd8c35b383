"""A call that met non-finite values leaves nothing behind in its handle: the next call on valid
data gives what a fresh handle gives (the same kernels in the same order: the same bits)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import sdp_instances as si  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2505_15775_gb300 import alm  # noqa: E402


def _instance(kind):
    if kind == "torus":  # fixed-width rows: the fused inner step
        return si.torus_maxcut(20, 21, seed=1)
    if kind == "er":  # CSR rows, diagonal selectors
        return si.er_maxcut(300, 0.1, seed=1)
    if kind == "mc":  # off-diagonal selectors
        return si.matrix_completion(60, 70, 2, seed=1)
    return si.theta_er(200, 8.0, seed=1)  # selectors, a general constraint, low-rank C


@pytest.mark.parametrize("prec", [alm.ALM_FP64, alm.ALM_FP32])
@pytest.mark.parametrize("first", ["eval", "grad", "linesearch", "solve"])
@pytest.mark.parametrize("kind", ["torus", "er", "mc", "theta"])
def test_solve_after_a_call_with_nan(kind, first, prec):
    inst = _instance(kind)
    r = 4
    rng = np.random.default_rng(0)
    R = rng.standard_normal((inst.n, r)) * (0.3 if kind == "mc" else 1.0 / np.sqrt(r * (inst.n if kind == "theta" else 1)))
    y = np.full(inst.m, -3.0) if inst.kind == "maxcut" else 0.1 * rng.standard_normal(inst.m)
    bad = R.copy()
    bad[3, 1] = np.nan
    options = dict(precision=prec, r_max=r, max_outer=2, max_inner=4, inner_start=1e-9)

    def solve(h):
        try:
            Rg, _, yg, st = alm.alm_solve(h, R, y)
        finally:
            alm.alm_destroy(h)
        return Rg, yg, st["objective"], st["inner_total"]

    want = solve(alm.alm_create(inst, **options))
    assert bool(torch.isfinite(want[0]).all())
    h = alm.alm_create(inst, **options)
    Rb, D = alm.factor_tensor(h, bad), alm.factor_tensor(h, 0.1 * R)
    calls = dict(eval=lambda: alm.alm_eval(h, Rb, r, y, 1.0), grad=lambda: alm.alm_grad(h, Rb, r, y, 1.0),
                 linesearch=lambda: alm.alm_linesearch(h, Rb, D, r, y, 1.0), solve=lambda: alm.alm_solve(h, bad, y))
    if first == "grad":
        assert not np.isfinite(calls[first]()[1])
    else:
        with pytest.raises(alm.AlmError):
            calls[first]()
    got = solve(h)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]) and got[2:] == want[2:]
