"""Norms of the short eigensolve (vectors of up to 8192 entries) in its FP32 form: the start vector's and the
Ritz vector's squares are summed in FP64.  With S = 0 the Krylov space ends at the start vector, and
the returned eigenvector is that vector, normalised twice: its bits follow from the two sums.
(Sums in FP32 within a warp give another factor at 3000 and 4000 entries.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import sdp_instances as si  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2505_15775_gb300 import alm  # noqa: E402


def _start(seed, n):
    """Uniform in [-1, 1): SplitMix64 as a counter, rounded to float."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (2.0 * ((z >> np.uint64(11)).astype(np.float64) / 9007199254740992.0) - 1.0).astype(np.float32)


def _normalised(x, squares):
    return x * np.float32(1.0 / np.sqrt(squares.astype(np.float64).sum()))


@pytest.mark.parametrize("n", [64, 997, 3000, 4000, 5000, 8192])
def test_norms_are_summed_in_fp64(n):
    inst = si.maxcut(n, np.array([0]), np.array([1]), np.array([1.0]))
    inst.c_i = inst.c_j = np.arange(n, dtype=np.int32)  # C = I, no off-diagonal entry
    inst.c_v = np.ones(n)
    h = alm.alm_create(inst, precision=alm.ALM_FP32)
    try:
        R = alm.factor_tensor(h, np.ones((n, 1)))
        lam, v, _ = alm.alm_lambda_min(h, R, 1, np.ones(n), 1.0)  # S = C - diag(1) = 0
        seed = h.options.seed
    finally:
        alm.alm_destroy(h)
    assert lam == 0.0
    x = _start(seed, n)
    q = _normalised(x, x.astype(np.float64) ** 2)
    assert np.array_equal(v.cpu().numpy().ravel(), _normalised(q, q * q))
