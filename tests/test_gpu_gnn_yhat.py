"""The multiplier head's sum of 64 products: pairs and halves, 7 roundings deep.  One product of 1 and 63 of just
under a quarter of its last place: added to it one at a time they are all lost."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import sdp_instances as si  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2505_15775_gb300 import alm  # noqa: E402


@pytest.mark.parametrize("storage", [alm.ALM_GNN_FP32, alm.ALM_GNN_BF16])
@pytest.mark.parametrize("n", [100, 30_000])  # tiles of 32 and of 128 rows
def test_yhat_error_bound(n, storage):
    small = np.float32(0.9 * 2.0**-25)
    parts, din = [], 8
    for _ in range(3):  # h = relu(bias) = 1 in every channel of every layer
        parts += [np.zeros(2 * 64 * din), np.ones(64)]
        din = 64
    wy = np.full(64, small, np.float32)
    wy[0] = 1.0
    parts += [np.zeros(32 * 64), wy, np.zeros(1)]
    g = alm.alm_gnn_create(storage, feat_seed=1)
    hb = alm.alm_batch_create([si.maxcut(n, *si.cycle_edges(n), np.ones(n))], r_max=32)
    try:
        alm.alm_gnn_set_params(g, np.concatenate(parts).astype(np.float32))
        _, yhat = alm.alm_gnn_forward(g, hb)
    finally:
        alm.alm_gnn_destroy(g)
        alm.alm_batch_destroy(hb)
    exact = wy.astype(np.float64).sum()
    assert np.abs(yhat.double().cpu().numpy() - exact).max() <= 8 * 2.0**-24 * exact  # the sum and the bias
