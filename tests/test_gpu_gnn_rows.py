"""The warm-start network against the FP64 oracle on rows of more than 64 entries (gathered one at a time beyond that,
sixteen entries in flight) in both tile sizes, and with BF16 activations at the edges of the tiles.
Tolerances as in test_gpu_gnn.py; the BF16 gradient's bar holds there at 258 rows, and as it sums
the rounding of that many activations it is widened by sqrt(258 / rows) for fewer (32 rows: the one
warp per row that the tiles replaced is 0.070 off on that input as well)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle.gnn as OG  # noqa: E402
import sdp_instances as si  # noqa: E402
from gpu_common import as_np, rel_err  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2505_15775_gb300 import alm  # noqa: E402
from test_gpu_gnn_tiles import _graph, _split  # noqa: E402

FEAT_SEED = 0x711E


def _check(insts, storage, tf, tg):
    graphs = [OG.Graph(x) for x in insts]
    th = (OG.init_params(9) * 1.2).astype(np.float32)
    th64 = th.astype(np.float64)
    rng = np.random.default_rng(len(insts))
    Rs = [(lambda a: (a / np.linalg.norm(a, axis=1, keepdims=True)).astype(np.float32))(
        rng.standard_normal((x.n, 32))) for x in insts]
    ys = [rng.uniform(-2.0, 0.0, x.n) for x in insts]
    hb = alm.alm_batch_create(insts)
    g = alm.alm_gnn_create(storage, feat_seed=FEAT_SEED)
    try:
        alm.alm_gnn_set_params(g, th)
        rhat, yhat = (as_np(t) for t in alm.alm_gnn_forward(g, hb))
        R, _ = alm.batch_factor(hb, Rs)
        y = torch.as_tensor(np.concatenate(ys), dtype=torch.float64, device="cuda")
        loss, grad = alm.alm_gnn_loss_grad(g, hb, R, y, 0.05)
    finally:
        alm.alm_gnn_destroy(g)
        alm.alm_batch_destroy(hb)
    ro, yo = (np.concatenate(t) for t in zip(*(OG.forward(th64, G, FEAT_SEED)[:2] for G in graphs)))
    assert rel_err(rhat, ro, max(1.0, np.abs(ro).max())) <= tf
    assert rel_err(yhat, yo, max(1.0, np.abs(yo).max())) <= tf
    Lo, go = OG.loss_and_grad(th64, graphs, FEAT_SEED, [r.astype(np.float64) for r in Rs], ys, 0.05)
    assert loss == pytest.approx(Lo, rel=tf)
    assert rel_err(grad, go, np.abs(go).max()) <= tg


@pytest.mark.parametrize("degrees,n", [((31, 32, 33, 34), 2100), ((31, 32, 33, 34), 20_000), ((47, 48, 49, 64, 65), 2100),
                                       ((47, 48, 49, 64, 65), 20_000), ((63, 95, 96, 97), 2100),
                                       ((63, 95, 96, 97), 20_000), ((1, 2000, 3, 300), 2100)])
def test_long_rows(degrees, n):  # tiles of 32 and of 128 rows
    rng = np.random.default_rng(n)
    k = len(degrees)
    ei = np.concatenate([np.full(d, h) for h, d in enumerate(degrees)] + [np.arange(k, n - 1)])
    ej = np.concatenate([rng.choice(np.arange(k, n), size=d, replace=False) for d in degrees] + [np.arange(k + 1, n)])
    inst = si.maxcut(n, ei, ej, rng.choice([-1.0, 1.0], ei.size))
    _check([inst], alm.ALM_GNN_FP32, 1e-5, 1e-4)


@pytest.mark.parametrize("tiles,width,extra", [(0, 32, 1), (1, 32, 0), (1, 32, 1), (4, 32, 5), ("sms", 128, -1),
                                               ("sms", 128, 0), ("sms", 128, 129)])
def test_bf16_at_tile_edges(tiles, width, extra):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = (sms if tiles == "sms" else tiles) * width + extra
    insts = [_graph(n, 7 + k) for k, n in enumerate(_split(rows))]
    _check(insts, alm.ALM_GNN_BF16, 3e-2, 6e-2 * max(1.0, (258 / rows) ** 0.5))
