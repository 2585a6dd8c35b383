"""The warm-start network's layers at the edges of their row tiles (32 rows, and 128 rows from
one tile a multiprocessor on), with tiles that span instances, against the FP64 oracle, with
FP32 activations.  Tolerances as in test_gpu_gnn.py."""
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

FEAT_SEED = 0x711E
TOL = (1e-5, 1e-4)


def _split(rows):
    """Instances of `rows` rows in all: a large one, then small ones of 1, 2, .. rows."""
    sizes, k = [], 1
    while rows > 40 and k < 8:
        sizes.append(k)
        k += 1
    return [rows - sum(sizes)] + sizes


def _graph(n, seed):
    rng = np.random.default_rng(seed)
    if n < 3:
        z = np.zeros(0, np.int64)
        return si.maxcut(n, z, z, np.zeros(0))
    code = np.unique(rng.integers(0, n, 2 * n) * n + rng.integers(0, n, 2 * n))
    i, j = code // n, code % n
    i, j = i[i < j], j[i < j]
    return si.maxcut(n, i, j, rng.choice([-1.0, 1.0], i.size))


@pytest.mark.parametrize("tiles,width,extra", [(0, 32, 1), (1, 32, -1), (1, 32, 0), (1, 32, 1), (4, 32, 5),
                                               ("sms", 128, -1), ("sms", 128, 0), ("sms", 128, 129)])
def test_layers_at_tile_edges(tiles, width, extra):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = (sms if tiles == "sms" else tiles) * width + extra
    insts = [_graph(n, 7 + k) for k, n in enumerate(_split(rows))]
    graphs = [OG.Graph(x) for x in insts]
    th = (OG.init_params(9) * 1.2).astype(np.float32)
    th64 = th.astype(np.float64)
    rng = np.random.default_rng(rows)
    Rs = [(lambda a: (a / np.linalg.norm(a, axis=1, keepdims=True)).astype(np.float32))(
        rng.standard_normal((x.n, 32))) for x in insts]
    ys = [rng.uniform(-2.0, 0.0, x.n) for x in insts]
    hb = alm.alm_batch_create(insts)
    g = alm.alm_gnn_create(alm.ALM_GNN_FP32, feat_seed=FEAT_SEED)
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
    tf, tg = TOL
    assert rhat.shape[0] == rows
    assert rel_err(rhat, ro, max(1.0, np.abs(ro).max())) <= tf
    assert rel_err(yhat, yo, max(1.0, np.abs(yo).max())) <= tf
    Lo, go = OG.loss_and_grad(th64, graphs, FEAT_SEED, [r.astype(np.float64) for r in Rs], ys, 0.05)
    assert loss == pytest.approx(Lo, rel=tf)
    assert rel_err(grad, go, np.abs(go).max()) <= tg
