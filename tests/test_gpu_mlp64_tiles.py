"""The H = 64 gradient where its tiles are shared out: single points, ragged
tiles, exactly eight tiles for each SM (one CTA each) and one more (two CTAs
that take groups of eight in turn).  Bounds as in the other H = 64 tests:
loss 1e-5, gradient 2e-3 relative L2 against the oracle's tensor-core form.
"""
import numpy as np
import pytest

from oracle import mlp as M
from paper_2003_01833_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import __graft_entry__ as g

    g.build()
    import paper_2003_01833_gb300.tagi as T

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return T


@pytest.mark.parametrize("tiles,extra", [(0, 1), (1, -1), (1, 1), (152, 1), (152 * 8, 0), (152 * 8, 1),
                                         (152 * 17, -5)])
def test_gradient_at_tile_edges(T, tiles, extra):
    n = 128 * tiles + extra
    rng = np.random.default_rng(n)
    nuc = [[-0.75, 0.0, 0.0], [0.75, 0.0, 0.0]]
    xyz = torch.tensor(rng.normal(size=(3, n)) * 2.0, dtype=torch.float64, device="cuda")
    feat = T.tagi_mlp_features(xyz, nuc)
    x = (feat.cpu().numpy().view(np.uint16).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    t = (0.3 * np.tanh(rng.normal(size=n))).astype(np.float32)
    wt = (rng.uniform(0.5, 1.5, size=n) / n).astype(np.float32)
    p = W.mlp_init(3, hidden=64) + 0.1
    with T.Mlp(p, hidden=64) as m:
        loss, g = m.gradient(feat, torch.tensor(t, device="cuda"), torch.tensor(wt, device="cuda"))
    lo, go = M.loss_grad_tc(p, x, t.astype(np.float64), wt.astype(np.float64), 64)
    assert abs(loss - lo) <= 1e-5 * lo
    assert np.linalg.norm(g - go) <= 2e-3 * np.linalg.norm(go)
