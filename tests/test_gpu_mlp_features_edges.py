"""The warm-start features' float32 path at its edges: bit for bit the float64
form (the oracle's) on a nucleus, on the bond and its extension, on the plane
between the nuclei, next to it, far out (underflowing exponentials, tangents of
one), and for many nuclei with ties.
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


def check(T, xyz, nuc, **kw):
    f = T.tagi_mlp_features(torch.tensor(np.ascontiguousarray(xyz), dtype=torch.float64, device="cuda"), nuc, **kw)
    bits = f.cpu().numpy().view(np.uint16).astype(np.uint32) << 16
    np.testing.assert_array_equal(bits.view(np.float32).astype(np.float64), M.features(xyz, nuc, **kw))


@pytest.mark.parametrize("kw", [{}, {"ordered": True}, {"ordered": True, "scale": np.array([5.7, 7.7])},
                                {"scale": np.array([1.0, 30.0])}])
def test_special_points(T, kw):
    R = 1.375
    nuc = np.array([[-0.5 * R, 0.0, 0.0], [0.5 * R, 0.0, 0.0]])
    rng = np.random.default_rng(6)
    t = np.concatenate([np.linspace(-30, 30, 4001), rng.uniform(-1, 1, 2000), [-0.5 * R, 0.5 * R, 0.0]])
    z = np.zeros_like(t)
    off = np.concatenate([10.0 ** -rng.uniform(1, 17, 3000), 1.0 + z[3000:]])
    pts = [np.stack([t, z, z]),                                  # the axis: nuclei, bond, extension
           np.stack([z, t, 0.3 * t]),                            # the plane between them
           np.stack([off, t, z]),                       # next to it
           np.stack([t, off, z]),                       # next to the axis
           rng.normal(size=(3, 20000)) * 10.0 ** rng.uniform(-3, 2.3, 20000)]
    check(T, np.concatenate(pts, axis=1), nuc, **kw)


def test_ring_of_nuclei(T):
    nuc = np.array([[x, y, 0.0] for x, y in W.BENZENE_C + W.BENZENE_H])
    rng = np.random.default_rng(8)
    xyz = np.concatenate([rng.normal(size=(3, 50000)) * 4.0, np.stack([np.zeros(500)] * 2 + [np.linspace(-5, 5, 500)]),
                          nuc.T, 0.5 * (nuc[::2] + nuc[1::2]).T], axis=1)
    check(T, xyz, nuc)
