"""The near/far kernel's items: batches whose target counts sit at the edges
of its warps and items (64 targets a warp, 128 an item), and lists cut into
items at other places.  Parity with the
float64 oracle within the stated FP32C tolerance, relative L2 1e-6 per field.
"""
import numpy as np
import pytest

import oracle
from paper_2003_01833_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FP32C_TOL = 1e-6


@pytest.fixture(scope="module")
def T():
    import __graft_entry__ as g

    g.build()
    import paper_2003_01833_gb300.tagi as T

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return T


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def check(T, n, leaf, degree, seed, ss=True):
    xyz, w = W.random_cube(n, seed=seed)
    f = 1.0 + 0.3 * np.sin(3 * xyz[0]) * np.cos(2 * xyz[1])
    rho = np.exp(-np.sum(xyz * xyz, axis=0))
    with T.Tree(dev(xyz), dev(w), theta=0.7, degree=degree, leaf_size=leaf, prec=T.TAGI_FP32C, ss=ss) as tr:
        u, vh = torch.empty((1, n), dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.float64,
                                                                                    device="cuda")
        T.tagi_fields_conv(tr.handle, dev(f), [1.7], u, rho=dev(rho), vh=vh)
        u, vh = u.cpu().numpy()[0], vh.cpu().numpy()
    ot = oracle.Tree(xyz, leaf)
    for got, ref in ((u, oracle.treecode_yukawa(ot, 0.7, degree, f, 1.7, w, ss=ss)),
                     (vh, oracle.treecode_coulomb(ot, 0.7, degree, rho, w, ss=ss))):
        assert np.linalg.norm(got - ref) <= FP32C_TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [2, 17, 33, 63, 64, 65, 127, 128, 129, 191, 193, 255, 256, 257, 300, 513])
def test_one_batch_at_the_edges(T, n):
    check(T, n, 600, 6, seed=n)


@pytest.mark.parametrize("degree", [5, 6, 8])  # record path, tensor-grid path with 7 and 9 nodes
@pytest.mark.parametrize("leaf", [40, 90, 180, 700])
def test_far_field_over_batch_sizes(T, degree, leaf):
    check(T, 12007, leaf, degree, seed=leaf + degree)


def test_without_subtraction(T):
    check(T, 5003, 90, 6, seed=4, ss=False)


@pytest.mark.parametrize("prec", ["FP32C", "FP64"])
@pytest.mark.parametrize("n,leaf,degree", [(12007, 3000, 8), (12007, 333, 6), (3001, 4000, 9)])
def test_items_may_cut_an_entry(T, n, leaf, degree, prec):
    """The item length regroups whole folds of 16 sources: two-float sums
    (2^-48 of the partial sums a fold, about 1e3 folds, SS cancellation of at
    most 1e2 on the cube) and float64 ones move by less than 1e-9."""
    xyz, w = W.random_cube(n, seed=7)
    f = 1.0 + 0.3 * np.sin(3 * xyz[0]) * np.cos(2 * xyz[1])
    out = []
    for segment in (0, 1024, 65536):
        with T.Tree(dev(xyz), dev(w), theta=0.6, degree=degree, leaf_size=leaf, prec=getattr(T, "TAGI_" + prec),
                    segment=segment) as tr:
            u = torch.empty((1, n), dtype=torch.float64, device="cuda")
            T.tagi_yukawa_conv(tr.handle, dev(f), [2.3], u)
            out.append(u.cpu().numpy()[0])
    for a in out[:2]:
        assert np.linalg.norm(a - out[2]) <= 1e-9 * np.linalg.norm(out[2])
