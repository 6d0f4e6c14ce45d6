"""The work items of the near/far kernel: a segment that the caller passes is
the one that the tree is cut with (whole entries until they hold that many
sources), the default one only on trees with enough items, and the sums of
every cut agree with the float64 oracle within the stated tolerances of the two
forms (relative L2 1e-6 per field, FP32C; 1e-12 of the largest value, FP64).
"""
import numpy as np
import pytest

import oracle
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


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def items_of(T, tr, segment):
    """Number of items where each takes whole list entries until they hold
    `segment` sources, padded to 8 each, for every 128 targets of a batch."""
    ex = T.tagi_tree_export(tr.handle)
    batch, cluster, kind = T.tagi_tree_lists(tr.handle)
    size = ex["end"] - ex["begin"]
    src = np.where(kind == 1, T.tagi_tree_info(tr.handle)["n_proxies"], size[cluster])
    total = 0
    for b in np.unique(batch):
        runs, held = 0, 0
        for s in src[batch == b]:
            held += (int(s) + 7) // 8 * 8
            if held >= segment:
                runs, held = runs + 1, 0
        total += (int(size[b]) + 127) // 128 * (runs + (held > 0))
    return total


@pytest.mark.parametrize("prec", ["FP32C", "FP64"])
@pytest.mark.parametrize("n,leaf,degree", [(12007, 3000, 8), (12007, 333, 6), (9001, 700, 5)])
def test_given_segment_holds(T, n, leaf, degree, prec):
    xyz, w = W.random_cube(n, seed=7)
    f = 1.0 + 0.3 * np.sin(3 * xyz[0]) * np.cos(2 * xyz[1])
    ref = oracle.treecode_yukawa(oracle.Tree(xyz, leaf), 0.6, degree, f, 2.3, w)
    items, u = [], torch.empty((1, n), dtype=torch.float64, device="cuda")
    for segment in (0, 1024, 65536):
        with T.Tree(dev(xyz), dev(w), theta=0.6, degree=degree, leaf_size=leaf, prec=getattr(T, "TAGI_" + prec),
                    segment=segment) as tr:
            items.append(T.tagi_tree_info(tr.handle)["n_items"])
            if segment:
                assert items[-1] == items_of(T, tr, segment)
            T.tagi_yukawa_conv(tr.handle, dev(f), [2.3], u)
        got = u.cpu().numpy()[0]
        if prec == "FP64":
            assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
        else:
            assert np.linalg.norm(got - ref) <= 1e-6 * np.linalg.norm(ref)
    assert items[0] > items[1] > items[2]  # three different cuts


def test_default_segment_on_a_large_tree(T):
    """8192 sources an item where that makes 2000 items or more."""
    xyz, w = W.random_cube(60000, seed=3)
    with T.Tree(dev(xyz), dev(w), theta=0.0, degree=1, leaf_size=500, prec=T.TAGI_FP64) as tr:
        assert T.tagi_tree_info(tr.handle)["n_items"] == items_of(T, tr, 8192)
