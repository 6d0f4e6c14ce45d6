"""The float64 pair forms (table-driven exponential, corrected reciprocal root)
where they can go wrong: the ends of their range, where the math library takes
over, exponents from 0 to underflow, coincident points, and field counts at the
edges of a launch group.  Against the float64 oracle's direct sum, 1e-12 of the
field's largest value (rounding order, as the other float64 parity tests).
"""
import numpy as np
import pytest

import oracle
from paper_2003_01833_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-12


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


def points(n, scale, seed):
    """Random points, some of them 1e-6 of the cube apart, two coincident."""
    xyz, w = W.random_cube(n, seed=seed)
    xyz[:, 1::7] = xyz[:, 0:-1:7][:, :xyz[:, 1::7].shape[1]] * (1 + 1e-6)
    xyz[:, 5] = xyz[:, 4]
    return np.ascontiguousarray(xyz * scale), w


# 1e-12 .. 1e9 lie inside the fast range of r (2^-35 to 2^35) in part or in
# whole, 1e-20 and 1e13 outside it
@pytest.mark.parametrize("scale", [1e-20, 1e-12, 1e-3, 1.0, 1e9, 1e13])
@pytest.mark.parametrize("nf", [1, 4, 5])
def test_direct_sums_over_ranges(T, scale, nf):
    n = 301
    xyz, w = points(n, scale, seed=nf)
    f = np.stack([1.0 + 0.3 * np.sin(np.arange(n) + o) for o in range(nf)])
    k = [v / scale for v in (1.3, 1e-9, 40.0, 700.0, 3e4)[:nf]]
    u, v = (torch.empty((nf, n), dtype=torch.float64, device="cuda") for _ in range(2))
    T.tagi_yukawa_direct_noalloc(dev(xyz), dev(w), dev(f), k, u)
    with T.Tree(dev(xyz), dev(w), theta=0.0, degree=2, leaf_size=100, prec=T.TAGI_FP64) as tr:
        T.tagi_yukawa_conv(tr.handle, dev(f), k, v)
    for o in range(nf):
        ref = oracle.direct_yukawa(xyz, w, f[o], k[o])
        for got in (u, v):
            assert np.abs(got[o].cpu().numpy() - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("ss", [True, False])
@pytest.mark.parametrize("nf_y", [0, 1, 3, 4, 5])
def test_groups_of_fields(T, ss, nf_y):
    """A field's sums do not depend on the fields it shares a launch with: bit
    for bit those of the field alone.  The Hartree field also against the
    oracle."""
    n = 1003
    xyz, w = points(n, 3.0, seed=9)
    rho = np.exp(-np.sum(xyz * xyz, axis=0))
    f = dev(np.stack([np.cos(xyz[0] + o) for o in range(nf_y)])) if nf_y else None
    k = [0.5 + o for o in range(nf_y)]
    u = torch.empty_like(f) if nf_y else None
    vh, alone = torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.float64, device="cuda")
    with T.Tree(dev(xyz), dev(w), theta=0.0, degree=2, leaf_size=300, prec=T.TAGI_FP64, ss=ss) as tr:
        T.tagi_fields_conv(tr.handle, f, k, u, rho=dev(rho), vh=vh)
        T.tagi_coulomb_conv(tr.handle, dev(rho), alone)
        assert torch.equal(alone, vh)
        for o in range(nf_y):
            T.tagi_yukawa_conv(tr.handle, f[o].contiguous(), [k[o]], alone)
            assert torch.equal(alone, u[o])
    ref = oracle.direct_coulomb(xyz, w, rho, ss=ss)
    assert np.abs(vh.cpu().numpy() - ref).max() <= TOL * np.abs(ref).max()
