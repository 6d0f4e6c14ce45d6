"""Single pairs of the float64 forms, one source seen by every target, where the
reciprocal root's approximation may lie on the other side of a power of two, and
where the exponential is below float64's normal range.  Against float64 and
extended arithmetic on the host.  Groups of fields against the float64 oracle.
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


def pair_values(T, r, k, weight):
    """4 pi times the field that a source of value 1 and quadrature weight
    `weight` at the origin makes at distances r along x, where nothing else has
    a weight: by the direct sum and by the tree form with and without subtraction."""
    n = len(r) + 1
    xyz = np.zeros((3, n))
    xyz[0, 1:] = r
    w, f = np.zeros(n), np.zeros((1, n))
    w[0], f[0, 0] = weight, 1.0
    u = torch.empty((1, n), dtype=torch.float64, device="cuda")
    T.tagi_yukawa_direct_noalloc(dev(xyz), dev(w), dev(f), [k], u)
    yield u.cpu().numpy()[0, 1:] * 4 * np.pi
    for ss in (True, False):
        with T.Tree(dev(xyz), dev(w), theta=0.0, degree=2, leaf_size=n, prec=T.TAGI_FP64, ss=ss) as tr:
            T.tagi_yukawa_conv(tr.handle, dev(f), [k], u)
        yield u.cpu().numpy()[0, 1:] * 4 * np.pi


def test_distances_next_to_powers_of_two(T):
    """32 float32 values of r^2 on each side of every power of four in the fast
    range.  Units of 2^-52: an ulp of the exponential, half of the final product
    and of k r (here below 2^-5), three roundings of the factor 4 pi and its
    quotient here."""
    p = np.arange(-34, 35)
    r2 = np.concatenate([(np.float32(4.0) ** p.astype(np.float32)).view(np.int32) + j for j in range(-32, 33)])
    r = np.sqrt(np.unique(r2).astype(np.int32).view(np.float32).astype(np.float64))
    k = 2.0 ** -40
    exact = np.exp(-k * r.astype(np.longdouble)) / r
    for got in pair_values(T, r, k, 1.0):
        assert np.max(np.abs(got / exact - 1)) <= 5 * 2.0 ** -52


def test_exponentials_below_the_normal_range(T):
    """k r from 690 to 750, a weight of 2^1000: the exponential's subnormal values
    (spacing 2^-1074) count.  Half a spacing beside the relative bound: an ulp of
    the exponential, half of the final product and of k r, four roundings of the
    weight, the factor 4 pi and its quotient here."""
    r = np.arange(690.0, 750.0, 0.25)
    e = np.exp(-r.astype(np.longdouble))
    exact = e / r * 2.0 ** 1000
    bound = (np.longdouble(2.0) ** -1075 + (6 + r) * 2.0 ** -52 * e) / r * 2.0 ** 1000
    for got in pair_values(T, r, 1.0, 2.0 ** 1000):
        assert np.all(np.abs(got - exact) <= bound)


@pytest.mark.parametrize("ss", [True, False])
@pytest.mark.parametrize("nf_y", [1, 3, 4, 5])
def test_groups_of_yukawa_fields(T, ss, nf_y):
    """With Hartree beside them, points 1e-6 apart and two coincident.  1e-12 of
    the field's largest value, as the other float64 parity tests, and beside it
    the rounding of the charges f w, which the tree form stores as float64 and the
    oracle does not form: 2^-53 of each |f w| times its kernel value."""
    n = 1003
    xyz, w = W.random_cube(n, seed=9)
    xyz[:, 1::7] = xyz[:, 0:-1:7][:, :xyz[:, 1::7].shape[1]] * (1 + 1e-6)
    xyz[:, 5] = xyz[:, 4]
    xyz *= 3.0
    rho = np.exp(-np.sum(xyz * xyz, axis=0))
    f = np.stack([np.cos(xyz[0] + o) for o in range(nf_y)])
    k = [0.5 + o for o in range(nf_y)]
    u, vh = torch.empty((nf_y, n), dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.float64,
                                                                                   device="cuda")
    with T.Tree(dev(xyz), dev(w), theta=0.0, degree=2, leaf_size=300, prec=T.TAGI_FP64, ss=ss) as tr:
        T.tagi_fields_conv(tr.handle, dev(f), k, u, rho=dev(rho), vh=vh)
    for o in range(nf_y):
        ref = oracle.direct_yukawa(xyz, w, f[o], k[o], ss=ss)
        charges = 2.0 ** -53 * oracle.direct_yukawa(xyz, np.abs(w), np.abs(f[o]), k[o], ss=False)
        assert np.all(np.abs(u[o].cpu().numpy() - ref) <= 1e-12 * np.abs(ref).max() + charges)
