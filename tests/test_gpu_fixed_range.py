"""The fixed-point LME solves at the ends of their range of separations, through the C ABI, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def otm():
    import paper_2206_08772_gb300 as g
    g.load()
    from paper_2206_08772_gb300 import otm as m
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("units", [2 ** 32 + 2 ** 30, 2 ** 33 - 1, 2 ** 33, 3 * 2 ** 32])
def test_gradient_of_a_node_beside_the_point(orc, otm, units, sign):
    """A node a few 2^32 units of the fixed-point grid from the point on every axis. Its gradient -N K d is compared to its
    own size: half a unit of the separation (2^-33 of it), K and N to 1e-11: 1e-9."""
    h = 1.3e-3
    rng = np.random.default_rng(units % 1000)
    beta = 0.8 / h ** 2
    fb = 63 - int(np.frexp(2.2 * np.sqrt(13.815510557964274 / beta))[1])
    g = np.stack(np.meshgrid(*[np.arange(-2, 3)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = (g + rng.uniform(-0.05, 0.05, g.shape)) * h
    x[62] = -sign * units * 2.0 ** -fb   # d = x_p - x_a, all components of one sign
    n = len(x)
    ids = np.arange(n, dtype=np.int32)[None]
    tol = 1e-14 * h
    shape, lam, _, st = otm.lme(dev(x), dev(np.zeros((1, 3))), dev(ids), dev(np.array([n], np.int32)), beta, tol)
    so, N, dN, _, _ = orc.lme(-x, beta, tol)
    assert st.item() == 0 and so == 0
    got = shape.cpu().numpy()[0]
    assert abs(got[62, 0] - N[62]) <= 1e-11 * N[62]
    assert np.abs(got[62, 1:] - dN[62]).max() <= 1e-9 * np.abs(dN[62]).max()


@pytest.mark.parametrize("far", [0.45, 0.55, 0.62, 0.64, 0.655, 0.665, 0.9, 1.1])
def test_caller_supports_wider_than_the_default(orc, otm, far):
    """A node `far` of the fixed-point range from the point on every axis (0.23 is the default support radius), and
    points close to the corner of the body, whose lambda moves the centre of the weights by as much as a radius away
    from that node. J is near-singular there (its condition is (distance / h)^-1, 1e4 at most), so N is good to
    1e4 times the 1e-14 of the Newton tolerance: 1e-9 with margin."""
    rho = np.sqrt(13.815510557964274 / 0.8)
    h = 2.0 ** -7 * 1.002 / (2.2 * rho)
    beta, span = 0.8 / h ** 2, 2.0 ** -6
    x = np.stack(np.meshgrid(*[np.arange(4)] * 3, indexing="ij"), -1).reshape(-1, 3) * h
    x = np.vstack([x, np.full((1, 3), far * span)])
    xp = np.array([[d, d, d] for d in (0.4, 0.1, 1e-2, 3e-3, 1e-3, 3e-4)]) * h
    n, m = len(x), len(xp)
    ids = np.tile(np.arange(n, dtype=np.int32), (m, 1))
    tol = 1e-14 * h
    shape, lam, _, st = otm.lme(dev(x), dev(xp), dev(ids), dev(np.full(m, n, np.int32)), beta, tol)
    assert st.item() == 0
    got = shape.cpu().numpy()
    for p in range(m):
        so, N, dN, _, _ = orc.lme(xp[p] - x, beta, tol)
        assert so == 0
        assert np.abs(got[p, :, 0] - N).max() <= 1e-9
        assert np.abs(got[p, :, 1:] - dN).max() <= 1e-8 * np.abs(dN).max()
        assert got[p, -1, 0] <= 1e-15
