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


def check_shapes(orc, sim, p, rows, bound=1e-12):
    x, xp, cnt = sim.get("node_x"), sim.get("mp_x"), sim.get("support_count")
    ids, sh = sim.get_rows("support_ids", rows), sim.get_rows("shape", rows)
    for r, q in enumerate(rows):
        n = cnt[q]
        st, N, dN, _, _ = orc.lme(xp[q] - x[ids[r, :n]], p.beta, p.newton_tol * p.h)
        assert st == 0
        assert np.abs(sh[r, :n, 0] - N).max() <= bound * N.max()
        assert np.abs(sh[r, :n, 1:] - dN).max() <= 10 * bound * np.abs(dN).max()


@pytest.mark.parametrize("how", ["padded", "csr", "moved"])
@pytest.mark.parametrize("precision,eps", [("fp64", 0.0), ("fp64", 1e-2), ("mixed", 0.0)])
def test_supports_beyond_the_search(orc, how, precision, eps):
    """Supports that no search gave: nodes 1.05 to 6 support radii away added to some points' own (4.4 to 8.8 radii are
    2^64 units of the fixed-point grid), replayed, then kept by frozen steps, each state restored from a snapshot;
    and positions moved by the caller before a snapshot. Bound as of searched steps: 1e-12 on N (1e-6 and FP32
    rounding of the gradients in the mixed path)."""
    import scenarios
    from paper_2206_08772_gb300.otm import OTM
    h = 0.8e-3
    p = scenarios.taylor_rod(h=h, R=3.2e-3, L=26 * h, material=scenarios.copper_jc(), v0=50.0)
    p.eps_stab = eps * p.materials[0].E * h ** 2
    bound = 1e-12 if precision == "fp64" else 1e-6
    base, sim = OTM(p, precision=precision), OTM(p, precision=precision)
    assert base.step(1) == 0
    cnt, ids = base.get("support_count"), base.get("support_ids")
    x, xp = base.get("node_x"), base.get("mp_x")
    rs = np.sqrt(p.rs2)
    rows = np.linspace(0, p.n_mps - 1, 40).astype(int)
    for k, q in enumerate(rows):
        d = np.sqrt(((xp[q] - x) ** 2).sum(1)) / rs
        want = [1.05, 1.2, 1.45, 2.2, 2.9, 3.6, 4.6, 4.7, 5.0, 6.0][: 1 + k % 10]
        add = sorted({int(np.argmin(np.abs(d - w))) for w in want} - set(ids[q, :cnt[q]].tolist()))
        add = add[: 384 - cnt[q]]
        ids[q, cnt[q]:cnt[q] + len(add)] = add
        cnt[q] += len(add)
    if how == "padded":
        assert sim.step_with_supports(cnt, ids) == 0, sim.error()
    elif how == "csr":
        off = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int32)
        flat = np.concatenate([ids[q, :cnt[q]] for q in range(p.n_mps)]).astype(np.int32)
        assert sim.step_with_supports_csr(dev(off), dev(flat)) == 0, sim.error()
    else:
        assert sim.step(1) == 0, sim.error()
        far = np.linspace(0, p.n_nodes - 1, 12).astype(int)
        x = sim.get("node_x")
        x[far, 2] += 19.53125 * h * np.linspace(0.3, 1.0, 12)
        sim.set("node_x", x)
        sim.restore(sim.snapshot())
    assert how == "moved" or np.array_equal(sim.get("support_count"), cnt)

    def check():
        check_shapes(orc, sim, p, rows, bound)
        before = sim.get("shape")
        sim.restore(sim.snapshot())
        assert np.array_equal(before, sim.get("shape"))

    check()
    if how != "moved":
        sim.freeze_topology()
        assert sim.step(2) == 0, sim.error()
        check()


@pytest.mark.parametrize("n", [40, 336, 337, 400])
def test_rows_of_a_failed_point_stay_as_they_were(orc, otm, n):
    """Points outside the hull of their supports fail: their rows, and the unused slots of the others, keep what the
    caller had there, on either side of the 336 nodes that the fixed-point kernel takes."""
    import ctypes as C
    import paper_2206_08772_gb300 as g
    h = 1.3e-3
    rng = np.random.default_rng(n)
    x = np.stack(np.meshgrid(*[np.arange(-4, 5)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = (x[np.argsort((x ** 2).sum(1), kind="stable")][:n] + rng.uniform(-0.02, 0.02, (n, 3))) * h
    m, S, tol, beta = 9, 416, 1e-14 * h, 0.8 / h ** 2
    xp = rng.uniform(0.1, 0.3, (m, 3)) * h
    bad = np.arange(m) % 3 == 1
    xp[bad] += 6.0 * h
    xd, pd, ids, cnt = dev(x), dev(xp), dev(np.tile(np.arange(S, dtype=np.int32) % n, (m, 1))), dev(np.full(m, n, np.int32))
    shape = torch.full((m, S, 4), 7.25, dtype=torch.float64, device="cuda")
    lam = torch.zeros(m, 3, dtype=torch.float64, device="cuda")
    iters = torch.full((m,), -1, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    P = lambda t: C.c_void_p(t.data_ptr())
    assert g.load().otm_lme(P(xd), P(pd), m, P(ids), P(cnt), S, beta, tol, 50, P(lam), P(shape), P(iters), P(status),
                            C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    assert status.item() == -4
    sh = shape.cpu().numpy()
    assert (iters.cpu().numpy() >= 0).all()
    for q in range(m):
        st, N, dN, _, _ = orc.lme(xp[q] - x, beta, tol)
        assert (st != 0) == bad[q]
        assert (sh[q, n:] == 7.25).all()
        if bad[q]:
            assert (sh[q] == 7.25).all()
        else:
            assert np.abs(sh[q, :n, 0] - N).max() <= 1e-12 and np.abs(sh[q, :n, 1:] - dN).max() <= 1e-11 * np.abs(dN).max()


@pytest.mark.parametrize("h", [1e-22, 1e40])
@pytest.mark.parametrize("n", [60, 400])
def test_length_scales_outside_the_fixed_point(orc, otm, h, n):
    """Length scales beyond the exponent arithmetic's are evaluated in FP64; 1e-12 on N as elsewhere."""
    rng = np.random.default_rng(n)
    x = np.stack(np.meshgrid(*[np.arange(-4, 5)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = (x[np.argsort((x ** 2).sum(1), kind="stable")][:n] + rng.uniform(-0.02, 0.02, (n, 3))) * h
    m, tol, beta = 5, 1e-14 * h, 0.8 / h ** 2
    xp = rng.uniform(0.1, 0.3, (m, 3)) * h
    shape, lam, _, st = otm.lme(dev(x), dev(xp), dev(np.tile(np.arange(n, dtype=np.int32), (m, 1))),
                                dev(np.full(m, n, np.int32)), beta, tol)
    assert st.item() == 0
    sh = shape.cpu().numpy()
    for q in range(m):
        so, N, dN, _, _ = orc.lme(xp[q] - x, beta, tol)
        assert so == 0
        assert np.abs(sh[q, :, 0] - N).max() <= 1e-12 and np.abs(sh[q, :, 1:] - dN).max() <= 1e-11 * np.abs(dN).max()
