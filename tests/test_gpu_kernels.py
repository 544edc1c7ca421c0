"""GPU parity of the individual kernels, called through the C ABI, against the oracle.

Bars: neighbour lists, counts and linked-cell grid bit-exact; FP64 fields within 1e-10 relative
(max |gpu - oracle| / max |oracle| per field); LME invariants to 1e-12 on the GPU output."""
import math

import numpy as np
import pytest

import scenarios

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    d = np.abs(a - b).max() if a.size else 0.0
    s = np.abs(b).max() if b.size else 1.0
    return d / (s if s > 0 else 1.0)


@pytest.fixture(scope="module")
def otm():
    import paper_2206_08772_gb300 as g
    g.load()
    from paper_2206_08772_gb300 import otm as m
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("seed,nn,nm,r,S", [(1, 300, 500, 0.21, 256), (2, 5000, 3000, 0.11, 384),
                                            (3, 40, 100, 0.6, 64), (4, 20000, 1000, 0.05, 128)])
def test_search_bit_exact(orc, otm, seed, nn, nm, r, S):
    node_x, mp_x = scenarios.random_cloud(nn, nm, seed)
    mp_x = np.vstack([mp_x, [[-0.3, 0.5, 0.5], [9.0, 9.0, 9.0]]])   # points outside the node box
    rs2 = r * r
    cell = 0.5 * r * (1 + 2 ** -20)
    ids, counts, grid, status = otm.support_search(dev(node_x), dev(mp_x), rs2, cell, S)
    torch.cuda.synchronize()
    off, ref = orc.search(node_x, mp_x, rs2, cell)
    cnt_ref = np.diff(off)
    counts = counts.cpu().numpy()
    assert np.array_equal(counts, cnt_ref)
    ids = ids.cpu().numpy()
    over = cnt_ref > S
    assert (status.item() == -8) == bool(over.any())
    for p in np.nonzero(~over)[0]:
        assert np.array_equal(ids[p, :counts[p]], ref[off[p]:off[p + 1]])
    origin, dims, _, _ = orc.grid(node_x, cell)
    g = grid.cpu().numpy()
    assert np.array_equal(g[:3], origin) and np.array_equal(g[3:].astype(np.int64), dims)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 127, 129, 256, 257, 511, 513, 1024])
def test_search_list_lengths(otm, n):
    """Supports of every sort length: all n nodes in one point's ball; a second point with no node; the rows
    hold exactly the IDs, ascending, and a truncated row still ascends."""
    node_x, _ = scenarios.random_cloud(n, 1, n)
    mp_x = np.array([[0.5, 0.5, 0.5], [9.0, 9.0, 9.0]])
    ids, counts, _, status = otm.support_search(dev(node_x), dev(mp_x), 4.0, 1.0, n)
    assert counts.cpu().tolist() == [n, 0] and int(status) == 0
    assert np.array_equal(ids.cpu().numpy()[0], np.arange(n))
    S = max(1, n // 2)
    ids, counts, _, status = otm.support_search(dev(node_x), dev(mp_x), 4.0, 1.0, S)
    assert counts.cpu().tolist() == [n, 0]
    row = ids.cpu().numpy()[0]
    assert (np.diff(row) > 0).all() and 0 <= row[0] and row[-1] < n


@pytest.mark.parametrize("cell,scale,shift", [(0.50001, 1.0, 0.0), (0.6, 1.0, 40.0), (0.51, 1e-4, -7.0), (0.9, 1e3, 300.0),
                                              (1.7, 1.0, 0.0), (12.0, 1.0, 5.0)])
def test_search_cells_of_the_ball(orc, otm, cell, scale, shift):
    """The cells a ball meets, for cells from half the radius to beyond the body, away from the origin;
    bit-equal to the oracle's full box."""
    node_x, mp_x = scenarios.random_cloud(3000, 400, 11)
    node_x, mp_x, r = (node_x + shift) * scale, (1.2 * mp_x - 0.1 + shift) * scale, 0.17 * scale
    ids, counts, _, _ = otm.support_search(dev(node_x), dev(mp_x), r * r, cell * r, 256)
    off, ref = orc.search(node_x, mp_x, r * r, cell * r)
    counts, ids = counts.cpu().numpy(), ids.cpu().numpy()
    assert np.array_equal(counts, np.diff(off)) and counts.max() <= 256
    for p in range(len(counts)):
        assert np.array_equal(ids[p, :counts[p]], ref[off[p]:off[p + 1]])


def test_search_ties_exact(orc, otm):
    r = 0.25
    rs2 = r * r
    rng = np.random.default_rng(7)
    node_x = rng.uniform(0, 1, (400, 3))
    mp = []
    for k in range(60):
        p = node_x[k].copy()
        p[k % 3] += r if p[k % 3] + r <= 1.5 else -r
        mp.append(p)
    mp_x = np.array(mp)
    cell = 0.5 * r * (1 + 2 ** -20)
    ids, counts, _, _ = otm.support_search(dev(node_x), dev(mp_x), rs2, cell, 256)
    off, ref = orc.search(node_x, mp_x, rs2, cell)
    ids, counts = ids.cpu().numpy(), counts.cpu().numpy()
    for p in range(len(mp)):
        assert np.array_equal(ids[p, :counts[p]], ref[off[p]:off[p + 1]])


def rod_supports(orc, h=0.8e-3, L=8e-3):
    p = scenarios.taylor_rod(h=h, R=3.2e-3, L=L)
    off, ids = orc.search(p.node_x, p.mp_x, p.rs2, p.cell_size)
    return p, off, ids


def test_lme_vs_oracle_and_invariants(orc, otm):
    p, off, ref_ids = rod_supports(orc)
    S = 384
    ids, counts, _, st = otm.support_search(dev(p.node_x), dev(p.mp_x), p.rs2, p.cell_size, S)
    assert st.item() == 0
    tol = p.newton_tol * p.h
    shape, lam, iters, status = otm.lme(dev(p.node_x), dev(p.mp_x), ids, counts, p.beta, tol)
    assert status.item() == 0
    shape, lam = shape.cpu().numpy(), lam.cpu().numpy()
    counts = counts.cpu().numpy()
    for q in range(0, p.n_mps, 17):
        n = counts[q]
        xa = p.node_x[ref_ids[off[q]:off[q + 1]]]
        d = p.mp_x[q] - xa
        s_, N, dN, lr, _ = orc.lme(d, p.beta, tol)
        assert s_ == 0
        Ng, dNg = shape[q, :n, 0], shape[q, :n, 1:]
        assert rel(Ng, N) <= 1e-10
        assert rel(dNg, dN) <= 1e-10
        assert rel(lam[q], lr) <= 1e-8 or np.abs(lam[q] - lr).max() * p.h <= 1e-10
        assert abs(Ng.sum() - 1) <= 1e-12
        assert np.linalg.norm(Ng @ xa - p.mp_x[q]) / p.h <= 1e-12
        assert np.abs(dNg.sum(0)).max() * p.h <= 1e-12
        assert np.abs((xa - p.mp_x[q]).T @ dNg - np.eye(3)).max() <= 1e-12


def test_lme_outside_hull_reports_noconv(otm):
    X = np.random.default_rng(0).uniform(0, 1e-3, (30, 3))
    xp = np.array([[2e-3, 0.5e-3, 0.5e-3], [0.5e-3, 0.5e-3, 0.5e-3]])
    ids = np.tile(np.arange(30, dtype=np.int32), (2, 1))
    ids = np.pad(ids, ((0, 0), (0, 2)), constant_values=0)
    counts = np.array([30, 30], np.int32)
    shape, lam, iters, status = otm.lme(dev(X), dev(xp), dev(ids), dev(counts), 0.8e6, 1e-16, 50)
    assert status.item() == -4


@pytest.mark.parametrize("model", ["j2", "jc", "jc_frac"])
def test_return_map_vs_oracle(orc, otm, model):
    mat = {"j2": scenarios.copper_j2, "jc": scenarios.copper_jc, "jc_frac": scenarios.ti64_jc}[model]()
    rng = np.random.default_rng(5)
    n = 600
    dt = 5e-9
    dF = np.eye(3)[None] + rng.normal(0, 0.02, (n, 3, 3))
    F = dF @ (np.eye(3)[None] + rng.normal(0, 0.03, (n, 3, 3)))
    be = np.tile([1.0, 1, 1, 0, 0, 0], (n, 1)) + np.concatenate([rng.normal(0, 0.002, (n, 3)),
                                                                rng.normal(0, 0.001, (n, 3))], 1)
    ebar = np.abs(rng.normal(0, 0.05, n))
    T = 298 + np.abs(rng.normal(0, 80, n))
    dF_t, F_t = dev(dF.reshape(n, 9)), dev(F.reshape(n, 9))
    be_t, eb_t, T_t = dev(be.copy()), dev(ebar.copy()), dev(T.copy())
    sig, rate, failed, status = otm.return_map(mat, dt, dF_t, F_t, be_t, eb_t, T_t)
    assert status.item() == 0
    sig, be_g, eb_g, T_g = sig.cpu().numpy(), be_t.cpu().numpy(), eb_t.cpu().numpy(), T_t.cpu().numpy()
    failed = failed.cpu().numpy()
    ref = [orc.return_map(mat, dt, dF[k], be[k], ebar[k], T[k], np.linalg.det(F[k])) for k in range(n)]
    assert all(r[0] == 0 for r in ref)
    assert rel(sig, np.array([r[1] for r in ref])) <= 1e-10
    assert rel(be_g, np.array([r[2] for r in ref])) <= 1e-10
    assert rel(eb_g, np.array([r[3] for r in ref])) <= 1e-10
    assert rel(T_g, np.array([r[4] for r in ref])) <= 1e-10
    assert np.array_equal(failed.astype(bool), np.array([r[6] for r in ref]))
    assert (eb_g > ebar).any()     # the sample crosses the yield surface


def test_empty_point_sets(otm):
    """Zero points: the stand-alone search, LME and return map launch nothing and report OK."""
    nodes = dev(np.random.default_rng(0).uniform(0, 1, (50, 3)))
    empty = torch.empty((0, 3), dtype=torch.float64, device="cuda")
    ids, counts, grid, status = otm.support_search(nodes, empty, 0.04, 0.2, max_support=64)
    torch.cuda.synchronize()
    assert ids.shape == (0, 64) and counts.numel() == 0 and int(status.item()) == 0
    shape, lam, iters, st = otm.lme(nodes, empty, ids, counts, beta=20.0, tol_abs=1e-14)
    torch.cuda.synchronize()
    assert shape.shape == (0, 64, 4) and int(st.item()) == 0
    z = torch.empty((0, 9), dtype=torch.float64, device="cuda")
    sig, rate, failed, st = otm.return_map(scenarios.copper_jc(), 1e-8, z, z.clone(),
                                           torch.empty((0, 6), dtype=torch.float64, device="cuda"),
                                           torch.empty(0, dtype=torch.float64, device="cuda"),
                                           torch.empty(0, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    assert sig.shape == (0, 6) and int(st.item()) == 0


def test_lme_degenerate_supports(orc, otm):
    """Degenerate cases of Eq. 14. One node, or a point on the far side of a plane of nodes: no
    finite lambda puts the point inside the hull, so the solve fails (LME_NOCONV) on both sides.
    Four affinely independent nodes: N are the barycentric coordinates and grad N the constant
    tetrahedron gradients for any beta (the consistency conditions fix them), on the GPU to 1e-12."""
    beta, tol = 0.8 / 0.01 ** 2, 1e-14 * 0.01
    tet = np.array([[0.0, 0.0, 0.0], [0.01, 0.0, 0.0], [0.0, 0.01, 0.0], [0.0, 0.0, 0.01]])
    cases = {"one_node": (tet[:1], np.array([0.002, 0.001, 0.0])),
             "outside_plane": (tet[1:], np.array([0.0, 0.0, -0.001])),
             "tet": (tet, np.array([0.002, 0.003, 0.001]))}
    for name, (nx, xp) in cases.items():
        n = nx.shape[0]
        ids = torch.full((1, 32), -1, dtype=torch.int32, device="cuda")
        ids[0, :n] = torch.arange(n, dtype=torch.int32, device="cuda")
        counts = torch.tensor([n], dtype=torch.int32, device="cuda")
        shape, lam, iters, st = otm.lme(dev(nx), dev(xp[None, :]), ids, counts, beta=beta, tol_abs=tol)
        torch.cuda.synchronize()
        so, No, dNo, _, _ = orc.lme(xp[None, :] - nx, beta, tol)
        if name == "tet":
            assert int(st.item()) == 0 and so == 0
            A = np.vstack([np.ones(4), nx.T])                      # barycentric: A N = (1, x_p)
            N = np.linalg.solve(A, np.concatenate([[1.0], xp]))
            G = np.linalg.inv(A)[:, 1:]                            # dN/dx_p, constant
            sh = shape.cpu().numpy()[0, :4]
            assert np.abs(sh[:, 0] - N).max() <= 1e-12
            assert np.abs(sh[:, 1:] - G).max() <= 1e-12 * np.abs(G).max()
            assert rel(sh[:, 0], No) <= 1e-12 and rel(sh[:, 1:], dNo) <= 1e-12
        else:
            assert int(st.item()) == -4 and so == -4, name


def test_internal_exp_against_cuda_exp():
    """The LME weights use the library's table-driven FP64 exp (after Tang 1989, its polynomial
    in double-float) on a scaled argument y = f 1024/ln2; it must agree with CUDA's exp of the
    same f to a few ulps over the whole range it serves, including the table's breakpoints and the
    range limits."""
    import ctypes as C
    import paper_2206_08772_gb300 as g
    L = g.load()
    rng = np.random.default_rng(11)
    K = 1024 / np.log(2)
    y = np.concatenate([rng.uniform(-700, 700, 200000) * K, rng.uniform(-40, 5, 800000) * K,
                        np.arange(-2048, 2049, dtype=np.float64), np.arange(-2048, 2049) + 0.5,
                        [0.0, -0.0, 1e-300, -1e-300, 700.0 * K, -700.0 * K, -1020.0 * 1024, 1021.0 * 1024 + 1023]])
    yt = torch.from_numpy(y).cuda()
    mine, ref = torch.empty_like(yt), torch.empty_like(yt)
    assert L.otm_exp_selftest(C.c_void_p(yt.data_ptr()), y.size, C.c_void_p(mine.data_ptr()),
                              C.c_void_p(ref.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    m, r = mine.cpu().numpy(), ref.cpu().numpy()
    relerr = np.abs(m - r) / r
    assert relerr.max() <= 1.1e-15, relerr.max()   # 5 ulp: 2.5 from the cubic, table and reference roundings
    # against numpy on the range the LME uses (the argument's own rounding: |f| 2^-53)
    f = y * (np.log(2) / 1024)
    sel = np.abs(f) <= 60
    assert (np.abs(m[sel] - np.exp(f[sel])) / np.exp(f[sel])).max() <= 2e-14
    # out of range: zero below, infinity above
    out = torch.tensor([-1.0e7, 1.0e7, -3.0e9, 3.0e9, -1e300, 1e300], dtype=torch.float64).cuda()
    mo, ro = torch.empty_like(out), torch.empty_like(out)
    assert L.otm_exp_selftest(C.c_void_p(out.data_ptr()), out.numel(), C.c_void_p(mo.data_ptr()),
                              C.c_void_p(ro.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    assert mo.cpu().numpy().tolist() == [0.0, np.inf, 0.0, np.inf, 0.0, np.inf]


@pytest.mark.parametrize("h,gamma,tol,offset,S", [
    (0.8e-3, 0.8, 1e-6, 0.0, 384), (0.8e-3, 0.8, 1e-6, 3.7, 384),      # the default, far from the origin
    (0.7e-3, 1.6, 1e-6, 0.0, 128), (0.9e-3, 4.0, 1e-6, 0.0, 64),       # small supports (32 slots and below)
    (0.8e-3, 0.72, 1e-6, -0.5, 384), (0.8e-3, 0.62, 1e-6, 0.0, 512),   # supports about and above 336 slots
    (0.8e-3, 1.2, 3e-10, 0.0, 384), (0.8e-3, 1.4, 1e-12, 0.0, 384)])   # at and past the fixed-point range
def test_step_shape_functions_vs_oracle(orc, h, gamma, tol, offset, S):
    """The FP64 step's shape functions (fixed-point evaluations where their range covers the problem, FP64
    elsewhere) against the oracle's LME at the GPU's own positions, after steps that deform the body, and
    with points moved close to the hull, where lambda leaves the fixed-point range. Bound: both
    solves stop at |r| <= 1e-14 h, which moves N by up to |J^-1 r . d| = 2 gamma 1e-14 sqrt(ln(1/tol)/gamma)
    of itself each (2.6e-13 at most here), times 4 for the condition of J near the surface: 1e-12."""
    from paper_2206_08772_gb300.otm import OTM
    p = scenarios.taylor_rod(h=h, L=8 * h, gamma=gamma, support_tol=tol, material=scenarios.copper_jc())
    p.node_x[:] += offset
    p.mp_x[:] += offset
    p.contact.wall_point = (0.0, 0.0, offset)
    rng = np.random.default_rng(3)
    p.node_du0[:] += rng.normal(0, 2e-3 * h, p.node_du0.shape)
    sim = OTM(p, max_support=S)
    assert sim.step(3) == 0, sim.error()

    def check(points, bound):
        x, xp, cnt = sim.get("node_x"), sim.get("mp_x"), sim.get("support_count")
        ids, sh = sim.get_rows("support_ids", points), sim.get_rows("shape", points)
        for r, q in enumerate(points):
            d = xp[q] - x[ids[r, :cnt[q]]]
            assert ((d * d).sum(1) <= p.rs2).all()
            st, N, dN, _, _ = orc.lme(d, p.beta, p.newton_tol * p.h)
            assert st == 0
            assert rel(sh[r, :cnt[q], 0], N) <= bound
            assert rel(sh[r, :cnt[q], 1:], dN) <= 10 * bound
        return cnt

    cnt = check(np.arange(0, p.n_mps, max(1, p.n_mps // 60)), 1e-12)
    if gamma < 0.75:
        assert (cnt > 336).any()
    # the first point of each of a few cells towards the nearest corner node of the bottom face: lambda grows
    x, xp = sim.get("node_x"), sim.get("mp_x")
    corner = x[np.argmax(x[:, 0] - x[:, 2])]
    near = np.argsort(((xp - corner) ** 2).sum(1))[:3]
    for k, q in enumerate(near):
        xp[q] = corner + (xp[q] - corner) * (0.3, 0.05, 0.01)[k]
    sim.set("mp_x", xp)
    assert sim.refresh() == 0, sim.error()
    lam = sim.get("lam")[near]
    check(near, 1e-9)     # J is near-singular there: conditioned by (distance / h)^-2, at most 1e4 above
    if gamma == 0.8:      # a sharper prior needs less lambda to reach the hull
        assert np.abs(lam).max() * h > 3.0
    # a restored state repeats the solve bit for bit, on whichever path it ran
    snap, before = sim.snapshot(), sim.get("shape")
    sim.restore(snap)
    assert np.array_equal(before, sim.get("shape"))


@pytest.mark.parametrize("model", ["j2", "jc", "ti64"])
@pytest.mark.parametrize("strain,pressure", [(0.0, 0.0), (1e-6, 0.0), (1e-3, 0.0), (7e-3, 0.0), (0.012, 0.0),
                                             (1e-3, 0.04), (1e-3, -0.2), (1e-3, 0.7), (0.3, 0.0)])
def test_return_map_series_and_eigenvectors_vs_oracle(orc, otm, model, strain, pressure):
    """Points on both sides of the bound |dev b| <= 1/32 between the series form and the eigen decomposition
    (strain 0.007 and 0.012 straddle it), under pressure, at rest, virgin and hardened, cold, hot and
    melted. Stress bound: the FP64 rounding of b^e about 1 is 1.1e-16, seen through the moduli (largest
    of K and 2 mu) in either implementation, times 20 for the sums; plus 1e-10 of the stress, the bar of
    the other return map tests."""
    mat = {"j2": scenarios.copper_j2, "jc": scenarios.copper_jc, "ti64": scenarios.ti64_jc}[model]()
    rng = np.random.default_rng(11)
    n, dt = 300, 5e-9
    dF = np.eye(3) + rng.normal(0, 1, (n, 3, 3)) * 0.3 * strain
    F = dF @ (np.eye(3) + rng.normal(0, 0.02, (n, 3, 3)))
    be = np.concatenate([1 + pressure + rng.normal(0, 1, (n, 3)) * strain, rng.normal(0, 0.5, (n, 3)) * strain], 1)
    be[:, :3] = np.maximum(be[:, :3], 0.2)
    ebar = np.where(rng.uniform(size=n) < 0.3, 0.0, np.abs(rng.normal(0, 0.1, n)))
    T = rng.choice([mat.T_room, mat.T_room + 60.0, 0.5 * (mat.T_room + mat.T_melt), mat.T_melt, mat.T_melt + 40.0], n)
    ref = [orc.return_map(mat, dt, dF[k], be[k], ebar[k], T[k], np.linalg.det(F[k])) for k in range(n)]
    good = np.array([r[0] == 0 for r in ref])
    assert good.mean() > 0.5
    dF, F, be, ebar, T = dF[good], F[good], be[good], ebar[good], T[good]
    ref = [r for r in ref if r[0] == 0]
    be_t, eb_t, T_t = dev(be.copy()), dev(ebar.copy()), dev(T.copy())
    sig, rate, failed, status = otm.return_map(mat, dt, dev(dF.reshape(-1, 9)), dev(F.reshape(-1, 9)), be_t, eb_t, T_t)
    assert status.item() == 0
    K, mu = mat.E / (3 * (1 - 2 * mat.nu)), mat.E / (2 * (1 + mat.nu))
    s_ref = np.array([r[1] for r in ref])
    floor = 20 * 1.1e-16 * max(K, 2 * mu)
    J = np.abs(np.linalg.det(F)).min()
    assert np.abs(sig.cpu().numpy() - s_ref).max() <= floor / J + 1e-10 * np.abs(s_ref).max()
    assert rel(be_t.cpu().numpy(), np.array([r[2] for r in ref])) <= 1e-13 + 1e-10 * strain
    assert np.abs(eb_t.cpu().numpy() - np.array([r[3] for r in ref])).max() <= 20 * 1.1e-16 + 1e-10 * max(strain, ebar.max())
    assert rel(T_t.cpu().numpy(), np.array([r[4] for r in ref])) <= 1e-10
    assert np.array_equal(failed.cpu().numpy().astype(bool), np.array([r[6] for r in ref]))


def test_return_map_bad_input_reports_the_same_errors(otm):
    """Non-finite and inverted input leaves the series form for the eigen decomposition and its codes."""
    n = 4
    eye = torch.eye(3, dtype=torch.float64, device="cuda").reshape(1, 9).repeat(n, 1)
    be0 = torch.tensor([1.0, 1, 1, 0, 0, 0], dtype=torch.float64, device="cuda").repeat(n, 1)
    z = torch.zeros(n, dtype=torch.float64, device="cuda")
    for bad, code in ((float("nan"), -5), (-3.0, -5)):
        be = be0.clone()
        be[2, 0] = bad
        _, _, _, st = otm.return_map(scenarios.copper_jc(), 5e-9, eye, eye.clone(), be, z.clone(), z + 300.0)
        assert st.item() == code
    F = eye.clone()
    F[1] = 0.0
    _, _, _, st = otm.return_map(scenarios.copper_jc(), 5e-9, eye, F, be0.clone() * 1.001, z.clone(), z + 300.0)
    assert st.item() == -6


@pytest.mark.parametrize("n,far", [(4, 0.0), (31, 0.0), (33, 0.0), (336, 0.0), (337, 0.0), (400, 0.0), (40, 30.0)])
def test_lme_support_sizes_and_ranges(orc, otm, n, far):
    """The stand-alone LME at the edges of its fixed-point form: 32-lane passes, 336 shared slots, and one node
    30 spacings away (outside the fixed-point range), each with a start far from the solution for
    half of the points. Bound: both solves stop at |r| <= 1e-14 h, 1e-12 on N as in the step's test."""
    h = 1.3e-3
    rng = np.random.default_rng(n)
    g = np.stack(np.meshgrid(*[np.arange(-5, 6)] * 3, indexing="ij"), -1).reshape(-1, 3)
    g = g[np.argsort((g ** 2).sum(1), kind="stable")]
    if n == 4:
        g = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]])
    x = (g[:n] + rng.uniform(-0.02, 0.02, (n, 3))) * h + 0.5
    if far:
        x[-1] = x[0] + far * h
    xp = 0.5 + rng.uniform(0.1, 0.3, (12, 3)) * h
    S, tol, beta = 416, 1e-14 * h, 0.8 / h ** 2
    ids = np.zeros((12, S), np.int32)
    ids[:, :n] = rng.permutation(n)
    lam0 = np.where(np.arange(12)[:, None] % 2, 0.4 / h, 0.0) * np.ones((12, 3))
    shape, lam, iters, st = otm.lme(dev(x), dev(xp), dev(ids), dev(np.full(12, n, np.int32)), beta, tol,
                                    lam0=dev(lam0))
    assert st.item() == 0
    sh = shape.cpu().numpy()
    for p in range(12):
        so, N, dN, _, _ = orc.lme(xp[p] - x[ids[p, :n]], beta, tol)
        assert so == 0
        assert rel(sh[p, :n, 0], N) <= 1e-12 and rel(sh[p, :n, 1:], dN) <= 1e-11
        assert not sh[p, n:].any()
