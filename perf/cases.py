"""Performance cases: the work a user of this package has it do, through its public entry points.

Kinds of case:
  rod / chip  resume a checkpoint and advance a few explicit steps (restore, step, read the state):
              the Taylor rods (J2, Johnson-Cook; FP64 and mixed; with node insertion, with the
              stabilisation term) and the eroding chip block of the tests and the benchmark
  adjoint     a backward pass over a few steps with their snapshots
  search      the stand-alone linked-cell support search
  lme         the stand-alone max-ent shape functions
  return_map  the stand-alone constitutive update

The rods start as an impact in progress: the axial velocity falls off towards the wall and the
section spreads accordingly, with a smooth perturbation, so that every material point deforms (the
state of most of a run; at rest the Newton solve of the shape functions has nothing to do). A few
steps are taken while the case is prepared; they fill the history the solver starts from.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2206_08772_gb300 import otm

DEV = "cuda"
KUHN = ((0, 1, 3, 7), (0, 1, 5, 7), (0, 2, 3, 7), (0, 2, 6, 7), (0, 4, 5, 7), (0, 4, 6, 7))


# ------------------------------------------------------------------------------------- the cases
def _rod(h_mm, L_mm=25.4, model="jc", precision="fp64", steps=4, insert=0, eps=0.0, **kw):
    return dict(kind="rod", h_mm=h_mm, L_mm=L_mm, model=model, precision=precision, steps=steps, insert=insert,
                eps=eps, **kw)


def listed():
    return [
        # the smallest stepping run of the tests: 9,984 points, one wave of blocks, launches count
        _rod(0.8, model="j2", steps=16, name="rod_j2_10k"),
        # a design-study rod (the adjoint's and the profiles' size): 202,752 points
        _rod(0.29, name="rod_jc_200k"),
        # the largest: a fine rod, pair arrays of tens of GB
        _rod(0.16, name="rod_jc_1200k"),
        # the mixed path on a fine rod
        _rod(0.2, precision="mixed", name="rod_mixed_600k"),
        # a parameter-sweep rod: node insertion on, the host checks every step
        _rod(0.5, steps=8, insert=64, name="rod_insert_38k"),
        # the stabilisation sweep's term on a J2 rod
        _rod(0.4, model="j2", eps=1e-3, name="rod_stabilised_75k"),
        # orthogonal cutting, erosion on, tool embedded: the benchmark's block at a coarser spacing
        dict(kind="chip", cells=40, precision="mixed", steps=4, embed_h=1.5, name="chip_mixed_600k"),
        # gradients: backward steps over stored states
        dict(kind="adjoint", h_mm=0.4, L_mm=25.4, steps=3, name="adjoint_75k"),
        # the smallest call: one search of a small cloud
        dict(kind="search", nodes=300, points=500, radius_nodes=20.0, slots=256, name="search_500"),
        # a full-size search of a scattered cloud
        dict(kind="search", nodes=180001, points=600007, radius_nodes=250.0, slots=384, name="search_600k"),
        # shape functions at many points of a body
        dict(kind="lme", h_mm=0.32, L_mm=25.4, name="lme_150k"),
        # constitutive update of many points, fracture on
        dict(kind="return_map", points=1000003, model="ti64", name="return_map_1000k"),
    ]


def draw(rng):
    def log(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    def spacing(n, L):   # the spacing (mm) that gives about n points in a rod of length L (mm), R 3.2 mm
        return round((6.0 * math.pi * 3.2 * 3.2 * L / n) ** (1.0 / 3.0), 4)

    kind = rng.choice(["rod"] * 6 + ["chip", "adjoint", "search", "lme", "return_map"])
    L = round(rng.uniform(6.0, 25.4), 2)
    if kind == "rod":
        n = log(4e3, 7e5)
        return _rod(spacing(n, L), L, model=rng.choice(["j2", "jc", "jc"]), precision=rng.choice(["fp64", "mixed"]),
                    steps=rng.randint(2, 5), insert=rng.choice([0, 0, 0, 32]), eps=rng.choice([0.0, 0.0, 0.0, 1e-3]))
    if kind == "chip":
        return dict(kind="chip", cells=rng.randint(12, 42), precision=rng.choice(["mixed", "fp64"]),
                    steps=rng.randint(2, 4), embed_h=rng.choice([0.0, 1.5]))
    if kind == "adjoint":
        return dict(kind="adjoint", h_mm=spacing(log(4e3, 7e4), L), L_mm=L, steps=rng.randint(1, 3))
    if kind == "search":
        return dict(kind="search", nodes=int(log(200, 2e5)), points=int(log(300, 6e5)),
                    radius_nodes=round(rng.uniform(15.0, 250.0), 1), slots=384)
    if kind == "lme":
        return dict(kind="lme", h_mm=spacing(log(4e3, 1.5e5), L), L_mm=L)
    return dict(kind="return_map", points=int(log(500, 1e6)), model=rng.choice(["j2", "jc", "ti64"]))


# ----------------------------------------------------------------------------------- the problems
def _material(model, rng):
    """Copper (J2 or Johnson-Cook) and Ti-6Al-4V of the rods and the chip, the flow stress varied as in a study."""
    f = rng.uniform(0.9, 1.1, 2)
    m = dict(E=117e9, nu=0.35, rho0=8930.0, model="j2", sigma_y0=400e6 * f[0], H=100e6, A=0.0, B=0.0, n=1.0, C=0.0,
             m=1.0, eps_dot0=1.0, T_room=298.0, T_melt=1356.0, chi=0.0, cp=385.0, fracture=False,
             d=(0.0, 0.0, 0.0, 0.0, 0.0))
    if model == "jc":
        m.update(model="jc", sigma_y0=0.0, H=0.0, A=90e6 * f[0], B=292e6 * f[1], n=0.31, C=0.025, m=1.09, chi=0.9)
    if model == "ti64":
        m.update(E=113.8e9, nu=0.342, rho0=4430.0, model="jc", sigma_y0=0.0, H=0.0, A=1098e6 * f[0], B=1092e6 * f[1],
                 n=0.93, C=0.014, m=1.1, T_room=298.15, T_melt=1903.15, chi=0.9, cp=526.0, fracture=True,
                 d=(-0.09, 0.25, -0.5, 0.014, 3.87))
    return SimpleNamespace(**m)


def _cloud(keep, h, origin, gen):
    """Nodes and material points of the kept hexes (nk, nj, ni): six tetrahedra per hex, one point at
    each barycentre, interior nodes jittered by one per cent of the spacing."""
    nk, nj, ni = keep.shape
    touch = torch.zeros(nk + 1, nj + 1, ni + 1, dtype=torch.int32, device=DEV)
    for c in range(8):
        dk, dj, di = (c >> 2) & 1, (c >> 1) & 1, c & 1
        touch[dk:dk + nk, dj:dj + nj, di:di + ni] += keep
    at = (touch > 0).nonzero()
    node_id = torch.full(touch.shape, -1, dtype=torch.int64, device=DEV)
    node_id[touch > 0] = torch.arange(at.shape[0], device=DEV)
    x = torch.tensor(origin, dtype=torch.float64, device=DEV) + at.flip(1).double() * h
    inner = (touch[touch > 0] == 8).unsqueeze(1)
    x = x.contiguous() + inner * (2.0 * torch.rand(x.shape, generator=gen, dtype=torch.float64, device=DEV) - 1.0) * (0.01 * h)
    ck, cj, ci = keep.nonzero().unbind(1)
    corner = torch.stack([node_id[ck + ((c >> 2) & 1), cj + ((c >> 1) & 1), ci + (c & 1)] for c in range(8)], 1)
    p = x[corner[:, torch.tensor(KUHN, device=DEV)].reshape(-1, 4)]
    a, b, c = p[:, 1] - p[:, 0], p[:, 2] - p[:, 0], p[:, 3] - p[:, 0]
    return x, p.mean(1), (a * torch.cross(b, c, dim=1)).sum(1).abs() / 6.0


def _problem(x, du0, flags, mp_x, vol, mat, h, dt, contact, eps=0.0, insert=0, host=True):
    beta = 0.8 / (h * h)
    rs2 = math.log(1e6) / beta
    c = dict(wall=False, wall_point=(0.0, 0.0, 0.0), wall_normal=(0.0, 0.0, 1.0), tool=False, tool_x0=0.0,
             tool_tip_y=0.0, tool_rake_deg=0.0, tool_clearance_deg=7.0, tool_velocity=0.0, friction=0.0)
    c.update(contact)
    put = (lambda t: t.cpu().numpy()) if host else (lambda t: t)
    return SimpleNamespace(h=h, beta=beta, rs2=rs2, cell_size=0.5 * math.sqrt(rs2) * (1.0 + 2.0 ** -20), dt=dt,
                           T0=mat.T_room, newton_tol=1e-14, max_newton=50, eps_stab=eps * mat.E * h * h,
                           max_insert=insert, materials=[mat], contact=SimpleNamespace(**c), n_nodes=x.shape[0],
                           n_mps=mp_x.shape[0], node_x=put(x), node_du0=put(du0), node_flags=put(flags),
                           mp_x=put(mp_x), mp_vol=put(vol), mp_mass=put(mat.rho0 * vol),
                           mp_material=put(torch.zeros(mp_x.shape[0], dtype=torch.int32, device=DEV)))


def _time_step(mat, h):
    lame = mat.E * (1.0 - mat.nu) / ((1.0 + mat.nu) * (1.0 - 2.0 * mat.nu))
    return 0.3 * h / math.sqrt(lame / mat.rho0)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed), np.random.default_rng(seed)


def _rod_body(case, gen):
    h, R = case["h_mm"] * 1e-3, 3.2e-3
    M, nk = int(math.ceil(R / h - 1e-12)), max(1, round(case["L_mm"] * 1e-3 / h))
    c = (torch.arange(-M, M, device=DEV).double() + 0.5) * h
    disc = (c[None, :] ** 2 + c[:, None] ** 2) <= R * R * (1.0 + 1e-12)
    return h, _cloud(disc.expand(nk, -1, -1).contiguous(), h, (-M * h, -M * h, 0.0), gen)


def _rod_problem(case, seed, host=True):
    gen, rng = _gen(seed)
    h, (x, mp_x, vol) = _rod_body(case, gen)
    mat = _material(case.get("model", "jc"), rng)
    dt = _time_step(mat, h)
    v0, reach, phase = rng.uniform(150.0, 300.0), rng.uniform(6e-3, 1e-2), rng.uniform(0.0, 2 * math.pi, 3)
    fall = torch.exp(-x[:, 2:] / reach)
    v = torch.cat([0.5 * v0 / reach * x[:, :2] * fall, -v0 * (1.0 - fall)], 1)
    wave = torch.sin(x.flip(1) * (2 * math.pi / 8e-3) + torch.tensor(phase, device=DEV))
    v = v + 0.03 * v0 * wave * torch.clamp(x[:, 2:] / 2e-3, max=1.0)
    flags = torch.zeros(x.shape[0], dtype=torch.uint8, device=DEV)
    return _problem(x, v * dt, flags, mp_x, vol, mat, h, dt, dict(wall=True), case.get("eps", 0.0),
                    case.get("insert", 0), host)


def _chip_problem(case, seed):
    gen, rng = _gen(seed)
    n, h = case["cells"], 1e-3 / case["cells"]
    keep = torch.ones(max(1, round(0.4 * n)), n, 4 * n, dtype=torch.bool, device=DEV)
    x, mp_x, vol = _cloud(keep, h, (0.0, 0.0, 0.0), gen)
    mat = _material("ti64", rng)
    flags = (x[:, 1] <= 0.5 * h).to(torch.uint8)
    tool = dict(tool=True, tool_x0=4 * n * h + h - case["embed_h"] * h, tool_tip_y=n * h - 0.2e-3,
                tool_velocity=rng.uniform(4.0, 6.0), friction=0.8)
    return _problem(x, torch.zeros_like(x), flags, mp_x, vol, mat, h, _time_step(mat, h), tool)


# ------------------------------------------------------------------------------- prepare and run
WARM = 5                        # steps before the checkpoint: the solver's start history is then full
NODE_FIELDS = ("node_x", "node_du")
MP_FIELDS = ("F", "sigma", "ebar", "T", "support_count")


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("rod", "chip"):
        prob = _rod_problem(case, seed) if kind == "rod" else _chip_problem(case, seed)
        sim = otm.OTM(prob, precision=case["precision"])
        _advance(sim, WARM)
        width = dict(node_x=3, node_du=3, F=9, sigma=6, ebar=1, T=1, support_count=1)
        room = {}               # page-locked result buffers, as a program that reads results often keeps them
        for f in NODE_FIELDS + MP_FIELDS:
            rows = prob.n_nodes + prob.max_insert if f in NODE_FIELDS else prob.n_mps
            kind_ = torch.int32 if f == "support_count" else torch.float64
            room[f] = torch.zeros(rows * width[f], dtype=kind_, pin_memory=True).numpy()
        return dict(kind=kind, sim=sim, steps=case["steps"], start=sim.snapshot(), room=room, width=width)
    if kind == "adjoint":
        prob = _rod_problem(case, seed)
        sim = otm.OTM(prob)
        _advance(sim, WARM)
        states = [sim.snapshot()]
        for _ in range(case["steps"]):
            _advance(sim, 1)
            states.append(sim.snapshot())
        x = sim.get("node_x")
        seedvec = np.zeros_like(x)
        seedvec[:, 2] = np.exp((x[:, 2] - x[:, 2].max()) / prob.h)   # a smooth measure of the rod's length
        du0 = np.zeros_like(x)
        du0[:, 2] = -prob.dt
        return dict(kind=kind, sim=sim, states=states, xbar=seedvec, du0=du0)
    if kind == "search":
        node_x, mp_x, rs2, cell = _search_inputs(case, seed)
        return dict(kind=kind, args=(node_x, mp_x, rs2, cell, case["slots"]))
    if kind == "lme":
        node_x, mp_x, h, beta, rs2, cell = _lme_inputs(case, seed)
        ids, counts, _, _ = otm.support_search(node_x, mp_x, rs2, cell, 384)
        return dict(kind=kind, args=(node_x, mp_x, ids, counts, beta, 1e-14 * h))
    return dict(kind=kind, args=_points(case, seed))


def _advance(sim, n):
    st = sim.step(n)
    if st != 0:
        raise RuntimeError("step failed: %s %s" % (st, sim.error()))


def run(state):
    kind = state["kind"]
    if kind in ("rod", "chip"):
        sim, w = state["sim"], state["width"]
        sim.restore(state["start"])
        _advance(sim, state["steps"])
        c, room = sim.counts(), state["room"]
        for f in NODE_FIELDS + MP_FIELDS:
            rows = c["n_nodes"] if f in NODE_FIELDS else c["n_mps"]
            sim.get(f, room[f][:rows * w[f]])
        return dict(room, nodes=c["n_nodes"], points=c["n_mps"])   # rows past the counts stay zero
    if kind == "adjoint":
        sim, states = state["sim"], state["states"]
        sim.restore(states[-1])
        sim.adjoint_begin(state["xbar"])
        for k in range(len(states) - 2, -1, -1):
            sim.restore(states[k])
            sim.adjoint_step(states[k + 1])
        theta, dub = sim.adjoint_result(state["du0"])
        return dict(theta=theta, dub=dub)
    if kind == "search":
        ids, counts, grid, status = otm.support_search(*state["args"])
        return dict(ids=ids, counts=counts, grid=grid, status=status)
    if kind == "lme":
        shape, lam, _, status = otm.lme(*state["args"])
        return dict(shape=shape, lam=lam, status=status)
    mat, dt, dF, F, be, ebar, T = state["args"]
    be, ebar, T = be.clone(), ebar.clone(), T.clone()          # updated in place
    sigma, rate, failed, status = otm.return_map(mat, dt, dF, F, be, ebar, T)
    return dict(sigma=sigma, rate=rate, failed=failed, be=be, ebar=ebar, T=T, status=status)


def _search_inputs(case, seed):
    """A uniform cloud in the unit box; a ball of the search radius holds radius_nodes nodes on average."""
    gen, _ = _gen(seed)
    n, m = case["nodes"], case["points"]
    node_x = torch.rand(n, 3, generator=gen, dtype=torch.float64, device=DEV)
    mp_x = torch.rand(m, 3, generator=gen, dtype=torch.float64, device=DEV)
    r = (case["radius_nodes"] / (n * 4.0 / 3.0 * math.pi)) ** (1.0 / 3.0)
    return node_x, mp_x, r * r, 0.5 * r * (1.0 + 2.0 ** -20)


def _lme_inputs(case, seed):
    gen, _ = _gen(seed)
    h, (x, mp_x, _) = _rod_body(case, gen)
    beta = 0.8 / (h * h)
    rs2 = math.log(1e6) / beta
    return x, mp_x, h, beta, rs2, 0.5 * math.sqrt(rs2) * (1.0 + 2.0 ** -20)


def _points(case, seed):
    """Increments and states about the yield surface, as an impact has them: elastic strains of a few
    per mille, plastic strains of some per cent, heated points."""
    gen, rng = _gen(seed)
    mat, n = _material(case["model"], rng), case["points"]

    def normal(*shape):
        return torch.randn(*shape, generator=gen, dtype=torch.float64, device=DEV)

    eye = torch.eye(3, dtype=torch.float64, device=DEV)
    dF = eye + 1.5e-3 * normal(n, 3, 3)
    F = dF @ (eye + 0.03 * normal(n, 3, 3))
    be = torch.cat([1.0 + 3e-3 * normal(n, 3), 1.5e-3 * normal(n, 3)], 1)
    ebar = (0.05 * normal(n)).abs() * (torch.rand(n, generator=gen, device=DEV) < 0.8)
    return mat, 5e-9, dF.reshape(n, 9), F.reshape(n, 9), be, ebar, mat.T_room + (80.0 * normal(n)).abs()


# ------------------------------------------------------------------------------------------ work
def work(case):
    kind = case["kind"]
    if kind in ("rod", "chip", "adjoint"):
        if kind == "chip":
            cells = max(1, round(0.4 * case["cells"])) * 4 * case["cells"] ** 2
        else:
            h = case["h_mm"]
            M = int(math.ceil(3.2 / h - 1e-12))
            c = (np.arange(-M, M) + 0.5) * h
            cells = int(((c[:, None] ** 2 + c[None, :] ** 2) <= 3.2 * 3.2 * (1 + 1e-12)).sum()) * max(1, round(case["L_mm"] / h))
        mps, nodes, pairs = 6 * cells, 1.1 * cells, 6 * cells * 280.0
        # per step: the points' state (x, F, b^e, sigma, v, m, ebar, T, lambda: 35 doubles) and the nodes'
        # (x, du, m, f: 10 doubles) in and out; 24 flops of kinematics, 57 of one shape-function
        # evaluation with its outputs and 8 of reduction a pair, 25 more for a second evaluation
        step = dict(bytes=2.0 * 8.0 * (35.0 * mps + 10.0 * nodes), flops=114.0 * pairs + 1500.0 * mps)
        n = case["steps"] * (4.0 if kind == "adjoint" else 1.0)
        return dict(bytes=n * step["bytes"], flops=n * step["flops"])
    if kind == "search":
        pairs = case["points"] * min(case["radius_nodes"], case["slots"])
        return dict(bytes=24.0 * (case["nodes"] + case["points"]) + 4.0 * (pairs + case["points"]), flops=8.0 * pairs)
    if kind == "lme":
        h = case["h_mm"]
        mps = 6.0 * math.pi * (3.2 / h) ** 2 * case["L_mm"] / h
        return dict(bytes=mps * 280.0 * (4.0 + 32.0), flops=mps * 280.0 * 4.0 * 25.0)
    return dict(bytes=8.0 * case["points"] * (9 + 9 + 2 * 8 + 6 + 1), flops=1500.0 * case["points"])


# ------------------------------------------------------------------------------ 64-bit references
def exact(case, seed):
    """Plain torch in 64 bits: the method's step written out, a brute-force search for its supports. None where
    points leave or nodes arrive (chip), for the backward pass and where the brute force would take too long."""
    kind = case["kind"]
    if kind == "rod":
        prob = _rod_problem(case, seed, host=False)
        if float(prob.n_mps) * prob.n_nodes * (WARM + case["steps"]) > 1.2e11:
            return None
        return _steps(prob, WARM + case["steps"])
    if kind == "search":
        node_x, _, _, cell = _search_inputs(case, seed)
        lo, hi = node_x.amin(0), node_x.amax(0)
        return dict(ids=None, counts=None, grid=torch.cat([lo, torch.floor((hi - lo) / cell) + 1.0]), status=None)
    if kind == "lme":
        node_x, mp_x, h, beta, rs2, _ = _lme_inputs(case, seed)
        if float(mp_x.shape[0]) * node_x.shape[0] > 1e11:
            return None
        ids, ok = _supports(node_x, mp_x, rs2, 384)
        N, dN, lam = _max_ent(node_x, mp_x, ids, ok, beta, 1e-15 * h)
        return dict(shape=torch.cat([N.unsqueeze(2), dN], 2), lam=lam, status=None)
    if kind == "return_map":
        mat, dt, dF, F, be, ebar, T = _points(case, seed)
        got = [_return_map(mat, dt, *(t[i:i + 100000] for t in (dF.reshape(-1, 3, 3), be, ebar, T)),
                           torch.linalg.det(F[i:i + 100000].reshape(-1, 3, 3))) for i in range(0, dF.shape[0], 100000)]
        be, sigma, ebar, T, rate = (torch.cat(t) for t in zip(*got))
        return dict(sigma=sigma, rate=rate, failed=None, be=be, ebar=ebar, T=T, status=None)
    return None


def _supports(x, xp, rs2, slots):
    """Padded ascending node lists of every point, and which slots are filled."""
    ids = torch.zeros(xp.shape[0], slots, dtype=torch.int64, device=DEV)
    ok = torch.zeros(xp.shape[0], slots, dtype=torch.bool, device=DEV)
    chunk = max(1, int(2e8 // x.shape[0]))
    for i in range(0, xp.shape[0], chunk):
        q = xp[i:i + chunk]
        dx, dy, dz = (q[:, None, k] - x[None, :, k] for k in range(3))
        inside = ((dx * dx + dy * dy) + dz * dz) <= rs2
        row, col = inside.nonzero().unbind(1)
        count = inside.sum(1)
        slot = torch.arange(row.numel(), device=DEV) - (count.cumsum(0) - count)[row]
        ids[i + row, slot] = col
        ok[i + row, slot] = True
    return ids, ok


def _max_ent(x, xp, ids, ok, beta, tol):
    got = []
    for i in range(0, xp.shape[0], 50000):
        s = slice(i, i + 50000)
        d, on = (xp[s, None, :] - x[ids[s]]) * ok[s].unsqueeze(2), ok[s]
        prior = -beta * (d * d).sum(2)

        def state(lam):
            f = (prior + (d * lam.unsqueeze(1)).sum(2)).masked_fill(~on, -math.inf)
            return torch.softmax(f, 1), torch.logsumexp(f, 1)

        lam = torch.zeros(d.shape[0], 3, dtype=torch.float64, device=DEV)
        for _ in range(60):
            N, logz = state(lam)
            r = (N.unsqueeze(2) * d).sum(1)
            if float(r.norm(dim=1).max()) <= tol:
                break
            J = (N.unsqueeze(2) * d).transpose(1, 2) @ d - r.unsqueeze(2) * r.unsqueeze(1)
            dl = -torch.linalg.solve(J, r.unsqueeze(2)).squeeze(2)
            t = torch.ones(d.shape[0], 1, dtype=torch.float64, device=DEV)
            for _ in range(40):
                Nt, lz = state(lam + t * dl)
                worse = (lz >= logz) & ((Nt.unsqueeze(2) * d).sum(1).norm(dim=1) >= r.norm(dim=1))
                if not bool((worse & (r.norm(dim=1) > tol)).any()):
                    break
                t = torch.where(worse.unsqueeze(1) & (r.norm(dim=1, keepdim=True) > tol), 0.5 * t, t)
            better = (r.norm(dim=1, keepdim=True) > tol) & ~worse.unsqueeze(1)
            lam = torch.where(better, lam + t * dl, lam)
            if not bool(better.any()):
                break
        N, _ = state(lam)
        r = (N.unsqueeze(2) * d).sum(1)
        J = (N.unsqueeze(2) * d).transpose(1, 2) @ d - r.unsqueeze(2) * r.unsqueeze(1)
        got.append((N, -N.unsqueeze(2) * torch.linalg.solve(J, d.transpose(1, 2)).transpose(1, 2), lam))
    return tuple(torch.cat(t) for t in zip(*got))


def _full(s):
    return torch.stack([torch.stack([s[:, a], s[:, b], s[:, c]], 1) for a, b, c in ((0, 3, 5), (3, 1, 4), (5, 4, 2))], 1)


def _six(A):
    return torch.stack([A[:, 0, 0], A[:, 1, 1], A[:, 2, 2], A[:, 0, 1], A[:, 1, 2], A[:, 0, 2]], 1)


def _return_map(mat, dt, dF, be, ebar, T, J):
    K, mu = mat.E / (3.0 * (1.0 - 2.0 * mat.nu)), mat.E / (2.0 * (1.0 + mat.nu))
    b = dF @ _full(be) @ dF.transpose(1, 2)
    parts = [torch.linalg.eigh(t) for t in (0.5 * (b + b.transpose(1, 2))).split(10000)]
    lam, Q = torch.cat([t[0] for t in parts]), torch.cat([t[1] for t in parts])
    e = 0.5 * torch.log(lam)
    tr = e.sum(1, keepdim=True)
    s = 2.0 * mu * (e - tr / 3.0)
    sn = s.norm(dim=1)
    q = math.sqrt(1.5) * sn
    if mat.model == "j2":
        f = sn - math.sqrt(2.0 / 3.0) * (mat.sigma_y0 + mat.H * ebar)
        dep = math.sqrt(2.0 / 3.0) * torch.clamp(f, min=0.0) / (2.0 * mu + 2.0 * mat.H / 3.0)
    else:
        therm = 1.0 - torch.clamp((T - mat.T_room) / (mat.T_melt - mat.T_room), 0.0, 1.0) ** mat.m

        def flow(x):
            rate = torch.clamp(x / dt / mat.eps_dot0, min=1.0)
            return (mat.A + mat.B * (ebar + x) ** mat.n) * (1.0 + mat.C * torch.log(rate)) * therm

        lo, hi = torch.zeros_like(q), q / (3.0 * mu)
        for _ in range(70):
            mid = 0.5 * (lo + hi)
            up = q - 3.0 * mu * mid - flow(mid) > 0.0
            lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
        dep = torch.where(q > flow(torch.zeros_like(q)), 0.5 * (lo + hi), torch.zeros_like(q))
    e = e - math.sqrt(1.5) * dep.unsqueeze(1) * s / sn.clamp(min=1e-300).unsqueeze(1)
    tau = K * tr + 2.0 * mu * (e - tr / 3.0)
    new_be = (Q * torch.exp(2.0 * e).unsqueeze(1)) @ Q.transpose(1, 2)
    sigma = (Q * (tau / J.unsqueeze(1)).unsqueeze(1)) @ Q.transpose(1, 2)
    heat = mat.chi * (q - 3.0 * mu * dep) * dep / (mat.rho0 * mat.cp) if mat.model == "jc" else 0.0
    return _six(new_be), _six(sigma), ebar + dep, T + heat, dep / dt


def _steps(P, steps):
    mat, x, du, xp = P.materials[0], P.node_x, P.node_du0, P.mp_x
    n = xp.shape[0]
    vol, ebar = P.mp_vol.clone(), torch.zeros(n, dtype=torch.float64, device=DEV)
    T = torch.full((n,), P.T0, dtype=torch.float64, device=DEV)
    eye = torch.eye(3, dtype=torch.float64, device=DEV).expand(n, 3, 3)
    F, dF, be, sigma = eye, eye, _six(eye), torch.zeros(n, 6, dtype=torch.float64, device=DEV)
    x_old, xp_old = x, xp
    ids, ok = _supports(x, xp, P.rs2, 384)
    N, dN, _ = _max_ent(x, xp, ids, ok, P.beta, 1e-15 * P.h)
    for _ in range(steps):
        m, f = torch.zeros(x.shape[0], dtype=torch.float64, device=DEV), torch.zeros_like(x)
        for i in range(0, n, 50000):
            s = slice(i, i + 50000)
            m.index_add_(0, ids[s].reshape(-1), (N[s] * P.mp_mass[s, None]).reshape(-1))
            g = -vol[s, None, None] * (dN[s] @ _full(sigma[s]))
            if P.eps_stab > 0.0:
                q = x_old[ids[s]] - xp_old[s, None, :]
                off = (x[ids[s]] - xp[s, None, :]) - q @ dF[s].transpose(1, 2)
                g = g - P.eps_stab * N[s].unsqueeze(2) * off / q.norm(dim=2, keepdim=True).clamp(min=1e-12 * P.h)
            f.index_add_(0, ids[s].reshape(-1), g.reshape(-1, 3))
        u = du + P.dt * P.dt * f / m.unsqueeze(1)
        new = x + u
        new = torch.cat([new[:, :2], new[:, 2:].clamp(min=0.0)], 1)     # the wall at z = 0
        du, x_old, x, xp_old = new - x, x, new, xp
        xp = torch.cat([(N[i:i + 50000].unsqueeze(1) @ x[ids[i:i + 50000]]).squeeze(1) for i in range(0, n, 50000)])
        dF = eye + torch.cat([du[ids[i:i + 50000]].transpose(1, 2) @ dN[i:i + 50000] for i in range(0, n, 50000)])
        F, vol = dF @ F, vol * torch.linalg.det(dF)
        be, sigma, ebar, T, _ = _return_map(mat, P.dt, dF, be, ebar, T, torch.linalg.det(F))
        ids, ok = _supports(x, xp, P.rs2, 384)
        N, dN, _ = _max_ent(x, xp, ids, ok, P.beta, 1e-15 * P.h)
    spare = torch.zeros(3 * P.max_insert, dtype=torch.float64, device=DEV)      # room for inserted nodes
    return dict(node_x=torch.cat([x.reshape(-1), spare]), node_du=torch.cat([du.reshape(-1), spare]),
                F=F.reshape(-1), sigma=sigma.reshape(-1), ebar=ebar, T=T, support_count=None, nodes=None, points=None)
