"""The FP64 path's kinematics gather (Eq. 9, Eq. 11) against exact fractions over the exported shape functions."""
from fractions import Fraction

import numpy as np
import pytest

import scenarios

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tol", [1e-14, 1e-4])
@pytest.mark.parametrize("amp", [0.3, 1e-2, 1e-3, 1e-5, 1e-7])
def test_kinematics_gather_is_as_precise_for_small_increments(amp, tol):
    """Eq. 9 and Eq. 11 of one step with random increments of `amp` spacings, over the exported shape functions: x_p is
    sum N x_a whatever the Newton tolerance, and the off-diagonal entries of dF (free of the 1) are good to FP64
    rounding of their own products. Bounds: at most 9 additions a lane and 5 of the warp, each of a partial sum below
    the largest |x| (sum N = 1): 14 2^-53 of that; the same, three products with K and the exported gradient's
    own 4 roundings: below 32 2^-53 of sum |du||K||e|."""
    from paper_2206_08772_gb300.otm import OTM
    p = scenarios.taylor_rod(h=0.8e-3, R=3.2e-3, L=6.4e-3, wall=False, material=scenarios.copper_j2())
    p.newton_tol = tol
    rng = np.random.default_rng(3)
    p.node_du0[:] = rng.normal(0, amp * p.h, p.node_du0.shape).clip(-1.5 * amp * p.h, 1.5 * amp * p.h) / 3
    sim = OTM(p)
    rows = np.arange(0, p.n_mps, 37)
    cnt, kinv = sim.get("support_count"), sim.get("kinv")
    xp0, x0 = sim.get("mp_x"), sim.get("node_x")
    ids, sh = sim.get_rows("support_ids", rows), sim.get_rows("shape", rows)
    assert sim.step(1) == 0, sim.error()
    x, du, xp, dF = sim.get("node_x"), sim.get("node_du"), sim.get("mp_x"), sim.get("dF").reshape(-1, 3, 3)
    off = ~np.eye(3, dtype=bool)
    for r, q in enumerate(rows):
        a, N, g = ids[r, :cnt[q]], sh[r, :cnt[q], 0], sh[r, :cnt[q], 1:]
        for i in range(3):
            ref = sum(Fraction(float(n)) * Fraction(float(c)) for n, c in zip(N, x[a, i]))
            assert abs(Fraction(float(xp[q, i])) - ref) <= 14 * 2.0 ** -53 * np.abs(x[a, i]).max()
        K = np.abs(kinv[q][[0, 3, 5, 3, 1, 4, 5, 4, 2]].reshape(3, 3))
        e = N[:, None] * np.abs(xp0[q] - x0[a])
        scale = np.abs(du[a]).T @ (e @ K)
        assert (np.abs(dF[q] - du[a].T @ g)[off] <= 32 * 2.0 ** -53 * scale[off]).all()
