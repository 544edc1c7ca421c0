"""J^-1 of the LME solves against the exported shape functions."""
import numpy as np
import pytest

import scenarios

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def inverse_hessians(sim, p, rows):
    """K = (sum N d d^T - r r^T)^-1 and |r| / h of the rows, from the handle's own positions and N."""
    x, xp, cnt = sim.get("node_x"), sim.get("mp_x"), sim.get("support_count")
    ids, sh = sim.get_rows("support_ids", rows), sim.get_rows("shape", rows)
    K, res = [], []
    for r, q in enumerate(rows):
        d, N = xp[q] - x[ids[r, :cnt[q]]], sh[r, :cnt[q], 0]
        rr = N @ d
        K.append(np.linalg.inv((N[:, None] * d).T @ d - np.outer(rr, rr)))
        res.append(np.abs(rr).max() / p.h)
    return np.array(K)[:, [0, 1, 2, 0, 1, 0], [0, 1, 2, 1, 2, 2]], np.array(res)


@pytest.mark.parametrize("tol", [0.2, 1e-2, 1e-14])
def test_inverse_hessian_at_any_newton_tolerance(tol):
    """K is exact for the r at which the solve stops, however loose the caller's tolerance: 1e-12 of its largest entry
    (A to 2e-15 of its trace, times the condition of H, at most about 30 at the surface, and numpy's own)."""
    p = scenarios.taylor_rod(h=0.8e-3, R=3.2e-3, L=6.4e-3, material=scenarios.copper_jc())
    p.newton_tol = tol
    from paper_2206_08772_gb300.otm import OTM
    sim = OTM(p)
    rows = np.arange(0, p.n_mps, 5)
    for steps in (0, 3):
        assert steps == 0 or sim.step(steps) == 0, sim.error()
        K, res = inverse_hessians(sim, p, rows)
        got = sim.get("kinv")[rows]
        assert (np.abs(got - K).max(1) <= 1e-12 * np.abs(K).max(1)).all()
        assert res.max() <= tol + 1e-14
        if tol > 1e-3 and steps == 0:
            assert res.max() > 0.05 * tol


@pytest.mark.parametrize("tol", [1e-2, 1e-14])
def test_double_float_hessian_sums_of_the_mixed_path(tol):
    """The mixed handle's own solves (its first and after steps), whose A is summed in double-float, 1e-14 of its trace:
    times the condition of H and three products, 1e-11. A snapshot of an FP64 handle regenerates in fixed point and
    does not reach these sums."""
    from paper_2206_08772_gb300.otm import OTM
    p = scenarios.taylor_rod(h=0.8e-3, R=3.2e-3, L=6.4e-3, material=scenarios.copper_jc())
    p.newton_tol = tol
    sim = OTM(p, precision="mixed")
    rows = np.arange(0, p.n_mps, 5)
    for steps in (0, 3):
        assert steps == 0 or sim.step(steps) == 0, sim.error()
        K, _ = inverse_hessians(sim, p, rows)
        err = (np.abs(sim.get("kinv")[rows] - K).max(1) / np.abs(K).max(1)).max()
        print("mixed J^-1 against the exported N:", steps, err)
        assert err <= 1e-11
