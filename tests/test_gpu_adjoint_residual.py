"""The adjoint where the LME solves stop well before r = 0."""
import numpy as np
import pytest

import scenarios

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

THETA0 = np.array([90e6, 292e6, 0.31, 0.025, 1.09, 227.0])


@pytest.mark.parametrize("tol", [1e-2, 1e-4])
def test_adjoint_at_loose_newton_tolerances(orc, tol):
    """Two steps from a Newton tolerance of 1e-2 and 1e-4 spacings, against the CPU reference adjoint, which carries
    r = sum N d in H and its adjoint. Both solve from the same starts up to the last state, whose shape functions
    the objectives do not see, so they stop at the same iterates; bounds as of the tight tolerance."""
    from paper_2206_08772_gb300.adjoint import rod_objectives

    def make(theta):
        A, B, n, C, m, v0 = theta
        p = scenarios.taylor_rod(h=0.8e-3, R=3.2e-3, L=4.0e-3, material=scenarios.copper_jc(A=A, B=B, n=n, C=C, m=m), v0=v0)
        p.newton_tol = tol
        return p

    th = torch.tensor(THETA0, dtype=torch.float64, requires_grad=True)
    vals = rod_objectives(th, make, 2, 1)
    ref_vals, ref_grads, _ = orc.reference_adjoint(make(THETA0), 2)
    for o in range(2):
        assert abs(vals[o].item() - ref_vals[o]) <= 1e-10 * abs(ref_vals[o])
        g = torch.autograd.grad(vals[o], th, retain_graph=True)[0].numpy()
        scale = np.abs(ref_grads[o] * THETA0)
        assert np.all(np.abs(g - ref_grads[o]) * THETA0 <= 1e-10 * scale.max() + 1e-8 * scale), (g, ref_grads[o])
