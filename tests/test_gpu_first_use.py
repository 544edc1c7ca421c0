"""Stand-alone entries as the first CUDA work of a process: nothing else has set up the library's device data."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import sys
import numpy as np
import torch
import oracle, scenarios
from paper_2206_08772_gb300 import otm
mode, model = sys.argv[1:3]
mat = scenarios.copper_j2() if model == "j2" else scenarios.copper_jc()
rng = np.random.default_rng(5)
n, dt = 64, 5e-9
dF = np.eye(3) + rng.normal(0, 1, (n, 3, 3)) * 3e-4
dF[:8] = np.eye(3)
be = np.concatenate([1 + rng.normal(0, 1, (n, 3)) * 1e-3, rng.normal(0, 0.5, (n, 3)) * 1e-3], 1)
be[:8] = [1, 1, 1, 0, 0, 0]
ebar = np.abs(rng.normal(0, 0.1, n))
T = np.full(n, mat.T_room + 100.0)
ref = [oracle.return_map(mat, dt, dF[k], be[k], ebar[k], T[k], np.linalg.det(dF[k])) for k in range(n)]
assert all(r[0] == 0 for r in ref) and (model == "j2" or any(r[3] > e for r, e in zip(ref, ebar)))
dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
a = [dev(dF.reshape(-1, 9)), dev(dF.reshape(-1, 9)), dev(be), dev(ebar), dev(T)]
if mode == "captured":
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        sig, rate, failed, status = otm.return_map(mat, dt, *a)
    g.replay()
else:
    sig, rate, failed, status = otm.return_map(mat, dt, *a)
torch.cuda.synchronize()
assert status.item() == 0
K, mu = mat.E / (3 * (1 - 2 * mat.nu)), mat.E / (2 * (1 + mat.nu))
s = np.array([r[1] for r in ref])
# the rounding of b^e about 1 through the moduli, times 20 for the sums, and 1e-10 of the stress
err = np.abs(sig.cpu().numpy() - s).max()
assert err <= 20 * 1.1e-16 * max(K, 2 * mu) / 0.99 + 1e-10 * np.abs(s).max(), (err, K)
'''


@pytest.mark.parametrize("mode", ["plain", "captured"])
@pytest.mark.parametrize("model", ["j2", "jc"])
def test_return_map_alone_in_a_fresh_process(orc, mode, model):
    r = subprocess.run([sys.executable, "-c", CHILD, mode, model], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
