"""Snapshots written before the header named the kind of evaluation."""
import numpy as np
import pytest

import scenarios

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MAGIC_AT, KIND_AT = 24, 64      # bytes into the header: nn, nm, step, magic; 8 words, then the kind
FIRST_MAGIC = 0x4F544D53


def test_snapshot_without_the_evaluation_kind():
    """Such a snapshot's bytes past its shorter header hold anything: it loads the same whatever they are, with the
    shape functions of an FP64 evaluation, 1e-12 from the fixed-point ones; another magic is refused."""
    from paper_2206_08772_gb300.otm import OTM
    p = scenarios.taylor_rod(h=0.8e-3, R=3.2e-3, L=6.4e-3, material=scenarios.copper_jc())
    sim = OTM(p)
    assert sim.step(3) == 0
    shape0, x0 = sim.get("shape"), sim.get("node_x")
    buf, ptr = sim.snapshot()
    head = buf[ptr - buf.data_ptr():][:128].view(torch.int64)
    head[MAGIC_AT // 8] = FIRST_MAGIC
    got = []
    for junk in (0, 1, 2, -1, 0x7FF8DEADBEEF0001):
        head[KIND_AT // 8] = junk
        sim.restore((buf, ptr))
        assert np.array_equal(sim.get("node_x"), x0)
        got.append(sim.get("shape"))
        assert np.array_equal(got[-1], got[0])
        assert np.abs(got[-1][..., 0] - shape0[..., 0]).max() <= 1e-12
        assert sim.step(1) == 0
    head[MAGIC_AT // 8] = FIRST_MAGIC + 7
    with pytest.raises(Exception):
        sim.restore((buf, ptr))
