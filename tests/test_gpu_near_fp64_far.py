"""FP64 near field with a particle so far outside an open box that its squared distance
overflows: the call reports PMMM_ERR_OUT_OF_BOX, and the particle, clamped into a corner
cell, adds nothing to the others (1 / infinity) instead of making them NaN.  Order 0 on
2^3 cells, so that every cell is a near one and the far field is zero up to the rounding
of the transforms (1e-13 of the sums)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cutoff", [1, 2])
def test_infinite_distance_adds_nothing(cutoff):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    n = 60
    g = synth.rng(7500 + cutoff)
    pos = g.random((n, 3))
    pos[0] = (1e160, 0.7, 0.6)
    q = 0.5 + g.random(n)
    plan = pk.Plan(pk.Config(mesh=(2, 2, 2), p=0, cutoff=cutoff, boundary=pk.OPEN, precision=pk.FP64))
    phi, force, _ = plan.compute(torch.tensor(pos, device="cuda"), torch.tensor(q, device="cuda"))
    assert plan.status() == pk.ERR_OUT_OF_BOX
    phi, force = phi.cpu().numpy(), force.cpu().numpy()
    d = pos[1:, None] - pos[None, 1:]
    r = np.sqrt((d ** 2).sum(-1))
    np.fill_diagonal(r, np.inf)
    rphi = (q[None, 1:] / r).sum(1)
    rforce = q[1:, None] * (q[None, 1:, None] * d / r[..., None] ** 3).sum(1)
    assert np.linalg.norm(phi[1:] - rphi) < 1e-12 * np.linalg.norm(rphi)
    assert np.linalg.norm(force[1:] - rforce) < 1e-12 * np.linalg.norm(rforce)
    plan.close()
