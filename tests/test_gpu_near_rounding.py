"""Rounding of the per-target FP32 near field: the potential is sign (far + sum / h) with
one rounding.  Pairs of particles at the centres of adjacent cells (distance exactly one
cell, so the sum is the partner's charge), h = 0.75 (1 / h is no FP32 number); the far
field is read back, so the exact value is known to every bit."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("timing", [False, True])  # far field beside the near field, one stream
def test_one_rounding(timing):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    mesh, h = 16, 0.75
    cells = np.array([(x + dx, y, z) for x in range(0, 16, 4) for y in range(0, 16, 4) for z in range(0, 16, 4)
                      for dx in (0, 1)])
    pos = ((cells + 0.5) * h).astype(np.float32)  # exact
    g = synth.rng(7400)
    q = (0.5 + g.random(len(pos))).astype(np.float32)
    plan = pk.Plan(pk.Config(box_len=(mesh * h,) * 3, mesh=(mesh,) * 3, p=3, boundary=pk.OPEN, precision=pk.FP32,
                             near_field=pk.NEAR_AUTO))
    plan.set_timing(timing)
    phi, force, _ = plan.compute(torch.tensor(pos, device="cuda"), torch.tensor(q, device="cuda"))
    assert plan.info(pk.INFO_SPLIT) == (0 if timing else 1)
    perm, far = plan.export(pk.EXPORT_PERM), plan.export(pk.EXPORT_FAR).reshape(-1, 4)
    plan.close()
    fp = np.empty(len(q))
    fp[perm] = far[:, 0]
    partner = q.reshape(-1, 2)[:, ::-1].reshape(-1).astype(np.float64)
    want = fp + partner * np.float64(np.float32(1.0 / h))  # 48 bits of product: exact in 64 bits
    got = phi.cpu().numpy()
    # half a unit in the last place, and 2^-50 for the rounding of the sum in 64 bits
    assert np.all(np.abs(got.astype(np.float64) - want) <= np.spacing(np.abs(got)) * (0.5 + 2.0 ** -20))
