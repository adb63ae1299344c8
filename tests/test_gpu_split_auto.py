"""The automatic near field of small FP32 systems runs the far field on the plan's second
stream: results, energies included, equal those of the one-stream sequence (stage timing
on) bit for bit, from plain calls, graph replays and batched calls, for the per-target
kernel (sparse) and the cell items (filled cells); above the size limit one stream."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mesh,cutoff,boundary", [(1, 8, 1, 0), (1500, 8, 1, 1), (7001, 8, 2, 0), (16400, 8, 1, 1),
                                                    (40007, 16, 2, 1), (131072, 16, 1, 0), (131073, 16, 1, 1)])
def test_auto_split_matches_one_stream(n, mesh, cutoff, boundary):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    g = synth.rng(9900 + n)
    pos = torch.tensor(g.random((n, 3)), dtype=torch.float32, device="cuda")
    q = torch.tensor(g.random(n) - 0.5, dtype=torch.float32, device="cuda")
    cfg = pk.Config(mesh=(mesh,) * 3, p=4, cutoff=cutoff, boundary=boundary, precision=pk.FP32)
    counts = [n // 3, 0, n - n // 3]
    ref = pk.Plan(cfg)
    ref.set_timing(True)
    rphi, rforce, re = ref.compute(pos, q, energy=True)
    bphi, bforce, be = ref.compute_batched(counts, pos, q, energies=True)
    assert ref.info(pk.INFO_SPLIT) == 0
    plan = pk.Plan(cfg)
    phi, force = torch.empty_like(q), torch.empty_like(pos)
    for k in range(3):  # plain, capture + launch, replay
        phi.zero_()
        force.zero_()
        _, _, e = plan.compute(pos, q, phi, force, energy=True)
        assert plan.info(pk.INFO_SPLIT) == (1 if n <= 1 << 17 else 0)
        assert torch.equal(phi, rphi) and torch.equal(force, rforce) and e == re, k
    phi2, force2, e2 = plan.compute_batched(counts, pos, q, energies=True)
    assert torch.equal(phi2, bphi) and torch.equal(force2, bforce) and np.array_equal(e2, be)
    plan.close()
    ref.close()
