"""Calls that do not ask for the energy skip its reduction: same potentials and forces,
bit for bit, for every near-field kernel (cell items, per target, FP64 blocks, split),
plain, graph-launched and batched, and alternating with calls that ask for it."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,mesh,n,near", [(1, 16, 140001, 0), (1, 8, 16384, 1), (1, 8, 3001, 2),
                                                   (1, 8, 16384, 3), (1, 8, 1500, 0), (0, 8, 3001, 0)])
def test_no_energy_same_results(precision, mesh, n, near):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    g = synth.rng(1234 + n)
    dt = torch.float64 if precision == pk.FP64 else torch.float32
    pos = torch.tensor(g.random((n, 3)), dtype=dt, device="cuda")
    q = torch.tensor(g.random(n) - 0.5, dtype=dt, device="cuda")
    plan = pk.Plan(pk.Config(mesh=(mesh,) * 3, p=3, boundary=pk.PERIODIC, precision=precision, near_field=near))
    rphi, rforce, re = plan.compute(pos, q, energy=True)
    phi, force = torch.empty_like(q), torch.empty_like(pos)
    for energy in (False, False, False, True, False, True, True):
        phi.zero_()
        force.zero_()
        _, _, e = plan.compute(pos, q, phi, force, energy=energy)
        torch.cuda.synchronize()
        assert torch.equal(phi, rphi) and torch.equal(force, rforce) and (e == re if energy else e is None)
    counts = [n - 5, 0, 5]
    bphi, bforce, be = plan.compute_batched(counts, pos, q, energies=True)
    phi2, force2, _ = plan.compute_batched(counts, pos, q)
    assert torch.equal(phi2, bphi) and torch.equal(force2, bforce)
    hphi, hforce, he = plan.compute_host(pos.cpu().numpy(), q.cpu().numpy())
    assert he is None and np.array_equal(hphi, rphi.cpu().numpy()) and np.array_equal(hforce, rforce.cpu().numpy())
    plan.close()
