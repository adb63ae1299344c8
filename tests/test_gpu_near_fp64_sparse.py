"""The FP64 near field with three blocks per SM (at least 2^14 particles, at most one to
three cells), on both sides of the line: a batch of sparse systems against their own
evaluations, where every sum has the same terms (1e-13: the M2L of a batch adds them in
another order)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nsys,per", [(97, 169), (97, 170), (97, 171), (96, 170)])  # 16393, 16490, 16587 of 49664 cells; 16320
@pytest.mark.parametrize("cutoff", [1, 2])
def test_sparse_batch_matches_single_systems(nsys, per, cutoff):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    g = synth.rng(8300 + nsys + per + cutoff)
    n = nsys * per
    pos = torch.tensor(g.random((n, 3)), device="cuda")
    q = torch.tensor(g.random(n) - 0.5, device="cuda")
    cfg = pk.Config(mesh=(8, 8, 8), p=2, cutoff=cutoff, boundary=pk.PERIODIC, precision=pk.FP64)
    batch, single = pk.Plan(cfg), pk.Plan(cfg)
    phi, force, e = batch.compute_batched([per] * nsys, pos, q, energies=True)
    for s in (0, nsys // 2, nsys - 1):
        a, b = s * per, (s + 1) * per
        sphi, sforce, se = single.compute(pos[a:b].contiguous(), q[a:b].contiguous(), energy=True)
        assert torch.linalg.norm(phi[a:b] - sphi) < 1e-13 * torch.linalg.norm(sphi)
        assert torch.linalg.norm(force[a:b] - sforce) < 1e-13 * torch.linalg.norm(sforce)
        assert abs(e[s] - se) < 1e-13 * 0.5 * float((q[a:b] * sphi).abs().sum())
    batch.close()
    single.close()
