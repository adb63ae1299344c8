"""The autotuner offers the schedule that the automatic choice takes for small sparse
systems, the per-target kernel with the far field beside it: chosen where it is the
fastest by a fifth or more (c = 2, 4 particles per cell), whatever the config asked for,
with the results of the automatic plan bit for bit; larger systems run on one stream."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh,near", [((32, 16, 16), "NEAR_AUTO"), ((32, 32, 32), "NEAR_AUTO"),
                                       ((32, 32, 32), "NEAR_CELL_ITEMS")])
def test_autotune_offers_the_automatic_schedule(mesh, near):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    n = 4 * int(np.prod(mesh))
    g = synth.rng(7600 + n)
    pos = torch.tensor(g.random((n + 200000, 3)), dtype=torch.float32, device="cuda")
    q = torch.tensor(g.random(n + 200000) - 0.5, dtype=torch.float32, device="cuda")

    def cfg(nf):
        return pk.Config(mesh=mesh, p=5, cutoff=2, boundary=pk.PERIODIC, precision=pk.FP32, near_field=nf)

    auto, plan = pk.Plan(cfg(pk.NEAR_AUTO)), pk.Plan(cfg(getattr(pk, near)))
    kernel, _ = plan.autotune([n], pos[:n].contiguous(), q[:n].contiguous(), reps=10)
    assert kernel == pk.NEAR_PER_TARGET
    phi, force = torch.empty_like(q[:n]), torch.empty_like(pos[:n])
    rphi, rforce, _ = auto.compute(pos[:n].contiguous(), q[:n].contiguous())
    tp, tq = pos[:n].contiguous(), q[:n].contiguous()
    for _ in range(3):  # plain, capture + launch, replay
        plan.compute(tp, tq, phi, force)
        assert plan.info(pk.INFO_SPLIT) == 1
        assert torch.equal(phi, rphi) and torch.equal(force, rforce)
    plan.compute(pos, q)
    assert plan.info(pk.INFO_SPLIT) == 0 and plan.status() == pk.OK
    plan.compute(tp, tq, phi, force)  # the workspace has grown
    assert plan.info(pk.INFO_SPLIT) == 1 and torch.equal(phi, rphi) and torch.equal(force, rforce)
    auto.close()
    plan.close()
