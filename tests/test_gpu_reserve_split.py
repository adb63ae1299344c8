"""After pmmm_plan_reserve the default evaluation allocates nothing, whatever the reserved
capacity: small FP32 systems still run the far field beside the near field, single and
batched, with the workspace unchanged and the results of the one-stream sequence."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap", [1 << 12, 1 << 17, (1 << 20) + 1])
def test_reserved_plan_allocates_nothing(cap):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    n, counts = 1500, [600, 0, 900]
    pos, q = synth.uniform_pm1(n, synth.seed(7, 40))
    tp = torch.tensor(pos.astype(np.float32), device="cuda")
    tq = torch.tensor(q.astype(np.float32), device="cuda")
    cfg = pk.Config(mesh=(8, 8, 8), p=2, boundary=pk.PERIODIC, precision=pk.FP32)
    ref = pk.Plan(cfg)
    ref.set_timing(True)  # one stream
    rphi, rforce, _ = ref.compute(tp, tq)
    bphi, bforce, _ = ref.compute_batched(counts, tp, tq)
    plan = pk.Plan(cfg)
    plan.reserve_batched(len(counts), cap)
    used = plan.info(pk.INFO_WORKSPACE_BYTES)
    phi, force = torch.empty_like(tq), torch.empty_like(tp)
    for _ in range(3):  # plain, capture + launch, replay
        plan.compute(tp, tq, phi, force)
        assert plan.info(pk.INFO_SPLIT) == 1
        assert torch.equal(phi, rphi) and torch.equal(force, rforce)
    assert plan.info(pk.INFO_WORKSPACE_BYTES) == used
    p2 = pk.Plan(cfg)
    p2.reserve_batched(len(counts), cap)
    plan.compute_batched(counts, tp, tq, phi, force)  # brings the M2L tables of batched calls
    used = plan.info(pk.INFO_WORKSPACE_BYTES)
    phi.zero_()
    plan.compute_batched_graph(counts, tp, tq, phi, force)
    assert plan.info(pk.INFO_SPLIT) == 1 and plan.info(pk.INFO_WORKSPACE_BYTES) == used
    assert torch.equal(phi, bphi) and torch.equal(force, bforce)
    p2.compute_batched_graph(counts, tp, tq, phi, force)  # captured by the first call already
    assert p2.info(pk.INFO_SPLIT) == 1
    assert torch.equal(phi, bphi) and torch.equal(force, bforce)
    for p in (ref, plan, p2):
        p.close()
