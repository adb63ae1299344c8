"""PMMM_INFO_LAUNCHES and PMMM_INFO_SPLIT describe the last call, also when it replayed a
graph that was captured before calls of another form (without the energy, another
batch)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_facts_follow_the_replayed_graph():
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    n = 1500
    pos, q = synth.uniform_pm1(n, synth.seed(7, 50))
    tp = torch.tensor(pos.astype(np.float32), device="cuda")
    tq = torch.tensor(q.astype(np.float32), device="cuda")
    phi, force = torch.empty_like(tq), torch.empty_like(tp)
    plan = pk.Plan(pk.Config(mesh=(8, 8, 8), p=3, boundary=pk.PERIODIC, precision=pk.FP32))

    def call(energy):
        plan.compute(tp, tq, phi, force, energy=energy)
        return plan.info(pk.INFO_LAUNCHES), plan.info(pk.INFO_SPLIT)

    with_e = call(True)                # plain
    assert call(True) == with_e        # captured
    without = call(False)              # the other graph, captured
    assert without[0] < with_e[0]      # no reduction
    for _ in range(2):                 # replays in turn
        assert call(True) == with_e
        assert call(False) == without
    # a batch replayed after a single-system call
    counts = [700, 800]
    plan.compute_batched_graph(counts, tp, tq, phi, force)
    batch = plan.info(pk.INFO_LAUNCHES), plan.info(pk.INFO_SYSTEMS)
    plan.set_timing(True)              # one stream: another number of launches
    assert call(False)[1] == 0
    plan.set_timing(False)
    plan.compute_batched_graph(counts, tp, tq, phi, force)
    assert (plan.info(pk.INFO_LAUNCHES), plan.info(pk.INFO_SYSTEMS)) == batch
    assert plan.info(pk.INFO_SPLIT) == 1
    plan.close()
