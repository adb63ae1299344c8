"""A caller's own capture of the plan's stream: default evaluations of small FP32 systems
record the fork to the plan's second stream and the join, larger ones one stream; replays
read new inputs, and results equal those of the one-stream sequence bit for bit, also of
a plain call between replays."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mesh,refine", [(3000, 8, 0), (6000, 8, 0), (3000, 8, 2), (140000, 16, 0)])
def test_captured_by_the_caller(n, mesh, refine):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    cfg = pk.Config(mesh=(mesh,) * 3, p=3, boundary=pk.PERIODIC, precision=pk.FP32, refine=refine)
    inputs = []
    ref = pk.Plan(cfg)
    ref.set_timing(True)
    for k in range(2):
        g = synth.rng(9100 + n + refine + k)
        pos = torch.tensor(g.random((n, 3)), dtype=torch.float32, device="cuda")
        q = torch.tensor(g.random(n) - 0.5, dtype=torch.float32, device="cuda")
        phi, force, _ = ref.compute(pos, q)
        inputs.append((pos, q, phi, force))
    assert ref.info(pk.INFO_SPLIT) == 0
    pos, q = inputs[0][0].clone(), inputs[0][1].clone()
    phi, force = torch.empty_like(q), torch.empty_like(pos)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    plan = pk.Plan(cfg, stream)
    plan.reserve(n)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        assert plan.compute_raw(n, pos.data_ptr(), q.data_ptr(), phi.data_ptr(), force.data_ptr()) == 0
    assert plan.info(pk.INFO_SPLIT) == (1 if n <= 1 << 17 else 0)

    def check(k):
        torch.cuda.synchronize()
        assert plan.status() == pk.OK
        assert torch.equal(phi, inputs[k][2]) and torch.equal(force, inputs[k][3])
        phi.zero_()
        force.zero_()
        torch.cuda.synchronize()

    for k in (0, 1, 1, 0):
        pos.copy_(inputs[k][0])
        q.copy_(inputs[k][1])
        torch.cuda.synchronize()
        graph.replay()
        check(k)
        assert plan.compute_raw(n, pos.data_ptr(), q.data_ptr(), phi.data_ptr(), force.data_ptr()) == 0
        check(k)
    del graph
    plan.close()
    ref.close()
