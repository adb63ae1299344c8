"""The rotated tensor-core M2L at the edges of its tiles: 1 to 65 systems past a tile of
64 (or 32), orders whose channels leave 64 partly empty, few wavevectors (tiles split over
blocks) and many, against the FP32 SIMT M2L of the same systems: the largest difference
of the locals below 1e-4 of the largest local, the bound of the split-BF16 test of whole
batches (products carry 3 * 2^-18 each)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nsys,mesh,p", [(2, 4, 7), (3, 8, 1), (31, 4, 4), (33, 4, 7), (64, 4, 3), (65, 4, 7),
                                         (129, 4, 6), (5, 16, 7), (66, 8, 5)])
def test_tiles_match_simt(nsys, mesh, p):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    g = synth.rng(9100 + nsys + p)
    counts = g.integers(0, 40, nsys)
    counts[0] = 25
    n = int(counts.sum())
    pos = torch.tensor(g.random((n, 3)), dtype=torch.float32, device="cuda")
    q = torch.tensor(2.0 * g.random(n) - 1.0, dtype=torch.float32, device="cuda")
    out = []
    for prec in (pk.FP32, pk.FP32_SPLITBF16_M2L):
        plan = pk.Plan(pk.Config(mesh=(mesh,) * 3, p=p, boundary=pk.PERIODIC, precision=prec))
        plan.compute_batched(counts, pos, q, energies=True)
        if prec == pk.FP32_SPLITBF16_M2L:
            assert plan.info(pk.INFO_M2L_ARITH) == pk.M2L_ARITH_SPLITBF16_TC
        out.append(plan.export(pk.EXPORT_LOCAL))
        plan.close()
    assert np.abs(out[1] - out[0]).max() < 1e-4 * np.abs(out[0]).max()
