"""The automatic near field runs the per-target kernel below 8 particles per cell and the
cell items from 8 on, where crowded cells of an uneven system would make the per-target
kernel up to 1.7 times slower: results bit for bit those of the chosen kernel, for a
uniform and a clustered system, with the far field beside the near field (small systems)
and on one stream, both cutoffs."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mesh,kernel", [(7 * 512 + 511, (8, 8, 8), "NEAR_PER_TARGET"), (8 * 512, (8, 8, 8), "NEAR_CELL_ITEMS"),
                                           (15 * 4096, (16, 16, 16), "NEAR_CELL_ITEMS"),
                                           (12 * 16384, (32, 32, 16), "NEAR_CELL_ITEMS")])
@pytest.mark.parametrize("cutoff", [1, 2])
def test_automatic_kernel(n, mesh, kernel, cutoff):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    g = synth.rng(7700 + n + cutoff)
    uniform = g.random((n, 3))
    clustered = np.where(np.arange(n)[:, None] % 4 == 0, uniform, 0.45 + 0.1 * uniform)
    q = torch.tensor(g.random(n) - 0.5, dtype=torch.float32, device="cuda")

    def cfg(near):
        return pk.Config(mesh=mesh, p=3, cutoff=cutoff, boundary=pk.OPEN, precision=pk.FP32, near_field=near)

    for pos in (uniform, clustered):
        tp = torch.tensor(pos, dtype=torch.float32, device="cuda")
        auto, ref = pk.Plan(cfg(pk.NEAR_AUTO)), pk.Plan(cfg(getattr(pk, kernel)))
        phi, force, _ = auto.compute(tp, q)
        assert auto.info(pk.INFO_SPLIT) == (1 if n <= 1 << 17 else 0)
        rphi, rforce, _ = ref.compute(tp, q)
        assert torch.equal(phi, rphi) and torch.equal(force, rforce)
        auto.close()
        ref.close()
