"""The cell sort of an evaluation: permutation, sorted cells and offsets against a
stable numpy sort by the oracle's cell ids, at the sizes where its kernels change
form: a cell below, at and above the size from which whole blocks rank it, crowded
cells at ragged positions, cells that fill scan blocks, input already sorted by cell,
and a second evaluation on the same plan (the per-cell counters are reused)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pk():
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    return pk


def _crowd(g, sizes, mesh, extra):
    """sizes[k] particles in cell (k, 1, 2) of the mesh and `extra` uniform ones, shuffled."""
    pos = [g.random((extra, 3))]
    for k, m in enumerate(sizes):
        pos.append((np.array([k, 1, 2]) + 0.02 + 0.96 * g.random((m, 3))) / mesh)
    pos = np.concatenate(pos)
    return pos[g.permutation(len(pos))].astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("sizes,mesh,extra", [
    ((1, 2, 3, 31, 32, 33, 255, 257), 8, 0),
    ((1023, 1024, 1025, 7, 1279, 1281), 8, 100),
    ((4099, 1, 2600), 8, 5),
    ((), 16, 3 * 4096 + 1),
    ((40000,), 4, 0),
])
@pytest.mark.parametrize("fp64", [False, True])
def test_cell_sort_is_stable(pk, sizes, mesh, extra, fp64):
    import torch
    g = synth.rng(4200 + mesh + extra + len(sizes))
    pos = _crowd(g, sizes, mesh, extra)
    cfg = pk.Config(mesh=(mesh,) * 3, p=1, boundary=pk.OPEN, precision=pk.FP64 if fp64 else pk.FP32)
    dt = torch.float64 if fp64 else torch.float32
    plan = pk.Plan(cfg)
    for order in ("shuffled", "sorted", "shuffled"):
        _, cell, perm, cs, _ = oracle.bin_particles(pos, (0, 0, 0), (1, 1, 1), (mesh,) * 3, False)
        x = pos if order == "shuffled" else pos[perm]
        _, cell, perm, cs, _ = oracle.bin_particles(x, (0, 0, 0), (1, 1, 1), (mesh,) * 3, False)
        plan.compute(torch.tensor(x, dtype=dt, device="cuda"), torch.ones(len(x), dtype=dt, device="cuda"), energy=True)
        assert np.array_equal(plan.export(pk.EXPORT_PERM), perm)
        assert np.array_equal(plan.export(pk.EXPORT_SORTED_CELL), cell[perm])
        assert np.array_equal(plan.export(pk.EXPORT_CELL_START), cs)
    plan.close()
