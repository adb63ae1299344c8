"""The FP64 near field at the block splits of its items: cells of 1 to 129 particles (128
down to 4 source phases, idle lanes, items that end a cell), empty cells, rows that wrap
or end, both cutoffs, against the FP64 oracle.  Jittered lattices keep every pair 0.07
cells apart, so 1e-12 leaves a factor of 50 over 2^-52 / 0.07 per pair."""
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


def _cell(g, cell, n, mesh):
    k = 5 if n <= 125 else 10
    idx = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[g.permutation(k ** 3)[:n]]
    return (np.asarray(cell) + (idx + 0.5 + 0.15 * (2.0 * g.random((n, 3)) - 1.0)) / k) / mesh


@pytest.mark.parametrize("sizes", [(1,), (1, 2, 3, 5, 7), (31, 32, 33, 16, 17), (64, 0, 43, 129)])
@pytest.mark.parametrize("boundary,cutoff", [(0, 1), (1, 1), (1, 2), (0, 2)])
def test_fp64_near_matches_oracle(pk, sizes, boundary, cutoff):
    import torch
    g = synth.rng(8100 + sum(sizes) + 7 * boundary + cutoff)
    mesh, p = 8, 3
    pos = np.concatenate([_cell(g, (k, 0, 7), m, mesh) for k, m in enumerate(sizes)]
                         + [_cell(g, (c % mesh, c // mesh, 3), 1, mesh) for c in g.permutation(mesh * mesh)[:20]])
    pos = pos[g.permutation(len(pos))]
    q = 0.5 + g.random(len(pos))
    plan = pk.Plan(pk.Config(mesh=(mesh,) * 3, p=p, cutoff=cutoff, boundary=boundary, precision=pk.FP64))
    phi, force, _ = plan.compute(torch.tensor(pos, device="cuda"), torch.tensor(q, device="cuda"))
    ref = oracle.pmmm(pos, q, (0, 0, 0), (1, 1, 1), (mesh,) * 3, p, cutoff, boundary == pk.PERIODIC)
    f = -q[:, None] * ref["grad"]
    assert np.linalg.norm(force.cpu().numpy() - f) < 1e-12 * np.linalg.norm(f)
    assert np.linalg.norm(phi.cpu().numpy() - ref["phi"]) < 1e-12 * np.linalg.norm(ref["phi"])
    plan.close()
