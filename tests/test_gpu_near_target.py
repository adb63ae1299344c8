"""The per-target FP32 near field where its warps change form: cells of 31 to 97
particles (a warp of 32 targets lies in one cell or does not), empty and odd cells,
rows that wrap around a periodic box or end at an open one, both cutoffs.  Against the
FP64 oracle; particles on jittered lattices inside their cells, so that no pair is
closer than 0.07 cells and the cell-relative FP32 coordinates (2^-24) bound the force
error by 3 * 2^-24 / 0.07 = 2.6e-6 of the closest pair, below the FP32 tolerance of
the order (3e-6 (1 + p / 4))."""
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
    u = (idx + 0.5 + 0.15 * (2.0 * g.random((n, 3)) - 1.0)) / k
    return (np.asarray(cell) + u) / mesh


@pytest.mark.parametrize("sizes", [(31, 32, 33, 1), (64, 0, 97, 2, 3), (700, 96)])
@pytest.mark.parametrize("boundary,cutoff", [(0, 1), (1, 1), (1, 2)])
def test_per_target_matches_oracle(pk, sizes, boundary, cutoff):
    import torch
    g = synth.rng(6100 + sum(sizes) + 7 * boundary + cutoff)
    mesh, p = 8, 3
    pos = [_cell(g, (k, 0, 7), m, mesh) for k, m in enumerate(sizes)]
    pos += [_cell(g, (c % mesh, c // mesh, 3), 1, mesh) for c in g.permutation(mesh * mesh)[:40]]
    pos = np.concatenate(pos)
    pos = pos.astype(np.float32).astype(np.float64)
    pos = pos[g.permutation(len(pos))]
    q = 0.5 + g.random(len(pos))
    q = q.astype(np.float32).astype(np.float64)
    plan = pk.Plan(pk.Config(mesh=(mesh,) * 3, p=p, cutoff=cutoff, boundary=boundary, precision=pk.FP32,
                             near_field=pk.NEAR_PER_TARGET))
    phi, force, _ = plan.compute(torch.tensor(pos, dtype=torch.float32, device="cuda"),
                                 torch.tensor(q, dtype=torch.float32, device="cuda"))
    ref = oracle.pmmm(pos, q, (0, 0, 0), (1, 1, 1), (mesh,) * 3, p, cutoff, boundary == pk.PERIODIC)
    f = -q[:, None] * ref["grad"]
    tol = 3e-6 * (1 + 0.25 * p)
    assert np.linalg.norm(force.double().cpu().numpy() - f) < tol * np.linalg.norm(f)
    assert np.linalg.norm(phi.double().cpu().numpy() - ref["phi"]) < tol * np.linalg.norm(ref["phi"])
    plan.close()
