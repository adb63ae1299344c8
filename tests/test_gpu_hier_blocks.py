"""Block transforms of two-level plans at their edges: fewer coarse cells than a block of
threads holds, every compile-time transform length and kept width (m, W) = (8, 6), (16, 12),
(16, 10), (32, 24), (32, 20), odd and even channel counts of the child matrices, against the
oracle's cell-pair definition with the tolerances of the two-level path."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-10
FP32_TOL = {p: 3e-6 * (1 + 0.25 * p) for p in range(0, 13)}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("mesh,refine,cutoff,p,boundary", [
    ((8, 8, 8), 2, 1, 4, 1), ((8, 4, 4), 2, 1, 3, 0), ((8, 8, 8), 4, 1, 4, 0), ((16, 16, 16), 4, 1, 3, 1),
    ((8, 16, 8), 2, 2, 4, 0), ((16, 16, 32), 8, 1, 2, 0), ((16, 8, 8), 4, 2, 3, 0)])
def test_blocks(precision, mesh, refine, cutoff, p, boundary):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    fp64 = precision == "fp64"
    pos, q = synth.uniform_pm1(1500, synth.seed(7, 70 + refine + cutoff + p))
    if not fp64:
        pos = pos.astype(np.float32).astype(np.float64)
    cfg = pk.Config(mesh=mesh, p=p, cutoff=cutoff, boundary=pk.PERIODIC if boundary else pk.OPEN,
                    precision=pk.FP64 if fp64 else pk.FP32, refine=refine)
    dt = torch.float64 if fp64 else torch.float32
    plan = pk.Plan(cfg)
    phi, force, _ = plan.compute(torch.tensor(pos, dtype=dt, device="cuda"), torch.tensor(q, dtype=dt, device="cuda"))
    phi, force = phi.cpu().numpy().astype(np.float64), force.cpu().numpy().astype(np.float64)
    alpha = cfg.ewald_alpha if cfg.ewald_alpha > 0 else None
    ref = oracle.pmmm_hier(pos, q, cfg.box_lo, cfg.box_len, mesh, p, refine, cutoff, bool(boundary), alpha=alpha,
                           nmax=cfg.ewald_nmax or 5)
    rf = -(q[:, None] * ref["grad"])
    bound = FP64_TOL if fp64 else FP32_TOL[p]
    assert np.linalg.norm(force - rf) < bound * np.linalg.norm(rf)
    assert np.linalg.norm(phi - ref["phi"]) < bound * np.linalg.norm(ref["phi"])
    plan.close()
