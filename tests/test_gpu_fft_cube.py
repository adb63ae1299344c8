"""One-CTA-per-channel transforms of cubic FP32 meshes (8, 16, 32 cells an axis, periodic;
8, 16 open, padded): local expansions of single systems and of a batch against the FP64
plan, whose transforms are the column passes, within the tolerance of the FP32 path."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

P = 3
TOL = 3e-6 * (1 + 0.25 * P)


@pytest.mark.parametrize("m,boundary", [(8, 1), (16, 1), (32, 1), (8, 0), (16, 0)])
def test_cube(m, boundary):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    counts = [700, 900]
    pos, q = synth.uniform_pm1(sum(counts), synth.seed(7, 90 + m + boundary))
    pos = pos.astype(np.float32).astype(np.float64)

    def plan(prec):
        return pk.Plan(pk.Config(mesh=(m,) * 3, p=P, boundary=pk.PERIODIC if boundary else pk.OPEN, precision=prec))

    def t(a, dt):
        return torch.tensor(a, dtype=dt, device="cuda")

    p64, p32 = plan(pk.FP64), plan(pk.FP32)
    n = counts[0]
    p64.compute(t(pos[:n], torch.float64), t(q[:n], torch.float64))
    p32.compute(t(pos[:n], torch.float32), t(q[:n], torch.float32))
    L64, L32 = p64.export(pk.EXPORT_LOCAL), p32.export(pk.EXPORT_LOCAL).astype(np.float64)
    assert np.linalg.norm(L32 - L64) < TOL * np.linalg.norm(L64)

    phi64, f64, _ = p64.compute_batched(counts, t(pos, torch.float64), t(q, torch.float64))
    phi32, f32, _ = p32.compute_batched(counts, t(pos, torch.float32), t(q, torch.float32))
    for a, b in ((phi32, phi64), (f32, f64)):
        a, b = a.double().cpu().numpy(), b.cpu().numpy()
        assert np.linalg.norm(a - b) < TOL * np.linalg.norm(b)
    p64.close()
    p32.close()
