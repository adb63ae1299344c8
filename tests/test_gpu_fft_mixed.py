"""The runtime-size one-CTA-per-channel transforms: batches of FP32 systems on non-cubic
meshes of up to 32 cells an axis (every radix, mixed axis lengths, padded and not), with
more channels than the GPU has SMs, against the FP64 plan, whose transforms are the column
passes, within the tolerance of the FP32 path; a system of its own, whose channels take
the plane kernels, agrees too."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

P = 3
TOL = 3e-6 * (1 + 0.25 * P)


@pytest.mark.parametrize("mesh,boundary", [((16, 8, 32), 1), ((32, 16, 8), 1), ((8, 32, 32), 1), ((4, 16, 32), 1),
                                           ((16, 8, 8), 0), ((4, 16, 8), 0), ((2, 8, 16), 0)])
def test_mixed_axes(mesh, boundary):
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nsys = sms // (P + 1) ** 2 + 1
    counts = [300 + 7 * s for s in range(nsys)]
    g = synth.rng(9000 + sum(mesh) + boundary)
    n = sum(counts)
    pos = (g.random((n, 3)) * np.asarray(mesh) / max(mesh)).astype(np.float32).astype(np.float64)
    q = np.where(np.arange(n) % 2, 1.0, -1.0)

    def plan(prec):
        return pk.Plan(pk.Config(box_len=tuple(m / max(mesh) for m in mesh), mesh=mesh, p=P, precision=prec,
                                 boundary=pk.PERIODIC if boundary else pk.OPEN))

    def t(a, dt):
        return torch.tensor(a, dtype=dt, device="cuda")

    p64, p32 = plan(pk.FP64), plan(pk.FP32)
    phi64, f64, _ = p64.compute_batched(counts, t(pos, torch.float64), t(q, torch.float64))
    phi32, f32, _ = p32.compute_batched(counts, t(pos, torch.float32), t(q, torch.float32))
    L64, L32 = p64.export(pk.EXPORT_LOCAL), p32.export(pk.EXPORT_LOCAL)
    for a, b in ((phi32, phi64), (f32, f64)):
        a, b = a.double().cpu().numpy(), b.cpu().numpy()
        assert np.linalg.norm(a - b) < TOL * np.linalg.norm(b)
    assert np.linalg.norm(L32 - L64) < TOL * np.linalg.norm(L64)
    m = counts[0]
    p32.compute(t(pos[:m], torch.float32), t(q[:m], torch.float32))
    K = int(np.prod(mesh))
    assert np.linalg.norm(p32.export(pk.EXPORT_LOCAL) - L64[:, :K]) < TOL * np.linalg.norm(L64[:, :K])
    p64.close()
    p32.close()
