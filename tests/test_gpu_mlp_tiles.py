"""The forms of the network's products (whole output rows or 128 columns per block in two
stages for large and medium batches, 64-column tiles in four stages for small ones): a
batch's outputs equal those of its parts bit for bit (the sums run over the same K in the
same order), at the last size of one form and the first of the next, and its gradient is the
mean of its parts' (a power-of-two number of parts, so only FP32 sums of K = rows
products separate the two: 2e-5 covers 16384 2^-24 / sqrt(16384))."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sur():
    import torch
    import paper_1409_5981_gb300 as pk
    from paper_1409_5981_gb300.surrogate import init_params
    pk.build()
    torch.cuda.set_device(0)
    s = pk.Surrogate(pk.Config(mesh=(8, 8, 8), p=3, boundary=pk.PERIODIC, precision=pk.FP32), 10)
    s.set(pk.SUR_PARAMS, init_params(121, 78))
    yield s
    s.close()


@pytest.mark.parametrize("rows", [11648, 11776, 29056, 29184, 38912])
def test_forward_equals_its_parts(sur, rows):
    import torch
    g = synth.rng(7800 + rows)
    X = torch.tensor(g.standard_normal((rows, 432)), dtype=torch.bfloat16, device="cuda")
    out = sur.forward(X, torch.empty((rows, 128), dtype=torch.float32, device="cuda"))
    for r in range(0, rows, 4096):
        part = X[r:r + 4096].contiguous()
        want = sur.forward(part, torch.empty((len(part), 128), dtype=torch.float32, device="cuda"))
        assert torch.equal(out[r:r + 4096], want)


def test_gradient_of_a_large_batch(sur):
    import torch
    rows, part = 16384, 4096
    g = synth.rng(7900)
    X = torch.tensor(g.standard_normal((rows, 432)), dtype=torch.bfloat16, device="cuda")
    T = torch.tensor(g.standard_normal((rows, 128)), dtype=torch.float32, device="cuda")
    T[:, 121:] = 0.0
    loss, grad = sur.gradients(X, T)
    parts = [sur.gradients(X[r:r + part], T[r:r + part]) for r in range(0, rows, part)]
    mean = np.mean([p[1].astype(np.float64) for p in parts], axis=0)
    assert np.linalg.norm(grad - mean) < 2e-5 * np.linalg.norm(mean)
    assert abs(loss - np.mean([p[0] for p in parts])) < 1e-6 * loss
