"""The weight and bias gradients summed over row slices (and the tile widths chosen by
the number of blocks): a batch's gradient against the mean of its 128-row parts, each
of which is one slice of two K chunks.  For a power-of-two number of parts the output
gradients differ by an exact scale, so only FP32 sums (K = rows products, and as many
partial sums) separate the two: 2e-5 covers 8192 2^-24 / sqrt(8192).  Otherwise their
BF16 rounding differs as well (2^-9 each, averaged over the rows): 5e-3."""
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
    s.set(pk.SUR_PARAMS, init_params(121, 77))
    yield s
    s.close()


@pytest.mark.parametrize("rows", [256, 384, 512, 640, 4096, 4224, 8192])
def test_gradient_is_the_mean_of_its_parts(sur, rows):
    import torch
    g = synth.rng(7100 + rows)
    X = torch.tensor(g.standard_normal((rows, 432)), dtype=torch.bfloat16, device="cuda")
    T = torch.tensor(g.standard_normal((rows, 128)), dtype=torch.float32, device="cuda")
    T[:, 121:] = 0.0
    loss, grad = sur.gradients(X, T)
    parts = [sur.gradients(X[r:r + 128], T[r:r + 128]) for r in range(0, rows, 128)]
    mean = np.mean([p[1].astype(np.float64) for p in parts], axis=0)
    tol = 2e-5 if rows & (rows - 1) == 0 else 5e-3
    for lo, hi in ((0, 256 * 432), (256 * 432, 256 * 433), (256 * 433, 256 * 433 + 65536),
                   (256 * 433 + 65536, 256 * 434 + 65536), (256 * 434 + 65536, 256 * 434 + 98304),
                   (256 * 434 + 98304, 256 * 434 + 98304 + 121)):
        d = np.linalg.norm(grad[lo:hi] - mean[lo:hi])
        assert d < tol * np.linalg.norm(mean[lo:hi]), (lo, d / np.linalg.norm(mean[lo:hi]))
    assert abs(loss - np.mean([p[0] for p in parts])) < 1e-6 * loss
