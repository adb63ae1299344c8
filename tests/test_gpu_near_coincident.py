"""Two particles on both sides of a cell face that coincide after the rounding of their
cell-relative FP32 coordinates (x = -1e-9 and x = 0 about a face at 0): the near field
drops such a pair, as it drops the self pair, and leaves every other pair alone.  In a
cell crowded enough that whole warps of targets lie in it and in a sparse one, against
FP64 evaluations without one or the other particle of the pair (open box: their mutual
term is in the near field only).  Every other pair is 0.05 cells apart, so 3 * 2^-24 /
0.05 = 3.6e-6 bounds the relative error of the closest pair's force; twice that, and the
FP32 far field's tolerance 3e-6 (1 + p / 4), bound the sums."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

MESH, P = 8, 3


@pytest.fixture(scope="module")
def pk():
    import torch
    import paper_1409_5981_gb300 as pk
    pk.build()
    torch.cuda.set_device(0)
    return pk


def _cell(g, cell, n):
    """n particles of cell (3 integers), 0.35/5 cells from its faces and each other."""
    idx = np.stack(np.meshgrid(*[np.arange(5)] * 3, indexing="ij"), -1).reshape(-1, 3)[g.permutation(125)[:n]]
    u = (idx + 0.5 + 0.15 * (2.0 * g.random((n, 3)) - 1.0)) / 5
    return -1.0 + (np.asarray(cell) + u) * (2.0 / MESH)


def _system(m, cutoff):
    g = synth.rng(7300 + m + cutoff)
    pair = np.array([[-1e-9, 0.115, 0.13], [0.0, 0.115, 0.13]])  # the face between cells 3 and 4, 4, 4
    cell = _cell(g, (3, 4, 4), m)  # the pair in the middle of the cell's order, inside a whole warp of it
    pos = np.concatenate([cell[:m // 2], pair, cell[m // 2:], _cell(g, (4, 4, 4), 5)]
                         + [_cell(g, (c % MESH, c // MESH, 1), 2) for c in g.permutation(MESH * MESH)[:20]])
    return pos.astype(np.float32), (0.5 + g.random(len(pos))).astype(np.float32), m // 2


def _eval(pk, pos, q, precision, cutoff, boundary, near=0):
    import torch
    dt = torch.float64 if precision == pk.FP64 else torch.float32
    plan = pk.Plan(pk.Config(box_lo=(-1.0,) * 3, box_len=(2.0,) * 3, mesh=(MESH,) * 3, p=P, cutoff=cutoff,
                             boundary=boundary, precision=precision, near_field=near))
    phi, force, e = plan.compute(torch.tensor(pos, dtype=dt, device="cuda"), torch.tensor(q, dtype=dt, device="cuda"),
                                 energy=True)
    plan.close()
    return phi.double().cpu().numpy(), force.double().cpu().numpy(), e


def _check(pk, near, m, cutoff):
    pos, q, i0 = _system(m, cutoff)
    n = len(q)
    phi, force, e = _eval(pk, pos, q, pk.FP32, cutoff, pk.OPEN, near)
    assert np.isfinite(phi).all() and np.isfinite(force).all() and np.isfinite(e)
    # everyone but the pair from the whole system, each of the pair from the system without the other
    rphi, rforce, _ = _eval(pk, pos, q, pk.FP64, cutoff, pk.OPEN)
    for a, b in ((i0, i0 + 1), (i0 + 1, i0)):
        keep = np.arange(n) != b
        pa, fa, _ = _eval(pk, pos[keep], q[keep], pk.FP64, cutoff, pk.OPEN)
        rphi[a], rforce[a] = pa[i0], fa[i0]
    tol = 7.2e-6 + 3e-6 * (1 + 0.25 * P)
    assert np.linalg.norm(force - rforce) < tol * np.linalg.norm(rforce)
    assert np.linalg.norm(phi - rphi) < tol * np.linalg.norm(rphi)
    assert abs(e - 0.5 * (q * rphi).sum()) < tol * 0.5 * np.abs(q * rphi).sum()
    # periodic: the same near-field pairs
    assert all(np.isfinite(v).all() for v in _eval(pk, pos, q, pk.FP32, cutoff, pk.PERIODIC, near))


@pytest.mark.parametrize("cutoff", [1, 2])
@pytest.mark.parametrize("m", [3, 100])
def test_per_target(pk, m, cutoff):
    _check(pk, pk.NEAR_PER_TARGET, m, cutoff)


@pytest.mark.parametrize("cutoff", [1, 2])
@pytest.mark.parametrize("m", [3, 100])
@pytest.mark.parametrize("split", [False, True])
def test_cell_items(pk, split, m, cutoff):
    _check(pk, pk.NEAR_CELL_ITEMS_SPLIT if split else pk.NEAR_CELL_ITEMS, m, cutoff)
