"""Performance cases of the particle mesh multipole library: what its users have it do.

A case is one pass through a public entry point of ``paper_1409_5981_gb300``:
``Plan.compute`` (one system, device arrays), ``Plan.compute_host`` (host arrays in
and out), ``Plan.compute_batched`` / ``compute_batched_graph`` (many systems at
once) and ``Surrogate.gradients`` (one backward pass of the learned correction).
Plans, weights and output buffers are made once, as a program that steps in time or
trains keeps them.

``exact`` is an independent FP64 evaluation in plain torch of what each call is
defined to return: the method at the same order, mesh, cutoff and Ewald splitting
(not the infinite-order limit), from its definitions.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1409_5981_gb300 as pk

_PRECISION = {"fp64": pk.FP64, "fp32": pk.FP32, "splitbf16": pk.FP32_SPLITBF16_M2L}


# ------------------------------------------------------------------------- the cases
def _single(name, n, mesh, p, boundary="periodic", precision="fp32", cutoff=1, refine=0, distribution="uniform",
            energy=False, form="single"):
    mx, my, mz = (mesh,) * 3 if isinstance(mesh, int) else mesh
    return {"name": name, "form": form, "n": n, "mx": mx, "my": my, "mz": mz, "p": p, "cutoff": cutoff,
            "boundary": boundary, "precision": precision, "refine": refine, "distribution": distribution,
            "energy": energy}


def listed():
    return [
        # the smallest call: a small isolated cluster in double precision, its energy read every step
        _single("open_n4096_m8_p4_fp64", 4096, 8, 4, "open", "fp64", energy=True),
        # a small periodic box (molecular-dynamics size, odd count, a few particles per cell), energy every step
        _single("periodic_n20011_m16_p5", 20011, 16, 5, energy=True),
        # the ordinary call: a periodic box of 2^20 charges, 32 per cell
        _single("periodic_n1M_m32_p7", 1 << 20, 32, 7),
        # the same physics called with host arrays (a program that keeps its particles on the host), ragged count
        _single("host_n300007_m32_p7", 300007, 32, 7, form="host"),
        # gravity of a centrally concentrated cluster: open boundary, very uneven cells
        _single("plummer_n1M_m64_p5", 1 << 20, 64, 5, "open", distribution="plummer"),
        # the largest single system
        _single("periodic_n16M_m64_p7", 1 << 24, 64, 7),
        # double precision, ordinary size: the reference run of a precision study
        _single("periodic_n131072_m16_p7_fp64", 1 << 17, 16, 7, precision="fp64"),
        # the wider cutoff (125 near cells) at lower order: the paper's recommended trade
        _single("periodic_n1M_m32_p5_c2", 1 << 20, 32, 5, cutoff=2),
        # a fine mesh with few particles per cell: the far field carries the time
        _single("periodic_n1M_m64_p7_sparse", 1000003, 64, 7),
        # two-level evaluation, tensor-core block M2L
        _single("hier_n1M_m32_r4_p7", 1 << 20, 32, 7, precision="splitbf16", refine=4),
        # many independent systems of uneven size in one graph-launched evaluation, tensor-core M2L
        {"name": "batched64_m32_p7_splitbf16", "form": "batched", "systems": 64, "lo": 14.0, "hi": 18.0, "draw": 4,
         "mesh": 32, "p": 7, "precision": "splitbf16", "graph": True},
        # one training step's backward pass of the learned correction
        {"name": "train_rows8192", "form": "train", "rows": 8192, "p_high": 10},
    ]


def draw(rng):
    kind = rng.random()
    if kind < 0.12:
        return {"form": "train", "rows": 128 * int(round(2 ** rng.uniform(2, 8))), "p_high": rng.randint(4, 10)}
    if kind < 0.27:
        mesh = rng.choice([8, 16, 32])
        lo = rng.uniform(8.0, 14.0)
        nsys = int(round(2 ** rng.uniform(1, 5 if mesh == 32 else 6)))
        return {"form": "batched", "systems": nsys, "lo": round(lo, 2), "hi": round(lo + rng.uniform(0.5, 4.0), 2),
                "draw": rng.randint(0, 1 << 20), "mesh": mesh, "p": rng.randint(3, 7),
                "precision": rng.choice(["fp32", "splitbf16"]), "graph": rng.random() < 0.5}
    boundary = rng.choice(["open", "periodic"])
    if kind < 0.37:
        m = rng.choice([16, 32])
        c = _single("", int(m ** 3 * 2 ** rng.uniform(1, 6)) | 1, m, rng.randint(3, 7), "periodic",
                    rng.choice(["fp32", "splitbf16"]), refine=rng.choice([2, 4]))
        del c["name"]
        return c
    precision = "fp64" if rng.random() < 0.25 else "fp32"
    m = rng.choice([8, 16, 32] if precision == "fp64" else [8, 16, 32, 64])
    mesh = [m if rng.random() < 0.75 else max(8, m // 2) for _ in range(3)]
    p = rng.randint(2, 7 if m == 64 else 11)
    plummer = boundary == "open" and rng.random() < 0.4
    n = int(mesh[0] * mesh[1] * mesh[2] * 2 ** rng.uniform(0, 6)) + rng.randint(0, 7)
    c = _single("", n, mesh, p, boundary, precision, 2 if rng.random() < 0.2 else 1, 0,
                "plummer" if plummer else "uniform", rng.random() < 0.3, "host" if rng.random() < 0.2 else "single")
    del c["name"]
    # no drawn case costs more than the largest listed ones (FP64 runs at about 1/64 of the FP32 rate)
    most = 2.5e9 if precision == "fp64" else 2.0e11
    while work(c)["flops"] > most:
        c["n"] = int(0.8 * c["n"])
    return c


def _box(case):
    """(box_lo, box_len) of a single-system case: cubic cells."""
    if case["distribution"] == "plummer":
        return (-1.0, -1.0, -1.0), (2.0, 2.0, 2.0)
    m = (case["mx"], case["my"], case["mz"])
    return (0.0, 0.0, 0.0), tuple(a / max(m) for a in m)


def _sizes(case):
    """Particle counts of a batched case: log-uniform, fixed by the case."""
    u = np.random.Generator(np.random.PCG64(case["draw"])).random(case["systems"])
    return [int(2.0 ** (case["lo"] + (case["hi"] - case["lo"]) * v)) for v in u]


# ------------------------------------------------------------------------- inputs
def _rand(n, k, gen, dtype):
    return torch.rand((n, k), generator=gen, dtype=dtype, device=gen.device)


def _charges(n, dtype, device):
    """n // 2 charges of each sign (one zero when n is odd): a neutral system of i.i.d. positions."""
    q = torch.zeros(n, dtype=dtype, device=device)
    q[: n // 2] = 1.0
    q[n // 2: 2 * (n // 2)] = -1.0
    return q


def _inputs(case, seed, device):
    """(pos, q) of a single-system case; (pos, q, counts) of a batched one."""
    gen = torch.Generator(device=device).manual_seed(int(seed))
    if case["form"] == "batched":
        counts = _sizes(case)
        pos = _rand(sum(counts), 3, gen, torch.float32)
        q = torch.cat([_charges(c, torch.float32, device) for c in counts])
        return pos, q, counts
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    n = case["n"]
    if case["distribution"] == "plummer":
        # Plummer sphere, scale radius 0.1, cut at 10 radii, equal masses
        a, top = 0.1, (1.0 + 0.01) ** -1.5
        u = _rand(n, 3, gen, torch.float64)
        r = a / torch.sqrt((top * (1.0 - u[:, 0])) ** (-2.0 / 3.0) - 1.0)
        ct, ph = 2.0 * u[:, 1] - 1.0, 2.0 * math.pi * u[:, 2]
        st = torch.sqrt(1.0 - ct * ct)
        pos = torch.stack([r * st * torch.cos(ph), r * st * torch.sin(ph), r * ct], dim=1) * 0.999
        return pos.to(dtype).contiguous(), torch.full((n,), 1.0 / n, dtype=dtype, device=device)
    _, length = _box(case)
    pos = _rand(n, 3, gen, dtype) * torch.tensor(length, dtype=dtype, device=device)
    return pos.contiguous(), _charges(n, dtype, device)


def _train_inputs(case, seed, device):
    """Unit-variance features and targets, and parameters of the usual scale."""
    gen = torch.Generator(device=device).manual_seed(int(seed))
    rows, c_high = case["rows"], (case["p_high"] + 1) ** 2

    def normal(*shape):
        return torch.randn(shape, generator=gen, device=device)

    X = normal(rows, pk.SUR_IN).to(torch.bfloat16)
    T = normal(rows, pk.SUR_OUT_ROWS)
    T[:, c_high:] = 0.0
    W3 = normal(128, 256) / 16.0
    W3[c_high:] = 0.0
    b3 = 0.1 * normal(128)
    b3[c_high:] = 0.0
    theta = torch.cat([(normal(256, 432) / math.sqrt(432)).reshape(-1), 0.1 * normal(256),
                       (normal(256, 256) / 16.0).reshape(-1), 0.1 * normal(256), W3.reshape(-1), b3])
    return X, T, theta


def _gravity(case):
    return case.get("distribution") == "plummer"


def prepare(case, seed):
    stream = torch.cuda.current_stream()
    if case["form"] == "train":
        X, T, theta = _train_inputs(case, seed, "cuda")
        sur = pk.Surrogate(pk.Config(mesh=(8, 8, 8), p=3, boundary=pk.PERIODIC, precision=pk.FP32),
                           p_high=case["p_high"], stream=stream)
        sur.set(pk.SUR_PARAMS, theta.cpu().numpy())
        return {"form": "train", "sur": sur, "X": X, "T": T}
    if case["form"] == "batched":
        pos, q, counts = _inputs(case, seed, "cuda")
        plan = pk.Plan(pk.Config(mesh=(case["mesh"],) * 3, p=case["p"], boundary=pk.PERIODIC,
                                 precision=_PRECISION[case["precision"]]), stream=stream)
        plan.reserve_batched(len(counts), int(q.shape[0]))
        return {"form": "batched", "plan": plan, "pos": pos, "q": q, "counts": counts, "graph": case["graph"],
                "phi": torch.empty_like(q), "force": torch.empty_like(pos)}
    pos, q = _inputs(case, seed, "cuda")
    lo, length = _box(case)
    plan = pk.Plan(pk.Config(box_lo=lo, box_len=length, mesh=(case["mx"], case["my"], case["mz"]), p=case["p"],
                             cutoff=case["cutoff"], boundary=pk.OPEN if case["boundary"] == "open" else pk.PERIODIC,
                             precision=_PRECISION[case["precision"]], sign=-1.0 if _gravity(case) else 1.0,
                             refine=case["refine"]), stream=stream)
    plan.reserve(case["n"])
    if case["form"] == "host":
        pos, q = pos.cpu().pin_memory(), q.cpu().pin_memory()
        return {"form": "host", "plan": plan, "pos": pos, "q": q,
                "phi": torch.empty_like(q, pin_memory=True), "force": torch.empty_like(pos, pin_memory=True)}
    return {"form": "single", "plan": plan, "pos": pos, "q": q, "energy": case["energy"],
            "phi": torch.empty_like(q), "force": torch.empty_like(pos)}


def run(state):
    s = state
    if s["form"] == "train":
        loss, grad = s["sur"].gradients(s["X"], s["T"])
        return {"loss": loss, "grad": grad}
    if s["form"] == "batched":
        call = s["plan"].compute_batched_graph if s["graph"] else s["plan"].compute_batched
        phi, force, _ = call(s["counts"], s["pos"], s["q"], s["phi"], s["force"])
        return {"phi": phi, "force": force}
    if s["form"] == "host":
        phi, force, _ = s["plan"].compute_host(s["pos"], s["q"], s["phi"], s["force"])
        return {"phi": phi, "force": force}
    phi, force, energy = s["plan"].compute(s["pos"], s["q"], s["phi"], s["force"], energy=s["energy"])
    return {"phi": phi, "force": force, "energy": energy} if s["energy"] else {"phi": phi, "force": force}


# ------------------------------------------------------------------------- work
def _near_pairs(n, mesh, cutoff, periodic, plummer):
    """Expected source-target pairs of the (2c+1)^3 near cells."""
    if plummer:
        sample = {"form": "single", "precision": "fp64", "n": 200000, "distribution": "plummer"}
        pos, _ = _inputs(sample, 1, "cpu")
        ix = torch.clamp(((pos + 1.0) * (torch.tensor(mesh) / 2.0)).long(), min=0)
        cnt = torch.bincount((ix[:, 2] * mesh[1] + ix[:, 1]) * mesh[0] + ix[:, 0], minlength=math.prod(mesh))
        cnt = cnt.double().reshape(1, 1, mesh[2], mesh[1], mesh[0])
        w = 2 * cutoff + 1
        near = torch.nn.functional.avg_pool3d(cnt, w, 1, cutoff, count_include_pad=True) * w ** 3
        return float((cnt * near).sum()) * (n / 200000.0) ** 2
    pairs = float(n) * n / math.prod(mesh)
    for m in mesh:
        pairs *= 2 * cutoff + 1 if periodic else (m * (2 * cutoff + 1) - cutoff * (cutoff + 1)) / m
    return pairs


def work(case):
    """Near field 19 flops a pair; P2M and L2P 5 and 10 a particle and coefficient; real FFTs; the M2L at 4
    flops a matrix entry and wavevector.  Bytes: particles in, potentials and forces out, kernel spectra in."""
    if case["form"] == "train":
        rows, mac = case["rows"], 432 * 256 + 256 * 256 + 256 * 128
        return {"bytes": rows * (432 * 2 + 128 * 4) + 2 * 4 * pk.SUR_NPARAM,
                "flops": 2.0 * rows * (3 * mac - 432 * 256)}
    if case["form"] == "batched":
        mesh, counts, p, size = (case["mesh"],) * 3, _sizes(case), case["p"], 4
        n, nsys = sum(counts), len(counts)
        pairs = sum(_near_pairs(c, mesh, 1, True, False) for c in counts)
        periodic, refine = True, 0
    else:
        mesh, n, p, nsys = (case["mx"], case["my"], case["mz"]), case["n"], case["p"], 1
        size = 8 if case["precision"] == "fp64" else 4
        periodic, refine = case["boundary"] == "periodic", case["refine"]
        pairs = _near_pairs(n, mesh, case["cutoff"], periodic, _gravity(case))
    C, CG = (p + 1) ** 2, (2 * p + 1) ** 2
    far_mesh = [m // refine for m in mesh] if refine else mesh
    L = [m if periodic else 2 * m for m in far_mesh]
    Kt = math.prod(L)
    Kh = L[2] * L[1] * (L[0] // 2 + 1)
    flops = 19.0 * pairs + 15.0 * n * C + nsys * (5.0 * C * Kt * math.log2(Kt) + 4.0 * C * C * Kh)
    nbytes = 8.0 * n * size + CG * Kh * size
    if refine:
        m = 1  # zero-padded block transforms of length m per axis, one block per coarse cell
        while m < 2 * (case["cutoff"] + 1) * refine:
            m *= 2
        blocks = math.prod(far_mesh)
        flops += blocks * (5.0 * C * m ** 3 * math.log2(m ** 3) + 4.0 * C * C * m * m * (m // 2 + 1))
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------- exact
# Solid harmonics with the 1/(l+m)! and (l-m)! normalisations of the method, complex, all m; index l*l + l + m.
def _h(l, m):
    return l * l + l + m


def _columns(p, col):
    """Stacks m >= 0 columns col[(l, m)] into all (p+1)^2 components; X_l^-m = (-1)^m conj(X_l^m)."""
    rows = []
    for l in range(p + 1):
        for m in range(-l, l + 1):
            rows.append(col[l, m] if m >= 0 else (-1.0) ** (-m) * col[l, -m].conj())
    return torch.stack(rows)


def _regular(p, x, y, z):
    """R_l^m, [(p+1)^2][n]."""
    xy, r2 = torch.complex(x, y), x * x + y * y + z * z
    col = {}
    for m in range(p + 1):
        col[m, m] = torch.ones_like(xy) if m == 0 else col[m - 1, m - 1] * xy * (-0.5 / m)
        for l in range(m + 1, p + 1):
            a = col[l - 1, m] * z * (2 * l - 1)
            if l > m + 1:
                a = a - col[l - 2, m] * r2
            col[l, m] = a / ((l - m) * (l + m))
    return _columns(p, col)


def _singular_columns(J, x, y, z):
    """S_l^m for m >= 0 as {(l, m): complex}."""
    ir2 = 1.0 / (x * x + y * y + z * z)
    xy, zr = torch.complex(x * ir2, y * ir2), z * ir2
    col = {}
    for m in range(J + 1):
        col[m, m] = torch.complex(ir2.sqrt(), torch.zeros_like(x)) if m == 0 else col[m - 1, m - 1] * xy * -(2 * m - 1)
        for l in range(m + 1, J + 1):
            a = col[l - 1, m] * zr * (2 * l - 1)
            if l > m + 1:
                a = a + col[l - 2, m] * ir2 * ((l + m - 1) * (l - m - 1))
            col[l, m] = -a
    return col


def _gamma_upper(J, x):
    """Gamma(l + 1/2, x) / Gamma(l + 1/2), l = 0..J."""
    q, t, out = torch.erfc(x.sqrt()), 2.0 / math.sqrt(math.pi) * x.sqrt() * torch.exp(-x), []
    for l in range(J + 1):
        out.append(q)
        q, t = q + t, t * x / (l + 1.5)
    return out


def _gamma_lower(J, x):
    """gamma(l + 1/2, x) / Gamma(l + 1/2), l = 0..J, from the power series at the top order."""
    term, total = torch.ones_like(x), torch.ones_like(x)
    for k in range(1, 200):
        term = term * x / (J + 0.5 + k)
        total = total + term
    t = torch.exp((J + 0.5) * x.log() - x - math.lgamma(J + 1.5))
    out = [t * total]
    for l in range(J - 1, -1, -1):
        t = t * (l + 1.5) / x
        out.append(out[-1] + t)
    return out[::-1]


def _grid(L, device):
    """Cell offsets of a transform grid (x fastest): (dx, dy, dz) flattened, minimum image."""
    ax = [torch.arange(m, device=device) for m in L]
    ax = [torch.where(2 * a <= m, a, a - m) for a, m in zip(ax, L)]
    dz, dy, dx = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    return dx.reshape(-1), dy.reshape(-1), dz.reshape(-1)


def _green(case_mesh, h, p, c, periodic, device):
    """Kernel components [(2p+1)^2][grid] in real space on the transform grid L; returns (G, L)."""
    J = 2 * p
    L = tuple(m if periodic else 2 * m for m in case_mesh)
    dx, dy, dz = _grid(L, device)
    K = dx.numel()
    masked = torch.maximum(dx.abs(), torch.maximum(dy.abs(), dz.abs())) <= c
    f64 = dict(dtype=torch.float64, device=device)
    if not periodic:
        ok = ~masked
        for d, m in zip((dx, dy, dz), case_mesh):
            ok &= d.abs() < m
        i = torch.nonzero(ok).reshape(-1)
        G = torch.zeros(((J + 1) ** 2, K), dtype=torch.complex128, device=device)
        col = _singular_columns(J, *(d[i].double() * a for d, a in zip((dx, dy, dz), h)))
        G[:, i] = _columns(J, col)
        return G, L
    b = [m * a for m, a in zip(case_mesh, h)]
    alpha, nmax = 1.5 / min(b), 5
    images = [(i, j, k) for i in range(-nmax, nmax + 1) for j in range(-nmax, nmax + 1) for k in range(-nmax, nmax + 1)
              if i * i + j * j + k * k <= nmax * nmax]
    col = {(l, m): torch.zeros(K, dtype=torch.complex128, device=device) for m in range(J + 1) for l in range(m, J + 1)}
    per = max(1, 2_000_000 // K)
    # real space: Q(l + 1/2, (alpha r)^2) S_l over the images, the masked image -P(l + 1/2, (alpha r)^2) S_l
    for s in range(0, len(images), per):
        im = torch.tensor(images[s:s + per], device=device)
        D = [d[None, :] + im[:, a:a + 1] * m for a, (d, m) in enumerate(zip((dx, dy, dz), L))]
        near = torch.maximum(D[0].abs(), torch.maximum(D[1].abs(), D[2].abs())) <= c
        r = [torch.where(near, 1.0e3 * b[a], D[a].double() * h[a]) for a in range(3)]
        w = _gamma_upper(J, alpha ** 2 * (r[0] ** 2 + r[1] ** 2 + r[2] ** 2))
        S = _singular_columns(J, *r)
        for (l, m) in col:
            col[l, m] += (w[l] * ~near * S[l, m]).sum(0)
    i = torch.nonzero(masked & ((dx != 0) | (dy != 0) | (dz != 0))).reshape(-1)
    r = [d[i].double() * a for d, a in zip((dx, dy, dz), h)]
    w = _gamma_lower(J, alpha ** 2 * (r[0] ** 2 + r[1] ** 2 + r[2] ** 2))
    S = _singular_columns(J, *r)
    for (l, m) in col:
        col[l, m][i] -= w[l] * S[l, m]
    # reciprocal space
    kv = torch.tensor([v for v in images if v != (0, 0, 0)], **f64)
    k = [kv[:, a] / b[a] for a in range(3)]
    kn = torch.sqrt(k[0] ** 2 + k[1] ** 2 + k[2] ** 2)
    phase = sum(kv[:, a:a + 1] * (d.double() / L[a])[None, :] for a, d in enumerate((dx, dy, dz)))
    phase = torch.polar(torch.ones_like(phase), 2.0 * math.pi * phase)
    S = _singular_columns(J, *k)
    gauss = torch.exp(-(math.pi * kn / alpha) ** 2) / (b[0] * b[1] * b[2])
    for (l, m) in col:
        f = (-1j) ** l * math.pi ** (l - 0.5) / math.gamma(l + 0.5)
        col[l, m] += (f * gauss * kn ** (2 * l - 1) * S[l, m]) @ phase
    return _columns(J, col), L


def _m2l_index(p):
    """Component of S_{l+lam}^{-(m+mu)} for output (l, m) and input (lam, mu)."""
    lm = [(l, m) for l in range(p + 1) for m in range(-l, l + 1)]
    return [[_h(l + a, -(m + b)) for a, b in lm] for l, m in lm]


def _convolve(M, G, L, mesh, p):
    """Locals [C][B * K] from multipoles [C][B * K] by the cyclic convolution on the grid L."""
    C, nx, ny, nz = (p + 1) ** 2, *mesh
    B = M.shape[1] // (nx * ny * nz)
    shape = (L[2], L[1], L[0])
    Gk = torch.fft.fftn(G.reshape(-1, *shape), dim=(1, 2, 3)).reshape(G.shape[0], -1)
    Mk = torch.fft.fftn(M.reshape(C * B, nz, ny, nx), s=shape, dim=(1, 2, 3)).reshape(C, B, -1)
    Lk = torch.empty_like(Mk)
    idx = torch.tensor(_m2l_index(p), device=M.device)
    step = 1 << 15
    for s in range(0, Mk.shape[2], step):
        A = Gk[:, s:s + step].t().contiguous()[:, idx]  # [k][C][C]
        Lk[:, :, s:s + step] = torch.matmul(A, Mk[:, :, s:s + step].permute(2, 0, 1)).permute(1, 2, 0)
    out = torch.fft.ifftn(Lk.reshape(C * B, *shape), dim=(1, 2, 3))[:, :nz, :ny, :nx]
    return out.reshape(C, -1)


def _p2m(u, q, cell, ncell, p):
    M = torch.zeros((ncell, 2 * (p + 1) ** 2), dtype=torch.float64, device=u.device)
    for s in range(0, q.numel(), 1 << 20):
        x = u[s:s + (1 << 20)]
        R = _regular(p, -x[:, 0], -x[:, 1], -x[:, 2]) * q[s:s + (1 << 20)]
        M.index_add_(0, cell[s:s + (1 << 20)], torch.view_as_real(R.t().contiguous()).reshape(x.shape[0], -1))
    return torch.view_as_complex(M.reshape(ncell, -1, 2)).t().contiguous()


def _l2p(u, cell, Lc, p):
    """(phi, grad [n][3]) of locals [C][cells] at offsets u from the cell centres."""
    n = u.shape[0]
    out = torch.empty((n, 4), dtype=torch.float64, device=u.device)
    rows = [(l, m) for l in range(p + 1) for m in range(-l, l + 1)]
    table = Lc.t().contiguous()
    for s in range(0, n, 1 << 20):
        x = u[s:s + (1 << 20)]
        R = _regular(p, x[:, 0], x[:, 1], x[:, 2])
        Lp = table[cell[s:s + (1 << 20)]].t()
        out[s:s + (1 << 20), 0] = (Lp * R).sum(0).real
        # d/dz R_l^m = R_{l-1}^m, (d/dx - i d/dy) R_l^m = -R_{l-1}^{m-1}
        gz, gm = torch.zeros_like(R[0]), torch.zeros_like(R[0])
        for i, (l, m) in enumerate(rows):
            if abs(m) <= l - 1:
                gz += Lp[i] * R[_h(l - 1, m)]
            if abs(m - 1) <= l - 1:
                gm -= Lp[i] * R[_h(l - 1, m - 1)]
        # phi is real, so (d/dx - i d/dy) phi has real part d/dx phi and imaginary part -d/dy phi
        out[s:s + (1 << 20), 1], out[s:s + (1 << 20), 2], out[s:s + (1 << 20), 3] = gm.real, -gm.imag, gz.real
    return out[:, 0], out[:, 1:]


def _wrap(j, m, periodic):
    """(valid, index) of cell coordinates j on an axis of m cells."""
    return (torch.ones_like(j, dtype=torch.bool) if periodic else (j >= 0) & (j < m)), j % m


def _near(u, q, cell, mesh, h, c, periodic, B):
    """Direct sums over the near cells for particles sorted by cell; (phi, grad)."""
    n, K = q.numel(), mesh[0] * mesh[1] * mesh[2]
    count = torch.bincount(cell, minlength=B * K)
    start = torch.cumsum(count, 0) - count
    out = torch.zeros((n, 4), dtype=torch.float64, device=u.device)
    sysc, lc = cell // K * K, cell % K
    ix, iy, iz = lc % mesh[0], lc // mesh[0] % mesh[1], lc // (mesh[0] * mesh[1])
    x, y, z = (u[:, a].contiguous() for a in range(3))
    offsets = range(-c, c + 1)
    for ez in offsets:
        vz, jz = _wrap(iz + ez, mesh[2], periodic)
        for ey in offsets:
            vy, jy = _wrap(iy + ey, mesh[1], periodic)
            for ex in offsets:
                vx, jx = _wrap(ix + ex, mesh[0], periodic)
                nb = sysc + jx + mesh[0] * (jy + mesh[1] * jz)
                cnt = torch.where(vx & vy & vz, count[nb], 0)
                cnt, order = torch.sort(cnt, descending=True)
                pos = 0
                while pos < n:
                    most = int(cnt[pos])
                    if most == 0:
                        break
                    t = order[pos:pos + max(1, (1 << 26) // most)]
                    e = torch.arange(most, device=u.device)[None, :]
                    live = e < cnt[pos:pos + t.numel(), None]
                    i = torch.where(live, start[nb[t]][:, None] + e, 0)
                    dx = x[t][:, None] - x[i] - ex * h[0]
                    dy = y[t][:, None] - y[i] - ey * h[1]
                    dz = z[t][:, None] - z[i] - ez * h[2]
                    r2 = dx * dx + dy * dy + dz * dz
                    ri = torch.where(live & (r2 > 0), torch.rsqrt(r2), 0.0)
                    qr = q[i] * ri
                    g = -qr * ri * ri
                    out[t] += torch.stack([qr.sum(1), (g * dx).sum(1), (g * dy).sum(1), (g * dz).sum(1)], dim=1)
                    pos += t.numel()
    return out[:, 0], out[:, 1:]


def _bin(pos, lo, length, mesh, periodic):
    """(cell coordinates [n][3], offsets from the cell centres [n][3]) by the binning definition."""
    idx, rel = [], []
    for a in range(3):
        t = pos[:, a] - lo[a]
        if periodic:
            t = torch.where((t >= 0) & (t < length[a]), t, t - length[a] * torch.floor(t / length[a]))
            t = torch.where(t >= length[a], t - length[a], t)
        i = torch.clamp(torch.floor(t * (mesh[a] / length[a])), 0, mesh[a] - 1)
        idx.append(i.long())
        rel.append(t - (2 * i + 1) * (0.5 * length[a] / mesh[a]))
    return torch.stack(idx, 1), torch.stack(rel, 1)


def _corrections(u, q, cell, ncell, B, V, alpha):
    """The periodic corrections of the potential and gradient: (phi, grad) per particle."""
    per = ncell // B
    sysi = cell // per

    def total(v):
        return torch.zeros(B, dtype=torch.float64, device=u.device).index_add_(0, sysi, v)[sysi]

    Q = total(q)
    Qcell = torch.zeros(ncell, dtype=torch.float64, device=u.device).index_add_(0, cell, q)[cell]
    f = 2.0 * math.pi / (3.0 * V)
    rr = (u * u).sum(1)
    dip = torch.stack([total(q * u[:, a]) for a in range(3)], 1)
    phi = f * total(q * rr) - 2.0 * f * (dip * u).sum(1) + f * Q * (rr - 1.5 / alpha ** 2) \
        - 2.0 * alpha / math.sqrt(math.pi) * Qcell
    return phi, -2.0 * f * dip + 2.0 * f * Q[:, None] * u


def _block_m2l(M, mesh, h, p, c, r, periodic):
    """Two-level fine part: locals [C][K] of the fine cells inside the masked coarse blocks, less the near cells."""
    C, J = (p + 1) ** 2, 2 * p
    nx, ny, nz = mesh
    out = torch.zeros_like(M)
    Mg = M.reshape(C, nz, ny, nx)
    idx = torch.tensor(_m2l_index(p), device=M.device)
    ax = [torch.arange(m, device=M.device) for m in mesh]
    reach = (c + 1) * r - 1
    for dz in range(-reach, reach + 1):
        for dy in range(-reach, reach + 1):
            for dx in range(-reach, reach + 1):
                if max(abs(dx), abs(dy), abs(dz)) <= c:
                    continue
                # target minus source = d; the source's coarse cell is within c of the target's
                ok = [(((a - d).div(r, rounding_mode="floor") - a.div(r, rounding_mode="floor")).abs() <= c)
                      & _wrap(a - d, m, periodic)[0] for a, d, m in zip(ax, (dx, dy, dz), mesh)]
                d = [torch.tensor([v * a], dtype=torch.float64, device=M.device) for v, a in zip((dx, dy, dz), h)]
                A = _columns(J, _singular_columns(J, *d))[:, 0][idx]
                src = torch.roll(Mg, (dz, dy, dx), (1, 2, 3)) * (ok[2][:, None, None] & ok[1][:, None] & ok[0])
                out += A @ src.reshape(C, -1)
    return out


def _pmmm(pos, q, sysid, B, lo, length, mesh, p, c, periodic, refine, sign):
    """(phi, force, energy) in FP64 by the definition of the method, all B systems."""
    K = mesh[0] * mesh[1] * mesh[2]
    h = [length[a] / mesh[a] for a in range(3)]
    idx, u = _bin(pos, lo, length, mesh, periodic)
    cell = sysid * K + idx[:, 0] + mesh[0] * (idx[:, 1] + mesh[1] * idx[:, 2])
    cell, order = torch.sort(cell, stable=True)
    u, qs, idx = u[order], q[order], idx[order]
    phi, grad = _near(u, qs, cell, mesh, h, c, periodic, B)
    V = length[0] * length[1] * length[2]
    alpha = 1.5 / min(length)
    if refine < 2:
        G, L = _green(mesh, h, p, c, periodic, pos.device)
        far = _convolve(_p2m(u, qs, cell, B * K, p), G, L, mesh, p)
        uc, cc, ncc = u, cell, B * K
    else:
        nf = _l2p(u, cell, _block_m2l(_p2m(u, qs, cell, K, p), mesh, h, p, c, refine, periodic), p)
        phi, grad = phi + nf[0], grad + nf[1]
        cmesh, hc = tuple(m // refine for m in mesh), [a * refine for a in h]
        ci = idx.div(refine, rounding_mode="floor")
        uc = u + ((idx - ci * refine).double() + 0.5 - 0.5 * refine) * torch.tensor(h, device=u.device)
        cc, ncc = ci[:, 0] + cmesh[0] * (ci[:, 1] + cmesh[1] * ci[:, 2]), cmesh[0] * cmesh[1] * cmesh[2]
        G, L = _green(cmesh, hc, p, c, periodic, pos.device)
        far = _convolve(_p2m(uc, qs, cc, ncc, p), G, L, cmesh, p)
    f = _l2p(uc, cc, far, p)
    phi, grad = phi + f[0], grad + f[1]
    if periodic:
        f = _corrections(uc, qs, cc, ncc, B, V, alpha)
        phi, grad = phi + f[0], grad + f[1]
    phi, force = sign * phi, -sign * qs[:, None] * grad
    out_phi, out_force = torch.empty_like(phi), torch.empty_like(force)
    out_phi[order], out_force[order] = phi, force
    return out_phi, out_force, float(0.5 * (qs * phi).sum())


def _mlp_exact(X, T, theta, c_high):
    """Loss and parameter gradient of the mean squared error, FP64."""
    t = theta.double().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = torch.split(t, [256 * 432, 256, 256 * 256, 256, 128 * 256, 128])
    gelu = torch.nn.functional.gelu
    y = gelu(X.double() @ W1.reshape(256, 432).t() + b1)
    y = gelu(y @ W2.reshape(256, 256).t() + b2)
    o = y @ W3.reshape(128, 256).t() + b3
    loss = ((o - T.double())[:, :c_high] ** 2).mean()
    loss.backward()
    return loss.detach(), t.grad


def exact(case, seed, device="cuda"):
    if case["form"] == "train":
        loss, grad = _mlp_exact(*_train_inputs(case, seed, device), (case["p_high"] + 1) ** 2)
        return {"loss": loss, "grad": grad}
    if case["form"] == "batched":
        pos, q, counts = _inputs(case, seed, device)
        sysid = torch.repeat_interleave(torch.arange(len(counts), device=device), torch.tensor(counts, device=device))
        phi, force, _ = _pmmm(pos.double(), q.double(), sysid, len(counts), (0.0,) * 3, (1.0,) * 3,
                              (case["mesh"],) * 3, case["p"], 1, True, 0, 1.0)
        return {"phi": phi, "force": force}
    pos, q = _inputs(case, seed, device)
    lo, length = _box(case)
    phi, force, energy = _pmmm(pos.double(), q.double(), torch.zeros_like(q, dtype=torch.long), 1, lo, length,
                               (case["mx"], case["my"], case["mz"]), case["p"], case["cutoff"],
                               case["boundary"] == "periodic", case["refine"], -1.0 if _gravity(case) else 1.0)
    out = {"phi": phi, "force": force}
    if case["form"] == "single" and case["energy"]:
        out["energy"] = energy
    return out
