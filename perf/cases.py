"""What is timed: the calls of a band-structure program, over the sizes that this package is used at.

A program computes permittivities, sets up a Solver for a structure and solves for the lowest bands at a batch of
Bloch vectors (`solve`, in the default FP64 precision or the mixed one). A program with an eigensolver of its own
calls the steps: the operator (`op`), the preconditioner (`precond`), the block products (`gram`, `update`) and the
small Rayleigh-Ritz problem (`rr`). A program that learns initial blocks runs training steps (`warmstart`).

Cases are dicts of plain values; `listed` gives the fixed ones, `draw` more of the same ranges.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_2503_19379_gb300 as pc

PI = math.pi
FCC_SITES = ((0.0, 0.0, 0.0), (0.0, 0.5, 0.5), (0.5, 0.0, 0.5), (0.5, 0.5, 0.0))
FCC_CELL = 0.5 * np.array([[0.0, 1.0, 1.0], [1.0, 0.0, 1.0], [1.0, 1.0, 0.0]])  # columns: lattice vectors
DTYPES = {"c64": torch.complex64, "c128": torch.complex128, "df": torch.complex128}


# ------------------------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # the headline use: a stretch of a band path of the diamond cell in mixed precision
        {"name": "solve-mixed-n64", "op": "solve", "precision": "mixed", "shape": "diamond", "N": 64, "nk": 8,
         "nbands": 12, "tol": 1e-6},
        # the smallest whole call, in the default precision: one k-point of a coarse simple-cubic cell
        {"name": "solve-fp64-n16", "op": "solve", "precision": "fp64", "shape": "sc", "N": 16, "nk": 1, "nbands": 8,
         "tol": 1e-8},
        # the operator on the search directions of four k-points (complex64: W and P of the mixed solve)
        {"name": "op-c64-n64", "op": "op", "dtype": "c64", "cell": "cube", "N": 64, "nb": 4, "m": 19},
        # the operator in double-float arithmetic on complex128 blocks, an odd number of k-points at N = 32
        {"name": "op-df-n32", "op": "op", "dtype": "df", "cell": "cube", "N": 32, "nb": 15, "m": 16},
        # the operator on the FCC primitive cell (the paper's diamond timing setting), default precision
        {"name": "op-c128-fcc-n64", "op": "op", "dtype": "c128", "cell": "fcc", "N": 64, "nb": 1, "m": 16},
        # the preconditioner on the residual blocks of four k-points
        {"name": "precond-c64-n64", "op": "precond", "dtype": "c64", "cell": "cube", "N": 64, "nb": 4, "m": 19},
        # the smallest step call: the FP64 preconditioner on one block of a coarse grid
        {"name": "precond-c128-n16", "op": "precond", "dtype": "c128", "cell": "cube", "N": 16, "nb": 1, "m": 13},
        # the Rayleigh-Ritz products of [X W P] in FP64, eight k-points at N = 32 (10 bands, 6 guard columns)
        {"name": "gram-c128-n32", "op": "gram", "dtype": "c128", "N": 32, "nb": 8, "p": 48},
        # the rotation of [X W P] to the new block in FP64, at N = 32, and in complex64 at N = 64 (12 bands)
        {"name": "update-c128-n32", "op": "update", "dtype": "c128", "N": 32, "nb": 8, "p": 48, "q": 16},
        {"name": "update-c64-n64", "op": "update", "dtype": "c64", "N": 64, "nb": 4, "p": 57, "q": 19},
        # the small dense problems of 15 k-points (a quarter of the 60-point path, 12 bands)
        {"name": "rr-n57", "op": "rr", "nb": 15, "n": 57, "m": 19},
        # one training step of the learned initial block on a batch of 16 samples
        {"name": "warmstart-n32", "op": "warmstart", "N": 32, "nb": 8, "S": 16, "nstruct": 4},
    ]


def _log(rng, lo, hi):
    """An integer of [lo, hi], spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["solve", "op", "op", "precond", "precond", "gram", "update", "update", "rr", "warmstart"])
    if op == "solve":
        precision = rng.choice(["mixed", "fp64"])
        N = rng.choice([8, 16, 32]) if precision == "mixed" else rng.choice([8, 16])
        nk = _log(rng, 1, 24) if precision == "mixed" else _log(rng, 1, 6)
        return {"op": op, "precision": precision, "shape": rng.choice(["sc", "fcc", "diamond"]), "N": N, "nk": nk,
                "nbands": rng.randint(4, 12), "tol": 1e-6 if precision == "mixed" else 1e-8}
    if op in ("op", "precond"):
        N = rng.choice([8, 16, 32, 64, 128])
        dtype = rng.choice(["c64", "c128", "df"] if op == "op" else ["c64", "c128"])
        fields = _log(rng, 1, max(2, (24 if dtype == "c64" else 12) * 64 ** 3 // N ** 3 * 3 if N >= 64 else 480))
        m = min(fields, rng.randint(1, 21))
        return {"op": op, "dtype": dtype, "cell": rng.choice(["cube", "cube", "fcc"]), "N": N,
                "nb": max(1, fields // m), "m": m}
    if op == "gram":
        N = rng.choice([8, 16, 32, 64])
        return {"op": op, "dtype": "c128", "N": N, "nb": rng.randint(1, 2) if N == 64 else _log(rng, 1, 16),
                "p": rng.randint(8, 64)}
    if op == "update":
        N = rng.choice([8, 16, 32, 64])
        p = rng.randint(8, 64)
        return {"op": op, "dtype": rng.choice(["c64", "c128"]), "N": N,
                "nb": rng.randint(1, 4) if N == 64 else _log(rng, 1, 16), "p": p, "q": rng.randint(4, min(21, p))}
    if op == "rr":
        m = rng.randint(4, 21)
        return {"op": op, "nb": _log(rng, 1, 64), "n": m * rng.choice([2, 3]), "m": m}
    return {"op": op, "N": rng.choice([16, 32, 64]), "nb": rng.randint(2, 12), "S": _log(rng, 1, 16),
            "nstruct": rng.randint(1, 4)}


# ----------------------------------------------------------------------------------------------------------- inputs
def _path(npts):
    """The Bloch vectors of Gamma-X-W-K-Gamma-L in the conventional cube's frame, evenly shared by segment length."""
    G, X, W, K, L = (0, 0, 0), (0, 2 * PI, 0), (PI, 2 * PI, 0), (1.5 * PI, 1.5 * PI, 0), (PI, PI, PI)
    v = np.array([G, X, W, K, G, L], dtype=np.float64)
    length = np.linalg.norm(np.diff(v, axis=0), axis=1)
    each = np.maximum(1, np.round(length / length.sum() * (npts - 1)).astype(int))
    pts = [v[0]]
    for a, b, n in zip(v[:-1], v[1:], each):
        pts += [a + (b - a) * (i + 1) / n for i in range(n)]
    return np.array(pts)


def _kpts(nk, seed):
    """nk points spread over the path of 60, starting at a place that the seed gives."""
    path = _path(60)
    first = np.random.default_rng(seed).integers(0, len(path))
    return path[(first + np.round(np.arange(nk) * (len(path) / max(nk, 1))).astype(int)) % len(path)]


def _kpts_inside(nb, seed):
    """Bloch vectors inside the first zone and away from 0, as the solver hands them to its steps."""
    k = np.random.default_rng(seed).uniform(-PI, PI, (nb, 3))
    return k * np.maximum(1.0, 0.5 / np.linalg.norm(k, axis=1, keepdims=True))


def _gammas(N, k):
    return 2.0 * np.maximum(float(N), 1.0 / np.sum(k * k, axis=1))


def _spheres(shape, g):
    """Centres, radius, permittivity inside and outside: the package's structures with radii that vary by the seed."""
    s = 1.0 + 0.04 * g.uniform(-1, 1)
    if shape == "sc":
        return [(0.5, 0.5, 0.5)], 0.25 * s, 13.0, 1.0
    if shape == "fcc":
        return list(FCC_SITES), 0.25 * s, 13.0, 1.0
    return list(FCC_SITES) + [tuple(x + 0.25 for x in c) for c in FCC_SITES], 0.3 * s, 1.0, 13.0


def _permittivity(shape, N, seed):
    """(3, N, N, N) permittivity at the edge midpoints of the unit cube, component x first, grid (z, y, x)."""
    centres, r, inside, outside = _spheres(shape, np.random.default_rng(seed + 17))
    eps = np.full((3, N, N, N), outside)
    i = np.arange(N) / N
    for c in range(3):
        x, y, z = (i + (0.5 / N if a == c else 0.0) for a in range(3))
        for cx, cy, cz in centres:
            dx, dy, dz = ((p - q) - np.round(p - q) for p, q in ((x, cx), (y, cy), (z, cz)))
            d2 = dz[:, None, None] ** 2 + dy[None, :, None] ** 2 + dx[None, None, :] ** 2
            eps[c][d2 <= r * r] = inside
    return eps


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _fields(shape, N, dtype, gen, noise):
    """Random face fields [..., 3, N, N, N]: smooth (the Bloch modes' spectrum) plus white noise of the given share."""
    x = torch.randn(*shape, 3, N, N, N, dtype=dtype, device="cuda", generator=gen)
    f = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
    s = 1.0 / (1.0 + (f[:, None, None] ** 2 + f[None, :, None] ** 2 + f[None, None, :] ** 2))
    s = (s / s.square().mean().sqrt() + noise).to(x.real.dtype)
    flat = x.view(-1, 3, N, N, N)
    for i in range(0, flat.shape[0], 64):
        flat[i:i + 64] = torch.fft.ifftn(torch.fft.fftn(flat[i:i + 64], dim=(2, 3, 4)) * s, dim=(2, 3, 4))
    return x


def _panel(c, gen):
    """A search panel [X W P] of p columns: smooth columns, those past the first third smaller (W and P)."""
    nb, p, N = c["nb"], c["p"], c["N"]
    S = _fields((nb, p), N, DTYPES[c["dtype"]], gen, 0.05).view(nb, p, 3 * N ** 3)
    S /= math.sqrt(3 * N ** 3)
    scale = torch.ones(nb, p, 1, dtype=torch.float64, device="cuda")
    late = p - (p + 2) // 3
    scale[:, p - late:] = 10.0 ** (-3.0 * torch.rand(nb, late, 1, dtype=torch.float64, device="cuda", generator=gen))
    return S.mul_(scale.to(S.real.dtype))


def _image(S, N):
    """H S for the Hermitian operator that multiplies each Fourier mode by 10 + 4 N^2 sum sin^2 (pi m / N)."""
    f = torch.arange(N, device="cuda", dtype=torch.float64)
    s = 4.0 * N * N * torch.sin(PI * f / N) ** 2
    s = 10.0 + s[:, None, None] + s[None, :, None] + s[None, None, :]
    out = torch.empty_like(S)
    a, b = S.view(-1, 3, N, N, N), out.view(-1, 3, N, N, N)
    for i in range(0, a.shape[0], 64):
        b[i:i + 64] = torch.fft.ifftn(torch.fft.fftn(a[i:i + 64], dim=(2, 3, 4)) * s.to(S.real.dtype), dim=(2, 3, 4))
    return out


def _ws_shapes(nb):
    return {"W1": (8, 3, 3, 3, 3), "b1": (8,), "W2": (16, 8, 3, 3, 3), "b2": (16,), "Fa": (16, 6), "fa": (16,),
            "Fc": (16, 6), "fc": (16,), "Wh": (6 * nb, 16), "bh": (6 * nb,), "Wv": (nb, 22), "bv": (nb,)}


def _ws_inputs(c, seed):
    N, nb, S = c["N"], c["nb"], c["S"]
    g = np.random.default_rng(seed)
    fan = {"W1": 81 / 2, "W2": 216 / 2, "Wh": 16, "Wv": 22}
    params = np.concatenate([(g.standard_normal(math.prod(s)) * (fan[k] ** -0.5 if k in fan else 0.2))
                             for k, s in _ws_shapes(nb).items()]).astype(np.float32)
    shapes = ("sc", "fcc", "diamond")
    m0 = np.stack([1.0 / _permittivity(shapes[i % 3], N, seed + i) for i in range(c["nstruct"])]).astype(np.float32)
    gen = _generator(seed)
    V = _fields((S, nb), N, torch.complex64, gen, 0.0).view(S, nb, -1)
    V = torch.linalg.qr(V.transpose(1, 2))[0].transpose(1, 2).contiguous()
    return {"params": torch.from_numpy(params).cuda(), "m0": torch.from_numpy(m0).cuda(),
            "sidx": torch.from_numpy(g.integers(0, c["nstruct"], S).astype(np.int32)).cuda(),
            "kpts": g.uniform(-PI, PI, (S, 3)), "V": V.view(S, nb, 3, N, N, N),
            "lam": torch.from_numpy(np.sort(g.uniform(2.0, 60.0, (S, nb)), axis=1)).cuda()}


def _inputs(c, seed):
    """The inputs of a case as tensors and arrays, before anything of the package has seen them."""
    op, gen = c["op"], _generator(seed)
    if op == "solve":
        return {"eps": _permittivity(c["shape"], c["N"], seed), "kpts": _kpts(c["nk"], seed)}
    if op in ("op", "precond"):
        k = _kpts_inside(c["nb"], seed)
        # noise 0.2: residuals and early search directions are rough
        return {"eps": _permittivity("diamond", c["N"], seed), "kpts": k, "gammas": _gammas(c["N"], k),
                "X": _fields((c["nb"], c["m"]), c["N"], DTYPES[c["dtype"]], gen, 0.2)}
    if op == "gram":
        S = _panel(c, gen)
        return {"S": S, "AS": _image(S, c["N"])}
    if op == "update":
        C = torch.randn(c["nb"], c["p"], c["q"], dtype=torch.complex128, device="cuda", generator=gen)
        return {"S": _panel(c, gen), "C": C / math.sqrt(c["p"])}
    if op == "rr":
        S = torch.randn(c["nb"], 300, c["n"], dtype=torch.complex128, device="cuda", generator=gen)
        lam = torch.linspace(1.0, 1e3, 300, dtype=torch.float64, device="cuda")
        G, H = S.mH @ S, S.mH @ (lam[None, :, None] * S)
        return {"G": ((G + G.mH) / 2).contiguous(), "H": ((H + H.mH) / 2).contiguous()}
    return _ws_inputs(c, seed)


def _lattice(c):
    return FCC_CELL if c.get("cell") == "fcc" else None


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    if case["op"] == "solve":
        s["solver"] = pc.Solver(case["N"], s["eps"], precision=1 if case["precision"] == "mixed" else 0)
    elif case["op"] in ("op", "precond"):
        s["solver"] = pc.Solver(case["N"], s["eps"], lattice=_lattice(case))
    elif case["op"] == "warmstart":
        s["net"] = pc.WarmStart(case["N"], case["nb"], case["S"], params=s["params"].clone())
    return s


def run(state):
    c = state["case"]
    op = c["op"]
    if op == "solve":
        return {"evals": state["solver"].solve(state["kpts"], c["nbands"], c["tol"])["evals"]}
    if op == "op":
        return state["solver"].apply_op(state["kpts"], state["gammas"], state["X"], double_float=c["dtype"] == "df")
    if op == "precond":
        return state["solver"].apply_precond(state["kpts"], state["gammas"], state["X"])
    if op == "gram":
        return list(pc.gram_pair(state["S"], state["AS"]))
    if op == "update":
        return pc.block_update(state["S"], state["C"])
    if op == "rr":
        theta, coef, rank = pc.rayleigh_ritz(state["G"], state["H"], c["m"])
        return {"theta": theta, "coef": coef, "rank": rank}
    net = state["net"]
    X, y = net.forward(state["m0"], state["sidx"], state["kpts"])
    grad, _ = net.backward(state["m0"], state["sidx"], X, y, state["V"], state["lam"])
    net.adam(grad)
    return {"X": X, "y": y, "grad": grad, "params": net.params}


# ------------------------------------------------------------------------------------------------------------- work
def work(case):
    """Bytes: every input once, every output once. Flops: real operations of the formulas (a complex multiply-add: 8).

    A solve needs at least about 30 block iterations here, whatever the path (LOBPCG takes 50 to 90): each applies the
    operator and the preconditioner to a block of nbands fields, forms its products and rotates it."""
    c = dict(case)
    op, N = c["op"], c.get("N", 0)
    L = 3 * N ** 3
    size = 8 if c.get("dtype") == "c64" else 16
    op_flops, fft_flops = 214.0 * N ** 3, 30.0 * N ** 3 * math.log2(max(N, 2) ** 3) + 60.0 * N ** 3
    if op == "solve":
        b = c["nbands"]
        each = b * (op_flops + fft_flops) + 8.0 * L * (2 * b * (2 * b + 1) + 2 * b * b)
        return {"bytes": 8.0 * L + 8.0 * c["nk"] * (3 + b), "flops": 30.0 * c["nk"] * each}
    if op in ("op", "precond"):
        fields = c["nb"] * c["m"]
        flops = op_flops * (2.5 if c["cell"] == "fcc" else 1.0) if op == "op" else fft_flops
        return {"bytes": 2.0 * fields * L * size + (8.0 * L if op == "op" else 0.0), "flops": flops * fields}
    if op == "gram":
        nb, p = c["nb"], c["p"]
        return {"bytes": 2.0 * nb * p * L * size + 32.0 * nb * p * p, "flops": 8.0 * nb * p * (p + 1) * L}
    if op == "update":
        nb, p, q = c["nb"], c["p"], c["q"]
        return {"bytes": nb * (p + q) * L * size + 16.0 * nb * p * q, "flops": 8.0 * nb * p * q * L}
    if op == "rr":
        nb, n, m = c["nb"], c["n"], c["m"]
        # Cholesky, two substitutions and the tridiagonalisation (complex), back-transformation of m vectors
        flops = 4.0 * (n ** 3 / 3 + 2 * n ** 3 + 4 * n ** 3 / 3 + 4 * n * n * m)
        return {"bytes": nb * (32.0 * n * n + 16.0 * n * m), "flops": nb * flops}
    nb, S, h, q = c["nb"], c["S"], (N // 2) ** 3, (N // 4) ** 3
    conv = 2.0 * (81 * 8 * h + 216 * 16 * q + 16 * 6 * nb * q)
    return {"bytes": 4.0 * c["nstruct"] * L + 2 * 8.0 * S * nb * L,
            "flops": S * (3.0 * conv + 4 * 8.0 * nb * nb * L + 3 * 2.0 * 14 * nb * L)}


# ------------------------------------------------------------------------------------------------------------ exact
def _shift(f, axis, off):
    """f at the neighbour `off` points up axis 0 (x), 1 (y) or 2 (z); the last three dimensions are (z, y, x)."""
    return torch.roll(f, -off, dims=-1 - axis)


def _difference(f, a, k, N, adjoint, b):
    """D_a f or its adjoint: sum_j b[j, a] N (difference along j) plus or minus i k_a times the average along a."""
    off = -1 if adjoint else 1
    out = (-0.5j if adjoint else 0.5j) * float(k[a]) * (f + _shift(f, a, off))
    for j in range(3):
        if b[j, a] != 0.0:
            out = out + float(b[j, a]) * N * (_shift(f, j, off) - f)
    return out


def _operator(v, k, gamma, m0, b):
    """A M0 A' v + gamma B'B v for fields v [m, 3, N, N, N] in 64 bits."""
    N = v.shape[-1]

    def fw(f, a):
        return _difference(f, a, k, N, False, b)

    def ad(f, a):
        return _difference(f, a, k, N, True, b)

    v1, v2, v3 = v.unbind(1)
    e = (m0[0] * (ad(v2, 2) - ad(v3, 1)), m0[1] * (ad(v3, 0) - ad(v1, 2)), m0[2] * (ad(v1, 1) - ad(v2, 0)))
    c = fw(v1, 0) + fw(v2, 1) + fw(v3, 2)
    return torch.stack([fw(e[2], 1) - fw(e[1], 2) + gamma * ad(c, 0), fw(e[0], 2) - fw(e[2], 0) + gamma * ad(c, 1),
                        fw(e[1], 0) - fw(e[0], 1) + gamma * ad(c, 2)], dim=1)


def _preconditioner(r, k, gamma, b):
    """The inverse of the operator at M0 = 1, mode by mode."""
    N = r.shape[-1]
    th = 2.0 * PI * torch.arange(N, device=r.device, dtype=torch.float64) / N
    half = 1j * torch.exp(0.5j * th)
    diff, avg = half * 2.0 * N * torch.sin(th / 2), half * torch.cos(th / 2)
    d = []
    for a in range(3):
        t = torch.zeros(N, N, N, dtype=torch.complex128, device=r.device)
        for j in range(3):
            part = float(b[j, a]) * diff + (float(k[a]) * avg if j == a else 0.0)
            t = t + part.view([N if 2 - j == i else 1 for i in range(3)])
        d.append(t)
    s = sum(x.abs() ** 2 for x in d)
    f = torch.fft.fftn(r, dim=(2, 3, 4))
    along = sum(d[i] * f[:, i] for i in range(3)) * ((gamma - 1.0) / gamma) / s
    return torch.fft.ifftn(torch.stack([(f[:, i] - d[i].conj() * along) / s for i in range(3)], dim=1), dim=(2, 3, 4))


def _mirrored(A):
    up = torch.triu(A)
    return up + torch.triu(A, 1).mH - 1j * torch.diag_embed(torch.diagonal(A, dim1=1, dim2=2).imag)


def _exact_solve(c, s):
    if c["N"] > 8:
        return None  # 12288 unknowns and more
    N, n = c["N"], 3 * c["N"] ** 3
    m0 = torch.from_numpy(1.0 / s["eps"]).cuda()
    eye = torch.eye(n, dtype=torch.complex128, device="cuda").view(n, 3, N, N, N)
    out = []
    for k in s["kpts"]:
        k = k - 2 * PI * np.round(k / (2 * PI))
        k2 = float(k @ k)
        gamma = 2.0 * (float(N) if k2 == 0.0 else max(float(N), 1.0 / k2))
        A = _operator(eye, k, gamma, m0, np.eye(3)).view(n, n).T
        w = torch.linalg.eigvalsh(((A + A.mH) / 2).cpu())
        skip = 3 if k2 == 0.0 else 0  # the constant fields
        out.append(w[skip:skip + c["nbands"]])
    return {"evals": torch.stack(out)}


def _exact_warmstart(c, s):
    N, nb, S = c["N"], c["nb"], c["S"]
    p, at = {}, 0
    flat = s["params"].double().requires_grad_(True)
    for name, shape in _ws_shapes(nb).items():
        n = math.prod(shape)
        p[name] = flat[at:at + n].view(shape)
        at += n

    def conv(u, W, b):
        # taps at 2 q + d - 1, periodic
        n, out = u.shape[-1], b[:, None, None, None]
        for d in itertools.product(range(3), repeat=3):
            w = torch.roll(u, [1 - x for x in d], dims=(-3, -2, -1))[..., ::2, ::2, ::2]
            out = out + torch.einsum("oc,czyx->ozyx", W[(slice(None), slice(None)) + d], w)
        return out

    U = torch.zeros(N, N // 4, dtype=torch.float64, device="cuda")
    for i in range(N):
        j, r = divmod(i, 4)
        U[i, j] += 1.0 - r / 4.0
        U[i, (j + 1) % (N // 4)] += r / 4.0
    Xs, ys, loss = [], [], 0.0
    for i in range(S):
        k = torch.from_numpy(s["kpts"][i]).cuda()
        phi = torch.cat([torch.sin(k), torch.cos(k)])
        u = torch.relu(conv(s["m0"][int(s["sidx"][i])].double(), p["W1"], p["b1"]))
        u = torch.relu(conv(u, p["W2"], p["b2"]))
        z = (1.0 + p["Fa"] @ phi + p["fa"])[:, None, None, None] * u + (p["Fc"] @ phi + p["fc"])[:, None, None, None]
        h = torch.einsum("oc,czyx->ozyx", p["Wh"], z) + p["bh"][:, None, None, None]
        h = torch.einsum("Zz,Yy,Xx,ozyx->oZYX", U, U, U, h).reshape(nb, 3, 2, N, N, N)
        X = torch.complex(h[:, :, 0], h[:, :, 1])
        y = p["Wv"] @ torch.cat([z.mean(dim=(1, 2, 3)), phi]) + p["bv"]
        x, v = X.reshape(nb, -1), s["V"][i].to(torch.complex128).reshape(nb, -1)
        B = x.conj() @ v.T
        loss = loss + nb - torch.trace(torch.linalg.solve(x.conj() @ x.T, B @ B.mH)).real
        loss = loss + 0.1 * torch.sum((y - torch.log(s["lam"][i])) ** 2)
        Xs.append(X.detach())
        ys.append(y.detach())
    grad, = torch.autograd.grad(loss / S, flat)
    step = flat.detach() - 1e-3 * grad / (grad.abs() + 1e-8)  # the first Adam step
    return {"X": torch.stack(Xs), "y": torch.stack(ys), "grad": grad, "params": step}


def exact(case, seed):
    c, s = case, _inputs(case, seed)
    op = c["op"]
    if op == "solve":
        return _exact_solve(c, s)
    if op in ("op", "precond"):
        b = np.eye(3) if _lattice(c) is None else np.linalg.inv(_lattice(c))
        m0 = torch.from_numpy(1.0 / s["eps"]).cuda()
        out = torch.empty(s["X"].shape, dtype=torch.complex128, device="cuda")
        for i in range(c["nb"]):
            for j in range(0, c["m"], 4):
                x = s["X"][i, j:j + 4].to(torch.complex128)
                k, g = s["kpts"][i], float(s["gammas"][i])
                out[i, j:j + 4] = _operator(x, k, g, m0, b) if op == "op" else _preconditioner(x, k, g, b)
        return out
    if op == "gram":
        S, AS = s["S"].to(torch.complex128), s["AS"].to(torch.complex128)
        return [_mirrored(S.conj() @ S.transpose(1, 2)), _mirrored(S.conj() @ AS.transpose(1, 2))]
    if op == "update":
        return s["C"].transpose(1, 2) @ s["S"].to(torch.complex128)
    if op == "rr":
        Linv = torch.linalg.inv(torch.linalg.cholesky(s["G"]))
        return {"theta": torch.linalg.eigvalsh(Linv @ s["H"] @ Linv.mH)[:, :c["m"]].contiguous(), "coef": None,
                "rank": None}  # eigenvectors are given up to a phase
    return _exact_warmstart(c, s)
