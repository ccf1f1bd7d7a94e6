"""The work that programs have this library do, as cases that a timer can run.

A case is a dict of plain values; ``kind`` says which entry point it goes through:

  apply    one operator apply y = A u on a structured or explicitly numbered hexahedral mesh;
  solve    one mixed-precision solve (iterative refinement) of one problem to 1e-10;
  batch    one solve of many small problems of uneven size and order together;
  precond  one application of the learned element preconditioner;
  train    one training step of its network (forward, backward, Adam);
  fd       two leapfrog steps of the finite-difference wave example (both buffers change hands);
  dg       one volume right-hand side of the discontinuous-Galerkin shallow-water example.

``prepare`` builds what a program holds before the call, ``run`` is the call, ``exact`` the same
result in plain FP64 torch and numpy.
"""
import math

import numpy as np
import torch

import paper_1403_0968_gb300 as sem

H = 256  # hidden widths of the preconditioner's network
GRAV = 9.81
FLOAT = {"fp32": torch.float32, "fp64": torch.float64}


def listed():
    return [
        # The smallest problem of the test suite, in the default precision: a call whose launches count.
        {"name": "apply_fp64_4cube_n7", "kind": "apply", "N": 7, "sx": 4, "sy": 4, "sz": 4, "prec": "fp64",
         "kappa": False, "alpha": False, "bc": "box", "glo": False},
        # The FP64-accurate apply that the outer residuals and FP64 solves spend their time in, at
        # the order and size of the variable-coefficient solve.
        {"name": "apply_emu_48cube_n7", "kind": "apply", "N": 7, "sx": 48, "sy": 48, "sz": 48, "prec": "fp64_emu",
         "kappa": True, "alpha": False, "bc": "box", "glo": False},
        # The same apply at a higher odd order on a box with uneven sides, with the screened term.
        {"name": "apply_emu_uneven_n9", "kind": "apply", "N": 9, "sx": 23, "sy": 19, "sz": 17, "prec": "fp64_emu",
         "kappa": True, "alpha": True, "bc": "box", "glo": False},
        # The inner apply of a mixed-precision solve, stored FP32 factors.
        {"name": "apply_fp32_48cube_n7", "kind": "apply", "N": 7, "sx": 48, "sy": 48, "sz": 48, "prec": "fp32",
         "kappa": True, "alpha": False, "bc": "box", "glo": False},
        # The inner apply at the lowest order of the sweep, uneven sides, pure Neumann.
        {"name": "apply_fp32_uneven_n3", "kind": "apply", "N": 3, "sx": 67, "sy": 61, "sz": 59, "prec": "fp32",
         "kappa": False, "alpha": False, "bc": "none", "glo": False},
        # The inner apply without stored factors, for problems that would not fit otherwise.
        {"name": "apply_otf_48cube_n7", "kind": "apply", "N": 7, "sx": 48, "sy": 48, "sz": 48, "prec": "fp32_otf",
         "kappa": False, "alpha": False, "bc": "box", "glo": False},
        # A whole solve: variable coefficient, refinement around FP32 iterations, to 1e-10.
        {"name": "solve_ir_16cube_n7", "kind": "solve", "N": 7, "sx": 16, "sy": 16, "sz": 16},
        # A whole batched solve: many small problems at once.
        {"name": "batch_24_problems", "kind": "batch", "nprob": 24, "smin": 4, "smax": 8},
        # The learned preconditioner inside one iteration of flexible CG.
        {"name": "precond_32cube_n7", "kind": "precond", "N": 7, "sx": 32, "sy": 32, "sz": 32},
        # One minibatch of its training.
        {"name": "train_n7_batch256", "kind": "train", "N": 7, "batch": 256},
        # The wave example on the benchmark's grid, the middle of the stencil sizes.
        {"name": "fd_fp32_16384_r4", "kind": "fd", "w": 16384, "h": 16384, "r": 4, "type": "fp32"},
        # The shallow-water volume kernel on a mesh of the published size.
        {"name": "dg_fp32_n7_212800", "kind": "dg", "N": 7, "nx": 280, "ny": 380, "type": "fp32"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: orders, sizes and options that a program may ask for."""
    kind = rng.choices(["apply", "solve", "batch", "precond", "train", "fd", "dg"], [9, 2, 1, 2, 2, 4, 4])[0]
    if kind == "apply":
        N = rng.choice([2, 3, 4, 5, 6, 7, 7, 8, 9, 10, 11, 13, 15])
        prec = rng.choices(["fp64_emu", "fp32", "fp32_otf", "bf16", "fp64"], [4, 4, 2, 1, 1])[0]
        # 1e4 to 3e7 local nodes, at most what the largest listed apply holds
        side = (math.exp(rng.uniform(math.log(1e4), math.log(3e7))) ** (1 / 3)) / (N + 1)
        s = [max(1, min(90, int(round(side * rng.uniform(0.7, 1.4))))) for _ in range(3)]
        glo = rng.random() < 0.1 and s[0] * s[1] * s[2] * (N + 1) ** 3 < 4e6
        return {"kind": kind, "N": N, "sx": s[0], "sy": s[1], "sz": s[2], "prec": prec, "kappa": rng.random() < 0.5,
                "alpha": rng.random() < 0.25, "bc": "box" if rng.random() < 0.8 else "none", "glo": glo}
    if kind == "solve":
        N = rng.choice([3, 4, 5, 6, 7, 8])
        s = _log_int(rng, 3, 90 // (N + 1))
        return {"kind": kind, "N": N, "sx": s, "sy": max(2, s - rng.randrange(3)), "sz": s + rng.randrange(2)}
    if kind == "batch":
        smin = rng.randrange(2, 5)
        return {"kind": kind, "nprob": rng.randrange(3, 22), "smin": smin, "smax": smin + rng.randrange(1, 4)}
    if kind == "precond":
        N = rng.choice([3, 5, 7, 7])
        s = _log_int(rng, 4, 240 // (N + 1))
        return {"kind": kind, "N": N, "sx": s, "sy": max(2, s - rng.randrange(4)), "sz": max(2, s - rng.randrange(4))}
    if kind == "train":
        return {"kind": kind, "N": rng.choice([3, 4, 5, 6, 7]), "batch": _log_int(rng, 33, 512)}
    if kind == "fd":
        real = rng.choices(["fp32", "fp64"], [3, 1])[0]
        top = 14000 if real == "fp32" else 6000
        return {"kind": kind, "w": _log_int(rng, 200, top) // (1 if rng.random() < 0.3 else 4) * 4 or 4,
                "h": _log_int(rng, 200, top), "r": rng.randrange(1, 8), "type": real}
    real = rng.choices(["fp32", "fp64"], [4, 1])[0]
    return {"kind": kind, "N": rng.randrange(1, 9), "nx": _log_int(rng, 20, 300), "ny": _log_int(rng, 20, 300),
            "type": real}


# ---- inputs -------------------------------------------------------------------------------------
def _rng(seed, salt=0):
    return np.random.Generator(np.random.PCG64([seed, salt]))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(shape, g, dtype=torch.float64):
    return (torch.rand(shape, generator=g, device="cuda", dtype=dtype) * 2 - 1).contiguous()


def _box(sx, sy, sz, seed):
    """Vertices [E][8][3] of a box mesh of the unit cube, interior vertices moved by up to 0.1 h."""
    n, h = (sx + 1, sy + 1, sz + 1), np.array([1 / sx, 1 / sy, 1 / sz])
    lat = np.stack(np.meshgrid(*(np.arange(k, dtype=float) for k in n[::-1]), indexing="ij")[::-1], -1) * h
    d = _rng(seed, 1).uniform(-0.1, 0.1, lat.shape) * h
    lat[1:-1, 1:-1, 1:-1] += d[1:-1, 1:-1, 1:-1]
    out = np.empty((sz, sy, sx, 8, 3))
    for v in range(8):
        a, b, c = v & 1, v >> 1 & 1, v >> 2
        out[..., v, :] = lat[c:c + sz, b:b + sy, a:a + sx]
    return out.reshape(-1, 8, 3)


def _modes(seed, amplitude=0.25):
    """Rows (k, phase, amplitude) of a random Fourier field, the coefficient being its exponential."""
    g = _rng(seed, 2)
    k = g.integers(-4, 5, (16, 3))
    k[~k.any(1)] = 1
    return np.concatenate([k, g.uniform(0, 2 * math.pi, (16, 1)), np.full((16, 1), amplitude)], 1).astype(float)


def _numbering(N, sx, sy, sz):
    """Global ids [E][n^3] of the box's nodes."""
    n = N + 1
    e, l = (torch.arange(k, device="cuda") for k in (sx * sy * sz, n ** 3))
    I = (e % sx * N)[:, None] + l % n
    J = (e // sx % sy * N)[:, None] + l // n % n
    K = (e // (sx * sy) * N)[:, None] + l // (n * n)
    return I + (sx * N + 1) * (J + (sy * N + 1) * K)


def _boundary(N, sx, sy, sz):
    g = torch.zeros((sz * N + 1, sy * N + 1, sx * N + 1), dtype=torch.bool, device="cuda")
    for d in range(3):
        g.select(d, 0).fill_(True)
        g.select(d, g.shape[d] - 1).fill_(True)
    return g.reshape(-1)


def _mesh(c, seed):
    """The description of an apply, solve or preconditioner case: keyword arguments of Problem."""
    box = (c["sx"], c["sy"], c["sz"])
    kw = {"vertices": _box(*box, seed), "box": box, "bc": c.get("bc", "box"),
          "kappa_modes": _modes(seed) if c.get("kappa", True) else None}
    if c.get("alpha"):
        kw["alpha"] = _rng(seed, 3).uniform(1, 2, (box[0] * box[1] * box[2], (c["N"] + 1) ** 3))
    return kw


def _nglobal(c):
    return (c["sx"] * c["N"] + 1) * (c["sy"] * c["N"] + 1) * (c["sz"] * c["N"] + 1)


def _vector(c, seed):
    return _uniform(_nglobal(c), _gen(seed))


def _network(N, seed):
    """He-normal weights of the element network (the last layer damped) and small biases."""
    g, n3 = _gen(seed + 7), (N + 1) ** 3
    parts = []
    for a, b, s in ((n3 + 6, H, 1.0), (H, H, 1.0), (H, n3, 0.3)):
        parts += [torch.randn(a * b, generator=g, device="cuda") * (s * math.sqrt(2 / a)),
                  torch.randn(b, generator=g, device="cuda") * 0.01]
    return torch.cat(parts)


def _layers(N, p):
    """The three (weight, bias) pairs of a parameter vector."""
    n3, at, out = (N + 1) ** 3, 0, []
    for a, b in ((n3 + 6, H), (H, H), (H, n3)):
        out.append((p[at:at + a * b].reshape(a, b), p[at + a * b:at + a * b + b]))
        at += a * b + b
    return out


def _train_inputs(c, seed):
    """A minibatch, and weights and Adam moments as in the midst of a training run."""
    N, B, n3, g = c["N"], c["batch"], (c["N"] + 1) ** 3, _gen(seed)
    X = torch.randn(B, n3 + 6, generator=g, device="cuda")
    X[:, :n3] /= X[:, :n3].norm(dim=1, keepdim=True)
    T = torch.randn(B, n3, generator=g, device="cuda") * 0.05
    p = _network(N, seed)
    m = torch.randn(p.shape, generator=g, device="cuda") * 1e-4
    v = (torch.rand(p.shape, generator=g, device="cuda") * 1e-3 + 2e-4) ** 2
    return X, T, p, m, v


def _wave(c, seed):
    g, t = _gen(seed), FLOAT[c["type"]]
    dx, dy = 2 / max(1, c["w"] - 1), 2 / max(1, c["h"] - 1)
    return _uniform((c["h"], c["w"]), g, t), _uniform((c["h"], c["w"]), g, t), 0.25 * min(dx, dy), dx, dy


def _triangles(nx, ny, seed):
    """Vertices [E][3][2] of a perturbed triangulation of the unit square, two per cell."""
    lat = np.stack(np.meshgrid(np.arange(ny + 1.0), np.arange(nx + 1.0), indexing="ij")[::-1], -1) / [nx, ny]
    d = _rng(seed, 4).uniform(-0.1, 0.1, lat.shape) / [nx, ny]
    lat[1:-1, 1:-1] += d[1:-1, 1:-1]
    a, b, u, v = lat[:-1, :-1], lat[:-1, 1:], lat[1:, :-1], lat[1:, 1:]
    return np.stack([np.stack([a, b, v], -2), np.stack([a, v, u], -2)], 2).reshape(-1, 3, 2)


def _water(c, seed):
    g, t, E = _gen(seed), FLOAT[c["type"]], 2 * c["nx"] * c["ny"]
    Np = (c["N"] + 1) * (c["N"] + 2) // 2
    Q = _uniform((E, 3, Np), g, t) * 0.5
    Q[:, 0] += 1.0
    return Q, _uniform((E, 2, Np), g, t)


def _batch_list(c, seed):
    """(order, side, seed of the mesh) of each problem: sizes and orders are the case's, not the seed's."""
    g = _rng(c["nprob"], 100 * c["smin"] + c["smax"])
    return [(int(g.choice([3, 5, 7, 9, 11])), int(g.integers(c["smin"], c["smax"] + 1)), seed + 17 * k)
            for k in range(c["nprob"])]


# ---- the cases ----------------------------------------------------------------------------------
FEATURES = {"fp64": sem.SEM_FEAT_FP64, "fp64_emu": sem.SEM_FEAT_EMU, "fp32": sem.SEM_FEAT_FP32,
            "bf16": sem.SEM_FEAT_FP32 | sem.SEM_FEAT_BF16, "fp32_otf": sem.SEM_FEAT_OTF}


def prepare(case, seed):
    k = case["kind"]
    if k == "apply":
        kw = _mesh(case, seed)
        if case["glo"]:
            kw |= {"glo_num": _numbering(case["N"], *kw["box"]).cpu().numpy(), "nglobal": _nglobal(case)}
        P = sem.Problem(case["N"], features=FEATURES[case["prec"]], **kw)
        u = _vector(case, seed)
        u = u if case["prec"].startswith("fp64") else u.float()
        return {"case": case, "P": P, "u": u, "y": torch.empty_like(u)}
    if k == "solve":
        kw = _mesh(case, seed)
        P = sem.Problem(case["N"], features=sem.SEM_FEAT_EMU | sem.SEM_FEAT_FP32 | sem.SEM_FEAT_PCG, **kw)
        A = _Operator(case["N"], **kw)
        return {"case": case, "P": P, "b": A.apply(A.smooth(seed))}
    if k == "batch":
        probs, b = [], []
        for N, s, sd in _batch_list(case, seed):
            probs.append({"N": N, "box": (s, s, s), "vertices": _box(s, s, s, sd)})
            A = _Operator(**probs[-1])
            b.append(A.apply(A.smooth(sd)))
        return {"case": case, "B": sem.Batch(probs), "b": torch.cat(b)}
    if k == "precond":
        P = sem.Problem(case["N"], features=sem.SEM_FEAT_EMU | sem.SEM_FEAT_PCG | sem.SEM_FEAT_MLP, **_mesh(case, seed))
        P.mlp_load(_network(case["N"], seed))
        return {"case": case, "P": P, "r": _vector(case, seed)}
    if k == "train":
        X, T, p, m, v = _train_inputs(case, seed)
        tr = sem.MlpTrainer(case["N"], p, case["batch"], lr=1e-3)
        tr.m.copy_(m)
        tr.v.copy_(v)
        tr.step_count = 100
        return {"case": case, "tr": tr, "X": X, "T": T, "grad": torch.empty_like(p)}
    if k == "fd":
        u, up, dt, dx, dy = _wave(case, seed)
        return {"case": case, "u": u, "up": up, "steps": (dt, dx, dy)}
    Q, B = _water(case, seed)
    geo = sem.dg_geometry(_triangles(case["nx"], case["ny"], seed), Q.dtype)
    return {"case": case, "Q": Q, "B": B, "geo": geo, "ops": sem.dg_load_operators(case["N"], Q.dtype),
            "rhs": torch.empty_like(Q)}


def run(state):
    c = state["case"]
    k = c["kind"]
    if k == "apply":
        return state["P"].apply(state["u"], state["y"], prec=c["prec"])
    if k == "solve":
        return state["P"].pcg(state["b"], rtol=1e-10, mode="ir", apply_prec="fp64_emu", inner_rtol=1e-3)[0]
    if k == "batch":
        return state["B"].pcg(state["b"], rtol=1e-10, inner_rtol=1e-3)[0]
    if k == "precond":
        return state["P"].mlp_precond(state["r"])
    if k == "train":
        tr = state["tr"]
        loss = tr.step(state["X"], state["T"], grad_out=state["grad"])
        # the loss as a training log keeps it; it is a sum over FP32 activations
        return {"params": tr.params, "m": tr.m, "v": tr.v, "grad": state["grad"], "loss": loss.float()}
    if k == "fd":
        return sem.fd_run(state["u"], state["up"], 2, c["r"], *state["steps"])
    return sem.dg_volume(c["N"], state["Q"], state["B"], state["geo"], GRAV, state["ops"], out=state["rhs"])


def work(case):
    """Each input read once, each output written once, and the arithmetic of the method."""
    k, N = case["kind"], case.get("N", 0)
    n = N + 1
    if k in ("apply", "solve", "precond"):
        E = case["sx"] * case["sy"] * case["sz"]
        G, L = _nglobal(case), E * n ** 3
        flops = E * (12 * n ** 4 + 15 * n ** 3)
        if k == "apply":
            s = 8 if case["prec"].startswith("fp64") else 4
            per_node = {"bf16": 12, "fp32_otf": 4 if case["kappa"] else 0}.get(case["prec"], 6 * s)
            data = L * (per_node + (s if case["alpha"] else 0)) + 2 * s * G
            return {"bytes": data + (96 * E if case["prec"] == "fp32_otf" else 0) + (4 * L if case["glo"] else 0),
                    "flops": flops}
        if k == "solve":  # both factor sets once and the two vectors; about 4 products of A per element row
            return {"bytes": 72 * L + 16 * G, "flops": flops * 4 * N * max(case["sx"], case["sy"], case["sz"])}
        return {"bytes": 24 * G, "flops": 2 * E * ((n ** 3 + 6) * H + H * H + H * n ** 3)}
    if k == "batch":
        data = flops = 0
        for N, s, _ in _batch_list(case, 0):
            n, E = N + 1, s ** 3
            data += 72 * E * n ** 3 + 16 * (s * N + 1) ** 3
            flops += E * (12 * n ** 4 + 15 * n ** 3) * 4 * N * s
        return {"bytes": data, "flops": flops}
    if k == "train":
        n3, B = n ** 3, case["batch"]
        count = (n3 + 6) * H + H + H * H + H + H * n3 + n3
        return {"bytes": 4 * (7 * count + B * (2 * n3 + 6)), "flops": 2 * B * (2 * (n3 + 6) * H + 3 * H * H + 3 * H * n3)}
    if k == "fd":
        nodes = case["w"] * case["h"]
        return {"bytes": 2 * nodes * 3 * (4 if case["type"] == "fp32" else 8), "flops": 2 * nodes * (8 * case["r"] + 3)}
    Np, E = n * (n + 1) // 2, 2 * case["nx"] * case["ny"]
    return {"bytes": (8 * Np + 4) * (4 if case["type"] == "fp32" else 8) * E, "flops": (12 * Np * Np + 36 * Np) * E}


# ---- the same results in plain FP64 -------------------------------------------------------------
def _gll(N):
    """Gauss-Lobatto-Legendre points, weights and the derivative matrix of the Lagrange basis."""
    P = np.polynomial.legendre.Legendre.basis(N)
    d1, d2 = P.deriv(), P.deriv(2)
    x = np.sort(np.concatenate([[-1, 1], d1.roots().real if N > 1 else []]))
    for _ in range(3):
        x[1:-1] -= d1(x[1:-1]) / d2(x[1:-1])
    w = 2 / (N * (N + 1) * P(x) ** 2)
    X = x[:, None] - x + np.eye(N + 1)
    a = X.prod(1)
    D = a[:, None] / a / X
    np.fill_diagonal(D, 0)
    np.fill_diagonal(D, -D.sum(1))
    return x, w, D


class _Operator:
    """The assembled operator M A M of one box problem, element by element in FP64."""

    def __init__(self, N, vertices, box, bc="box", kappa_modes=None, alpha=None):
        t = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
        x, w, D = _gll(N)
        self.N, self.n, self.box, self.E = N, N + 1, box, len(vertices)
        self.x, self.D, self.V = t(x), t(D), t(vertices)
        self.w = t(np.einsum("c,b,a->cba", w, w, w).reshape(-1))
        self.modes, self.alpha = kappa_modes, None if alpha is None else t(alpha)
        self.ids = _numbering(N, *box)
        self.G = int(self.ids.max()) + 1
        self.free = ~_boundary(N, *box) if bc == "box" else torch.ones(self.G, dtype=torch.bool, device="cuda")
        r, s, q = (g.reshape(-1) for g in torch.meshgrid(self.x, self.x, self.x, indexing="ij")[::-1])
        sg = [t([1 if v >> d & 1 else -1 for v in range(8)]) for d in range(3)]
        f = [1 + r[:, None] * sg[0], 1 + s[:, None] * sg[1], 1 + q[:, None] * sg[2]]
        self.shape = f[0] * f[1] * f[2] / 8  # [n^3][8]
        self.grad = [sg[0] * f[1] * f[2] / 8, f[0] * sg[1] * f[2] / 8, f[0] * f[1] * sg[2] / 8]
        self.step = max(1, 4_000_000 // self.n ** 3)  # elements at a time

    def pieces(self):
        return [slice(e, min(e + self.step, self.E)) for e in range(0, self.E, self.step)]

    def coords(self, at):
        return torch.einsum("pv,evd->epd", self.shape, self.V[at])

    def factors(self, at):
        """(rr, rs, rt, ss, st, tt) [6][e][n^3] and w det J."""
        J = [torch.einsum("pv,evd->dep", g, self.V[at]) for g in self.grad]  # d x / d r, d s, d t
        C = [torch.linalg.cross(J[1], J[2], dim=0), torch.linalg.cross(J[2], J[0], dim=0),
             torch.linalg.cross(J[0], J[1], dim=0)]
        det = (J[0] * C[0]).sum(0)
        k = self.w / det
        if self.modes is not None:
            xyz, g = self.coords(at), 0
            for kx, ky, kz, phase, a in self.modes:
                g = g + a * torch.cos(2 * math.pi * (kx * xyz[..., 0] + ky * xyz[..., 1] + kz * xyz[..., 2]) + phase)
            k = k * torch.exp(g)
        return [k * (C[i] * C[j]).sum(0) for i, j in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))], self.w * det

    def apply(self, u):
        y, u, n, D = torch.zeros_like(u), torch.where(self.free, u, 0.0), self.n, self.D
        for at in self.pieces():
            ue = u[self.ids[at]].reshape(-1, n, n, n)  # [e][t][s][r]
            g, wj = self.factors(at)
            g = [f.reshape(-1, n, n, n) for f in g]
            d = [torch.einsum("am,ecbm->ecba", D, ue), torch.einsum("bm,ecma->ecba", D, ue),
                 torch.einsum("cm,emba->ecba", D, ue)]
            q = [g[0] * d[0] + g[1] * d[1] + g[2] * d[2], g[1] * d[0] + g[3] * d[1] + g[4] * d[2],
                 g[2] * d[0] + g[4] * d[1] + g[5] * d[2]]
            ye = (torch.einsum("ma,ecbm->ecba", D, q[0]) + torch.einsum("mb,ecma->ecba", D, q[1])
                  + torch.einsum("mc,emba->ecba", D, q[2]))
            if self.alpha is not None:
                ye = ye + (wj * self.alpha[at]).reshape(ue.shape) * ue
            y.index_add_(0, self.ids[at].reshape(-1), ye.reshape(-1))
        return torch.where(self.free, y, 0.0)

    def smooth(self, seed):
        """A smooth field of the seed's own, zero on the boundary of the cube."""
        g, x = _rng(seed, 5), torch.zeros(self.G, dtype=torch.float64, device="cuda")
        terms = [(g.integers(1, 4, 3), g.uniform(-1, 1)) for _ in range(4)] + [((1, 1, 1), 1.0)]
        for at in self.pieces():
            xyz = self.coords(at)
            x[self.ids[at]] = sum(a * torch.sin(math.pi * xyz * torch.tensor(k, device="cuda")).prod(-1)
                                  for k, a in terms)
        return torch.where(self.free, x, 0.0)


def _exact_precond(c, seed):
    A, r = _Operator(c["N"], **_mesh(c, seed)), _vector(c, seed)
    n, n3, D = A.n, A.n ** 3, A.D
    r = torch.where(A.free, r, 0.0)
    diag, corr, mult = torch.zeros_like(r), torch.zeros_like(r), torch.zeros_like(r)
    (W1, b1), (W2, b2), (W3, b3) = ((W.double(), b.double()) for W, b in _layers(c["N"], _network(c["N"], seed)))
    D2, dd = (D * D).t().contiguous(), torch.diagonal(D)
    for at in A.pieces():
        g, _ = A.factors(at)
        f = [q.reshape(-1, n, n, n) for q in g]
        de = (torch.einsum("am,ecbm->ecba", D2, f[0]) + torch.einsum("bm,ecma->ecba", D2, f[3])
              + torch.einsum("cm,emba->ecba", D2, f[5]))
        de = de + 2 * (f[1] * dd * dd[:, None] + f[2] * dd * dd[:, None, None] + f[4] * dd[:, None] * dd[:, None, None])
        ids, re = A.ids[at], r[A.ids[at]]
        diag.index_add_(0, ids.reshape(-1), de.reshape(-1))
        mean = torch.stack([q.mean(1) for q in g], 1)
        geo = mean / (mean[:, [0, 3, 5]].sum(1, keepdim=True) / 3)
        norm = re.norm(dim=1, keepdim=True)
        X = torch.cat([re / norm, geo], 1)
        out = torch.relu(torch.relu(X @ W1 + b1) @ W2 + b2) @ W3 + b3
        out = out * norm / de.reshape(-1, n3).mean(1, keepdim=True)
        corr.index_add_(0, ids.reshape(-1), out.reshape(-1))
        mult.index_add_(0, ids.reshape(-1), torch.ones_like(out).reshape(-1))
    return torch.where(A.free, r / diag + corr / mult, 0.0)


def _exact_train(c, seed):
    X, T, p, m, v = (a.double() for a in _train_inputs(c, seed))
    p.requires_grad_()
    (W1, b1), (W2, b2), (W3, b3) = _layers(c["N"], p)
    O = torch.relu(torch.relu(X @ W1 + b1) @ W2 + b2) @ W3 + b3
    loss = ((O - T) ** 2).mean()
    (g,) = torch.autograd.grad(loss, p)
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    p = p.detach() - 1e-3 * (m / (1 - 0.9 ** 101)) / (torch.sqrt(v / (1 - 0.999 ** 101)) + 1e-8)
    return {"params": p, "m": m, "v": v, "grad": g, "loss": loss.detach().reshape(1)}


def _exact_wave(c, seed):
    u, up, dt, dx, dy = _wave(c, seed)
    u, up, r = u.double(), up.double(), c["r"]
    f = math.factorial
    w = [0] + [2 * (-1) ** (k + 1) * f(r) ** 2 / (k * k * f(r - k) * f(r + k)) for k in range(1, r + 1)]
    for _ in range(2):
        nxt = 2 * u - up
        for d, h in ((1, dx), (0, dy)):
            for k in range(1, r + 1):
                nxt += dt * dt / (h * h) * w[k] * (torch.roll(u, k, d) + torch.roll(u, -k, d) - 2 * u)
        u, up = nxt, u
    return u, up


def _exact_water(c, seed):
    N, (Q, B) = c["N"], _water(c, seed)
    Q, B = Q.double(), B.double()
    nodes = np.array([(-1 + 2 * a / N, -1 + 2 * b / N) for b in range(N + 1) for a in range(N + 1 - b)])
    leg = np.polynomial.legendre.Legendre.basis

    def basis(r, s):  # P_i(r) P_j(s), i + j <= N, and its two derivatives
        ij = [(i, j) for i in range(N + 1) for j in range(N + 1 - i)]
        return [np.stack([leg(i).deriv(a)(r) * leg(j).deriv(b)(s) for i, j in ij], -1) for a, b in ((0, 0), (1, 0), (0, 1))]

    g, w = np.polynomial.legendre.leggauss(2 * N + 2)
    a, s = (q.reshape(-1) for q in np.meshgrid(g, g, indexing="ij"))
    wt = (w[:, None] * w).reshape(-1) * (1 - s) / 2
    V = basis(*nodes.T)[0]
    L, Lr, Ls = (np.linalg.solve(V.T, q.T) for q in basis((1 + a) * (1 - s) / 2 - 1, s))  # Lagrange functions at the points
    M = (L * wt) @ L.T
    Dr, Ds = (torch.tensor(np.linalg.solve(M, (q * wt) @ L.T), device="cuda") for q in (Lr, Ls))
    v = torch.tensor(_triangles(c["nx"], c["ny"], seed), device="cuda")
    e1, e2 = (v[:, 1] - v[:, 0]) / 2, (v[:, 2] - v[:, 0]) / 2
    J = e1[:, 0] * e2[:, 1] - e2[:, 0] * e1[:, 1]
    rx, ry, sx, sy = (q[:, None, None] for q in (e2[:, 1] / J, -e2[:, 0] / J, -e1[:, 1] / J, e1[:, 0] / J))
    h, hu, hv = Q.unbind(1)
    p = GRAV * h * h / 2
    F, G = torch.stack([hu, hu * hu / h + p, hu * hv / h], 1), torch.stack([hv, hu * hv / h, hv * hv / h + p], 1)
    rhs = (rx * F + ry * G) @ Dr.T + (sx * F + sy * G) @ Ds.T
    rhs[:, 1:] -= GRAV * h[:, None] * B
    return rhs


def exact(case, seed):
    k = case["kind"]
    if k == "apply":
        u = _vector(case, seed)
        u = u if case["prec"].startswith("fp64") else u.float().double()
        return _Operator(case["N"], **_mesh(case, seed)).apply(u)
    if k == "solve":  # the right-hand side is made from this solution
        return _Operator(case["N"], **_mesh(case, seed)).smooth(seed)
    if k == "batch":
        return torch.cat([_Operator(N, _box(s, s, s, sd), (s, s, s)).smooth(sd) for N, s, sd in _batch_list(case, seed)])
    return {"precond": _exact_precond, "train": _exact_train, "fd": _exact_wave, "dg": _exact_water}[k](case, seed)
