"""Performance cases of the TT-S_N library: the work its users have it do, through its public entry points.

Kinds (``case["kind"]``):

* ``gemm``, ``gram``: the FP64 (or precision-form) contractions as library calls (``dgemm``, ``gram``,
  ``gemm_nt_mixed``, ``gram_mixed``).
* ``round``: ``TensorTrain.round`` of a TT whose ranks a sum has doubled, by any of the three roundings.
* ``step``: ``TTSN.step`` from a held state: the state is put back (``set_cores``, ``set_T``), stepped, and the
  energies are read, as a run resumed from a checkpoint does.
* ``batch``: ``TTSNBatch`` steps of uneven problems, as host-driven or captured steps.
* ``adjoint``: ``escape_energy`` forward and backward.

States are built from the seed alone (no step of the library runs in ``prepare``): an isotropic field in
equilibrium with a hot region plus smooth angular and spatial modes with geometrically decaying weights, which is
the spectrum that a rounded solution has.
"""
import math

import numpy as np
import torch

import paper_2503_18056_gb300 as ttsn

FOUR_PI = 4.0 * math.pi


def listed():
    return [
        # small ragged product: launch and host latency of one call
        dict(name="gemm-small", kind="gemm", mixed=False, m=133, n=97, k=389, ta=False, tb=True),
        # core update A' = A P_A of a tall grown core
        dict(name="gemm-update", kind="gemm", mixed=False, m=200000, n=96, k=577, ta=False, tb=True),
        # left Gram of a tall grown core, the dominant contraction of the method
        dict(name="gram-tall", kind="gram", mixed=False, m=500000, n=449),
        # a bare tensor train rounded to tolerance (no physics)
        dict(name="round-gram-4d", kind="round", method="gram", n0=64, n1=48, n2=32, n3=48, r=20, eps=1e-5),
        # the 2D pulse problem: two steps on a small grid, bound by launches and small factorisations
        dict(name="step-pulse-32", kind="step", nx=32, ny=32, nz=0, nt=8, np=16, r1=12, r2=8, eps=3e-5, cap=128,
             steps=2, bc="periodic", sigma="uniform", scatter=False, flux="upwind", mixed=False, split=False,
             sources=0),
        # scattering-dominated diffusion: small ranks, a general (non-upwind) flux
        dict(name="step-diffusion-128", kind="step", nx=128, ny=128, nz=0, nt=8, np=16, r1=6, r2=5, eps=3e-5, cap=0,
             steps=4, bc="vacuum", sigma="thick", scatter=True, flux="rusanov", mixed=False, split=False, sources=0),
        # precision form on the crossing-beam grid, with fixed sources
        dict(name="step-beams-mixed", kind="step", nx=256, ny=256, nz=0, nt=64, np=128, r1=32, r2=20, eps=1e-4,
             cap=96, steps=1, bc="vacuum", sigma="thin", scatter=False, flux="upwind", mixed=True, split=False,
             sources=2),
        # line-source grid at the ranks its run reaches: wide Gram, large eigensolve
        dict(name="step-line-500", kind="step", nx=500, ny=500, nz=0, nt=32, np=64, r1=175, r2=41, eps=1e-4, cap=0,
             steps=1, bc="vacuum", sigma="thin", scatter=False, flux="upwind", mixed=False, split=False, sources=0),
        # the 3D two-region problem, FP64, ranks growing to the cap
        dict(name="step-blob-128", kind="step", nx=128, ny=128, nz=128, nt=32, np=64, r1=64, r2=24, eps=1e-5,
             cap=128, steps=1, bc="vacuum", sigma="blobs", scatter=False, flux="upwind", mixed=False, split=False,
             sources=0),
        # one core per spatial axis
        dict(name="step-split-64", kind="step", nx=64, ny=64, nz=64, nt=16, np=32, r1=14, r2=8, eps=3e-5, cap=96,
             steps=1, bc="vacuum", sigma="uniform", scatter=False, flux="upwind", mixed=False, split=True, sources=0),
        # uneven problems stepped together as one captured graph
        dict(name="batch-graph-16", kind="batch", count=16, steps=4, graph=True),
        # gradient of the escape energy with respect to the opacity field
        dict(name="adjoint-128", kind="adjoint", nx=128, ny=128, nt=16, np=32, eps=1e-5, steps=6, every=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gemm", "gram", "round", "step", "step", "step", "step", "batch", "adjoint"])
    if kind == "gemm":
        mixed = rng.random() < 0.25
        return dict(kind="gemm", mixed=mixed, m=_log(rng, 100, 200000), n=_log(rng, 60, 400), k=_log(rng, 60, 600),
                    ta=False if mixed else rng.random() < 0.5, tb=True if mixed else rng.random() < 0.5)
    if kind == "gram":
        n = _log(rng, 40, 640)
        return dict(kind="gram", mixed=rng.random() < 0.25, m=_log(rng, 1000, min(500000, int(1e11 / n ** 2))), n=n)
    if kind == "round":
        return dict(kind="round", method=rng.choice(["gram", "gram", "ttsvd", "randomized"]), n0=_log(rng, 24, 64),
                    n1=_log(rng, 24, 64), n2=_log(rng, 16, 32), n3=_log(rng, 16, 48), r=_log(rng, 6, 24),
                    eps=10.0 ** rng.uniform(-5, -3))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 16), steps=rng.randint(2, 4), graph=rng.random() < 0.5)
    if kind == "adjoint":
        return dict(kind="adjoint", nx=_log(rng, 40, 128), ny=_log(rng, 40, 128), nt=16, np=32,
                    eps=10.0 ** rng.uniform(-5, -4), steps=rng.randint(3, 6), every=rng.randint(1, 3))
    three = rng.random() < 0.4
    split = rng.random() < 0.15
    if split:
        n = (_log(rng, 24, 64), _log(rng, 24, 64), _log(rng, 24, 64) if three else 0)
        r1, r2 = rng.randint(4, 14), rng.randint(3, 8)
    elif three:
        n = (_log(rng, 24, 128), _log(rng, 24, 128), _log(rng, 24, 128))
        r1, r2 = _log(rng, 6, 64), rng.randint(4, 20)
    else:
        n = (_log(rng, 32, 500), _log(rng, 32, 500), 0)
        r1, r2 = _log(rng, 6, 120), rng.randint(4, 24)
    nt, npp = rng.choice([(8, 16), (16, 32), (32, 64)])
    r2 = min(r2, npp // 2)
    r1 = min(r1, nt * r2 // 2)
    flux = "upwind" if split else rng.choice(["upwind", "upwind", "rusanov", "hll"])
    return dict(kind="step", nx=n[0], ny=n[1], nz=n[2], nt=nt, np=npp, r1=r1, r2=r2, eps=10.0 ** rng.uniform(-4.5, -3),
                cap=rng.choice([64, 96, 128]), steps=rng.randint(1, 2), bc=rng.choice(["vacuum", "periodic"]),
                sigma="uniform" if split else rng.choice(["uniform", "thin", "blobs", "smooth"]), scatter=False,
                flux=flux, mixed=(not split) and rng.random() < 0.3, split=split,
                sources=0 if split or flux != "upwind" else rng.choice([0, 0, 2]))


# ------------------------------------------------------------------ inputs


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _grid(c):
    return tuple(m for m in (c["nx"], c["ny"], c.get("nz", 0)) if m)


def _centres(m):
    return (torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) / m


def _outer(vs):
    """Separable fields: vs[a] is (n_a, k); the (N_c, k) products in C order."""
    out = vs[0]
    for v in vs[1:]:
        out = (out[:, None, :] * v[None, :, :]).reshape(-1, v.shape[1])
    return out


def _pulse(n, g):
    """T = 0.5 + a Gaussian hot region, on the grid; also its per-axis factors."""
    centre = 0.3 + 0.4 * _rand(g, len(n))
    width = 0.08 + 0.07 * _rand(g, 1)
    f = [torch.exp(-(_centres(m) - centre[a]) ** 2 / (2 * width ** 2))[:, None] for a, m in enumerate(n)]
    return 0.5 + 0.5 * _outer(f)[:, 0]


def _opacity(kind, n, g):
    nc = int(np.prod(n))
    if kind in ("uniform", "thin", "thick"):
        v = {"uniform": 1.0, "thin": 1e-3, "thick": 1e3}[kind]
        return torch.full((nc,), v * (0.75 + 0.5 * float(_rand(g, 1))), device="cuda", dtype=torch.float64)
    if kind == "smooth":  # exp of a smooth random field
        h = torch.zeros(nc, device="cuda", dtype=torch.float64)
        for _ in range(12):
            f = torch.randint(1, 6, (len(n),), generator=g, device="cuda")
            ph = 2 * math.pi * _rand(g, len(n))
            h += _randn(g, 1) * _outer([torch.cos(2 * math.pi * f[a] * _centres(m) + ph[a])[:, None]
                                        for a, m in enumerate(n)])[:, 0]
        return torch.exp(h / 3.0)
    mask = torch.zeros(nc, device="cuda", dtype=torch.bool)  # union of spheres, thick in thin
    for _ in range(16):
        ctr, rad = _rand(g, len(n)), 0.05 + 0.1 * _rand(g, 1)
        d2 = torch.zeros((), device="cuda", dtype=torch.float64)
        for a, m in enumerate(n):
            d2 = (d2[..., None] + (_centres(m) - ctr[a]) ** 2)
        mask |= d2.reshape(-1) <= rad ** 2
    return 1e-2 + (1e2 - 1e-2) * mask.double()


def _modes(n, r, g, top=12):
    """Per-axis factors of r smooth separable modes: a list of (n_a, r)."""
    out = []
    for m in n:
        f = torch.randint(0, top + 1, (r,), generator=g, device="cuda")
        ph = 2 * math.pi * _rand(g, r)
        out.append(torch.cos(2 * math.pi * _centres(m)[:, None] * f[None, :] + ph[None, :]))
    return out


def _angular(c, first, g):
    """theta core (r1 x nt x r2) and phi core (r2 x np); row `a` carries weight 10^(-p a / r1); the first `first`
    rows are isotropic, the others have no angular mean (they carry no energy density)."""
    nt, npp, r1, r2 = c["nt"], c["np"], c["r1"], c["r2"]
    phi = (torch.arange(npp, device="cuda", dtype=torch.float64) + 0.5) * (2 * math.pi / npp)
    rows = [torch.ones_like(phi)]
    for k in range(1, r2):
        rows.append(math.sqrt(2.0) * (torch.cos if k % 2 else torch.sin)((k + 1) // 2 * phi))
    modes = min(nt, 16)
    l = (torch.arange(nt, device="cuda", dtype=torch.float64) + 0.5) / nt
    basis = torch.cos(math.pi * torch.arange(modes, device="cuda", dtype=torch.float64)[:, None] * l[None, :])
    coef = _randn(g, r1, modes, r2) / math.sqrt(modes)
    coef[:, 0, 0] = 0.0
    p = -math.log10(c["eps"])
    wa = 10.0 ** (-p * torch.arange(r1, device="cuda", dtype=torch.float64) / r1)
    wb = 10.0 ** (-0.5 * p * torch.arange(r2, device="cuda", dtype=torch.float64) / r2)
    th = 1.5e-3 * torch.einsum("a,amb,ml,b->alb", wa, coef, basis, wb)
    th[:first] = 0.0
    th[:first, :, 0] = 1.0
    return th.contiguous(), torch.stack(rows)[:, :, None].contiguous()


def _problem(c, seed):
    """Fields, sources and cores of a step case."""
    g = _gen(seed)
    n = _grid(c)
    nc = int(np.prod(n))
    T = _pulse(n, g)
    sig = _opacity(c["sigma"], n, g)
    p = dict(n=n, L=(1.0,) * len(n), n_theta=c["nt"], n_phi=c["np"], cv=torch.ones_like(T), T0=T, Tr0=T,
             sigma_a=torch.zeros_like(sig) if c["scatter"] else sig, sigma_s=sig if c["scatter"] else None,
             bc=ttsn.TT_BC_VACUUM if c["bc"] == "vacuum" else ttsn.TT_BC_PERIODIC, eps=c["eps"],
             max_rank=c["cap"], cfl=0.5, precision=ttsn.TT_MIXED if c["mixed"] else ttsn.TT_FP64,
             layout=ttsn.TT_LAYOUT_SPLIT if c["split"] else ttsn.TT_LAYOUT_GROUPED, flux=c["flux"],
             rusanov_s=0.0 if c["scatter"] else 1.0)
    r1 = c["r1"]
    if c["split"]:
        # I = const + a separable hot region + modes: the spatial cores after the first are diagonal
        ctr, f = 0.3 + 0.4 * _rand(g, len(n)), _modes(n, r1, g)
        for a, m in enumerate(n):
            f[a][:, 0] = 1.0
            f[a][:, 1] = torch.exp(-(_centres(m) - ctr[a]) ** 2 / 0.02)
        f[0][:, 0] *= 0.0625 / FOUR_PI
        f[0][:, 1] *= 0.5 / FOUR_PI
        cores = [f[0][None]] + [torch.diag_embed(v).permute(1, 0, 2) for v in f[1:]]
        th, ph = _angular(c, 2, g)
    else:
        X = _outer(_modes(n, r1, g))
        X[:, 0] = T ** 4 / FOUR_PI
        cores = [X[None]]
        th, ph = _angular(c, 1, g)
    cores = [x.contiguous() for x in cores] + [th, ph]
    sources = []
    for k in range(c["sources"]):  # a patch on an edge emitting into a cone
        x = torch.zeros(n, device="cuda", dtype=torch.float64)
        at = int(_rand(g, 1).item() * (n[1] - 8))
        x[0:4, at:at + 8] = 0.5 + 0.5 * float(_rand(g, 1))
        wt, wp = (_rand(g, c["nt"]) < 0.2).double(), (_rand(g, c["np"]) < 0.1).double()
        sources.append((x.reshape(nc).cpu(), wt, wp))
    return p, cores, T, sources


def _matrix(g, rows, cols, grade, axis):
    """Normal entries, graded over `grade` decades along an axis: a grown core's columns carry decaying weights."""
    A = _randn(g, rows, cols)
    m = A.shape[axis]
    w = 10.0 ** (-grade * torch.arange(m, device="cuda", dtype=torch.float64) / m)
    w = w[torch.randperm(m, generator=g, device="cuda")]
    return A.mul_(w[:, None] if axis == 0 else w[None, :])


def _gemm_inputs(c, seed):
    g = _gen(seed)
    A = _matrix(g, c["k"], c["m"], 2.0, 0) if c["ta"] else _matrix(g, c["m"], c["k"], 2.0, 1)
    B = _randn(g, c["n"], c["k"]) if c["tb"] else _randn(g, c["k"], c["n"])
    return A, B


def _round_cores(c, seed):
    """X + 1e-2 Y, the sum of two smooth TTs of ranks r: block cores of ranks 2 r with a decaying spectrum."""
    g = _gen(seed)
    n, r = (c["n0"], c["n1"], c["n2"], c["n3"]), c["r"]
    w = 10.0 ** (-1.5 * torch.arange(r, device="cuda", dtype=torch.float64) / r)
    cores = []
    for k in range(4):
        a, b = (1 if k == 0 else r), (1 if k == 3 else r)
        pair = [_randn(g, a, n[k], b) * (w[None, None, :] if b > 1 else 1.0) / math.sqrt(a) for _ in range(2)]
        if k == 0:
            cores.append(torch.cat([pair[0], 1e-2 * pair[1]], 2))
        elif k == 3:
            cores.append(torch.cat(pair, 0))
        else:
            z = torch.zeros_like(pair[0])
            cores.append(torch.cat([torch.cat([pair[0], z], 2), torch.cat([z, pair[1]], 2)], 0))
    return [x.contiguous() for x in cores]


def _batch_problems(c, seed):
    rng = np.random.default_rng(seed)
    out = []
    for i in range(c["count"]):  # the sizes are the case's, the fields the seed's
        size = np.random.default_rng(1000 * c["count"] + i)
        m = int(size.choice([48, 64, 96, 128]))
        nt, npp = [(8, 16), (16, 32)][int(size.integers(0, 2))]
        eps, cap = float(size.choice([1e-4, 1e-5])), int(size.integers(8, 49))
        x = (np.arange(m) + 0.5) / m
        cx, cy, w = rng.uniform(0.3, 0.7), rng.uniform(0.3, 0.7), rng.uniform(0.05, 0.15)
        T0 = 0.3 + rng.uniform(0.4, 0.7) * np.exp(-((x[:, None] - cx) ** 2 + (x[None, :] - cy) ** 2) / (2 * w * w))
        out.append(dict(n=(m, m), L=(1.0, 1.0), n_theta=nt, n_phi=npp, bc=[0, 0], eps=eps, max_rank=cap, cfl=0.5,
                        c=1.0, a_r=1.0, dt=0.5 / m, T0=T0, Tr0=T0.copy(), sigma_s=np.zeros((m, m)),
                        sigma_a=np.full((m, m), 10.0 ** rng.uniform(-2, 2)), cv=np.ones((m, m))))
    return out


def prepare(case, seed):
    c = case
    st = dict(case=c)
    if c["kind"] == "gemm":
        st["A"], st["B"] = _gemm_inputs(c, seed)
    elif c["kind"] == "gram":
        st["A"] = _matrix(_gen(seed), c["m"], c["n"], 4.0, 1)
    elif c["kind"] == "round":
        st["cores"] = _round_cores(c, seed)
        st["tt"] = ttsn.TensorTrain(st["cores"])
        if c["method"] == "randomized":
            g = _gen(seed + 7)
            n, r = (c["n0"], c["n1"], c["n2"], c["n3"]), [1] + [c["r"]] * 3 + [1]
            st["tt"].set_sketch([_randn(g, r[k], n[k], r[k + 1]) for k in range(4)])
        st["tt"].set_rounding(c["method"])
    elif c["kind"] == "step":
        p, st["cores"], st["T"], sources = _problem(c, seed)
        st["tt"] = ttsn.TTSN(**p)
        if sources:
            st["tt"].set_sources(sources)
    elif c["kind"] == "batch":
        problems = _batch_problems(c, seed)
        st["batch"] = ttsn.TTSNBatch(problems, threads=8)
        st["handles"] = [st["batch"].problem(i) for i in range(c["count"])]
        st["start"] = [h.state_dict() for h in st["handles"]]
        if c["graph"]:
            st["batch"].set_graph(True)
    elif c["kind"] == "adjoint":
        g = _gen(seed)
        n = _grid(c)
        T = _pulse(n, g)
        st["sigma"] = _opacity("smooth", n, g)
        st["problem"] = dict(n=n, L=(1.0, 1.0), n_theta=c["nt"], n_phi=c["np"], cv=torch.ones_like(T), T0=T, Tr0=T,
                             bc=ttsn.TT_BC_VACUUM, eps=c["eps"], cfl=0.5)
    else:
        raise ValueError(c["kind"])
    return st


# ------------------------------------------------------------------ one pass


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "gemm":
        if c["mixed"]:
            return ttsn.gemm_nt_mixed(state["A"], state["B"])
        return ttsn.dgemm(state["A"], state["B"], trans_a=c["ta"], trans_b=c["tb"])
    if kind == "gram":
        return (ttsn.gram_mixed if c["mixed"] else ttsn.gram)(state["A"])
    if kind == "round":
        tt = state["tt"]
        tt.set_cores(state["cores"])
        if c["method"] == "randomized":
            info = tt.round(forced=[c["r"]] * 3)
        else:
            info = tt.round(eps=c["eps"])
        return {"full": tt.full(), "ranks": list(info["ranks"])}
    if kind == "step":
        tt = state["tt"]
        tt.set_cores(state["cores"])
        tt.set_T(state["T"])
        info = tt.step(c["steps"])
        E, T, totals = tt.energy()
        out = {"E": E, "T": T, "totals": np.array(totals), "ranks": list(info["ranks"])}
        if E.numel() * c["nt"] * c["np"] <= 1 << 18:
            out["full"] = tt.full()
        return out
    if kind == "batch":
        for h, s in zip(state["handles"], state["start"]):
            h.load_state_dict(s)
        infos = state["batch"].step(c["steps"])
        E, T = [], []
        for h in state["handles"]:
            e, t, _ = h.energy(totals=False)
            E.append(e)
            T.append(t)
        return {"E": torch.cat(E), "T": torch.cat(T), "ranks": [r for i in infos for r in i["ranks"][1:-1]][:32]}
    sigma = state["sigma"].clone().requires_grad_(True)
    q = ttsn.escape_energy(sigma, state["problem"], c["steps"], c["every"])
    q.backward()
    return {"Q": q.detach(), "grad": sigma.grad}


# ------------------------------------------------------------------ what a pass cannot do without


def work(case):
    c = case
    kind = c["kind"]
    if kind == "gemm":
        m, n, k = c["m"], c["n"], c["k"]
        return {"bytes": 8.0 * (m * k + n * k + m * n), "flops": 2.0 * m * n * k}
    if kind == "gram":
        m, n = c["m"], c["n"]
        return {"bytes": 8.0 * (m * n + n * n), "flops": 1.0 * m * n * (n + 1)}
    if kind == "round":
        n, R = (c["n0"], c["n1"], c["n2"], c["n3"]), [1] + [2 * c["r"]] * 3 + [1]
        size = sum(R[k] * n[k] * R[k + 1] for k in range(4))
        flops = sum(3.0 * R[k] * n[k] * R[k + 1] ** 2 + 2.0 * R[k] ** 2 * n[k] * R[k + 1] for k in range(4))
        return {"bytes": 8.0 * (size + np.prod(n)), "flops": flops}
    if kind == "batch":
        return {"bytes": c["count"] * c["steps"] * 8.0 * 96 * 96 * 40, "flops": c["count"] * c["steps"] * 2e8}
    if kind == "adjoint":
        nc, r = c["nx"] * c["ny"], 24
        return {"bytes": 8.0 * nc * (4 + 2 * r), "flops": c["steps"] * nc * (3.0 * (5 * r) ** 2 + 10.0 * r * r)}
    n = _grid(c)
    nc, r1, terms = int(np.prod(n)), c["r1"], 1 + 2 * len(n)
    out = min(c["cap"] or 2 * r1, 2 * r1)
    if c["split"]:
        R = [1] + [terms * r1 + n[0]] + ([terms * r1 + n[2]] if len(n) == 3 else []) + [terms * r1 + 1]
        flops = sum(3.0 * R[k] * n[k] * R[k + 1] ** 2 for k in range(len(n)))
        return {"bytes": c["steps"] * 8.0 * (nc * 6 + sum(n) * r1 * r1), "flops": c["steps"] * flops}
    R1, R2 = terms * r1 + 1, terms * c["r2"] + 1
    flops = nc * (1.0 * R1 * (R1 + 1) + 2.0 * R1 * out) + 2.0 * R1 * c["nt"] * R2 * (R1 + R2)
    return {"bytes": c["steps"] * 8.0 * nc * (r1 + out + 6), "flops": c["steps"] * flops}


# ------------------------------------------------------------------ the same in plain 64-bit torch


def _ttsvd(G, eps, cap):
    """QR sweep from the right, truncated SVDs from the left (delta = eps ||X|| / sqrt(d - 1) per bond)."""
    d, G = len(G), list(G)
    for k in range(d - 1, 0, -1):
        a, m, b = G[k].shape
        Q, R = torch.linalg.qr(G[k].reshape(a, m * b).T)
        G[k] = Q.T.reshape(-1, m, b)
        G[k - 1] = torch.einsum("amb,cb->amc", G[k - 1], R)
    delta2 = (eps * torch.linalg.norm(G[0])) ** 2 / (d - 1)
    for k in range(d - 1):
        a, m, b = G[k].shape
        Q, R = torch.linalg.qr(G[k].reshape(a * m, b))
        U, S, Vt = (x.to(G[k].device) for x in torch.linalg.svd(R.cpu(), full_matrices=False))  # LAPACK's
        tail = torch.flip(torch.cumsum(torch.flip(S ** 2, (0,)), 0), (0,))
        r = max(1, int((tail > delta2).sum()))
        r = min(r, cap) if cap else r
        G[k] = (Q @ U[:, :r]).reshape(a, m, r)
        G[k + 1] = torch.einsum("ab,bmc->amc", S[:r, None] * Vt[:r], G[k + 1])
    return G


def _full(G):
    out = G[0].reshape(G[0].shape[1], -1)
    for x in G[1:]:
        out = (out @ x.reshape(x.shape[0], -1)).reshape(-1, x.shape[2])
    return out.reshape([x.shape[1] for x in G])


def _exact_step(c, seed):
    p, cores, T, sources = _problem(c, seed)
    n, nc, dim = p["n"], T.numel(), len(p["n"])
    dt = 0.5 / max(n)
    nt, npp = c["nt"], c["np"]
    w, v = 2.0 / nt, 2 * math.pi / npp
    mu = -1.0 + (torch.arange(nt, device="cuda", dtype=torch.float64) + 0.5) * w
    sin = torch.sqrt(1.0 - mu * mu)
    phi = (torch.arange(npp, device="cuda", dtype=torch.float64) + 0.5) * v
    one_t, one_p = torch.ones_like(mu), torch.ones_like(phi)
    normal = [(sin, torch.cos(phi)), (sin, torch.sin(phi)), (mu, one_p)]
    X, Th, Ph = cores[0][0], cores[1], cores[2][:, :, 0]
    ka = dt * p["sigma_a"]
    ks = dt * p["sigma_s"] if p["sigma_s"] is not None else torch.zeros_like(ka)

    def shift(Y, a, off):
        Z = torch.roll(Y.reshape(n + (-1,)), -off, a)
        if c["bc"] == "vacuum":
            Z.select(a, n[a] - 1 if off > 0 else 0).zero_()
        return Z.reshape(nc, -1)

    for _ in range(c["steps"]):
        xs, ths, phs = [X], [Th], [Ph]
        for a in range(dim):
            nu, (tf, pf) = dt * n[a], normal[a]
            lo, hi = shift(X, a, -1), shift(X, a, 1)
            if c["flux"] == "upwind":
                if a < 2:
                    facs = [(tf, pf.clamp(min=0.0)), (tf, pf.clamp(max=0.0))]
                else:
                    facs = [(tf.clamp(min=0.0), pf), (tf.clamp(max=0.0), pf)]
                diffs = [X - lo, hi - X]
            else:  # Rusanov with S+ = s c
                s = p["rusanov_s"]
                facs = [(tf, pf), (one_t, one_p)]
                diffs = [0.5 * (hi - lo), 0.5 * s * (2.0 * X - hi - lo)]
            for D, (ft, fp) in zip(diffs, facs):
                xs.append(-nu * D)
                ths.append(Th * ft[None, :, None])
                phs.append(Ph * fp[None, :])
        bar = [torch.einsum("alb,b->a", w * t, v * q.sum(1)) for t, q in zip(ths, phs)]
        E = sum(x @ b for x, b in zip(xs, bar))
        for x, st, sp in sources:
            x = dt * x.cuda()
            xs.append(x[:, None])
            ths.append(st[None, :, None])
            phs.append(sp[None, :])
            E = E + x * (w * st.sum()) * (v * sp.sum())
        gam = ka / (1.0 + ka)
        rhs, Td = T + gam * E, torch.maximum(T, E.clamp(min=0.0) ** 0.25) + 1.0
        for _ in range(100):  # Newton from above: convex and increasing
            Td = Td - (gam * Td ** 4 + Td - rhs) / (4.0 * gam * Td ** 3 + 1.0)
        B = Td ** 4 / FOUR_PI
        J = (E / FOUR_PI + ka * B) / (1.0 + ka)
        s = 1.0 / (1.0 + ka + ks)
        xs = [x * s[:, None] for x in xs] + [(s * (ks * J + ka * B))[:, None]]
        ths.append(one_t[None, :, None])
        phs.append(one_p[None, :])
        Xg, Pg = torch.cat(xs, 1), torch.cat(phs, 0)
        Tg = torch.zeros(Xg.shape[1], nt, Pg.shape[0], device="cuda", dtype=torch.float64)
        i = j = 0
        for t in ths:
            Tg[i:i + t.shape[0], :, j:j + t.shape[2]] = t
            i, j = i + t.shape[0], j + t.shape[2]
        G = _ttsvd([Xg[None], Tg, Pg[:, :, None]], c["eps"], c["cap"])
        X, Th, Ph = G[0][0], G[1], G[2][:, :, 0]
        En = X @ torch.einsum("alb,b->a", w * Th, v * Ph.sum(1))
        T = T + (E - En)
    vol = 1.0 / nc
    out = {"E": En, "T": T, "totals": np.array([float(En.sum()) * vol, float(T.sum()) * vol]), "ranks": None}
    if nc * nt * npp <= 1 << 18:
        out["full"] = _full(G).reshape(n + (nt, npp))
    return out


def _parts(A):
    """A (k x n) as three exact addends of at most 24 bits each below a power of two per column."""
    top = torch.exp2(torch.ceil(torch.log2(A.abs().amax(0, keepdim=True).clamp(min=1e-300))))
    out, rest = [], A
    for bits in (23, 46):
        q = torch.round(rest / top * 2.0 ** bits) / 2.0 ** bits * top
        out.append(q)
        rest = rest - q
    return out + [rest]


def _product(A, B, symmetric=False):
    """A^T B for A (k x m), B (k x n) to the last bits: the leading parts' products over 32 terms are exact in 64
    bits and added with their rounding errors kept."""
    m, n = A.shape[1], B.shape[1]
    hi = torch.zeros(m, n, device="cuda", dtype=torch.float64)
    lo = torch.zeros_like(hi)
    a = _parts(A)
    b = a if symmetric else _parts(B)
    step = 32
    for i, j in ((0, 0), (0, 1), (1, 0)):
        for k in range(0, A.shape[0], step):
            x = a[i][k:k + step].T @ b[j][k:k + step]
            s = hi + x
            t = s - hi
            lo += (hi - (s - t)) + (x - t)
            hi = s
    lo += a[1].T @ b[1] + (a[0] + a[1]).T @ b[2] + a[2].T @ (b[0] + b[1] + b[2])
    return hi + lo


def exact(case, seed):
    c = case
    if c["kind"] == "gemm":
        A, B = _gemm_inputs(c, seed)
        return _product(A if c["ta"] else A.T, B.T if c["tb"] else B)
    if c["kind"] == "gram":
        A = _matrix(_gen(seed), c["m"], c["n"], 4.0, 1)
        return _product(A, A, symmetric=True)
    if c["kind"] == "round" and c["method"] != "randomized":
        return {"full": _full(_ttsvd(_round_cores(c, seed), c["eps"], 0)), "ranks": None}
    if c["kind"] == "step" and not c["split"] and c["flux"] != "hll":
        return _exact_step(c, seed)
    return None
