"""Timed cases of the convexification library, through its Python binding.

Twelve listed cases cover what a program asks of the library: the per-point
form (from a material routine's few points to a million), an implicit
finite-element step with its tangent, meshes and load steps with fine angle
grids and long lines, the learned proposal, many meshes in one call, the
network's own inference and gradient, and the global-grid form in two and
three dimensions with its queries.  ``draw`` gives further cases of the same
kinds over the same ranges.  Sizes and distributions are those of the
repository's benchmark, tests and input generators.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2211_14318_gb300 import api, inputs

MAT = dict(mu=1.0, lambda_L=5.0, D_inf=0.99, D0=0.5)          # the per-point workloads
GRID_MAT = dict(mu=1.0, lambda_L=0.5, D_inf=0.9, D0=0.3)      # the global-grid studies
DEV = "cuda:0"

# angles: n_a x n_b directions; line: samples per line; depth: lamination depth
LISTED = [
    # a material routine called for a handful of quadrature points (one element
    # patch): launches and latency are what it costs
    dict(name="points_64", kind="points", n=64, na=16, nb=16, line=201, depth=2),
    # a million material points on the coarse angle grid: a large mesh's
    # constitutive update
    dict(name="points_1m", kind="points", n=1048576, na=16, nb=16, line=201, depth=2),
    # an implicit finite-element step on a ragged mesh: history update, adaptive
    # line window, Newton-refined splits, tree and consistent tangent
    dict(name="fe_step", kind="fe", n=20011, na=24, nb=20, line=333, depth=2, doublings=3),
    # a mesh with a finer angle grid, longer lines and three orders of laminates
    dict(name="mesh_64", kind="mesh", nx=64, na=64, line=1025, depth=3, stretch=1.3),
    # the full scan of a load step on the finest angle grid: labels for the
    # network, and the reference that the proposal is judged against
    dict(name="load_full", kind="load_full", n=3001, step=10, na=128, line=2049, depth=3),
    # the same load path by the learned proposal (windows, re-centring, mirror
    # windows, fallback): the headline workload on a 128 x 128 mesh
    dict(name="load_propose", kind="propose", nx=128, step=15, na=128, line=2049, depth=3,
         window=4, recentre=4),
    # many meshes of uneven size and their own parameters in one captured run,
    # replayed as a load-stepping program does
    dict(name="batch_12", kind="batch", problems=12, n_lo=1000, n_hi=20000),
    # the network alone: proposals for a million tree nodes
    dict(name="net_forward", kind="net_forward", n=1000000),
    # the network's training step: loss and gradient of one batch
    dict(name="net_grad", kind="net_grad", n=8192),
    # the paper's global grid in two dimensions, iterated to its tolerance
    dict(name="grid_2d", kind="grid", dim=2, nd=23, no=35, kmax=20),
    # ... and in three dimensions (nine components, 169 directions)
    dict(name="grid_3d", kind="grid", dim=3, nd=17, no=3, kmax=20),
    # relaxed energy, stress and tangent at arbitrary points of a converged grid
    dict(name="grid_query", kind="query", n=1048576, nd=23, no=35, tangent=True),
]


def listed():
    return [dict(c) for c in LISTED]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["points", "points", "fe", "mesh", "load_full", "propose", "batch",
                       "net_forward", "net_grad", "grid", "grid", "query"])
    if kind == "points":
        na, nb = rng.randint(6, 32), rng.randint(6, 32)
        line, depth = 2 * rng.randint(25, 256) + 1, rng.randint(1, 3)
        most = 1.6e11 / (na * nb * line * (2 ** depth - 1))
        return dict(kind=kind, n=_log(rng, 16, max(64, min(1048576, most))), na=na, nb=nb,
                    line=line, depth=depth)
    if kind == "fe":
        return dict(kind=kind, n=_log(rng, 50, 20011), na=rng.randint(10, 22),
                    nb=rng.randint(10, 22), line=2 * rng.randint(50, 166) + 1,
                    depth=rng.randint(1, 2), doublings=rng.randint(0, 3))
    if kind == "mesh":
        return dict(kind=kind, nx=_log(rng, 5, 60), na=rng.randint(24, 62),
                    line=2 * rng.randint(200, 512) + 1, depth=rng.randint(2, 3),
                    stretch=round(rng.uniform(1.1, 1.8), 3))
    if kind == "load_full":
        return dict(kind=kind, n=_log(rng, 40, 1400), step=rng.randint(1, 20), na=128,
                    line=2 * rng.randint(400, 1024) + 1, depth=rng.randint(2, 3))
    if kind == "propose":
        return dict(kind=kind, nx=_log(rng, 8, 120), step=rng.randint(1, 20), na=128,
                    line=2 * rng.randint(500, 1024) + 1, depth=rng.randint(2, 3),
                    window=rng.randint(3, 5), recentre=rng.randint(3, 5))
    if kind == "batch":
        return dict(kind=kind, problems=rng.randint(3, 11), n_lo=400, n_hi=rng.randint(2000, 15000))
    if kind == "net_forward":
        return dict(kind=kind, n=_log(rng, 100, 1000000))
    if kind == "net_grad":
        return dict(kind=kind, n=_log(rng, 30, 65000))
    if kind == "query":
        return dict(kind=kind, n=_log(rng, 500, 1000000), nd=rng.randint(8, 23),
                    no=rng.randint(7, 33), tangent=rng.random() < 0.5)
    if rng.random() < 0.3:
        return dict(kind=kind, dim=3, nd=rng.randint(6, 16), no=rng.randint(2, 3), kmax=20)
    return dict(kind=kind, dim=2, nd=rng.randint(6, 23), no=rng.randint(5, 35), kmax=20)


# ------------------------------------------------------------------- inputs
_kept = {}  # what a program keeps over its calls: its handle, the trained weights


def _handle(kind):
    if kind not in _kept:
        _kept[kind] = api.Convexifier(0)
    return _kept[kind]


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def _params(case, **kw):
    na = case["na"]
    return api.Params(n_theta_a=na, n_theta_b=case.get("nb", na), line_points=case["line"],
                      depth=case["depth"], **MAT, **kw)


def _material(n, seed):
    """Material points (stretch up to 2) and the previous step's F, on the device."""
    F, Fp = inputs.material_points(n, seed=seed % (1 << 31), lam_lo=1.0, lam_hi=2.0)
    return _dev(F), _dev(Fp)


def _load_step(cv, p, nx, step, seed):
    """F at a load step of a path of 20 to stretch 1.8, and the history before it."""
    path = inputs.load_path(nx, n_steps=20, stretch_end=1.8, seed=seed % (1 << 31))
    beta = None
    for k in range(step - 1):
        beta = cv.history_update(p, _dev(path[k]), beta)
    F = _dev(path[step - 1])
    if beta is None:
        beta = torch.zeros(F.shape[0], dtype=torch.float64, device=DEV)
    return F, beta


def _weights():
    """A proposal network (flat weights, input mean and deviation) fitted to
    full scans of material points and load steps, once per process."""
    if "weights" in _kept:
        return _kept["weights"]
    cv = api.Convexifier(0)
    pl = api.Params(n_theta_a=128, n_theta_b=128, line_points=257, depth=2, **MAT)
    F, Fp = _material(16384, 100)
    sets = [(F, cv.history_update(pl, Fp))]
    for mesh in (7, 8, 9):
        sets += [_load_step(cv, pl, 32, k, mesh) for k in (2, 6, 10, 14, 17, 20)]
    X, Y = [], []
    for F, b in sets:
        o = cv.convexify_points(pl, F, b, want_tree=True)
        x, y = cv.surrogate_labels(pl, b, o["tree"], F.shape[0])
        X.append(x.clone())
        Y.append(y.clone())
    X, Y = torch.cat(X), torch.cat(Y)
    cv.close()
    mean, std = X.mean(0), X.std(0).clamp_min(1e-6)
    Xn = (X - mean) / std
    g = torch.Generator(device=DEV).manual_seed(0)
    ws = []
    for i, o in ((6, 256), (256, 256), (256, 256), (256, 256), (256, 7)):
        for shape in ((o, i), (o,)):
            w = (torch.rand(shape, generator=g, device=DEV) * 2 - 1) / math.sqrt(i)
            ws.append(w.requires_grad_())
    opt = torch.optim.Adam(ws, lr=1e-3)
    steps = 1500
    for k in range(steps):
        for q in opt.param_groups:
            q["lr"] = 1e-3 * (0.5 + 0.5 * math.cos(math.pi * k / steps)) + 1e-5
        idx = torch.randint(0, Xn.shape[0], (8192,), generator=g, device=DEV)
        h, y = Xn[idx], Y[idx]
        for j in range(0, 8, 2):
            h = torch.nn.functional.gelu(h @ ws[j].T + ws[j + 1])
        loss = _loss(h @ ws[8].T + ws[9], y)
        opt.zero_grad()
        loss.backward()
        opt.step()
    flat = torch.cat([w.detach().reshape(-1) for w in ws]).cpu().numpy()
    _kept["weights"] = (flat, mean.cpu().numpy(), std.cpu().numpy())
    return _kept["weights"]


def _loss(o, y):
    """The network's documented loss: masked angles and fraction, jump."""
    a = torch.where(torch.isnan(y[:, :2]), 0.0, 1 - torch.cos(2 * (o[:, :2] - torch.nan_to_num(y[:, :2]))))
    x = torch.where(torch.isnan(y[:, 2]), 0.0, (torch.sigmoid(o[:, 2]) - torch.nan_to_num(y[:, 2])) ** 2)
    return (a.sum(1) + x + ((o[:, 3:] - y[:, 3:]) ** 2).sum(1)).mean()


def _net_weights(seed):
    """Weights of the fresh network's scale from a seed, standardisation of material points."""
    rng = np.random.default_rng(seed)
    w = []
    for i, o in ((6, 256), (256, 256), (256, 256), (256, 256), (256, 7)):
        w += [rng.uniform(-1, 1, o * i) / math.sqrt(i), rng.uniform(-1, 1, o) / math.sqrt(i)]
    return (np.concatenate(w).astype(np.float32),
            np.array([1.0, 0.0, 0.0, 1.0, 0.3, 0.2], np.float32),
            np.array([0.4, 0.3, 0.3, 0.4, 0.4, 0.2], np.float32))


def _net_rows(n, seed):
    """Features and labels (a third of the nodes do not split) as the library lays them out."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    F = torch.randn(n, 4, generator=g, device=DEV) * 0.25
    F[:, 0] += 1.2
    F[:, 3] += 1.2
    J = (F[:, 0] * F[:, 3] - F[:, 1] * F[:, 2]).clamp_min(0.05)
    X = torch.cat([F, torch.rand(n, 1, generator=g, device=DEV), torch.log(J)[:, None]], 1)
    Y = torch.rand(n, 7, generator=g, device=DEV)
    Y[:, :2] *= math.pi
    Y[:, 3:] -= 0.5
    flat = torch.rand(n, generator=g, device=DEV) < 1 / 3
    Y[flat, :3] = float("nan")
    Y[flat, 3:] = 0.0
    return X.contiguous(), Y.contiguous()


def _grid(case, seed):
    """The study grid of the case's shape (full size: 0.1 .. 3.4 by -2.55 .. 2.55
    in steps of 0.15, or 1 .. 3.4 by +-0.15 in three dimensions) and its history."""
    nd, no = case["nd"], case["no"]
    beta = 0.055 + 0.01 * np.random.default_rng(seed).random()
    if case.get("dim", 2) == 2:
        diag, off = (0.1, 0.1 + 0.15 * (nd - 1)), (-0.075 * (no - 1), 0.075 * (no - 1))
        return api.GridSpec.from_bounds(diag, off, (0.15, 0.15)), float(beta), 1
    diag, off = (1.0, 1.0 + 0.15 * (nd - 1)), (-0.075 * (no - 1), 0.075 * (no - 1))
    return api.GridSpec.from_bounds(diag, off, (0.15, 0.15), dim=3), float(beta), 0


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind in ("points", "fe"):
        s["cv"] = cv = _handle("points")
        s["p"] = p = _params(case) if kind == "points" else \
            _params(case, newton=True, window_doublings=case["doublings"])
        s["F"], Fp = _material(case["n"], seed)
        s["beta"] = cv.history_update(p, Fp)
    elif kind == "mesh":
        s["cv"] = cv = _handle("points")
        s["p"] = p = _params(case)
        F, Fp = inputs.mesh_points(case["nx"], stretch=case["stretch"], seed=seed % (1 << 31))
        s["F"], s["beta"] = _dev(F), cv.history_update(p, _dev(Fp))
    elif kind == "load_full":
        s["cv"] = cv = _handle("points")
        s["p"] = p = _params(case)
        F, b = _load_step(cv, p, 32, case["step"], seed)
        at = _dev(np.random.default_rng(seed).choice(F.shape[0], case["n"], replace=False))
        s["F"], s["beta"] = F[at].contiguous(), b[at].contiguous()
    elif kind == "propose":
        s["cv"] = cv = _handle("propose")
        if not getattr(cv, "has_weights", False):
            cv.surrogate_set_weights(*_weights())
            cv.has_weights = True
        s["p"] = p = _params(case, recentre=case["recentre"], mirror=True)
        s["window"] = case["window"]
        s["F"], s["beta"] = _load_step(cv, p, case["nx"], case["step"], seed)
    elif kind == "batch":
        s["cv"] = cv = api.Convexifier(0)  # a captured run belongs to its handle
        s["problems"] = []
        # the stretches, angle grids, lines, depths and log-uniform sizes of a
        # batch of meshes, drawn from the case alone so that every seed costs
        # alike; the displacement fields come from the seed
        shapes = np.random.default_rng(case["problems"] * 100003 + case["n_hi"])
        for k in range(case["problems"]):
            n = math.exp(shapes.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))
            nx, stretch = max(1, round(math.sqrt(n / 4))), float(shapes.uniform(1.1, 1.8))
            na, line, depth = (int(shapes.choice(v)) for v in ((32, 64), (513, 1025), (2, 3)))
            F, Fp = inputs.mesh_points(nx, stretch=stretch, seed=(seed * 1009 + k) % (1 << 31))
            p = api.Params(n_theta_a=na, n_theta_b=na, line_points=line, depth=depth, **MAT)
            s["problems"].append((p, _dev(F), cv.history_update(p, _dev(Fp))))
        s["outs"] = cv.convexify_batch(s["problems"])  # the plan: launch shape, captured run
    elif kind in ("net_forward", "net_grad"):
        s["cv"] = cv = _handle("net")
        if "net" not in _kept.get("loaded", ()):
            cv.surrogate_set_weights(*_net_weights(5))
            _kept["loaded"] = ("net",)
        s["X"], s["Y"] = _net_rows(case["n"], seed)
    else:
        s["cv"] = cv = _handle("grid")
        s["p"] = p = api.Params(**GRID_MAT)
        s["grid"], s["beta"], s["rule"] = g, beta, rule = _grid(case, seed)
        s["off"] = api.grid_r11(g.dim)
        kmax = s["kmax"] = case.get("kmax", 20)
        # rows of steps that are not taken stay as the program set them
        s["out"] = dict(W=torch.empty(g.count, dtype=torch.float64, device=DEV),
                        forest=torch.full((kmax, g.count, 3), -1, dtype=torch.int32, device=DEV),
                        decs=torch.zeros(kmax, dtype=torch.float64, device=DEV),
                        iters=torch.zeros(1, dtype=torch.int32, device=DEV))
        if kind == "query":
            cv.grid_convexify(p, g, beta, s["off"], kmax=kmax, det_rule=rule, out=s["out"])
            K = int(s["out"]["iters"].item())
            s["W"], s["forest"] = s["out"]["W"], s["out"]["forest"][:K].clone()
            lo = np.array(g.lo)
            hi = lo + (np.array(g.n) - 1) * np.array(g.delta)
            s["F"] = _dev(inputs.cuboid_points(lo, hi, case["n"], seed=seed % (1 << 31)))
            s["tangent"] = case["tangent"]
            del s["out"]
    return s


def run(s):
    cv, kind = s["cv"], s["kind"]
    if kind in ("points", "mesh", "load_full"):
        o = cv.convexify_points(s["p"], s["F"], s["beta"])
        return {k: o[k] for k in ("W_R", "P", "status")}
    if kind == "fe":
        o = cv.convexify_points(s["p"], s["F"], s["beta"], want_tree=True)
        A = cv.tree_tangent(s["p"], s["beta"], o["tree"], s["F"].shape[0])
        new = cv.history_update(s["p"], s["F"], s["beta"])
        return dict(W_R=o["W_R"], P=o["P"], status=o["status"], A=A, beta=new)
    if kind == "propose":
        o = cv.surrogate_propose(s["p"], s["F"], s["beta"], window=s["window"], gap_tol=1e30)
        return {k: o[k] for k in ("W_R", "P", "status", "fell_back")}
    if kind == "batch":
        return [{k: o[k] for k in ("W_R", "P", "status")}
                for o in cv.convexify_batch(s["problems"], outs=s["outs"])]
    if kind == "net_forward":
        return cv.surrogate_forward(s["X"])
    if kind == "net_grad":
        return cv.surrogate_loss_grad(s["X"], s["Y"])
    if kind == "grid":
        return cv.grid_convexify(s["p"], s["grid"], s["beta"], s["off"], kmax=s["kmax"],
                                 det_rule=s["rule"], out=s["out"])
    return cv.grid_query(s["p"], s["grid"], s["beta"], s["off"], s["W"], s["forest"], s["F"],
                         det_rule=s["rule"], want_A=s["tangent"])


def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: of the
    per-point form, 30 for each sample of the roots' lines (22 for the energy, 8
    for the hull), as every point is scanned at least once; of the proposal, the
    same for one window; of the network, its products; of the grid, 12 for each
    point, direction and one step (two predicates, one chord)."""
    kind, n = case["kind"], case.get("n", 0)
    if kind in ("points", "fe", "load_full"):
        extra = 8 * 16 + 8 if kind == "fe" else 0
        nb = case.get("nb", case["na"])
        return dict(bytes=n * (40 + 44 + extra), flops=30.0 * n * case["na"] * nb * case["line"])
    if kind in ("mesh", "propose"):
        n = 4 * case["nx"] ** 2
        d = case["na"] ** 2 if kind == "mesh" else (2 * case["window"] + 1) ** 2
        return dict(bytes=n * 84, flops=30.0 * n * d * case["line"])
    if kind == "batch":
        n = case["problems"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        return dict(bytes=n * 84, flops=30.0 * n * 32 ** 2 * 513)
    mac = 6 * 256 + 3 * 256 * 256 + 256 * 7
    if kind == "net_forward":
        return dict(bytes=n * 52 + 4 * 200967, flops=2.0 * n * mac)
    if kind == "net_grad":
        return dict(bytes=n * 52 + 8 * 200967, flops=6.0 * n * mac)
    g, _, _ = _grid(case, 0)
    if kind == "grid":
        dirs = 16 if g.dim == 2 else 169
        return dict(bytes=g.count * (8 + 12), flops=12.0 * g.count * dirs)
    A = 128 if case["tangent"] else 0
    return dict(bytes=n * (32 + 16 + 32 + 8 + A) + g.count * 8, flops=16.0 * n * 5)


# -------------------------------------------------------------------- exact
def _psi0(F):
    J = F[..., 0] * F[..., 3] - F[..., 1] * F[..., 2]
    lj = torch.log(J)
    s = 0.5 * MAT["mu"] * ((F * F).sum(-1) - 2) - MAT["mu"] * lj + 0.5 * MAT["lambda_L"] * lj * lj
    return s, J, lj


def _w_of(s, beta, m):
    ek = torch.exp(-beta / m["D0"])
    lo = (1 - m["D_inf"] * (1 - ek)) * (s - beta)
    hi = (1 - m["D_inf"]) * (s - beta) + m["D_inf"] * m["D0"] * (ek - torch.exp(-s / m["D0"]))
    return torch.where(s <= beta, lo, hi)


def _stress(F, beta):
    s, J, lj = _psi0(F)
    g = 1 - MAT["D_inf"] * (1 - torch.exp(-torch.maximum(s, beta) / MAT["D0"]))
    G = torch.stack([F[:, 3], -F[:, 2], -F[:, 1], F[:, 0]], 1) / J[:, None]
    return g[:, None] * (MAT["mu"] * (F - G) + MAT["lambda_L"] * lj[:, None] * G)


def _relax(F, beta, na, nb, L, t_half, K):
    """The per-point method in 64 bits: lower hull of every line read at 0,
    minimum over directions, split, recursion, leaves."""
    n = F.shape[0]
    ta = math.pi * torch.arange(na, device=DEV, dtype=torch.float64) / na
    tb = math.pi * torch.arange(nb, device=DEV, dtype=torch.float64) / nb
    a, b = torch.stack([ta.cos(), ta.sin()], 1), torch.stack([tb.cos(), tb.sin()], 1)
    R = (a[:, None, :, None] * b[None, :, None, :]).reshape(na * nb, 4)
    m0 = (L - 1) // 2
    x = torch.arange(-m0, m0 + 1, device=DEV, dtype=torch.float64)
    t = x * (2 * t_half / (L - 1))
    W = torch.zeros(n, dtype=torch.float64, device=DEV)
    P = torch.zeros(n, 4, dtype=torch.float64, device=DEV)

    def leaf(pt, Fl, wt):
        W.index_add_(0, pt, wt * _w_of(_psi0(Fl)[0], beta[pt], MAT))
        P.index_add_(0, pt, wt[:, None] * _stress(Fl, beta[pt]))

    pt, Fn, wt = torch.arange(n, device=DEV), F, torch.ones(n, dtype=torch.float64, device=DEV)
    for _ in range(K):
        nxt = []
        for c in torch.arange(pt.numel(), device=DEV).split(max(1, int(1.5e7 / (na * nb * L)))):
            f, bt, k = Fn[c], beta[pt[c]], c.numel()
            G = f[:, None, None, :] + t[None, None, :, None] * R[None, :, None, :]
            s, J, _ = _psi0(G)
            v = torch.where(J > 0, _w_of(s, bt[:, None, None], MAT), math.inf).reshape(-1, L)
            del G, s, J
            sl = torch.zeros(v.shape[0], 1, dtype=torch.float64, device=DEV)
            A = B = None
            for _it in range(64):
                e = v - sl * x
                A2, B2 = e[:, :m0].argmin(1, True), e[:, m0 + 1:].argmin(1, True) + m0 + 1
                if A is not None and bool((A2 == A).all()) and bool((B2 == B).all()):
                    break
                A, B = A2, B2
                sl = (v.gather(1, B) - v.gather(1, A)) / (B - A)
                sl = torch.where(torch.isfinite(sl), sl, 0.0)
            va, vb = v.gather(1, A), v.gather(1, B)
            q = ((B - m0) * va + (m0 - A) * vb) / (B - A)
            q = torch.where(torch.isfinite(q), q, math.inf).reshape(k, -1)
            d = q.argmin(1)
            split = q.gather(1, d[:, None])[:, 0] < _w_of(_psi0(f)[0], bt, MAT)
            am = A.reshape(k, -1).gather(1, d[:, None])[:, 0]
            bm = B.reshape(k, -1).gather(1, d[:, None])[:, 0]
            xi = (m0 - am).double() / (bm - am).double()
            leaf(pt[c][~split], f[~split], wt[c][~split])
            for tt, w in ((t[am], 1 - xi), (t[bm], xi)):
                nxt.append((pt[c][split], (f + tt[:, None] * R[d])[split], (wt[c] * w)[split]))
        pt, Fn, wt = (torch.cat(z) for z in zip(*nxt))
        if pt.numel() == 0:
            break
    leaf(pt, Fn, wt)
    return W, P


def _net_exact(X, weights):
    flat, mean, std = (torch.from_numpy(v).to(DEV).double() for v in weights)
    h, at = (X.double() - mean) / std, 0
    flat.requires_grad_()
    for j, (i, o) in enumerate(((6, 256), (256, 256), (256, 256), (256, 256), (256, 7))):
        w, b = flat[at:at + o * i].reshape(o, i), flat[at + o * i:at + o * i + o]
        at += o * i + o
        h = h @ w.T + b
        if j < 4:
            h = torch.nn.functional.gelu(h)
    return h, flat


def _grid_w(F, beta, rule):
    """Neo-Hooke with damage on a grid (plane strain, or three dimensions)."""
    m = GRID_MAT
    d = 2 if F.shape[-1] == 4 else 3
    J = torch.linalg.det(F.reshape(-1, d, d)).reshape(F.shape[:-1]) if d == 3 else \
        F[..., 0] * F[..., 3] - F[..., 1] * F[..., 2]
    lj = torch.log(J.abs())
    I1 = (F * F).sum(-1) + (1 if d == 2 else 0)
    s = 0.5 * m["mu"] * (I1 - 3) - m["mu"] * lj + 0.5 * m["lambda_L"] * lj * lj
    w = _w_of(s, torch.tensor(beta, dtype=torch.float64, device=DEV), m)
    return torch.where((J > 0) | ((J != 0) & (rule == 1)), w, math.nan)


def _grid_points(g):
    ax = [g.lo[c] + g.delta[c] * torch.arange(g.n[c], device=DEV, dtype=torch.float64)
          for c in range(g.D)]
    idx = torch.cartesian_prod(*[torch.arange(k, device=DEV) for k in g.n])
    return torch.stack([ax[c][idx[:, c]] for c in range(g.D)], 1), idx


def _grid_exact(g, off, beta, rule, kmax, tol):
    """Eq. (4.3) iterated in 64 bits: on every grid line the least chord over
    each point, over all pairs of line points."""
    F, idx = _grid_points(g)
    W = _grid_w(F, beta, rule)
    del F
    n = torch.tensor(g.n, device=DEV)
    stride = torch.tensor([int(np.prod(g.n[c + 1:])) for c in range(g.D)], device=DEV)
    o_all = torch.from_numpy(np.asarray(off)).to(DEV).long()
    lines = []
    for o in o_all:
        prev = idx - o
        p = torch.nonzero(((prev < 0) | (prev >= n)).any(1))[:, 0]
        room = torch.where(o > 0, n - 1 - idx[p], torch.where(o < 0, idx[p], 1 << 20))
        lines.append((p, int((o * stride).sum()), room.min(1).values + 1))
    decs = torch.zeros(kmax, dtype=torch.float64, device=DEV)
    for k in range(kmax):
        best = torch.where(torch.isfinite(W), W, math.inf)
        src = best.clone()
        for p, step, ln in lines:
            m = int(ln.max())
            l = torch.arange(m, device=DEV)
            at = p[:, None] + l * step
            ok = l < ln[:, None]
            v = torch.where(ok, src[torch.where(ok, at, p[:, None])], math.inf)
            h = v.clone()
            for i in range(m - 2):
                for j in range(i + 2, m):
                    x = torch.arange(1, j - i, device=DEV, dtype=torch.float64) / (j - i)
                    ch = v[:, i:i + 1] * (1 - x) + v[:, j:j + 1] * x
                    h[:, i + 1:j] = torch.minimum(h[:, i + 1:j], ch.nan_to_num(math.inf))
            best.index_put_((at[ok],), torch.minimum(best[at[ok]], h[ok]))
        new = torch.where(torch.isfinite(W), best, W)
        decs[k] = (W - new).nan_to_num(0.0).max()
        W = new
        if float(decs[k]) <= tol:
            break
    return W, decs


def _query_exact(s):
    """Interpolation of W and Algorithm 3 over the given forest in 64 bits:
    W, P and A of the leaves, combined order by order."""
    g, rule = s["grid"], s["rule"]
    G, _ = _grid_points(g)
    G.requires_grad_()
    w = _grid_w(G, s["beta"], rule)
    P, = torch.autograd.grad(w.nan_to_num(0.0).sum(), G, create_graph=True)
    cols = [w.detach()[:, None], P.detach()]
    if s["tangent"]:
        cols += [torch.autograd.grad(P[:, a].sum(), G, retain_graph=True)[0] for a in range(4)]
    T = torch.cat(cols, 1).detach()
    stride = torch.tensor([int(np.prod(g.n[c + 1:])) for c in range(g.D)], device=DEV)
    step = (torch.from_numpy(np.asarray(s["off"])).to(DEV).long() * stride).sum(1)
    for rec in s["forest"].long():
        p = torch.nonzero(rec[:, 0] >= 0)[:, 0]
        d, lm, lp = rec[p].unbind(1)
        xi = (-lm.double() / (lp - lm).double())[:, None]
        new = (1 - xi) * T[p + lm * step[d]] + xi * T[p + lp * step[d]]
        T = T.clone()
        T[p] = new
    lo = torch.tensor(g.lo, device=DEV, dtype=torch.float64)
    u = (s["F"] - lo) / torch.tensor(g.delta, device=DEV, dtype=torch.float64)
    n = torch.tensor(g.n, device=DEV)
    i0 = torch.minimum(u.floor().long().clamp_min(0), n - 2)
    t = u - i0
    out, wi = 0.0, 0.0
    for c in range(16):
        up = torch.tensor([(c >> (3 - k)) & 1 for k in range(4)], device=DEV)
        wt = torch.where(up == 1, t, 1 - t).prod(1)
        f = ((i0 + up) * stride).sum(1)
        out = out + wt[:, None] * T[f]
        wi = wi + wt * s["W"][f]
    r = [wi, out[:, 0], out[:, 1:5], None]
    return tuple(r + [out[:, 5:].reshape(-1, 4, 4)]) if s["tangent"] else tuple(r)


def exact(case, seed):
    """What run() returns, in 64 bits; None where the plain method takes too
    long (large scans) and for whole numbers."""
    kind = case["kind"]
    if kind == "points":
        cost = case["n"] * case["na"] * case["nb"] * case["line"] * (2 ** case["depth"] - 1)
        if cost > 6e8:
            return None
        s = prepare(case, seed)
        W, P = _relax(s["F"], s["beta"], case["na"], case["nb"], case["line"], 0.5, case["depth"])
        return dict(W_R=W, P=P, status=None)
    if kind == "fe":
        s = prepare(case, seed)
        new = torch.maximum(s["beta"], _psi0(s["F"])[0])
        return dict(W_R=None, P=None, status=None, A=None, beta=new)
    if kind == "net_forward":
        X, _ = _net_rows(case["n"], seed)
        with torch.no_grad():
            return torch.cat([_net_exact(x, _net_weights(5))[0] for x in X.split(1 << 17)])
    if kind == "net_grad":
        X, Y = _net_rows(case["n"], seed)
        out, flat = _net_exact(X, _net_weights(5))
        loss = _loss(out, Y.double())
        loss.backward()
        return loss.detach().reshape(1), flat.grad
    if kind == "grid":
        g, beta, rule = _grid(case, seed)
        W, decs = _grid_exact(g, api.grid_r11(g.dim), beta, rule, case["kmax"], 1e-4)
        return dict(W=W, forest=None, decs=decs, iters=None)
    if kind == "query":
        return _query_exact(prepare(case, seed))
    return None
