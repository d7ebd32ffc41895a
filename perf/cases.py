"""Workloads for timing the library through its public entry points.

A case is a dict of plain sizes and options.  ``prepare`` makes what a user's program holds
before the call (mesh, model or session handle, wavelets, observed traces), ``run`` is one
pass of the calls that the program repeats, and ``exact`` computes the same outputs in plain
64-bit torch: the paper's elimination written as batched dense algebra and one dense LU of
the boundary system, with the gradient of the exact adjoint taken by automatic
differentiation of that time loop.
"""

import functools
import math

import numpy as np
import torch

import sbfwi_inputs as inputs
from sbfwi_inputs import mesh3d
from paper_2501_06748_gb300 import sbfwi

XI0, BETA, GAMMA = 1e-3, 0.25, 0.5


def _case(kind, name=None, **kw):
    c = {"kind": kind, "mesh": "square", "nx": 4, "ny": 4, "p": 2, "n_r": 8, "shots": 1, "recs": 4, "steps": 100,
         "grid": 64, "ckpt": 0, "exact_adjoint": False}
    c.update(kw)
    return {"name": name, **c} if name else c


def listed():
    return [
        # the misfit of one batch of shots (traces of the 64 x 64 recipe), called on its own by a line search
        _case("misfit", "misfit_traces", shots=8, recs=32, steps=2000),
        # the smallest inversion evaluation: the 4 x 4 plate with one source and four receivers
        _case("gradient", "tiny_gradient", steps=200),
        # one shot on the 64 x 64 recipe, traces only: what a single request or a modelling user waits for
        _case("forward", "one_shot_forward", nx=64, ny=64, p=4, n_r=32, recs=32, steps=100, grid=256),
        # a serving session: five requests of uneven lengths in eight slots, windows of 32 steps
        _case("session", "session_requests", nx=24, ny=24, p=4, n_r=16, shots=5, recs=16, steps=80, grid=128),
        # a line-search evaluation on a new density: set-up, forward of a batch of shots, misfit
        _case("search", "line_search", nx=64, ny=64, p=4, n_r=32, shots=8, recs=32, steps=64, grid=256),
        # the flagship evaluation: misfit and gradient of eight shots, forward field stored
        _case("gradient", "batch_gradient", nx=64, ny=64, p=4, n_r=32, shots=8, recs=32, steps=96, grid=256),
        # the 128 x 128 recipe, whose forward field does not fit: checkpoints, recomputed in the adjoint
        _case("gradient", "checkpoint_gradient", nx=128, ny=128, p=4, n_r=32, shots=8, recs=64, steps=40, grid=512,
              ckpt=-1),
        # an odd plate: 37 x 23 elements of order 3, 13 radial points, five shots
        _case("gradient", "ragged_gradient", nx=37, ny=23, p=3, n_r=13, shots=5, recs=19, steps=100, grid=96),
        # the order-5 quadtree mesh of the batching recipe: hanging vertices, 20 to 30 nodes per element
        _case("gradient", "quadtree_gradient", mesh="quadtree", nx=16, ny=16, p=5, n_r=48, shots=8, recs=32, steps=48,
              grid=256),
        # one epoch of the paper's plate experiment: set-up, forward, misfit and adjoint on Voronoi polygons
        _case("epoch", "plate_epoch", mesh="voronoi", nx=1000, ny=1, p=2, n_r=6, shots=2, recs=100, steps=200, grid=256),
        # the solid cube: 16^3 hexahedral elements, 26 boundary nodes, eight shots
        _case("gradient", "solid_gradient", mesh="cube", nx=16, ny=16, p=2, n_r=16, shots=8, recs=30, steps=24, grid=64),
        # the exact derivative of the discrete misfit, which gradient checks and L-BFGS on it use
        _case("gradient", "exact_gradient", nx=24, ny=24, p=4, n_r=32, shots=8, recs=32, steps=40, grid=128,
              exact_adjoint=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh_nodes(c):
    """About how many elements, boundary nodes per element and global nodes the mesh has."""
    p = c["p"]
    if c["mesh"] == "cube":
        n = c["nx"] ** 3
        return n, 6 * p * p + 2, (c["nx"] * p + 1) ** 3 - n * (p - 1) ** 3
    if c["mesh"] == "voronoi":
        return c["nx"], 6 * p, c["nx"] * (3 * p - 1)
    if c["mesh"] == "quadtree":
        n = int(2.7 * c["nx"] * c["nx"])
        return n, 4 * p + 2, n * (2 * p)
    n = c["nx"] * c["ny"]
    return n, 4 * p, n * (2 * p - 1) + (c["nx"] + c["ny"]) * p


def _loops(c):
    """Time loops over all steps: forward, and adjoint (with a recompute where checkpoints are kept)."""
    if c["kind"] in ("forward", "session", "search"):
        return 1
    return 3 if c["ckpt"] else 2


def _cost(c):
    """Matrix products of the time loops, in flops."""
    E, nb, _ = _mesh_nodes(c)
    return _loops(c) * c["steps"] * E * c["n_r"] * 6.0 * nb * nb * c["shots"] * (4 if c["exact_adjoint"] else 1)


def draw(rng):
    kind = rng.choice(["misfit", "forward", "session", "search", "gradient", "gradient", "gradient", "epoch", "quadtree",
                       "cube", "exact"])
    if kind == "misfit":
        return _case("misfit", shots=rng.randint(1, 16), recs=_log_int(rng, 1, 200), steps=_log_int(rng, 50, 4000))
    if kind in ("forward", "session", "search", "gradient", "exact"):
        hi = 64 if kind in ("forward", "search", "gradient") else 32
        c = _case("gradient" if kind == "exact" else kind, nx=_log_int(rng, 2, hi), ny=_log_int(rng, 2, hi),
                  p=rng.randint(1, 4), n_r=rng.randint(5, 32), shots=rng.randint(1, 8), recs=rng.randint(1, 48),
                  steps=rng.randint(40, 200), grid=rng.randint(16, 256), exact_adjoint=kind == "exact")
        if kind == "gradient":
            c["ckpt"] = rng.choice([0, 0, -1])
            c["shots"] = rng.randint(1, 12)          # beyond eight shots a pass takes another element kernel
    elif kind == "quadtree":
        p = rng.randint(2, 5)
        c = _case("gradient", mesh="quadtree", nx=rng.randint(6, 16), p=p, n_r=rng.randint(8, 48), shots=rng.randint(1, 8),
                  recs=rng.randint(4, 32), steps=rng.randint(40, 100), grid=rng.randint(64, 256))
        c["ny"] = c["nx"]
    elif kind == "cube":
        c = _case("gradient", mesh="cube", nx=rng.randint(2, 14), p=rng.randint(1, 2), n_r=rng.randint(5, 16),
                  shots=rng.randint(1, 8), recs=rng.randint(5, 40), steps=rng.randint(20, 60), grid=rng.randint(16, 64))
        c["ny"] = c["nx"]
    else:
        c = _case("epoch", mesh=rng.choice(["voronoi", "square"]), nx=_log_int(rng, 40, 800), ny=1, p=2,
                  n_r=rng.randint(6, 8), shots=rng.randint(1, 2), recs=rng.randint(10, 300), steps=rng.randint(50, 200),
                  grid=rng.randint(64, 256))
        if c["mesh"] == "square":
            c["nx"] = c["ny"] = max(3, int(math.sqrt(c["nx"])))
    most = max(_cost(x) for x in listed() if x["kind"] != "misfit" and not x["exact_adjoint"])
    while _cost(c) > 0.7 * most and c["steps"] > 8:
        c["steps"] = max(8, c["steps"] // 2)
    while _cost(c) > 0.7 * most and c["shots"] > 1:
        c["shots"] -= 1
    return c


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=4)
def _mesh_of(kind, nx, ny, p):
    """The mesh arrays; they depend on the sizes only and a program keeps them."""
    if kind == "cube":
        return mesh3d.structured_mesh3d(nx, nx, nx, p)
    if kind == "voronoi":
        return inputs.voronoi_mesh(nx, p, lx=0.1, ly=0.1, seed=3, lloyd_iters=12)
    if kind == "quadtree":
        def near_a_flaw(x0, y0, x1, y1, level):      # two circles, as the recipe refines around its flaws
            m = 0.5 * (x1 - x0)
            x, y = 0.5 * (x0 + x1), 0.5 * (y0 + y1)
            return any(math.hypot(x - cx, y - cy) < r + m for cx, cy, r in ((0.35, 0.6, 0.08), (0.7, 0.3, 0.1)))
        return inputs.quadtree_mesh(nx, 2, near_a_flaw, p)
    return inputs.structured_mesh(nx, ny, p)


def _coords(m):
    return m.node_xyz if getattr(m, "dim", 2) == 3 else m.node_xy


def _problem(case, seed):
    """Host arrays: mesh, time axis, density grid, sources, receivers, wavelets, observed traces."""
    rng = np.random.default_rng(seed)
    m = _mesh_of(case["mesh"], case["nx"], case["ny"], case["p"])
    dim, g, B, R, K = getattr(m, "dim", 2), case["grid"], case["shots"], case["recs"], case["steps"]
    if case["mesh"] == "voronoi":
        c, f0, dt, rho0, amp = 6000.0, 500e3, 0.2e-6, 2700.0, 1e12       # the plate recipe
    else:
        c, rho0, amp = 1.0, 1.0, 1.0
        ln = m.face_nodes[:, :case["p"] + 1] if dim == 3 else m.line_nodes
        s = np.linalg.norm(_coords(m)[ln[:, 1:]] - _coords(m)[ln[:, :-1]], axis=-1).min()
        f0, dt = c / (10 * s), 0.5 * s / c                               # ten nodes per dominant wavelength
    f0 = f0 * rng.uniform(0.9, 1.1)
    # density: a background with a few weak inclusions (half the density)
    ax = [(np.arange(g) + 0.5) / g] * dim
    X = np.meshgrid(*ax, indexing="ij")
    rho = np.full((g,) * dim, rho0)
    for _ in range(2):
        q, r = rng.uniform(0.2, 0.8, dim), rng.uniform(0.05, 0.15)
        rho[sum((x - t) ** 2 for x, t in zip(X, q)) <= r * r] = 0.5 * rho0
    # sources on the top side, receivers on the whole outline and next to the sources
    xy = _coords(m)
    ext = np.array([m.lx, m.ly, getattr(m, "lz", 0.0)][:dim])
    tol = 1e-9 * ext.max()
    top = np.nonzero(np.abs(xy[:, dim - 1] - ext[dim - 1]) < tol)[0]
    edge = np.nonzero(((np.abs(xy) < tol) | (np.abs(xy - ext) < tol)).any(axis=1))[0]
    src = rng.choice(top, B, replace=B > top.size)
    rec = np.unique(src)[:max(1, R // 4)]
    rec = np.concatenate([rec, rng.permutation(np.setdiff1d(edge, rec))[:R - rec.size]])[:R]
    if case["mesh"] == "voronoi":
        wav = np.stack([inputs.sine_burst(f0, dt, K, amplitude=amp * rng.uniform(0.5, 1.5)) for _ in range(B)])
    else:
        wav = np.stack([inputs.ricker(f0, dt, K, t0=rng.uniform(0.9, 1.1) / f0, amplitude=amp * rng.uniform(0.5, 1.5))
                        for _ in range(B)])
    # recorded data: one arrival per receiver at its travel time
    dist = np.linalg.norm(xy[rec][None] - xy[src][:, None], axis=-1) / c + 1.0 / f0
    t = (np.arange(1, K + 1) * dt)[None, None, :]
    a = (np.pi * f0 * (t - dist[..., None])) ** 2
    obs = 0.1 * rng.uniform(0.5, 1.5, (B, rec.size, 1)) * (1 - 2 * a) * np.exp(-a)
    return m, c, dt, rho, src.astype(np.int64), rec.astype(np.int64), wav, obs


def _lib_model(lm, m, c, rho, dt):
    return sbfwi.Model(lm, c, rho, dt, BETA, GAMMA, lx=m.lx, ly=m.ly, lz=getattr(m, "lz", 1.0))


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    if case["kind"] == "misfit":
        gen = torch.Generator(device=dev).manual_seed(seed)
        shape = (case["shots"], case["recs"], case["steps"])
        tr, ob = (torch.randn(shape, generator=gen, device=dev, dtype=torch.float64) for _ in range(2))
        return {"case": case, "traces": tr, "observed": ob}
    m, c, dt, rho, src, rec, wav, obs = _problem(case, seed)
    on = lambda a: torch.tensor(a, device=dev, dtype=torch.float64)  # noqa: E731
    s = {"case": case, "mesh": m, "c": c, "dt": dt, "rho": on(rho), "src": src, "rec": rec, "wav": on(wav), "obs": on(obs),
         "lib_mesh": sbfwi.Mesh.from_inputs(m, case["n_r"], XI0)}
    if case["kind"] not in ("search", "epoch"):       # those set a new density up in every pass
        s["model"] = _lib_model(s["lib_mesh"], m, c, s["rho"], dt)
        if case["exact_adjoint"]:
            sbfwi.set_gradient_mode(s["model"], sbfwi.GRAD_EXACT)
    if case["kind"] == "session":
        s["session"] = sbfwi.Session(s["model"], sbfwi.SESSION_FORWARD, 8, rec, window=32)
        s["lengths"] = _lengths(case)
    return s


def _lengths(case):
    """Steps of a session's requests: uneven, the longest first."""
    return [max(1, case["steps"] - 7 * k) for k in range(case["shots"])]


def run(state):
    case = state["case"]
    if case["kind"] == "misfit":
        E, res = sbfwi.misfit(state["traces"], state["observed"], 1e-3)
        return {"misfit": E, "residual": res}
    if case["kind"] == "session":
        return _run_session(state)
    model = state.get("model")
    if model is None:
        model = _lib_model(state["lib_mesh"], state["mesh"], state["c"], state["rho"], state["dt"])
    gradient = case["kind"] in ("gradient", "epoch")
    traces, fwd = sbfwi.forward(model, state["src"], state["wav"], state["rec"], keep=gradient, ckpt_every=case["ckpt"])
    if case["kind"] == "forward":
        return {"traces": traces}
    E, res = sbfwi.misfit(traces, state["obs"], state["dt"])
    if not gradient:
        return {"traces": traces, "misfit": E}
    mode = sbfwi.GRAD_EXACT if case["exact_adjoint"] else sbfwi.GRAD_KERNEL
    g = sbfwi.adjoint_gradient(model, fwd, res, mode=mode)
    return {"traces": traces, "misfit": E, "gradient": g}


def _run_session(state):
    ses, out = state["session"], {}
    for k, n in enumerate(state["lengths"]):
        ses.admit(k, state["wav"][k, :n].contiguous(), int(state["src"][k]))
    while len(out) < len(state["lengths"]):
        for slot in ses.step():
            out[slot] = ses.collect(slot)
    return {"traces%d" % k: out[k] for k in sorted(out)}


def work(case):
    """Per step and element the three operators of every radial point are read once for all shots and multiply the
    shots' vectors, the Newmark state (two arrays) and the condensed load are read and written, and a gradient pass
    writes or reads one velocity per nodal point; the boundary factors are dense fronts of about 8 N log2 N entries."""
    if case["kind"] == "misfit":
        n = case["shots"] * case["recs"] * case["steps"]
        return {"bytes": 24.0 * n, "flops": 3.0 * n}
    E, nb, N = _mesh_nodes(case)
    B, pts = case["shots"], E * (case["n_r"] - 1)
    factors = 8.0 * N * max(1.0, math.log2(max(2.0, N)))
    field = 8.0 * nb * B if case["kind"] in ("gradient", "epoch") else 0.0
    per_step = pts * (24.0 * nb * nb + 48.0 * nb * B + field) + 8.0 * factors
    n = _loops(case) * case["steps"]
    flops = n * (pts * 6.0 * nb * nb * B + 2.0 * factors * B)
    if case["exact_adjoint"]:
        flops *= 2.0
    return {"bytes": n * per_step, "flops": flops}


# ---------------------------------------------------------------------------------------
# the same outputs in plain 64-bit torch
# ---------------------------------------------------------------------------------------
def _lagrange(p, x):
    """Shape functions of equally spaced nodes on [-1, 1] and their derivatives at x, [g][p+1]."""
    t = [-1.0 + 2.0 * k / p for k in range(p + 1)]
    phi, dphi = np.ones((x.size, p + 1)), np.zeros((x.size, p + 1))
    for a in range(p + 1):
        others = [b for b in range(p + 1) if b != a]
        for b in others:
            phi[:, a] *= (x - t[b]) / (t[a] - t[b])
        for k in others:
            term = np.full(x.size, 1.0 / (t[a] - t[k]))
            for b in others:
                if b != k:
                    term *= (x - t[b]) / (t[a] - t[b])
            dphi[:, a] += term
    return phi, dphi


def _rule(p, dim):
    """Gauss rule of one boundary line or face: weights [g], N [g][nodes], derivatives of N [dim-1][g][nodes]."""
    x, w = np.polynomial.legendre.leggauss((3 * p + 2) // 2 if dim == 2 else (3 * p + 4) // 2)
    f, d = _lagrange(p, x)
    if dim == 2:
        return w, f, d[None]
    both = lambda a, b: np.einsum("ia,jb->jiba", a, b).reshape(x.size ** 2, -1)  # noqa: E731
    return np.outer(w, w).ravel(), both(f, f), np.stack([both(d, f), both(f, d)])


class _Group:
    """Elements with the same numbers of boundary lines (faces) and nodes, batched."""

    def __init__(self, m, elems, pts):
        dim = getattr(m, "dim", 2)
        surf = m.face_nodes if dim == 3 else m.line_nodes
        ids = np.stack([surf[m.elem_ptr[e]:m.elem_ptr[e + 1]] for e in elems])              # [e][lines][nodes]
        pairs = [np.unique(i, return_inverse=True) for i in ids]
        self.dofs = torch.tensor(np.stack([u for u, _ in pairs]), device=pts)               # [e][nb]
        self.loc = torch.tensor(np.stack([v.reshape(ids.shape[1:]) for _, v in pairs]), device=pts)
        self.x = torch.tensor(_coords(m)[ids], device=pts)                                  # [e][lines][nodes][dim]
        ctr = m.centre_xyz if dim == 3 else m.centre_xy
        self.ctr = torch.tensor(ctr[np.asarray(elems)], device=pts)
        self.xn = torch.tensor(_coords(m), device=pts)[self.dofs]                           # [e][nb][dim]


def _groups(m, dev):
    surf = m.face_nodes if getattr(m, "dim", 2) == 3 else m.line_nodes
    by = {}
    for e in range(m.n_elem):
        ids = surf[m.elem_ptr[e]:m.elem_ptr[e + 1]]
        by.setdefault((ids.shape[0], np.unique(ids).size), []).append(e)
    return [_Group(m, v, dev) for _, v in sorted(by.items())]


def _interpolate(rho, x, ext):
    """Multilinear interpolation of a cell-centred grid (axes from the last coordinate to the first), clamped."""
    dim = x.shape[-1]
    base, frac = [], []
    for d in range(dim):
        n = rho.shape[dim - 1 - d]
        f = x[..., d] * n / ext[d] - 0.5
        i = f.floor().clamp(0, n - 2)
        base.append(i.long())
        frac.append((f - i).clamp(0.0, 1.0))
    out = 0.0
    for corner in range(2 ** dim):
        at, w = 0, 1.0
        for d in reversed(range(dim)):
            k = (corner >> d) & 1
            at = at * rho.shape[dim - 1 - d] + base[d] + k
            w = w * (frac[d] if k else 1.0 - frac[d])
        out = out + w * rho.reshape(-1)[at]
    return out


def _condense(grp, m, p, n, c, dt, rho):
    """The element operators of one group: per radial point P, Q, H, then R, T and the dynamic stiffness S."""
    dim = grp.x.shape[-1]
    dev, e, nb = grp.x.device, grp.dofs.shape[0], grp.dofs.shape[1]
    ext = (m.lx, m.ly, getattr(m, "lz", 0.0))
    w, N, dN = (torch.tensor(a, device=dev) for a in _rule(p, dim))
    xi = torch.tensor([XI0 + (1 - XI0) / n * i for i in range(n)] + [1.0], device=dev, dtype=torch.float64)
    h = (1 - XI0) / n
    pts = grp.ctr[:, None, None] + xi[None, :, None, None] * (grp.xn - grp.ctr[:, None])[:, None]   # [e][n+1][nb][dim]
    r = _interpolate(rho, pts, ext)
    rb = torch.einsum("ga,elad->elgd", N, grp.x) - grp.ctr[:, None, None]
    J = torch.stack([rb] + [torch.einsum("ga,elad->elgd", dN[k], grp.x) for k in range(dim - 1)], dim=-2)
    wd = w * torch.linalg.det(J)                                                            # [e][lines][g]
    Ji = torch.linalg.inv(J)                                                                # columns b1, b2, ..
    b1 = Ji[..., 0]
    B2 = sum(Ji[..., k + 1][..., None, :] * dN[k][None, None, :, :, None] for k in range(dim - 1))   # [e][l][g][a][dim]
    idx = grp.loc
    rl = torch.gather(r[:, :, None, :].expand(-1, -1, idx.shape[1], -1), 3, idx[:, None].expand(-1, n + 1, -1, -1))
    rg = torch.einsum("eila,ga->eilg", rl, N)
    kw = c * c * rg * wd[:, None]
    q11 = (b1 * b1).sum(-1)
    b21 = torch.einsum("elgad,elgd->elga", B2, b1)
    parts = [torch.einsum("eilg,elg,ga,gb->eilab", kw, q11, N, N), torch.einsum("eilg,elga,gb->eilab", kw, b21, N),
             torch.einsum("eilg,elgad,elgbd->eilab", kw, B2, B2),
             torch.einsum("eilg,ga,gb->eilab", rg * wd[:, None], N, N)]
    at = (idx[:, :, :, None] * nb + idx[:, :, None, :]).reshape(e, 1, -1).expand(-1, n + 1, -1)
    E0, E1, E2, M0 = (torch.zeros(e, n + 1, nb * nb, device=dev, dtype=torch.float64)
                      .scatter_add(2, at, q.reshape(e, n + 1, -1)).reshape(e, n + 1, nb, nb) for q in parts)

    def slope(A):
        return torch.cat([(A[:, 1:2] - A[:, :1]) / h, (A[:, 2:] - A[:, :-2]) / (2 * h), (A[:, -1:] - A[:, -2:-1]) / h], 1)

    t = lambda A: A.transpose(-1, -2)  # noqa: E731
    x = xi[None, :, None, None]
    D = (dim - 1) * E0 + t(E1) - E1 + x * slope(E0)
    mass = x * x * M0
    th, ps = x * x * E0 / (h * h) - x * D / (2 * h), x * x * E0 / (h * h) + x * D / (2 * h)
    ph = -2 * x * x * E0 / (h * h) - E2 + x * t(slope(E1)) - mass / (BETA * dt * dt) + (t(E1) if dim == 3 else 0.0)
    edge = lambda i: (-xi[i] * E0[:, i] / (2 * h), t(E1[:, i]), xi[i] * E0[:, i] / (2 * h))  # noqa: E731
    solve, right = torch.linalg.solve, lambda A, B: t(torch.linalg.solve(t(B), t(A)))       # A B^-1
    t0, p0, s0 = edge(0)
    first = right(th[:, 0], t0)
    P, Q, H = [], [], []
    phi, psi = ph[:, 0] - first @ p0, ps[:, 0] - first @ s0
    for i in range(n):
        if i:
            phi, psi = ph[:, i] - th[:, i] @ H[-1], ps[:, i]
        H.append(solve(phi, psi))
        P.append(solve(phi, mass[:, i]))
        Q.append(solve(phi, th[:, i]) if i else torch.zeros_like(phi))
    tn, pn, sn = edge(n)
    W = right(sn, ps[:, n])
    S = pn - tn @ H[-1] - W @ (ph[:, n] - th[:, n] @ H[-1])
    return P, Q, H, W @ th[:, n] - tn, W @ mass[:, n], S, pts


def _exact_loop(m, p, n_r, c, dt, rho, dev):
    """Set-up, and a function that runs the time loop on sources [K][N][B] and gives the boundary displacements of
    every step and, where asked, calls back with the velocities of every step."""
    n, N = n_r - 1, int(m.n_nodes)
    groups = _groups(m, dev)
    ops = [_condense(g, m, p, n, c, dt, rho) for g in groups]
    A = torch.zeros(N * N, device=dev, dtype=torch.float64)
    for g, o in zip(groups, ops):
        A = A.index_add(0, (g.dofs[:, :, None] * N + g.dofs[:, None, :]).reshape(-1), o[5].reshape(-1))
    A = A.reshape(N, N)
    if not rho.requires_grad:
        lu = torch.linalg.lu_factor(A)
        back = lambda F: torch.linalg.lu_solve(*lu, F)  # noqa: E731
    else:
        inv = torch.linalg.inv(A)
        back = lambda F: inv @ F  # noqa: E731
    a0, a1, a2 = 1 / (BETA * dt * dt), 1 / (BETA * dt), 1 / (2 * BETA) - 1

    def loop(source, K, B, seen=None):
        zero = lambda *s: torch.zeros(*s, device=dev, dtype=torch.float64)  # noqa: E731
        parts = [zero(n, g.dofs.shape[0], g.dofs.shape[1], B) for g in groups]
        u, ud, udd = list(parts), list(parts), list(parts)
        ub = udb = uddb = zero(N, B)
        out = []

        def newmark(new, x, xd, xdd):
            acc = a0 * (new - x) - a1 * xd - a2 * xdd
            return xd + dt * ((1 - GAMMA) * xdd + GAMMA * acc), acc

        for k in range(K):
            F = source(k)
            vb = a0 * ub + a1 * udb + a2 * uddb
            qs = []
            for j, (g, (P, Q, H, R, T, S, _)) in enumerate(zip(groups, ops)):
                v = a0 * u[j] + a1 * ud[j] + a2 * udd[j]
                q = [-(P[0] @ v[0])]
                for i in range(1, n):
                    q.append(-(P[i] @ v[i] + Q[i] @ q[-1]))
                qs.append(q)
                f = R @ q[-1] + T @ vb[g.dofs]
                F = F.index_add(0, g.dofs.reshape(-1), f.reshape(-1, B))
            new = back(F)
            for j, (g, (P, Q, H, R, T, S, _)) in enumerate(zip(groups, ops)):
                x, ui = new[g.dofs], [None] * n
                for i in range(n - 1, -1, -1):
                    x = ui[i] = qs[j][i] - H[i] @ x
                ui = torch.stack(ui)
                vel, acc = newmark(ui, u[j], ud[j], udd[j])
                u[j], ud[j], udd[j] = ui, vel, acc
            udb, uddb = newmark(new, ub, udb, uddb)
            ub = new
            out.append(ub)
            if seen is not None:
                seen(k, ud, udb)
        return out

    return groups, ops, loop


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "misfit":
        s = prepare(case, seed)
        d = s["observed"] - s["traces"]
        return {"misfit": 0.5e-3 * float((d * d).sum()), "residual": d}
    E, nb, N = _mesh_nodes(case)
    stored = 8.0 * case["steps"] * E * case["n_r"] * nb * case["shots"]
    # the dense boundary system, the batched element products and the kept velocities bound what 20 seconds allow
    if N > 14000 or _loops(case) * case["steps"] * case["n_r"] > 40000 or stored > 2e10:
        return None
    m, c, dt, rho, src, rec, wav, obs = _problem(case, seed)
    ext, (B, K) = (m.lx, m.ly, getattr(m, "lz", 0.0)), wav.shape
    on = lambda a: torch.tensor(a, device=dev)  # noqa: E731
    rho, src, rec, wav, obs = on(rho), on(src), on(rec), on(wav), on(obs)
    auto = case["exact_adjoint"]
    if auto and (stored > 3e9 or N > 4500):
        return None
    rho.requires_grad_(auto)
    groups, ops, loop = _exact_loop(m, case["p"], case["n_r"], c, dt, rho, dev)
    shots = torch.arange(B, device=dev)
    blank = torch.zeros(int(m.n_nodes), B, device=dev, dtype=torch.float64)
    shot_source = lambda k: blank.index_put((src, shots), wav[:, k])  # noqa: E731
    gradient, kept = case["kind"] in ("gradient", "epoch"), {}

    def keep(k, ud, udb):
        kept[k] = (list(ud), udb)

    ub = loop(shot_source, K, B, keep if gradient and not auto else None)
    traces = torch.stack([x[rec].T for x in ub], dim=-1)
    if case["kind"] == "session":
        return {"traces%d" % k: traces[k, :, :n].detach() for k, n in enumerate(_lengths(case))}
    if case["kind"] == "forward":
        return {"traces": traces}
    res = obs - traces
    value = 0.5 * dt * (res * res).sum()
    out = {"traces": traces.detach(), "misfit": float(value.detach())}
    if not gradient:
        return out
    if auto:
        value.backward()
        return {**out, "gradient": rho.grad}
    # the paper's kernel: dt times the sum of forward and reversed-time adjoint velocities, on the nodal points
    acc = [torch.zeros(g.dofs.shape[0], g.dofs.shape[1], len(o[0]), device=dev, dtype=torch.float64)
           for g, o in zip(groups, ops)]
    acc_b = torch.zeros(int(m.n_nodes), device=dev, dtype=torch.float64)

    def correlate(k, ud, udb):
        fwd, fwd_b = kept.pop(K - 1 - k)
        for a, x, y in zip(acc, fwd, ud):
            a += (x * y).sum(-1).permute(1, 2, 0)
        acc_b.add_((fwd_b * udb).sum(-1))

    loop(lambda k: blank.index_put((rec,), res[:, :, K - 1 - k].T), K, B, correlate)
    # the transpose of the grid interpolation, by differentiating it
    grid = rho.detach().clone().requires_grad_(True)
    total = (_interpolate(grid, torch.tensor(_coords(m), device=dev), ext) * acc_b).sum()
    for a, o in zip(acc, ops):
        total = total + (_interpolate(grid, o[6][:, :-1], ext) * a.permute(0, 2, 1)).sum()
    total.backward()
    return {**out, "gradient": dt * grid.grad}

