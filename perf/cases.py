"""What the framework is used for, as cases to time.

A case is one pass of a program that has a handle, a model and observed data:
it sets the coefficients, runs the forward solve, the functional, the adjoint
solve and fetches the gradient (or the same through a batch, torch's autograd or the
conjugate gradient loop).  Grids, FEM cubes, detector grids and options are those of
this repository's workloads, tests and benchmark; the long runs are cut to fewer steps,
with a pulse early enough that the wave crosses the FEM cube and its adjoint meets it.

Handles of FP32 fields hand their results over in doubles; a program that works with
FP32 keeps them as FP32, and so does run() here.

The reference values of exact() come from a separate torch FP64 solver at the end.
"""
import math
import random

import numpy as np
import torch

import paper_2508_07780_gb300 as ddfd
from paper_2508_07780_gb300.autograd import ddfd_loss

DEV = "cuda"


def listed():
    short = dict(t0=0.2, width=0.07, freq=5.0)    # pulses of the runs cut to a short horizon
    shorter = dict(t0=0.1, width=0.035, freq=10.0)
    full = dict(t0=0.75, width=0.25, freq=2.0)    # the library's default pulse
    return [
        # the allocation-free misfit of a caller that owns every buffer: the smallest call
        dict(name="misfit_41", kind="misfit", n_src=1, steps=300, n_det=64),
        # a smoke-sized inversion step, FP64: launches and host calls
        dict(name="fp64_13", kind="pass", prec="fp64", n=13, fem=9, steps=40, det=3, **full),
        # the plain FP64 workload in full: 41^3, FEM cube 21^3, 300 steps, 64 detectors
        dict(name="fp64_41", kind="pass", prec="fp64", n=41, fem=21, steps=300, det=8, **full),
        # the same problem on FP32 fields, two oblique waves summed by one handle
        dict(name="fp32_41_2src", kind="pass", prec="fp32", n=41, fem=21, steps=300, det=8, n_src=2, oblique=True,
             **full),
        # an even, ragged grid with a regulariser, absorbing side faces and the sine pulse
        dict(name="fp32_100_ragged", kind="pass", prec="fp32", n=100, fem=63, steps=200, det=16, sides=True, gamma=1e-3,
             sine=True, **short),
        # one FP64 member of the batch workload (161^3, FEM cube 121^3): the reference arm of FP32
        dict(name="fp64_161", kind="pass", prec="fp64", n=161, fem=121, steps=160, det=32, **short),
        # the single-source FP32 workload: 201^3, FEM cube 101^3, 1024 detectors
        dict(name="fp32_201", kind="pass", prec="fp32", n=201, fem=101, steps=460, det=32, **shorter),
        # the differentiable run: 301^3, FEM cube 151^3, checkpointed, through torch's autograd
        dict(name="fp32_301_loss", kind="loss", prec="fp32", n=301, fem=151, steps=700, det=32, snapshots=32,
             **shorter),
        # the headline batch: 16 oblique waves on 161^3, FEM cubes 61 / 81 / 101 / 121
        dict(name="batch16_161", kind="batch", prec="fp32", n=161, members=16, fem=121, steps=400, det=32, oblique=True,
             **shorter),
        # element gather over the explicit Kuhn tetrahedra
        dict(name="ebe_81", kind="pass", prec="fp32", n=81, fem=41, steps=240, det=16, ebe=True, **short),
        # a locally refined FEM mesh with new nodes (the time step of refined runs)
        dict(name="mesh_81", kind="pass", prec="fp32", n=81, fem=41, steps=280, det=16, refine=16, cfl=0.25, **short),
        # conjugate gradient iterations over four incident waves, from and to host arrays
        dict(name="cg_4x65", kind="cg", prec="fp32", n=65, members=4, fem=33, steps=160, det=16, oblique=True, iters=2,
             **short),
    ]


def _weight(c):
    """Rough cost of a pass in FP32 node steps, to keep drawn cases below the largest listed one."""
    per = 24.0 if c["prec"] == "fp64" else 1.0
    per *= 12.0 if c.get("ebe") or c.get("refine") else 1.5 if c.get("snapshots") or c.get("literal") else 1.0
    return per * (c["n"] + 20) ** 3 * c["steps"] * c.get("n_src", 1) * c.get("members", 1) * c.get("iters", 1)


def draw(rng):
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    kind = rng.choice(["pass"] * 6 + ["batch"] * 2 + ["element", "cg", "misfit", "loss"])
    if kind == "misfit":
        return dict(kind="misfit", n_src=rng.randint(1, 8), steps=log(40, 2000), n_det=log(4, 1024))
    top = dict(batch=161, element=97, cg=81).get(kind, 301)
    prec = rng.choice(["fp32", "fp32", "fp64"])
    n = log(13, top if prec == "fp32" else min(top, 161))
    part = rng.uniform(0.35 if n < 160 else 0.5, 0.78)
    t0 = 0.2 if n < 120 else 0.1
    # the horizon lets the wave reach the FEM cube and its adjoint meet it there
    c = dict(kind=kind, prec=prec, n=n, fem=max(7, min(n - 2, int(n * part))), det=max(2, min(32, n // 5)),
             steps=max(log(40, 400), int((1 - part + 2.2 * t0) * (n - 1) / 0.3)), oblique=rng.random() < 0.5,
             sine=rng.random() < 0.2, sides=rng.random() < 0.25, gamma=rng.choice([0.0, 0.0, 1e-3]),
             t0=t0, width=0.35 * t0, freq=1.0 / t0)
    if kind == "batch":
        c["members"] = log(2, 18)
    elif kind == "cg":
        c.update(members=rng.randint(2, 6), iters=rng.randint(1, 3), gamma=0.0)
    elif kind == "element":
        c["kind"] = "pass"
        c["cfl"] = 0.25
        if rng.random() < 0.5:
            c["ebe"] = True
        else:
            c["refine"] = max(1, (c["fem"] - 6) // 2)
    else:
        if rng.random() < 0.25:
            c["n_src"] = rng.randint(2, 3)
        option = rng.choice(["", "", "snapshots", "literal"])
        if option == "snapshots" or n > 220:
            c["snapshots"] = rng.randint(4, 24)
        elif option == "literal":
            c["literal"] = True
    most = 0.9 * max(_weight(x) for x in listed() if "prec" in x)
    for key, least in (("members", 2), ("n_src", 1), ("steps", 8)):  # the horizon is cut last: a wave has to reach the cube
        while c.get(key, 0) > least and _weight(c) > most:
            c[key] -= max(1, c[key] // 20)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


def _box(c, fem):
    a = (c["n"] - fem) // 2
    return a, a + fem - 1


def _members(c):
    """FEM cube sizes of the problems of a case (a batch mixes four sizes)."""
    m = c.get("members", 1)
    if c["kind"] != "batch":
        return [c["fem"]] * m
    return [max(5, c["fem"] * f // 121) | 1 for f in (61, 81, 101, 121)][:4] * (m // 4) + \
        [max(5, c["fem"] * f // 121) | 1 for f in (61, 81, 101, 121)][:m % 4]


def _model(n, fem, rng, inclusions):
    """Layered skin (three layers) with ellipsoidal inclusions on the free nodes, x fastest."""
    a = (n - fem) // 2
    x = torch.arange(a + 2, a + fem - 2, device=DEV, dtype=torch.float64) / (n - 1)
    lo, hi = (a + 2) / (n - 1), (a + fem - 3) / (n - 1)
    eps = torch.empty(len(x), len(x), len(x), device=DEV, dtype=torch.float64)
    sig = torch.empty_like(eps)
    frac = (x - lo) / max(hi - lo, 1e-9)
    for sel in (frac >= 0.9, (frac < 0.9) & (frac >= 0.55), frac < 0.55):
        eps[sel] = rng.uniform(4, 12)
        sig[sel] = rng.uniform(0, 0.5)
    for _ in range(inclusions):
        r = [rng.uniform(0.1, 0.2) for _ in range(3)]
        m = [rng.uniform(min(lo + q, (lo + hi) / 2), max(hi - q, (lo + hi) / 2)) for q in r]
        e, s = rng.uniform(15, 25), rng.uniform(0.5, 1)
        inside = (((x[None, None, :] - m[0]) / r[0]) ** 2 + ((x[None, :, None] - m[1]) / r[1]) ** 2
                  + ((x[:, None, None] - m[2]) / r[2]) ** 2) <= 1
        eps[inside] = e
        sig[inside] = s
    return eps.reshape(-1), sig.reshape(-1)


def _detectors(c, fem):
    a, b = _box(c, fem)
    q = np.arange(c["det"])
    pos = np.floor(a + (b - a) * (q + 0.5) / c["det"] + 0.5).astype(np.int32)
    jj, ii = np.meshgrid(pos, pos, indexing="ij")
    return np.stack([ii.ravel(), jj.ravel()], axis=1).astype(np.int32)


def _refined(c):
    """The Kuhn split of the FEM cube with the body diagonals of the central `refine`^3
    cubes bisected (the first bisection of a marked cube: its six tetrahedra become
    twelve).  (parents, tets) in the library's node numbering."""
    n, (a, b) = c["n"], _box(c, c["fem"])
    p = np.arange(a, b)
    k, j, i = (v.ravel() for v in np.meshgrid(p, p, p, indexing="ij"))
    nid = lambda i, j, k: i + n * (j + n * k)  # noqa: E731
    lo = a + (b - a - c["refine"]) // 2
    mark = np.ones(i.size, bool)
    for v in (i, j, k):
        mark &= (v >= lo) & (v < lo + c["refine"]) & (v >= a + 3) & (v < b - 3)
    base, far = nid(i, j, k), nid(i + 1, j + 1, k + 1)
    parents = np.stack([base[mark], far[mark]], axis=1)
    new = np.full(i.size, -1, np.int64)
    new[mark] = n ** 3 + np.arange(mark.sum())
    tets = []
    for pm in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        step = (1, n, n * n)
        v1 = base + step[pm[0]]
        v2 = v1 + step[pm[1]]
        whole = np.stack([base, v1, v2, far], axis=1)
        tets.append(whole[~mark])
        for keep in ((base, v1, v2, new), (new, v1, v2, far)):
            tets.append(np.stack(keep, axis=1)[mark])
    return parents.astype(np.int32), np.concatenate(tets).astype(np.int32)


def _inputs(c, seed):
    """The problems of a case: configurations, models and observed data, from the seed."""
    rng = random.Random(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    fems, ns = _members(c), c.get("n_src", 1)
    n, nt, cfl = c["n"], c["steps"], c.get("cfl", 0.3)
    tau = cfl / (n - 1)
    mesh = _refined(c) if c.get("refine") else None
    if c["kind"] == "cg":  # one physical model seen by every wave
        model = _model(n, fems[0], rng, 0)
    out = []
    for fem in fems:
        if c["kind"] != "cg":
            model = _model(n, fem, rng, rng.randint(1, 3))
        eps, sig = model
        if mesh is not None:  # new nodes: the mean of their parents
            a, _ = _box(c, fem)
            g = torch.as_tensor(mesh[0], device=DEV).long()
            nf = fem - 4
            at = (g % n - a - 2) + nf * ((g // n % n - a - 2) + nf * (g // (n * n) - a - 2))
            eps, sig = torch.cat([eps, eps[at].mean(1)]), torch.cat([sig, sig[at].mean(1)])
        dirs = np.array([[0.0, 0.0, -1.0]] * ns)
        if c.get("oblique"):
            for s in range(ns):
                ct, ph = rng.uniform(0.3, 1.0), rng.uniform(0, 2 * math.pi)
                st = math.sqrt(1 - ct * ct)
                dirs[s] = (st * math.cos(ph), st * math.sin(ph), -ct)
        cfg = dict(n=n, fem_n=fem, n_steps=nt, cfl=cfl, precision=c["prec"], src_dir=dirs, det_ij=_detectors(c, fem),
                   freq=c["freq"], t0=c["t0"], width=c["width"], source_kind=1 if c.get("sine") else 0,
                   gamma_eps=c.get("gamma", 0.0), gamma_sig=c.get("gamma", 0.0), n_snapshots=c.get("snapshots", 0))
        if c.get("sides"):
            cfg["absorbing_faces"] = 63
        if c.get("literal"):
            cfg["grad_variant"] = "literal"
        if c.get("ebe"):
            cfg["fem_kind"] = 1
        if mesh is not None:
            cfg["mesh"] = mesh
        # observations: the pulse with a detector-wise amplitude, a delay and 1 % noise
        t = torch.arange(nt + 1, device=DEV, dtype=torch.float64) * tau - c["t0"] - rng.uniform(0.0, 0.05)
        wave = 0.05 * torch.cos(2 * math.pi * c["freq"] * t) * torch.exp(-(t / c["width"]) ** 2)
        nd = c["det"] ** 2
        amp = 1 + 0.1 * torch.randn(ns, 1, nd, 3, generator=gen, device=DEV, dtype=torch.float64)
        amp = amp * torch.tensor([0.1, 1.0, 0.1], device=DEV, dtype=torch.float64)
        noise = 1 + 0.01 * torch.randn(ns, nt + 1, nd, 3, generator=gen, device=DEV, dtype=torch.float64)
        out.append(dict(cfg=cfg, eps=eps, sig=sig, eobs=(amp * wave[None, :, None, None] * noise).contiguous()))
    return out


def _misfit_inputs(c, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    shape = (c["n_src"], c["steps"] + 1, c["n_det"], 3)
    trace = torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64)
    return trace, trace + 0.1 * torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64)


def _cg_params(ge, gs, h3):
    """Step sizes from a first gradient, as a reconstruction sets them: the first update moves
    eps by half a unit at most and sigma by a twentieth, gamma^0 = 1 / alpha^0."""
    a = [float("%.1e" % (step * h3 / max(float(g.abs().max()), 1e-300))) for step, g in ((0.5, ge), (0.05, gs))]
    return dict(alpha_eps0=a[0], alpha_sig0=a[1], gamma_eps0=1 / a[0], gamma_sig0=1 / a[1], eps_max=30.0, sig_max=5.0)


def prepare(case, seed):
    c = case
    if c["kind"] == "misfit":
        trace, eobs = _misfit_inputs(c, seed)
        return dict(case=c, trace=trace, eobs=eobs, J=torch.empty(1, device=DEV, dtype=torch.float64))
    P = _inputs(c, seed)
    torch.cuda.synchronize()
    st = dict(case=c, P=P, type=torch.float32 if c["prec"] == "fp32" else torch.float64)
    if c["kind"] in ("batch", "cg"):
        st["batch"] = ddfd.Batch([p["cfg"] for p in P])
        if c["kind"] == "cg":
            _, _, g = _batch_pass(st["batch"], P)
            st["params"] = _cg_params(sum(v[0] for v in g), sum(v[1] for v in g), (1.0 / (c["n"] - 1)) ** 3)
            st["host"] = ([p["eobs"].cpu().numpy() for p in P], P[0]["eps"].cpu().numpy(), P[0]["sig"].cpu().numpy())
    else:
        st["problem"] = ddfd.Problem(**P[0]["cfg"])
    return st


# ---------------------------------------------------------------------------
# passes
# ---------------------------------------------------------------------------


def _like_trace(h):
    return torch.empty(h.trace_shape, device=DEV, dtype=torch.float64)


def _batch_pass(b, P):
    for h, p in zip(b.members, P):
        h.set_coeffs_dev(p["eps"], p["sig"])
    traces = b.forward_dev([_like_trace(h) for h in b.members])
    J = [h.functional_dev(p["eobs"]) for h, p in zip(b.members, P)]
    b.adjoint_dev([p["eobs"] for p in P])
    grads = []
    for h in b.members:
        g = torch.empty(2, h.n_free, device=DEV, dtype=torch.float64)
        h.gradient_dev(g[0], g[1])
        grads.append(g)
    return J, traces, grads


def run(state):
    c = state["case"]
    if c["kind"] == "misfit":
        ddfd.misfit_noalloc(state["trace"], state["eobs"], c["n_src"], c["steps"], c["n_det"], 1e-3, 0.1, state["J"])
        return state["J"]
    P, kept = state["P"], state["type"]
    if c["kind"] == "pass":
        h, p = state["problem"], P[0]
        h.set_coeffs_dev(p["eps"], p["sig"])
        trace = h.forward_dev(_like_trace(h))
        J = h.functional_dev(p["eobs"])
        h.adjoint_dev(p["eobs"])
        ge = torch.empty(h.n_free, device=DEV, dtype=torch.float64)
        gs = torch.empty_like(ge)
        h.gradient_dev(ge, gs)
        return dict(trace=trace.to(kept), J=torch.tensor(J, dtype=kept), g_eps=ge.to(kept), g_sig=gs.to(kept))
    if c["kind"] == "loss":
        p = P[0]
        eps, sig = p["eps"].requires_grad_(), p["sig"].requires_grad_()
        loss = ddfd_loss(eps, sig, state["problem"], p["eobs"])
        g = torch.autograd.grad(loss, (eps, sig))
        return dict(J=loss.detach().to(kept), g_eps=g[0].to(kept), g_sig=g[1].to(kept))
    if c["kind"] == "batch":
        J, traces, grads = _batch_pass(state["batch"], P)
        return dict(J=torch.tensor(J, dtype=kept), traces=[t.to(kept) for t in traces], grads=[g.to(kept) for g in grads])
    eobs, eps0, sig0 = state["host"]
    eps, sig, log = state["batch"].cg_run(eobs, eps0, sig0, max_iter=c["iters"], **state["params"])
    return dict(eps=torch.from_numpy(eps).to(kept), sig=torch.from_numpy(sig).to(kept),
                J=torch.tensor([r["J"] for r in log], dtype=kept),
                norms=torch.tensor([(r["gnorm_eps"], r["gnorm_sig"]) for r in log], dtype=kept))


def work(case):
    """Bytes and operations of one pass.  Inputs (coefficients, observed data) are read
    and outputs (trace, gradient) written once; E on the free nodes is written by the
    forward solve for the adjoint, which reads it.  Where the two field levels and the
    coefficients are larger than the 126 MB of L2, every time step also reads two levels
    and writes one (and a replayed step of a checkpointed run does so again).  Operations:
    per component, 9 for a finite-difference node, 27 for a node of the FEM cube."""
    c = case
    if c["kind"] == "misfit":
        v = c["n_src"] * (c["steps"] + 1) * c["n_det"] * 3
        return dict(bytes=16 * v + 8, flops=3 * v)
    e = 4 if c["prec"] == "fp32" else 8
    n3, nt, rounds = c["n"] ** 3, c["steps"], c.get("iters", 1) * c.get("n_src", 1)
    total, flops = 0, 0
    fems = _members(c)
    resident = 9 * e * n3 * len(fems) <= 126e6
    for fem in fems:
        free, inner, obs = (fem - 4) ** 3, (fem - 2) ** 3, 8 * 3 * c["det"] ** 2 * (nt + 1)
        new = c.get("refine", 0) ** 3
        sweeps = 3 if c.get("snapshots") else 2
        total += rounds * 3 * obs + 32 * (free + new) + rounds * 2 * nt * 3 * e * (free + new)
        if not resident:
            total += rounds * nt * sweeps * (9 * e * n3 + 2 * e * inner)
        flops += rounds * nt * sweeps * 3 * (9 * n3 + 18 * inner + 24 * new) + rounds * nt * 24 * (free + new)
    return dict(bytes=total, flops=flops)


# ---------------------------------------------------------------------------
# the same in torch, 64 bits
# ---------------------------------------------------------------------------


class _Solver:
    """The scheme written with whole-array operations on (3, n, n, n) fields (z, y, x)."""

    def __init__(self, p):
        cfg = p["cfg"]
        self.n, self.nt = cfg["n"], cfg["n_steps"]
        n = self.n
        self.h = 1.0 / (n - 1)
        self.tau = cfg["cfl"] * self.h
        self.a = (n - cfg["fem_n"]) // 2
        self.b = self.a + cfg["fem_n"] - 1
        self.fs = slice(self.a + 2, self.b - 1)
        self.nf = cfg["fem_n"] - 4
        self.cfg, self.dirs = cfg, cfg["src_dir"]
        self.faces = cfg.get("absorbing_faces", 3)
        self.literal = cfg.get("grad_variant") == "literal"
        self.mesh = cfg.get("mesh")
        self.nodes = n ** 3 + (len(self.mesh[0]) if self.mesh else 0)
        self.det = torch.as_tensor(cfg["det_ij"], device=DEV).long()
        if self.mesh:
            self._mesh()

    def _mesh(self):
        n = self.n
        par, tets = (torch.as_tensor(v, device=DEV).long() for v in self.mesh)
        at = torch.arange(n ** 3, device=DEV)
        X = torch.stack([at % n, at // n % n, at // (n * n)], 1).double()
        X = torch.cat([X, X[par].mean(1)])
        V = X[tets]
        A = torch.cat([torch.ones_like(V[..., :1]), V], -1)
        self.g = torch.linalg.inv(A)[:, 1:, :].transpose(1, 2).contiguous()     # (T, 4, 3), units of 1/h
        self.vol = torch.linalg.det(V[:, 1:] - V[:, :1]).abs() / 6
        self.tets = tets
        m = torch.zeros(self.nodes, device=DEV, dtype=torch.float64)
        m.index_add_(0, tets.reshape(-1), (self.vol / 4).repeat_interleave(4))
        i, j, k = X[:, 0], X[:, 1], X[:, 2]
        rows = torch.ones(self.nodes, device=DEV, dtype=torch.bool)
        for v in (i, j, k):
            rows &= (v > self.a) & (v < self.b)
        self.rows, self.m = rows, torch.where(rows, m, torch.ones_like(m))

    def coeffs(self, eps, sig):
        n = self.n
        full = lambda v, x: torch.full((self.nodes,), v, device=DEV, dtype=torch.float64).index_put_((self.free(),), x)  # noqa: E731,E501
        self.eps, self.sig = full(1.0, eps), full(0.0, sig)
        self.s = self.eps - 1
        self.g3 = lambda v: v[..., : n ** 3].unflatten(-1, (n, n, n))

    def free(self):
        n = self.n
        r = torch.arange(self.a + 2, self.b - 1, device=DEV)
        grid = (r[None, None, :] + n * (r[None, :, None] + n * r[:, None, None])).reshape(-1)
        return torch.cat([grid, torch.arange(n ** 3, self.nodes, device=DEV)])

    def lap(self, E):
        P = torch.nn.functional.pad(E[None], (1, 1, 1, 1, 1, 1), mode="reflect")[0]
        m = slice(1, -1)
        return 6 * E - (P[:, m, m, 2:] + P[:, m, m, :-2] + P[:, m, 2:, m] + P[:, m, :-2, m] + P[:, 2:, m, m] + P[:, :-2, m, m])

    PERMS = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))

    def divs(self, w):
        """Divergences (times h) of the six tetrahedra of every cube of the FEM box."""
        r = w[:, self.a: self.b + 1, self.a: self.b + 1, self.a: self.b + 1]
        d = [r[0].diff(dim=2), r[1].diff(dim=1), r[2].diff(dim=0)]
        L = r.shape[1]

        def at(p, o):  # edge difference along p starting at cube corner offset o (x, y, z)
            v = d[p]
            return v[tuple(slice(o[ax], o[ax] + L - 1) for ax in (2, 1, 0))]

        out = []
        for pm in self.PERMS:
            o, acc = [0, 0, 0], 0
            for p in pm:
                acc = acc + at(p, o)
                o[p] += 1
            out.append(acc)
        return out

    def gauss(self, w):
        """(1/6) sum_K g_a (div w)_K at the nodes strictly inside the FEM cube, zero elsewhere."""
        dv = self.divs(w)
        L = self.b - self.a + 1
        out = torch.zeros_like(w)
        for c in range(3):
            shape = [L, L, L]
            shape[2 - c] = L - 1
            edge = torch.zeros(shape, device=DEV, dtype=torch.float64)
            for pm, q in zip(self.PERMS, dv):
                o = [0, 0, 0]
                for p in pm:
                    if p == c:
                        edge[tuple(slice(o[ax], o[ax] + L - 1) for ax in (2, 1, 0))] += q
                    o[p] += 1
            e = -edge.diff(dim=2 - c)                     # flux(below) - flux(above) at inner nodes
            cut = [slice(1, -1)] * 3
            cut[2 - c] = slice(None)
            i = slice(self.a + 1, self.b)
            out[c, i, i, i] = e[tuple(cut)] / 6
        return out

    def apply(self, E, adj):
        """R = h^2 M^-1 K E (forward) or its transpose, and q = h^2 M^-1 D^T D E (adjoint)."""
        if not self.mesh:
            E3, s3 = self.g3(E), self.g3(self.s)
            if adj:
                q = self.gauss(E3)
                return (self.lap(E3) + s3 * q).flatten(1), q.flatten(1)
            return (self.lap(E3) + self.gauss(s3 * E3)).flatten(1), None
        R = torch.zeros(3, self.nodes, device=DEV, dtype=torch.float64)
        R[:, : self.n ** 3] = self.lap(self.g3(E)).flatten(1)
        Ev = E[:, self.tets]                                              # (3, T, 4)
        gg = torch.einsum("tac,tbc->tab", self.g, self.g) * self.vol[:, None, None]
        lapl = torch.einsum("tab,ctb->cta", gg, Ev)
        sv = torch.ones_like(self.g[..., 0]) if adj else self.s[self.tets]
        div = torch.einsum("tbc,ctb,tb->t", self.g, Ev, sv) * self.vol
        q = self.g.permute(2, 0, 1) * div[None, :, None]
        at = self.tets.reshape(-1)
        add = lambda v: torch.zeros_like(R).index_add_(1, at, v.reshape(3, -1)) / self.m  # noqa: E731
        q = add(q)
        F = add(lapl) + (self.s if adj else 1.0) * q
        return torch.where(self.rows, F, R), torch.where(self.rows, q, torch.zeros_like(q))

    # sources and boundary
    def wave(self, s):
        n, k = self.n, self.dirs[s] / np.linalg.norm(self.dirs[s])
        p = np.array([0.0, 1.0, 0.0]) - k[1] * k
        p /= np.linalg.norm(p)
        x = torch.arange(n, device=DEV, dtype=torch.float64) * self.h - 0.5
        d = float(k[0]) * x[None, :] + float(k[1]) * x[:, None]
        d = d - d.min()
        c = self.cfg
        end = 1 / c["freq"] if c["source_kind"] else c["t0"] + 3 * c["width"]
        n1 = math.floor((end + float(d.max())) / self.tau + 1e-9)
        return d, p, n1

    def pulse(self, t):
        c = self.cfg
        if c["source_kind"]:
            return torch.where((t > 0) & (t < 1 / c["freq"]), torch.sin(2 * math.pi * c["freq"] * t), torch.zeros_like(t))
        t = t - c["t0"]
        return torch.sin(2 * math.pi * c["freq"] * t) * torch.exp(-(t / c["width"]) ** 2)

    def damping(self, step, n1):
        f = torch.zeros(self.n, self.n, self.n, device=DEV, dtype=torch.float64)
        f[0] += bool(self.faces & 1)
        f[-1] += bool(self.faces & 2) and step > n1
        f[:, :, 0] += bool(self.faces & 4)
        f[:, :, -1] += bool(self.faces & 8)
        f[:, 0] += bool(self.faces & 16)
        f[:, -1] += bool(self.faces & 32)
        c = self.sig * self.tau / 2
        c[: self.n ** 3] += f.reshape(-1) * (self.tau / self.h)
        return c

    def dampings(self, n1):
        lo, hi = self.damping(-1, n1), self.damping(1 << 40, n1)
        return lambda step: hi if step > n1 else lo

    def forward(self, s):
        d, pol, n1 = self.wave(s)
        damp, n, r2 = self.dampings(n1), self.n, (self.tau / self.h) ** 2
        old, cur = (torch.zeros(3, self.nodes, device=DEV, dtype=torch.float64) for _ in range(2))
        at = self.free() if not self.literal else slice(None)
        at_det = self.det[:, 0] + n * (self.det[:, 1] + n * (n - 1))
        trace = torch.zeros(self.nt + 1, len(self.det), 3, device=DEV, dtype=torch.float64)
        hist = [cur[:, at]]
        for k in range(self.nt):
            R = self.apply(cur, False)[0] * r2
            if k <= n1:
                v = 2 * self.tau ** 2 / self.h * self.pulse(k * self.tau - d)
                top = R[:, : n ** 3].unflatten(-1, (n, n, n))[:, -1]
                top -= torch.as_tensor(pol, device=DEV)[:, None, None] * v
            c = damp(k)
            V = cur - old
            old, cur = cur, cur + ((self.eps - c) * V - R) / (self.eps + c)
            trace[k + 1] = cur[:, at_det].T
            hist.append(cur[:, at].clone())
        return trace, hist

    def taper(self):
        t = torch.arange(self.nt + 1, device=DEV, dtype=torch.float64) * self.tau
        T, dl = self.nt * self.tau, 0.1 * self.nt * self.tau
        z = 0.5 * (1 + torch.cos(math.pi * (t - T + dl) / dl))
        z = torch.where(t <= T - dl, torch.ones_like(t), z)
        return z

    def adjoint(self, s, trace, eobs, hist):
        _, _, n1 = self.wave(s)
        damp, n, r2, z = self.dampings(n1), self.n, (self.tau / self.h) ** 2, self.taper()
        nxt, cur = (torch.zeros(3, self.nodes, device=DEV, dtype=torch.float64) for _ in range(2))
        free = self.free()
        at = self.det[:, 0] + n * (self.det[:, 1] + n * (n - 1))
        edge = lambda v: torch.where((v == 0) | (v == n - 1), 0.5, 1.0).double()  # noqa: E731
        scale = self.tau ** 2 / self.h ** 3 / (edge(self.det[:, 0]) * edge(self.det[:, 1]) * 0.5)
        ge = torch.zeros(len(free), device=DEV, dtype=torch.float64)
        gs = torch.zeros_like(ge)
        for k in range(self.nt, 0, -1):
            R, q = self.apply(cur, True)
            R = R * r2
            j = (scale * self.tau * z[k])[:, None] * (trace[k] - eobs[k])
            R.index_add_(1, at, j.T.contiguous())
            cn, cp = damp(k + 1), damp(k - 1)
            new = (2 * self.eps * cur - R - (self.eps - cn) * nxt) / (self.eps + cp)
            E = hist[k]
            gauss = self.literal_term(E, cur) if self.literal else (E * q[:, free]).sum(0)
            E = E[:, free] if self.literal else E
            ge += (E * (new[:, free] - 2 * cur[:, free] + nxt[:, free])).sum(0) + r2 * gauss
            gs += (E * (new[:, free] - nxt[:, free])).sum(0)
            nxt, cur = cur, new
        m = torch.full_like(ge, self.h ** 3)
        if self.mesh:
            m = self.m[free] * self.h ** 3
        return ge * m / self.tau ** 2, gs * m / (2 * self.tau)

    def literal_term(self, E, mu):
        """sum_K |K|/4 div E div mu over the tetrahedra of each free node, in units of h."""
        prod = [p * q / 24 for p, q in zip(self.divs(self.g3(E)), self.divs(self.g3(mu)))]
        L = self.b - self.a + 1
        out = torch.zeros(L, L, L, device=DEV, dtype=torch.float64)
        for pm, v in zip(self.PERMS, prod):
            o = [0, 0, 0]
            for p in (None,) + pm:
                if p is not None:
                    o[p] += 1
                out[tuple(slice(o[ax], o[ax] + L - 1) for ax in (2, 1, 0))] += v
        i = slice(2, -2)
        return out[i, i, i].reshape(-1)

    def regular(self, eps, sig):
        m = self.m[self.free()] * self.h ** 3 if self.mesh else self.h ** 3
        ga = self.cfg["gamma_eps"]
        return 0.5 * ga * float((m * ((eps - 1) ** 2 + sig ** 2)).sum()), ga * m * (eps - 1), ga * m * sig

    def solve(self, eps, sig, eobs):
        self.coeffs(eps, sig)
        J, ge, gs = self.regular(eps, sig)
        ge, gs, traces = ge + 0 * eps, gs + 0 * sig, []
        for s in range(len(self.dirs)):
            trace, hist = self.forward(s)
            d = ((trace - eobs[s]) ** 2).sum((1, 2)) * self.taper()
            J += 0.5 * self.tau * float(d[1:].sum())
            e, g = self.adjoint(s, trace, eobs[s], hist)
            ge, gs = ge + e, gs + g
            traces.append(trace)
        return torch.stack(traces), J, ge, gs


def _cg(solvers, P, iters):
    """The conjugate gradient loop: Fletcher-Reeves directions, clamped updates."""
    eps, sig = P[0]["eps"].clone(), P[0]["sig"].clone()
    ref, m = (eps.clone(), sig.clone()), solvers[0].h ** 3
    first = [sv.solve(eps, sig, p["eobs"])[2:] for sv, p in zip(solvers, P)]
    C = _cg_params(sum(g[0] for g in first), sum(g[1] for g in first), m)
    gam, alp = [C["gamma_eps0"], C["gamma_sig0"]], [C["alpha_eps0"], C["alpha_sig0"]]
    hi, lo = (C["eps_max"], C["sig_max"]), (1.0, 0.0)
    d, gg_prev, Js, norms = [None, None], [0.0, 0.0], [], []
    for it in range(iters):
        J, G = 0.0, [torch.zeros_like(eps), torch.zeros_like(sig)]
        for sv, p in zip(solvers, P):
            _, Ji, e, g = sv.solve(eps, sig, p["eobs"])
            J, G = J + Ji, [G[0] + e, G[1] + g]
        new, nrm = [], []
        for q, (x, x0) in enumerate(((eps, ref[0]), (sig, ref[1]))):
            g = G[q] / m + gam[q] * (x - x0)
            J += 0.5 * gam[q] * m * float(((x - x0) ** 2).sum())
            gg = m * float((g * g).sum())
            beta = gg / gg_prev[q] if it and gg_prev[q] > 0 else 0.0
            d[q] = -g if it == 0 else -g + beta * d[q]
            new.append((x + alp[q] * d[q]).clamp(lo[q], hi[q]))
            dd, gd = m * float((d[q] * d[q]).sum()), m * float((g * d[q]).sum())
            if gam[q] > 0 and dd > 0:
                alp[q] = -gd / (gam[q] * dd)
            gam[q] = (C["gamma_eps0"], C["gamma_sig0"])[q] / math.sqrt(it + 1)
            gg_prev[q] = gg
            nrm.append(math.sqrt(gg))
        eps, sig = new
        Js.append(J)
        norms.append(nrm)
    return dict(eps=eps, sig=sig, J=torch.tensor(Js, dtype=torch.float64), norms=torch.tensor(norms, dtype=torch.float64))


def exact(case, seed):
    c = case
    if c["kind"] == "misfit":
        trace, eobs = _misfit_inputs(c, seed)
        nt, tau = c["steps"], 1e-3
        t = torch.arange(nt + 1, device=DEV, dtype=torch.float64) * tau
        dl = 0.1 * nt * tau
        z = torch.where(t <= nt * tau - dl, torch.ones_like(t), 0.5 * (1 + torch.cos(math.pi * (t - nt * tau + dl) / dl)))
        z[0] = 0
        return (0.5 * tau * (((trace - eobs) ** 2).sum((2, 3)) * z).sum()).reshape(1)
    if (c["n"] + 10.0) ** 3 * c["steps"] * c.get("members", 1) * c.get("n_src", 1) * c.get("iters", 1) > 3.5e10:
        return None  # minutes in whole-array FP64
    P = _inputs(c, seed)
    S = [_Solver(p) for p in P]
    if c["kind"] == "cg":
        return _cg(S, P, c["iters"])
    out = [s.solve(p["eps"], p["sig"], p["eobs"]) for s, p in zip(S, P)]
    if c["kind"] == "batch":
        return dict(J=torch.tensor([o[1] for o in out], dtype=torch.float64), traces=[o[0] for o in out],
                    grads=[torch.stack([o[2], o[3]]) for o in out])
    trace, J, ge, gs = out[0]
    J = torch.tensor(J, dtype=torch.float64)
    return dict(J=J, g_eps=ge, g_sig=gs) if c["kind"] == "loss" else dict(trace=trace, J=J, g_eps=ge, g_sig=gs)
