"""Performance cases of the solver: calls that a simulation program makes
through the package's public entry points, from one 1,024-DoF time step to
full-size 2D and 3D steps, with the reverse (adjoint) step, a plain PCG solve,
a single operator product and the pointwise ionic update.

A case is a dict of plain values:
  kind    "step" (Monodomain.step), "adjoint" (Monodomain.adjoint_step and
          Hierarchy.theta_gradient), "pcg" (Hierarchy.pcg_solve), "operator"
          (Hierarchy.operator_apply, level 0), "ionic" (ionic_update)
  mesh    "square", "jsquare", "jcube", "cube" or "shell" (the generators of
          workloads.py), n elements per side ("shell": n = circumferential
          elements, the longitudinal and transmural ones in proportion)
  degree, levels, group (2D/3D block agglomerates; "jsquare" bisects),
  form    V-cycle precision "f64", "f32" or "bf16s"; fine: "mf" or "bsr"
  model   "fhn", "ap" or "bo"; scheme 0 (backward Euler) or 1 (BDF2);
  steps   time steps per call

A program sets up its mesh and hierarchy once and then advances many states
with them, so prepare() keeps the hierarchy of a case (the last few cases') and
makes new states from the seed: a travelling front across the domain with its
gates, random load vectors, random loss derivatives.
"""
from __future__ import annotations

import collections
import math

import numpy as np
import torch

from paper_2602_16312_gb300 import aggmg
from paper_2602_16312_gb300 import workloads as W

MODELS = {"fhn": W.FHN, "ap": W.ALIEV_PANFILOV, "bo": W.BUENO_OROVIO}


def _case(name, kind, mesh="", n=0, degree=0, levels=0, form="", fine="", model="fhn", group=2, scheme=0, steps=1,
          rtol=1e-8):
    c = dict(kind=kind, mesh=mesh, n=n, degree=degree, levels=levels, group=group, form=form, fine=fine, model=model,
             scheme=scheme, steps=steps, rtol=rtol)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the plain float64 configuration of 1,024 DoFs: latency and launches
        _case("step_square_q1_16_f64", "step", "square", 16, 1, 2, "f64", "bsr", group=4, rtol=1e-10),
        # the benchmark workload: 2.36M DoFs, float32 matrix-free V-cycle
        _case("step_jsquare_q2_512_f32", "step", "jsquare", 512, 2, 4, "f32", "mf"),
        # the plain float64 form in 2D, ragged element count (62,500)
        _case("step_jsquare_q2_250_f64", "step", "jsquare", 250, 2, 4, "f64", "bsr"),
        # cubic elements and the paper's BDF2 scheme, two steps per call, odd size
        _case("step_jsquare_q3_101_bdf2", "step", "jsquare", 101, 3, 3, "f32", "mf", scheme=1, steps=2),
        # the full-size 3D workload: 7.08M DoFs
        _case("step_jcube_q2_64_f32", "step", "jcube", 64, 2, 4, "f32", "mf", "ap", group=4),
        # bf16-stored smoother blocks, ragged cube (27,000 elements)
        _case("step_jcube_q2_30_bf16s", "step", "jcube", 30, 2, 3, "bf16s", "mf", "ap", group=4),
        # cubic hexahedra, forward
        _case("step_cube_q3_24_f32", "step", "cube", 24, 3, 4, "f32", "mf", "ap"),
        # ventricle-like shell with the three-gate model
        _case("step_shell_bo_64_f32", "step", "shell", 64, 2, 4, "f32", "mf", "bo"),
        # one reverse step of the adjoint workload (float64 forward form)
        _case("adjoint_cube_q3_18_f64", "adjoint", "cube", 18, 3, 4, "f64", "bsr", "ap"),
        # a single linear solve with the assembled float32 smoother, odd size
        _case("pcg_jsquare_q2_181_bsr", "pcg", "jsquare", 181, 2, 3, "f32", "bsr", rtol=1e-10),
        # the float64 operator alone (outer CG product, residual checks)
        _case("operator_jcube_q2_40_f64", "operator", "jcube", 40, 2, 3, "f32", "mf", group=4),
        # the pointwise gate update of the full-size shell (5.3M DoFs)
        _case("ionic_bo_5m", "ionic", n=5308416, model="bo"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "pcg", "operator", "ionic", "adjoint"])
    if kind == "ionic":
        return _case("", kind, n=_log_int(rng, 1000, 5000000), model=rng.choice(sorted(MODELS)))
    if kind == "adjoint":
        mesh = rng.choice(["jsquare", "jcube", "cube"])
    else:
        mesh = rng.choice(["square", "jsquare", "jsquare", "jcube", "jcube", "cube", "shell"])
    degree = rng.choice([1, 2, 2, 3])
    if mesh in ("square", "jsquare"):
        n, dim = _log_int(rng, 12, {1: 300, 2: 250, 3: 160}[degree]), 2
    elif mesh == "shell":
        n, dim = 8 * _log_int(rng, 2, {1: 8, 2: 6, 3: 4}[degree]), 3
    else:
        n, dim = _log_int(rng, 5, {1: 40, 2: 28, 3: 16}[degree]), 3
    group = rng.choice([2, 4]) if n >= 12 else 2
    # coarsen until the coarsest level, solved directly, is small
    g = 3 if mesh == "jsquare" else 2 if mesh in ("cube", "shell") else group
    levels, units = 2, -(-n // g)
    while (units * (degree + 1)) ** dim > 2000:
        levels, units = levels + 1, -(-units // g)
    form = "f64" if kind == "adjoint" else rng.choice(["f64", "f32", "f32", "bf16s"])
    fine = "bsr" if form == "f64" else rng.choice(["mf", "mf", "bsr"])
    model = rng.choice(["fhn", "ap"] if kind == "adjoint" else sorted(MODELS))
    return _case("", kind, mesh, n, degree, levels, form, fine, model, group=group,
                 scheme=rng.choice([0, 0, 1]) if kind == "step" else 0, steps=rng.choice([1, 1, 2, 3]) if kind == "step" else 1,
                 rtol=1e-10 if kind == "pcg" else 1e-8)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _workload(case):
    """The workload (mesh, conductivity, maps) of a case."""
    n, p, lv, g = case["n"], case["degree"], case["levels"], case["group"]
    mesh = case["mesh"]
    if mesh == "square":
        wl = W.square_2d_fhn(n, p)
        wl.maps = W.block_hierarchy(wl.mesh.grid_shape, (g, g), lv)
    elif mesh == "jsquare":
        wl = W.jittered_square_2d(n, p, lv)
    elif mesh == "jcube":
        wl = W.jittered_cube_3d(n, p, lv, group=g)
    elif mesh == "cube":
        wl = W.cube_3d_adjoint(n, p, lv, n_sensors=1)
    elif case["model"] == "bo":
        wl = W.ventricle_shell_bo(n, 3 * n // 4, n // 8, p, lv)
    else:
        wl = W.ventricle_shell(n, 3 * n // 4, n // 8, p, lv)
    if (case["model"] == "bo") != (wl.ionic["model"] == 2):
        # the three-gate model runs in seconds: its own time step elsewhere
        wl.dt = 1e-4 if case["model"] == "bo" else 0.05
    wl.ionic = dict(MODELS[case["model"]])
    return wl


_kept = collections.OrderedDict()   # handles of the last cases, by case
_KEEP = 12


def _handles(case):
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key in _kept:
        _kept.move_to_end(key)
        return _kept[key]
    wl = _workload(case)
    adj = case["kind"] == "adjoint"
    theta = tmap = None
    if adj:
        nt = 64
        theta = np.exp(0.2 * np.random.default_rng(3).standard_normal(nt))
        tmap = (np.arange(wl.mesh.n_elements) * nt) // wl.mesh.n_elements
    mesh = aggmg.Mesh.from_workload(wl, adjoint_data=adj, theta=theta, theta_map=tmap)
    c = (1.5 if case["scheme"] == 1 else 1.0) / wl.dt
    hier = aggmg.Hierarchy(mesh, c, wl.maps, precision=case["form"], fine=case["fine"], cheb_range=wl.cheb_range)
    mask = torch.tensor(wl.stim_mask_nodal(), dtype=torch.float64, device="cuda")
    sim = None
    if case["kind"] in ("step", "adjoint"):
        sim = aggmg.Monodomain(hier, wl.dt, wl.ionic, iapp_mask=mask, iapp_value=wl.iapp_value,
                               iapp_steps=wl.iapp_steps, rtol=case["rtol"], flexible=case["form"] != "f64",
                               scheme=case["scheme"])
    h = dict(wl=wl, mesh=mesh, hier=hier, sim=sim, mask=mask, theta=theta, tmap=tmap)
    _kept[key] = h
    while len(_kept) > _KEEP:
        _kept.popitem(last=False)
    return h


def _gll(p):
    return {1: [0.0, 1.0], 2: [0.0, 0.5, 1.0],
            3: [0.0, 0.5 - 0.5 / math.sqrt(5.0), 0.5 + 0.5 / math.sqrt(5.0), 1.0]}[p]


def _grid(x, dim):
    """Tensor points (x fastest), (len(x)**dim, dim)."""
    g = np.meshgrid(*([np.asarray(x)] * dim), indexing="ij")
    return np.stack([a.ravel() for a in g[::-1]], axis=1)


def _multilinear(xi):
    """Corner shape functions (Q, 2^d) and derivatives (Q, 2^d, d) at xi."""
    q, d = xi.shape
    N, dN = np.ones((q, 2 ** d)), np.ones((q, 2 ** d, d))
    for c in range(2 ** d):
        for k in range(d):
            b = (c >> k) & 1
            v = xi[:, k] if b else 1.0 - xi[:, k]
            N[:, c] *= v
            for l in range(d):
                dN[:, c, l] *= (1.0 if b else -1.0) if l == k else v
    return N, dN


def _corners(wl, dev):
    return torch.tensor(wl.mesh.vertices[wl.mesh.elements], dtype=torch.float64, device=dev)   # (E, V, d)


def _nodes(wl, dev):
    N, _ = _multilinear(_grid(_gll(wl.degree), wl.mesh.dim))
    return torch.einsum("iv,evk->eik", torch.tensor(N, device=dev), _corners(wl, dev)).reshape(-1, wl.mesh.dim)


def _sigmoid(x):
    return 1.0 / (1.0 + torch.exp(-x))


def _front(x, rng, model):
    """A travelling front at the points x: potential and gates."""
    lo, hi = x.min(0).values, x.max(0).values
    size = float((hi - lo).max())
    d = torch.tensor(rng.standard_normal(x.shape[1]), device=x.device)
    d = d / torch.linalg.norm(d)
    s = ((x - 0.5 * (lo + hi)) @ d) / size
    at = rng.uniform(-0.2, 0.2)
    u = _sigmoid((at - s) / 0.03)
    for _ in range(3):                     # a little unevenness behind and ahead of the front
        k = torch.tensor(rng.uniform(3.0, 12.0, x.shape[1]) / size, device=x.device)
        u = u + 0.01 * torch.sin(x @ k + rng.uniform(0.0, 6.0))
    late = _sigmoid((at - 0.15 - s) / 0.06)
    if model != "bo":
        return u, 0.3 * late
    return 1.3 * u, torch.cat([1.0 - 0.9 * u.clamp(0.0, 1.0), 1.0 - 0.6 * late, 0.02 + 0.8 * u.clamp(0.0, 1.0)])


def _inputs(case, seed, wl, dev):
    """The seeded input vectors of a case (also what exact() starts from)."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "ionic":
        x = torch.tensor(rng.uniform(0.0, 1.0, (case["n"], 1)), device=dev)
        u, w = _front(x, rng, case["model"])
        return dict(u=u, w=w)
    n = wl.n_dofs
    gen = torch.Generator(device="cpu").manual_seed(int(seed))
    if case["kind"] == "pcg":
        return dict(b=torch.randn(n, dtype=torch.float64, generator=gen).to(dev))
    if case["kind"] == "operator":
        return dict(x=torch.randn(n, dtype=torch.float64, generator=gen).to(dev))
    x = _nodes(wl, dev)
    u, w = _front(x, rng, case["model"])
    out = dict(u=u, w=w, clock=int(rng.integers(0, 2)) * 50)
    if case["kind"] == "adjoint":
        out["u1"] = u + 0.02 * torch.sin(7.0 * u)
        out["ubar"] = torch.randn(n, dtype=torch.float64, generator=gen).to(dev)
        out["wbar"] = torch.randn(n, dtype=torch.float64, generator=gen).to(dev)
    return out


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "ionic":
        v = _inputs(case, seed, None, dev)
        return dict(kind="ionic", prm=dict(MODELS[case["model"]]), dt=1e-4 if case["model"] == "bo" else 0.05,
                    wrk=torch.empty_like(v["w"]), **v)
    h = _handles(case)
    v = _inputs(case, seed, h["wl"], dev)
    s = dict(kind=case["kind"], steps=case["steps"], rtol=case["rtol"], flexible=case["form"] != "f64", h=h, **v)
    if case["kind"] == "step":
        s.update(un=torch.empty_like(v["u"]), wn=torch.empty_like(v["w"]))
    elif case["kind"] == "adjoint":
        ne = h["wl"].mesh.n_elements
        s.update(ua=torch.empty_like(v["u"]), wa=torch.empty_like(v["w"]),
                 grad=torch.zeros(ne, dtype=torch.float64, device=dev),
                 gtheta=torch.zeros(len(h["theta"]), dtype=torch.float64, device=dev))
    else:
        s.update(y=torch.empty_like(v["b"] if case["kind"] == "pcg" else v["x"]))
    return s


def run(state):
    kind = state["kind"]
    if kind == "ionic":
        state["wrk"].copy_(state["w"])
        aggmg.ionic_update(state["prm"], state["dt"], state["u"], state["wrk"])
        return state["wrk"]
    h = state["h"]
    if kind == "operator":
        h["hier"].operator_apply(0, state["x"], state["y"])
        return state["y"]
    if kind == "pcg":
        state["y"].zero_()
        h["hier"].pcg_solve(state["b"], state["y"], rtol=state["rtol"], flexible=state["flexible"])
        return state["y"]
    if kind == "step":
        # the caller's state is advanced in place: start from the input state
        state["un"].copy_(state["u"])
        state["wn"].copy_(state["w"])
        h["sim"].set_clock(state["clock"])
        h["sim"].step(state["un"], state["wn"], state["steps"], iters=False)
        return dict(u=state["un"], w=state["wn"])
    state["ua"].copy_(state["ubar"])
    state["wa"].copy_(state["wbar"])
    state["grad"].zero_()
    state["gtheta"].zero_()
    h["sim"].adjoint_step(state["u"], state["w"], state["u1"], state["ua"], state["wa"], state["grad"])
    h["hier"].theta_gradient(state["grad"], state["gtheta"])
    return dict(ubar=state["ua"], wbar=state["wa"], grad=state["grad"], gtheta=state["gtheta"])


# --------------------------------------------------------------------------
# work
# --------------------------------------------------------------------------
def _elements(case):
    n = case["n"]
    if case["mesh"] == "shell":
        return n * (3 * n // 4) * (n // 8), 3
    dim = 2 if case["mesh"] in ("square", "jsquare") else 3
    return n ** dim, dim


def work(case):
    """Bytes and operations of a call that no implementation of the same
    method can do without, per element: the float64 operator's distinct
    entries (a symmetric operator: the upper triangle of the diagonal block,
    and each coupling block once for its two elements), a V-cycle's six level-0
    products (3 before, 3 after the coarse correction) with the same entries
    in the V-cycle's precision, their vectors, and the state in and out. A solve
    counts a nominal 10 iterations (2D: 20)."""
    gates = 3 if case["model"] == "bo" else 1
    if case["kind"] == "ionic":
        n = case["n"]
        return {"bytes": 8.0 * n * (1 + 2 * gates), "flops": (60.0 if gates == 3 else 12.0) * n}
    ne, dim = _elements(case)
    N = case["degree"] + 1
    B, NF = N ** dim, N ** (dim - 1)
    entries = B * (B + 1) / 2 + dim * (2 * NF * B - NF * NF)
    flops = 2.0 * (B * B + 2 * dim * (2 * NF * B - NF * NF))
    op = ne * (8.0 * entries + 16.0 * B)
    if case["kind"] == "operator":
        return {"bytes": op, "flops": ne * flops}
    st = 8.0 if case["form"] == "f64" else 4.0
    it = 20.0 if dim == 2 else 10.0
    cycle = 6.0 * ne * st * (entries + 4.0 * B)
    solve = it * (op + cycle + 8.0 * 9.0 * ne * B)
    solve_flops = it * 7.0 * ne * flops
    if case["kind"] == "pcg":
        return {"bytes": solve, "flops": solve_flops}
    state = 8.0 * ne * B * 2 * (1 + gates) + 4.0 * ne * B * (B + 1)
    if case["kind"] == "adjoint":
        forms = ne * (4.0 * B * (B + 1) + 8.0 * 2 * dim * 4 * NF * B)
        return {"bytes": solve + 2 * state + forms, "flops": solve_flops + 4.0 * forms / 8.0}
    return {"bytes": case["steps"] * (solve + state), "flops": case["steps"] * solve_flops}


# --------------------------------------------------------------------------
# 64-bit values, by dense element blocks in torch
# --------------------------------------------------------------------------
def _lagrange(nodes, x):
    """Values and derivatives (len(x), n) of the Lagrange basis at x."""
    n = len(nodes)
    v, d = np.ones((len(x), n)), np.zeros((len(x), n))
    for i in range(n):
        others = [j for j in range(n) if j != i]
        for j in others:
            v[:, i] *= (x - nodes[j]) / (nodes[i] - nodes[j])
        for m in others:
            t = np.full(len(x), 1.0 / (nodes[i] - nodes[m]))
            for j in others:
                if j != m:
                    t = t * (x - nodes[j]) / (nodes[i] - nodes[j])
            d[:, i] += t
    return v, d


def _basis(p, xi):
    """Tensor basis (Q, B) and gradients (Q, B, d) at reference points xi."""
    dim = xi.shape[1]
    one = [_lagrange(_gll(p), xi[:, k]) for k in range(dim)]
    phi = np.ones((len(xi), 1))
    for k in range(dim):
        phi = (one[k][0][:, :, None] * phi[:, None, :]).reshape(len(xi), -1)
    grads = []
    for l in range(dim):
        g = np.ones((len(xi), 1))
        for k in range(dim):
            g = (one[k][1 if k == l else 0][:, :, None] * g[:, None, :]).reshape(len(xi), -1)
        grads.append(g)
    return phi, np.stack(grads, axis=2)


class _Forms:
    """Mass blocks, and the SIPG operator c M + A as dense element blocks."""

    def __init__(self, wl, D, dev):
        self.dim, self.p = wl.mesh.dim, wl.degree
        dim, p = self.dim, self.p
        self.B = (p + 1) ** dim
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        self.t = t
        X = _corners(wl, dev)
        self.X, self.D = X, t(D)
        gx, gw = np.polynomial.legendre.leggauss(p + 2)
        gx, gw = 0.5 * (gx + 1.0), 0.5 * gw
        self.xi = _grid(gx, dim)
        wq = np.prod(_grid(gw, dim), axis=1)
        _, dN = _multilinear(self.xi)
        phi, gh = _basis(p, self.xi)
        self.phi, self.gh = t(phi), t(gh)
        J = torch.einsum("qvl,evk->eqkl", t(dN), X)
        self.wJ = t(wq)[None] * torch.linalg.det(J)
        self.Ji = torch.linalg.inv(J)
        self.vol = self.wJ.sum(1)
        self.Me = torch.einsum("eq,qi,qj->eij", self.wJ, self.phi, self.phi)
        # faces: the neighbour across local face f lists the shared corners in
        # the same order on its opposite face
        el = wl.mesh.elements
        nv = int(el.max()) + 1
        self.nbr, self.area, self.n, self.wdS, self.flux, self.tr = [], [], [], [], [], []
        keys = []
        for f in range(2 * dim):
            k, s = divmod(f, 2)
            cs = [c for c in range(2 ** dim) if ((c >> k) & 1) == s]
            keys.append(el[:, cs[0]].astype(np.int64) * nv + el[:, cs[-1]])
        for f in range(2 * dim):
            k, s = divmod(f, 2)
            other = keys[f ^ 1]
            order = np.argsort(other)
            pos = np.searchsorted(other[order], keys[f])
            hit = order[np.minimum(pos, len(order) - 1)]
            self.nbr.append(torch.tensor(np.where(other[hit] == keys[f], hit, -1), device=dev))
            fx = np.insert(_grid(gx, dim - 1), k, float(s), axis=1)
            fw = np.prod(_grid(gw, dim - 1), axis=1)
            _, dNf = _multilinear(fx)
            ph, g = _basis(p, fx)
            Jf = torch.einsum("qvl,evk->eqkl", t(dNf), X)
            Jfi = torch.linalg.inv(Jf)
            nh = np.zeros(dim)
            nh[k] = 2.0 * s - 1.0
            nvec = torch.einsum("eqlk,l->eqk", Jfi, t(nh))
            ln = torch.linalg.norm(nvec, dim=2)
            nrm = nvec / ln[..., None]
            wdS = t(fw)[None] * torch.linalg.det(Jf) * ln
            self.area.append(wdS.sum(1))
            self.n.append(nrm)
            self.wdS.append(wdS)
            self.tr.append(t(ph))
            # D grad phi_j . n at the face points
            a = torch.einsum("eqlk,ekm,eqm->eql", Jfi, self.D, nrm)
            self.flux.append(torch.einsum("qjl,eql->eqj", t(g), a))
        self.c_pen = float(p * (p + 1)) if wl.penalty_mode == 0 else float(wl.penalty_coeff) * p * p

    def _alpha(self, f, e):
        nb = self.nbr[f][e]
        return self.c_pen * torch.maximum(self.area[f][e] / self.vol[e], self.area[f][e] / self.vol[nb]), nb

    def _nDn(self, f, e, D):
        return torch.einsum("eqk,ekm,eqm->eq", self.n[f][e], D, self.n[f][e])

    def assemble(self, c):
        """Diagonal blocks, and the coupling blocks of each face's interior elements."""
        E = self.X.shape[0]
        self.diag = c * self.Me
        for s in range(0, E, 16384):
            sl = slice(s, s + 16384)
            G = torch.einsum("eqlk,ekm,eqnm->eqln", self.Ji[sl], self.D[sl], self.Ji[sl]) * self.wJ[sl][..., None, None]
            DG = torch.einsum("eqln,qjn->eqlj", G, self.gh)
            left = self.gh.permute(1, 0, 2).reshape(self.B, -1)
            self.diag[sl] += left @ DG.reshape(DG.shape[0], -1, self.B)
        self.off = []
        for f in range(2 * self.dim):
            e = torch.nonzero(self.nbr[f] >= 0).flatten()
            blk = torch.empty((len(e), self.B, self.B), dtype=torch.float64, device=self.X.device)
            for s in range(0, len(e), 32768):
                es = e[s:s + 32768]
                al, nb = self._alpha(f, es)
                sg = (al[:, None] * self._nDn(f, es, 0.5 * (self.D[es] + self.D[nb])) * self.wdS[f][es])[..., None]
                wf = self.wdS[f][es][..., None]
                ti, tj = self.tr[f], self.tr[f ^ 1]
                Fe, Fn = self.flux[f][es] * wf, -self.flux[f ^ 1][nb] * wf
                pen = torch.einsum("qi,eqj->eij", ti, sg * ti)
                con = torch.einsum("qi,eqj->eij", ti, Fe)
                self.diag[es] += pen - 0.5 * (con + con.transpose(1, 2))
                blk[s:s + 32768] = (0.5 * torch.einsum("eqi,qj->eij", Fe, tj) - 0.5 * torch.einsum("qi,eqj->eij", ti, Fn)
                                    - torch.einsum("qi,eqj->eij", ti, sg * tj))
            self.off.append((e, self.nbr[f][e], blk))

    def apply(self, x):
        x = x.view(-1, self.B, 1)
        y = self.diag @ x
        for e, nb, blk in self.off:
            y[e] += blk @ x[nb]
        return y.flatten()

    def mass(self, x):
        return (self.Me @ x.view(-1, self.B, 1)).flatten()

    def solve(self, b, x):
        """Block-Jacobi CG to the rounding level."""
        inv = torch.linalg.inv(self.diag)
        pre = lambda r: (inv @ r.view(-1, self.B, 1)).flatten()  # noqa: E731
        x = x.clone()
        for _ in range(2):                       # the second pass removes the recurrence's drift
            r = b - self.apply(x)
            z = pre(r)
            p, rz, stop = z.clone(), r @ z, 1e-15 * float(torch.linalg.norm(b))
            for it in range(3000):
                q = self.apply(p)
                a = rz / (p @ q)
                x += a * p
                r -= a * q
                if it % 10 == 9 and float(torch.linalg.norm(r)) <= stop:
                    break
                z = pre(r)
                rz, old = r @ z, rz
                p = z + (rz / old) * p
        return x

    def own_share(self, lam, u):
        """lam^T A_e u of every element e, A_e the part of A built with D_e."""
        L, U = lam.view(-1, self.B), u.view(-1, self.B)
        gl = torch.einsum("ei,qil,eqlk->eqk", L, self.gh, self.Ji)
        gu = torch.einsum("ei,qil,eqlk->eqk", U, self.gh, self.Ji)
        g = torch.einsum("eq,eqk,ekm,eqm->e", self.wJ, gl, self.D, gu)
        for f in range(2 * self.dim):
            e = torch.nonzero(self.nbr[f] >= 0).flatten()
            al, nb = self._alpha(f, e)
            jl = L[e] @ self.tr[f].T - L[nb] @ self.tr[f ^ 1].T
            ju = U[e] @ self.tr[f].T - U[nb] @ self.tr[f ^ 1].T
            fl = torch.einsum("eqj,ej->eq", self.flux[f][e], L[e])
            fu = torch.einsum("eqj,ej->eq", self.flux[f][e], U[e])
            sg = 0.5 * al[:, None] * self._nDn(f, e, self.D[e])
            g[e] += (self.wdS[f][e] * (sg * jl * ju - 0.5 * (fu * jl + fl * ju))).sum(1)
        return g


def _ionic(m, u, w):
    """I_ion and the gate rates at DoFs u with gates w (rows)."""
    if m["model"] == 2:
        on = lambda z0: (u >= z0).double()  # noqa: E731
        sm = lambda z0, k: 0.5 * (1.0 + torch.tanh(k * (u - z0)))  # noqa: E731
        h1, h1m, h2, ho = on(m["V1"]), on(m["V1m"]), on(m["V2"]), on(m["Vo"])
        a0 = (1 - h1) / (h1m * (m["tau1pp"] - m["tau1p"]) + m["tau1p"])
        a1 = (1 - h2) / (sm(m["V2m"], m["k2"]) * (m["tau2pp"] - m["tau2p"]) + m["tau2p"])
        a2 = 1 / (h2 * (m["tau3pp"] - m["tau3p"]) + m["tau3p"])
        H = torch.stack([(-h1 / m["tau1plus"] - a0) * w[0] + a0 * (1 - h1m),
                         (-h2 / m["tau2plus"] - a1) * w[1] + a1 * (ho * (m["winf_star"] - 1 + u / m["tau2inf"]) + 1 - u / m["tau2inf"]),
                         a2 * (sm(m["V3"], m["k3"]) - w[2])])
        cur = (-h1 * (u - m["V1"]) * (m["Vhat"] - u) * w[0] / m["taufi"]
               + (1 - h2) * (u - m["uo"]) / (ho * (m["tauo_pp"] - m["tauo_p"]) + m["tauo_p"])
               + h2 / (sm(m["Vso"], m["kso"]) * (m["tauso_pp"] - m["tauso_p"]) + m["tauso_p"]) - h2 * w[1] * w[2] / m["tausi"])
        return cur, H
    cub = m["k"] * u * (u - m["a"]) * (u - 1)
    if m["model"] == 0:
        return cub + w[0], m["eps"] * (u - m["gamma"] * w)
    return cub + u * w[0], (m["eps"] + m["mu1"] * w / (u + m["mu2"])) * (-w - m["k"] * u * (u - m["a"] - 1))


def _ionic_jac(m, u, w):
    dc = m["k"] * (3 * u * u - 2 * (m["a"] + 1) * u + m["a"])
    if m["model"] == 0:
        return dc, torch.ones_like(u), m["eps"] * torch.ones_like(u), -m["eps"] * m["gamma"] * torch.ones_like(u)
    den = u + m["mu2"]
    e, g = m["eps"] + m["mu1"] * w / den, -w - m["k"] * u * (u - m["a"] - 1)
    return dc + w, u, -m["mu1"] * w / den ** 2 * g - e * m["k"] * (2 * u - m["a"] - 1), m["mu1"] / den * g - e


def exact(case, seed, dev="cuda"):
    dev = torch.device(dev)
    m = MODELS[case["model"]]
    if case["kind"] == "ionic":
        v = _inputs(case, seed, None, dev)
        w = v["w"].view(-1, case["n"])
        return (w + (1e-4 if case["model"] == "bo" else 0.05) * _ionic(m, v["u"], w)[1]).flatten()
    wl = _workload(case)
    v = _inputs(case, seed, wl, dev)
    D = np.asarray(wl.conductivity)
    if case["kind"] == "adjoint":
        theta = np.exp(0.2 * np.random.default_rng(3).standard_normal(64))
        tmap = (np.arange(len(D)) * 64) // len(D)
        D = theta[tmap][:, None, None] * D
    dt, n = wl.dt, wl.n_dofs
    c = (1.5 if case["scheme"] == 1 else 1.0) / dt
    F = _Forms(wl, D, dev)
    F.assemble(c)
    if case["kind"] == "operator":
        return F.apply(v["x"])
    if case["kind"] == "pcg":
        return F.solve(v["b"], torch.zeros_like(v["b"]))
    if case["kind"] == "adjoint":
        u, w = v["u"], v["w"]
        lam = F.solve(v["ubar"], torch.zeros_like(u))
        q = F.mass(lam)
        w1 = w + dt * _ionic(m, u, w[None])[1][0]
        Iu, Iw, _, _ = _ionic_jac(m, u, w1)
        _, _, Hu, Hw = _ionic_jac(m, u, w)
        wt = v["wbar"] - Iw * q
        grad = -F.own_share(lam, v["u1"])
        gt = torch.zeros(64, dtype=torch.float64, device=dev)
        gt.index_add_(0, F.t(tmap).long(), grad / F.t(theta[tmap]))
        return dict(ubar=q * (c - Iu) + dt * Hu * wt, wbar=wt * (1 + dt * Hw), grad=grad, gtheta=gt)
    u, w = v["u"], v["w"].view(-1, n)
    mask = F.t(wl.stim_mask_nodal())
    up = wp = None
    for k in range(case["steps"]):
        ia = wl.iapp_value * mask if v["clock"] + k < wl.iapp_steps else 0.0 * mask
        if case["scheme"] == 1:
            if k == 0:
                cur, H = _ionic(m, u, w)
                Au = torch.linalg.solve(F.Me, F.apply(u).view(-1, F.B, 1)).flatten() - c * u
                up, wp = u - dt * (ia - cur - Au), w - dt * H
            us, ws = 2 * u - up, 2 * w - wp
            wn = (4 * w - wp) / 3 + (2 * dt / 3) * _ionic(m, us, ws)[1]
            b = F.mass((4 * u - up) / (2 * dt) + ia - _ionic(m, us, wn)[0])
        else:
            wn = w + dt * _ionic(m, u, w)[1]
            b = F.mass(c * u + ia - _ionic(m, u, wn)[0])
        up, wp = u, w
        u, w = F.solve(b, u), wn
    return dict(u=u, w=w.flatten())
