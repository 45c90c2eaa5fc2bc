"""Performance cases: what a user of the library has it do, through the public
binding (paper_2501_11767_gb300.chnss), over the range of sizes and options
in use.  Each case is a dict of plain values; prepare() makes its inputs from
a seed, run() is one pass, work() its unavoidable traffic, exact() the same
result in 64 bits from plain torch where that is affordable.

Kinds
  step     one semi-implicit time step of a film (2D)
  step3d   the same on a Kuhn tetrahedral mesh of the unit box
  sweep    one step of every instance of a parameter sweep, in one call
  adjoint  the reverse sweep of one step (gradients of a trajectory)
  solve    assembly and one linear system with a given right-hand side
  amg      smoothed aggregation: new matrix values, re-setup, one solve
  mass     the allocation-free mass solve

A time-stepping program builds its mesh and context once and steps many
fields through them, so the context of the last configuration is kept here
and prepare() makes fields; the sweep's contexts belong to its state, because
their step graphs are recorded for fixed field arrays.
"""
import math

import numpy as np
import torch

from paper_2501_11767_gb300 import chnss, inputs

# sizes a 2D mesh hierarchy accepts: m 2^k cells per side, m <= 25 odd or 2
SIZES = sorted({m << k for m in (1, 3, 5, 7, 9, 11, 13, 15, 17, 19, 21, 23, 25) for k in range(1, 11)
                if 24 <= m << k <= 1024})


def listed():
    return [
        # the 32 x 32 FP64 parity workload: launches and host round trips count
        {"name": "step_32_fp64", "kind": "step", "n": 32, "precision": 0, "tau": 1e-3, "eps": 0.02},
        # the paper's 2D mesh (n = 100, 25^2 coarsest level) with its solver settings:
        # rtol 1e-6 / 1e-4 and multigrid blocks solved to 1e-4
        {"name": "step_100_paper_solver", "kind": "step", "n": 100, "precision": 1, "tau": 1e-4, "eps": 0.02,
         "paper_solver": True},
        # the 256 x 256 FP64 workload with concentration-dependent mobility
        {"name": "step_256_mobility_fp64", "kind": "step", "n": 256, "precision": 0, "tau": 1e-3, "eps": 0.01,
         "mobility": 1},
        # mixed precision, open (do-nothing) top, the paper's time step
        {"name": "step_512_open_mixed", "kind": "step", "n": 512, "precision": 1, "tau": 1e-4, "eps": 0.005,
         "top": 1},
        # the benchmark's workload: about a million P1 nodes, mixed precision
        {"name": "step_1024_mixed", "kind": "step", "n": 1024, "precision": 1, "tau": 5e-4, "eps": 0.005},
        # a shard of the evaporation-rate sweep: uneven meshes of 128^2 to 512^2, one graph an instance
        {"name": "sweep_8", "kind": "sweep", "count": 8, "draw": 0},
        # the 3D film at the size of the 3D benchmark
        {"name": "step3d_32_mixed", "kind": "step3d", "n": 32, "precision": 1},
        # one reverse step of a gradient computation, FP64, concentration-dependent mobility
        {"name": "adjoint_128", "kind": "adjoint", "n": 128, "mobility": 1},
        # the Oseen system alone, mixed precision, a right-hand side of the caller's
        {"name": "solve_ns_384_mixed", "kind": "solve", "system": "ns", "n": 384, "precision": 1},
        # the Allen-Cahn system alone, FP64: assembly carries most of the call
        {"name": "solve_ac_640_fp64", "kind": "solve", "system": "ac", "n": 640, "precision": 0},
        # an unstructured operator: re-setup of the hierarchy for new values, then one solve
        {"name": "amg_512", "kind": "amg", "n": 512, "precision": 1},
        # the mass solve of a caller whose device memory is all taken
        {"name": "mass_240", "kind": "mass", "n": 240},
    ]


def _size(rng, lo, hi):
    """An accepted mesh size, spread over the logarithm of [lo, hi]."""
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((s for s in SIZES if lo <= s <= hi), key=lambda s: abs(math.log(s / t)))


def draw(rng):
    kind = rng.choice(["step"] * 8 + ["step3d", "sweep", "adjoint", "solve", "solve", "amg", "mass"])
    if kind == "step":
        precision = rng.choice([0, 1, 1, 2])
        n = _size(rng, 24, 512 if precision == 0 else 1024)
        top = rng.choice([0, 0, 1])
        c = {"kind": kind, "n": n, "precision": precision, "top": top,
             "tau": 1e-4 if top or n > 512 else rng.choice([1e-4, 5e-4, 1e-3]),
             "eps": rng.choice([0.005, 0.01, 0.02]), "mobility": 0}
        if n <= 512:
            c["mobility"] = rng.choice([0, 0, 1])
        if n <= 256 and precision and not c["mobility"]:
            c["paper_solver"] = rng.choice([False, False, True])
        return c
    if kind == "step3d":
        return {"kind": kind, "n": rng.choice([8, 12, 16, 20, 24, 28, 32]), "precision": rng.choice([0, 1, 1])}
    if kind == "sweep":
        return {"kind": kind, "count": rng.randint(3, 8), "draw": rng.randint(1, 1000)}
    if kind == "adjoint":
        return {"kind": kind, "n": _size(rng, 32, 192), "mobility": rng.choice([0, 1])}
    if kind == "solve":
        return {"kind": kind, "system": rng.choice(["ns", "ac", "ch"]), "n": _size(rng, 32, 640),
                "precision": rng.choice([0, 1])}
    if kind == "amg":
        return {"kind": kind, "n": rng.randint(40, 700), "precision": rng.choice([0, 1])}
    return {"kind": kind, "n": _size(rng, 32, 256)}


# ---------------------------------------------------------------------------
# parameters, fields, contexts
def _params(c):
    p = inputs.default_params()
    precision = c.get("precision", 0)
    p.update(tau=c.get("tau", 5e-4), beta=inputs.film_betas(c.get("eps", 0.01)), precision=precision,
             ortho=1 if precision else 0, mobility_kind=c.get("mobility", 0), top_bc=c.get("top", 0))
    if c.get("paper_solver"):
        p.update(rtol=1e-6, atol=1e-8, ns_rtol=1e-4, ns_atol=1e-8, inner_rtol=1e-4, inner_maxit=20)
    if c["kind"] == "step3d":
        p.update(tau=1e-4)
    return p


_kept = {}


def _keep(key, make):
    """The value of the last key only: a program holds one configuration."""
    if key not in _kept:
        _kept.clear()
        _kept[key] = make()
    return _kept[key]


def _context(c):
    key = tuple(sorted((k, v) for k, v in c.items() if k != "name"))
    if c["kind"] == "step3d":
        return _keep(key, lambda: chnss.Context3(c["n"], _params(c)))
    return _keep(key, lambda: chnss.Context(chnss.Mesh(c["n"], top_bc=c.get("top", 0)), _params(c)))


def _waves(gen, x, terms=4):
    """A smooth random field of size one on the coordinates x (tuple of tensors)."""
    out = torch.zeros_like(x[0])
    for _ in range(terms):
        k = torch.randint(1, 5, (len(x),), generator=gen).tolist()
        a, s = (torch.rand(2, generator=gen, dtype=torch.float64) * 2 - 1).tolist()
        w = torch.ones_like(out)
        for kd, xd in zip(k, x):
            w = w * torch.cos(math.pi * kd * xd + s)
        out += a * w
    return out / terms


def _fields(n, dim, seed, speed=0.05):
    """A film some way into its drying: noise and composition waves about
    0.3 / 0.3 / 0.4, vapour near the top, a slow vortex flow that vanishes on
    the walls, smooth potentials and a zero-mean pressure."""
    gen = torch.Generator().manual_seed(seed)
    dev = torch.Generator(device="cuda").manual_seed(seed)

    def lattice(m):
        ax = torch.linspace(0, 1, m + 1, dtype=torch.float64, device="cuda")
        return [g.reshape(-1) for g in torch.meshgrid(*([ax] * dim), indexing="ij")][::-1]

    x, x2 = lattice(n), lattice(2 * n)
    noise = lambda: 0.01 * (2 * torch.rand(x[0].numel(), generator=dev, dtype=torch.float64, device="cuda") - 1)  # noqa: E731
    phi = torch.stack([0.3 + 0.05 * _waves(gen, x) + noise(), 0.3 + 0.05 * _waves(gen, x) + noise(),
                       0.4 + 0.02 * _waves(gen, x)])
    wall = torch.ones_like(x2[0])
    for xd in x2:
        wall = wall * torch.sin(math.pi * xd) ** 2
    vortex = [wall * _waves(gen, x2) for _ in range(dim)]
    p = _waves(gen, x)
    return {"phi": phi, "mu": torch.stack([_waves(gen, x) for _ in range(4)]),
            "Phi_v": 0.1 * x[-1] ** 2 * (1 + _waves(gen, x)), "v": speed * torch.stack(vortex, 1).reshape(-1),
            "p": p - p.mean()}


def _sweep(c):
    """Instances of the sweep with other draws: (n, params) per instance."""
    return [(i["n"], i["params"]) for i in inputs.sweep_instances(c["count"], c["draw"])]


def _amg_matrix(c, seed):
    """M + tau K + tau C(w) on an unstructured triangulation, CSR on the device."""
    x, tri = inputs.unstructured_square(c["n"], seed % 1000)
    x, tri = torch.as_tensor(x, device="cuda"), torch.as_tensor(tri, device="cuda")
    area, g = _geometry(x[tri])
    gen = torch.Generator().manual_seed(seed)
    wind = (torch.rand(2, generator=gen, dtype=torch.float64) - 0.5).cuda()
    tau = 5e-4
    mass = (torch.ones(3, 3, dtype=torch.float64) + torch.eye(3, dtype=torch.float64)).cuda() / 12
    loc = area[:, None, None] * (mass + tau * torch.einsum("ead,ebd->eab", g, g)
                                 + tau / 3 * torch.einsum("d,ebd->eb", wind, g)[:, None, :])
    return _csr(loc, tri, tri, x.shape[0], x.shape[0])


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "sweep":
        meshes = _keep(("sweep", c["count"], c["draw"]), lambda: {n: chnss.Mesh(n) for n, _ in _sweep(c)})
        ctx, ins, outs = [], [], []
        for k, (n, p) in enumerate(_sweep(c)):
            ctx.append(chnss.Context(meshes[n], p, stream=torch.cuda.Stream()))
            ctx[-1].set_step_mode(1)
            ins.append(_fields(n, 2, seed + 7919 * k))
            outs.append(ctx[-1].new_state())
        return {"kind": kind, "ctx": ctx, "in": ins, "out": outs, "meshes": meshes}
    if kind == "amg":
        A = _amg_matrix(c, seed)
        rp, col, val = A.crow_indices().int(), A.col_indices().int(), A.values()
        b = torch.rand(rp.numel() - 1, generator=torch.Generator(device="cuda").manual_seed(seed), dtype=torch.float64,
                       device="cuda") - 0.5
        return {"kind": kind, "h": chnss.Amg(rp, col, val, c["precision"]), "val": val, "b": b,
                "x": torch.empty_like(b)}
    ctx = _context(c)
    st = {"kind": kind, "ctx": ctx}
    if kind == "mass":
        st["b"] = _fields(c["n"], 2, seed)["phi"][0] / c["n"] ** 2
        st["x"] = torch.empty_like(st["b"])
        return st
    st["in"] = _fields(c["n"], 3 if kind == "step3d" else 2, seed)
    st["out"] = ctx.new_state()
    if kind == "adjoint":
        st["out"] = _fields(c["n"], 2, seed + 2)      # the state after the step
        # adjoints as a reverse sweep carries them: mu enters a step only through
        # alpha = 1e-8, the pressure not at all
        size = {"phi": 1.0, "mu": 1e-8, "Phi_v": 1.0, "v": 1.0, "p": 0.0}
        st["adj"] = {k: size[k] * v / c["n"] ** 2 for k, v in _fields(c["n"], 2, seed + 1).items()}
        st["back"] = ctx.new_state()
    if kind == "solve":
        st["system"] = {"ns": chnss.SYS_NS, "ac": chnss.SYS_AC, "ch": chnss.SYS_CH_P}[c["system"]]
        f = _fields(c["n"], 2, seed + 1)
        st["b"] = torch.cat({"ns": [f["v"], 0 * f["p"]], "ac": [f["phi"][0]],
                             "ch": [f["phi"][0], 1e-3 * f["phi"][1]]}[c["system"]]) / c["n"] ** 2
        st["x"] = torch.empty_like(st["b"])
    return st


def run(state):
    kind = state["kind"]
    if kind == "sweep":
        chnss.step_batched(state["ctx"], state["in"], state["out"])
        return state["out"]
    if kind == "amg":
        state["h"].update(state["val"])
        return state["h"].solve(state["b"], state["x"])[0]
    ctx = state["ctx"]
    if kind == "mass":
        return ctx.mass_solve_noalloc(state["b"], state["x"])[0]
    if kind == "adjoint":
        back, grads, _, _ = ctx.adjoint_step(state["in"], state["out"], state["adj"], state["back"])
        return {"adj": back, "grads": grads}
    if kind == "solve":
        ctx.assemble(state["in"])
        return ctx.solve(state["system"], state["b"], state["x"])[0]
    return ctx.step(state["in"], state["out"])[0]


def work(case):
    """Bytes: every field, matrix value and right-hand side read once, every
    result written once.  The linear systems need far more, by an amount that
    depends on the method; flops are left at one multiply-add per byte read."""
    c, kind, n = case, case["kind"], case.get("n", 0)
    fields = lambda m, d: 8.0 * (9 * (m + 1) ** d + d * (2 * m + 1) ** d)   # noqa: E731
    if kind == "step":
        b = 2 * fields(n, 2)
    elif kind == "step3d":
        b = 2 * fields(n, 3)
    elif kind == "sweep":
        b = sum(2 * fields(m, 2) for m, _ in _sweep(c))
    elif kind == "adjoint":
        b = 4 * fields(n, 2)
    elif kind == "solve":
        b = fields(n, 2) + 16.0 * {"ns": 2 * (2 * n + 1) ** 2 + (n + 1) ** 2, "ac": (n + 1) ** 2,
                                   "ch": 2 * (n + 1) ** 2}[c["system"]]
    elif kind == "amg":
        b = (n + 1) ** 2 * (7 * 12 + 4 + 16.0)
    else:
        b = 16.0 * (n + 1) ** 2
    return {"bytes": b, "flops": 2 * b / 8}


# ---------------------------------------------------------------------------
# 64-bit results: the discretisation of include/chnss.h written out with
# quadrature, solved by dense LU or a Krylov method run to rounding level.
def _geometry(x):
    """Areas and barycentric gradients (E, 3, 2) of triangles x (E, 3, 2)."""
    d1, d2 = x[:, 1] - x[:, 0], x[:, 2] - x[:, 0]
    det = d1[:, 0] * d2[:, 1] - d1[:, 1] * d2[:, 0]
    g1 = torch.stack([d2[:, 1], -d2[:, 0]], 1) / det[:, None]
    g2 = torch.stack([-d1[:, 1], d1[:, 0]], 1) / det[:, None]
    return det / 2, torch.stack([-g1 - g2, g1, g2], 1)


def _csr(loc, rows, cols, nr, nc):
    """Element matrices (E, a, b) summed into a CSR matrix."""
    r = rows[:, :, None].expand(loc.shape)
    k = cols[:, None, :].expand(loc.shape)
    A = torch.sparse_coo_tensor(torch.stack([r.reshape(-1), k.reshape(-1)]), loc.reshape(-1), (nr, nc))
    return A.coalesce().to_sparse_csr()


class _Film:
    """Mesh, quadrature and forms of one 2D state, in float64."""

    def __init__(self, n, params, st):
        self.n, self.p, self.st, h = n, params, st, 1.0 / n
        j, i = (t.reshape(-1) for t in torch.meshgrid(*([torch.arange(n, device="cuda")] * 2), indexing="ij"))
        a, b, d, e = (j * (n + 1) + i), (j * (n + 1) + i + 1), ((j + 1) * (n + 1) + i + 1), ((j + 1) * (n + 1) + i)
        self.tri = torch.cat([torch.stack([a, b, d], 1), torch.stack([a, d, e], 1)])
        I, J = self.tri % (n + 1), self.tri // (n + 1)
        mid = lambda u, v: (J[:, u] + J[:, v]) * (2 * n + 1) + I[:, u] + I[:, v]   # noqa: E731
        self.tri2 = torch.stack([mid(0, 0), mid(1, 1), mid(2, 2), mid(1, 2), mid(0, 2), mid(0, 1)], 1)
        self.N1, self.N2 = (n + 1) ** 2, (2 * n + 1) ** 2
        self.area, self.g = _geometry(torch.stack([I, J], 2).double() * h)
        s, ws = np.polynomial.legendre.leggauss(6)
        s, ws = (s + 1) / 2, ws / 2
        S, T = (t.reshape(-1) for t in np.meshgrid(s, s, indexing="ij"))
        self.w = torch.as_tensor(2 * np.outer(ws, ws).reshape(-1) * (1 - S), device="cuda")
        self.lam = torch.as_tensor(np.stack([1 - S - T * (1 - S), S, T * (1 - S)], 1), device="cuda")
        l0, l1, l2 = self.lam.T
        self.z = torch.stack([l0 * (2 * l0 - 1), l1 * (2 * l1 - 1), l2 * (2 * l2 - 1), 4 * l1 * l2, 4 * l0 * l2,
                              4 * l0 * l1], 1)
        self.aw = self.area[:, None] * self.w

    def form(self, loc):
        return _csr(loc, self.tri, self.tri, self.N1, self.N1)

    # element matrices (E, 3, 3) of mass, (weighted) stiffness and convection
    def M(self):
        return torch.einsum("eq,qa,qb->eab", self.aw, self.lam, self.lam)

    def K(self, kappa=None):
        k = self.area if kappa is None else (self.aw * kappa).sum(1)
        return k[:, None, None] * torch.einsum("ead,ebd->eab", self.g, self.g)

    def at(self, f):
        return f[self.tri] @ self.lam.T                                   # (E, Q)

    def C(self):
        v = torch.einsum("qa,ead->eqd", self.z, self.st["v"].view(-1, 2)[self.tri2])
        return torch.einsum("eqa,ebd,eqd->eab", self.aw[:, :, None] * self.lam, self.g, v)

    def load(self, f):
        out = torch.zeros(self.N1, dtype=torch.float64, device="cuda")
        return out.index_add_(0, self.tri.reshape(-1), torch.einsum("eq,eq,qa->ea", self.aw, f, self.lam).reshape(-1))

    def flux(self):
        """Evaporation flux and the top edge's hat integrals."""
        t = torch.zeros(self.N1, dtype=torch.float64, device="cuda")
        t[self.n * (self.n + 1):] = 1.0 / self.n
        t[self.n * (self.n + 1)] = t[-1] = 0.5 / self.n
        ref = self.n * (self.n + 1) + self.n // 2
        return self.p["evap_rate"] * (self.st["phi"][2][ref] - self.p["phi_s_inf"]) * t

    def partials(self):
        """Loads of the partial derivatives of the potential (p, N, s, a, Phi_v)."""
        a, b, s = (self.at(f) for f in self.st["phi"])
        r, Ph = 1 - a - b - s, self.at(self.st["Phi_v"])
        q, dq = Ph * Ph * (3 - 2 * Ph), 6 * Ph * (1 - Ph)
        liquid = 3.5 * a**2 * b**2 + 0.3 * s**2 + 0.3 * r**2 - 10 * s * r
        gas = 3.5 * a**2 + 3.5 * b**2 + 2 * s**2 + 0.1 * r**2
        return [self.load(f) for f in ((1 - q) * 7 * a * b**2 + q * 7 * a, (1 - q) * 7 * a**2 * b + q * 7 * b,
                                       (1 - q) * (0.6 * s - 10 * r) + q * 4 * s,
                                       (1 - q) * (0.6 * r - 10 * s) + q * 0.2 * r, dq * (gas - liquid))]

    def allen_cahn(self):
        p = self.p
        A = self.form(self.M() + p["tau"] * p["delta_v"] * self.K() + p["tau"] * self.C())
        rhs = self.form(self.M()) @ self.st["Phi_v"] - p["tau"] * p["gamma_v"] * self.partials()[4]
        return A, rhs + (p["tau"] * p["delta_v"] * self.flux() if p["ac_top_flux"] else 0)

    def cahn_hilliard(self, k):
        p = self.p
        tg, c = p["tau"] * p["gamma"][k], p["tau"] * p["gamma"][k] / p["beta"][k]
        phi = self.at(self.st["phi"][k])
        kap = p["gamma"][k] * (phi * (1 - phi) + p["mobility_m0"]) if p["mobility_kind"] else None
        dense = lambda loc: self.form(loc).to_dense()                     # noqa: E731
        K, M = dense(self.K()), dense(self.M())
        K12 = p["tau"] * dense(self.K(kap)) if p["mobility_kind"] else tg * K
        f = self.partials()[k] - (p["beta"][2] * self.flux() if k == 2 else 0)
        A = torch.cat([torch.cat([M + p["tau"] * dense(self.C()), K12], 1), torch.cat([tg * K, -c * M], 1)])
        return A, torch.cat([M @ self.st["phi"][k], -c * f])

    def oseen(self):
        """Dense Oseen matrix (enclosed flow: with the zero-mean row) and right-hand side."""
        p, n, nv = self.p, self.n, 2 * self.N2
        mu = torch.einsum("f,fea,ead->ed", torch.tensor(p["alpha"], dtype=torch.float64, device="cuda"),
                          self.st["mu"][:, self.tri], self.g)
        l, g = self.lam, self.g
        dl = torch.zeros(l.shape[0], 6, 3, dtype=torch.float64, device="cuda")   # d zeta / d lambda
        for a in range(3):
            dl[:, a, a] = 4 * l[:, a] - 1
        for a, (u, v) in enumerate(((1, 2), (0, 2), (0, 1))):
            dl[:, 3 + a, u], dl[:, 3 + a, v] = 4 * l[:, v], 4 * l[:, u]
        dz = torch.einsum("qak,ekd->eqad", dl, g)
        v = torch.einsum("qa,ead->eqd", self.z, self.st["v"].view(-1, 2)[self.tri2]) - mu[:, None]
        m2 = torch.einsum("eq,qa,qb->eab", self.aw, self.z, self.z)
        s = m2 / p["tau"] + torch.einsum("eq,qa,eqd,eqbd->eab", self.aw, self.z, v, dz)
        s = s + p["eta"] * torch.einsum("eq,eqad,eqbd->eab", self.aw, dz, dz)
        eye = torch.eye(2, dtype=torch.float64, device="cuda")
        loc = torch.einsum("eab,cd->eacbd", s, eye) + p["eta"] * torch.einsum("eq,eqbc,eqad->eacbd", self.aw, dz, dz)
        dof = (2 * self.tri2[:, :, None] + torch.arange(2, device="cuda")).reshape(-1, 12)
        A = _csr(loc.reshape(-1, 12, 12), dof, dof, nv, nv).to_dense()
        B = _csr(-torch.einsum("eq,qa,eqbd->eabd", self.aw, l, dz).reshape(-1, 3, 12), self.tri, dof, self.N1,
                 nv).to_dense()
        grads = [torch.einsum("ea,ead->ed", f[self.tri], g) for f in self.st["phi"]]
        grads += [-(grads[0] + grads[1] + grads[2]), torch.einsum("ea,ead->ed", self.st["Phi_v"][self.tri], g)]
        G = sum(b * torch.einsum("ec,ed->ecd", q, q) for b, q in zip(p["beta"] + [p["beta_v"]], grads))
        rhs = torch.zeros(nv, dtype=torch.float64, device="cuda")
        rhs.index_add_(0, dof.reshape(-1), (torch.einsum("eq,ecb,eqab->eac", self.aw, G, dz)
                                            + torch.einsum("eab,ebd->ead", m2, self.st["v"].view(-1, 2)[self.tri2])
                                            / p["tau"]).reshape(-1))
        J, I = (t.reshape(-1) for t in torch.meshgrid(*([torch.arange(2 * n + 1, device="cuda")] * 2), indexing="ij"))
        wall = (I == 0) | (I == 2 * n) | (J == 0) | ((J == 2 * n) & (p["top_bc"] == 0))
        free = (~wall).repeat_interleave(2).double()
        A = A * free[:, None] * free + torch.diag(1 - free)
        B = B * free
        rows = [torch.cat([A, B.T], 1), torch.cat([B, torch.zeros(self.N1, self.N1, dtype=torch.float64, device="cuda")], 1)]
        S = torch.cat(rows)
        rhs = torch.cat([rhs * free, torch.zeros(self.N1, dtype=torch.float64, device="cuda")])
        if p["top_bc"] == 0:
            m = torch.cat([torch.zeros(nv, dtype=torch.float64, device="cuda"),
                           self.form(self.M()) @ torch.ones(self.N1, dtype=torch.float64, device="cuda")])
            S = torch.cat([torch.cat([S, m[:, None]], 1), torch.cat([m, m.new_zeros(1)])[None]])
            rhs = torch.cat([rhs, rhs.new_zeros(1)])
        return S, rhs, nv


def _krylov(A, b, sweeps=6):
    """A x = b by Jacobi-scaled BiCGSTAB with iterative refinement to rounding level."""
    rows = torch.repeat_interleave(torch.arange(b.numel(), device="cuda"), A.crow_indices().diff())
    on = rows == A.col_indices()
    d = torch.zeros_like(b)
    d[rows[on]] = A.values()[on]
    x = torch.zeros_like(b)
    for _ in range(sweeps):
        r = (b - A @ x) / d
        stop, it = 1e-7 * float(r.norm()), 0
        s0, q, v, e = r.clone(), torch.zeros_like(r), torch.zeros_like(r), torch.zeros_like(r)
        rho = alpha = omega = torch.ones((), dtype=torch.float64, device="cuda")
        while float(r.norm()) > stop and it < 4000:
            it += 1
            rho, old = s0 @ r, rho
            q = r + (rho / old) * (alpha / omega) * (q - omega * v)
            v = (A @ q) / d
            alpha = rho / (s0 @ v)
            s = r - alpha * v
            t = (A @ s) / d
            omega = (t @ s) / (t @ t)
            e = e + alpha * q + omega * s
            r = s - omega * t
        if not bool(torch.isfinite(e).all()):
            break
        x = x + e
    return x


DENSE = 36      # largest mesh whose Oseen and Cahn-Hilliard systems are solved densely here


def _exact_step(n, params, st):
    f = _Film(n, params, st)
    out = {"phi": None, "mu": None, "Phi_v": _krylov(*f.allen_cahn()), "v": None, "p": None}
    if n > DENSE:
        return out
    N1 = f.N1
    ch = [torch.linalg.solve(*f.cahn_hilliard(k)) for k in range(3)]
    out["phi"] = torch.stack([x[:N1] for x in ch])
    fa = f.partials()[3] + params["beta"][3] * f.flux()
    mu_a = _krylov(f.form(f.M()), fa + params["beta"][3] * (f.form(f.K()) @ (1 - out["phi"].sum(0))))
    out["mu"] = torch.stack([x[N1:] for x in ch] + [mu_a])
    S, rhs, nv = f.oseen()
    x = torch.linalg.solve(S, rhs)
    out["v"], out["p"] = x[:nv], x[nv:nv + N1]
    return out


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "step":
        return _exact_step(c["n"], _params(c), _fields(c["n"], 2, seed))
    if kind == "sweep":
        return [_exact_step(n, p, _fields(n, 2, seed + 7919 * k)) for k, (n, p) in enumerate(_sweep(c))]
    if kind == "amg":
        A = _amg_matrix(c, seed)
        b = torch.rand(A.shape[0], generator=torch.Generator(device="cuda").manual_seed(seed), dtype=torch.float64,
                       device="cuda") - 0.5
        return _krylov(A, b)
    if kind == "mass":
        st = _fields(c["n"], 2, seed)
        f = _Film(c["n"], _params(c), st)
        return _krylov(f.form(f.M()), st["phi"][0] / c["n"] ** 2)
    if kind == "solve":
        f = _Film(c["n"], _params(c), _fields(c["n"], 2, seed))
        g = _fields(c["n"], 2, seed + 1)
        if c["system"] == "ac":
            return _krylov(f.allen_cahn()[0], g["phi"][0] / c["n"] ** 2)
        if c["n"] > DENSE:
            return None
        if c["system"] == "ch":
            return torch.linalg.solve(f.cahn_hilliard(0)[0], torch.cat([g["phi"][0], 1e-3 * g["phi"][1]]) / c["n"] ** 2)
        S, rhs, nv = f.oseen()
        rhs.zero_()
        rhs[:nv] = g["v"] / c["n"] ** 2
        return torch.linalg.solve(S, rhs)[:nv + f.N1]
    return None                     # the adjoint and the 3D step: no affordable restatement
