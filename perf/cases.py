"""The work that a user of this library has it do, as cases that can be timed.

A case is one generalized Stokes operator (mesh size, mu, dt, gamma, options)
and one pass through a public entry point with it: a solve with one or several
right-hand sides, a batch of uneven instances, a solve with its adjoint
through autograd, a setup followed by a single solve, or one operator product
through ``Stokes.apply``. Meshes are Kuhn meshes of the unit cube with interior
vertices jittered by up to 0.16 h, the most for which no tetrahedron can invert
whatever the seed (the edge vectors then differ from the unjittered ones by a
matrix of norm below 1; the parity configuration has none); body forces are
N(0,1) per nodal component. Solves ask for a relative residual of 1e-12,
the tolerance at which two solutions of one system can be compared to 1e-9.
"""

import math

import numpy as np
import torch

import paper_2407_01783_gb300 as sk

TOL = 1e-12
DEVICE = "cuda"


def _case(name, kind, n, **kw):
    c = dict(kind=kind, n=n, mu=1e-2, dt=1e-3, gamma=0.0, jitter=0.16, method="schur", mixed=True, vcycles=1,
             block_lu=True, rhs=1, load=False, op="", instances=1)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the parity configuration: FP64, default options, unjittered 8^3
        _case("fp64-schur-8", "solve", 8, dt=1e-2, jitter=0.0, mixed=False, vcycles=2),
        # the default (FP64) solver on an ordinary mesh
        _case("fp64-schur-24", "solve", 24, mixed=False, vcycles=2),
        # the smallest instance of the uneven batch, alone: latency and launches
        _case("mixed-schur-12", "solve", 12, mu=1e-3),
        # the benchmark's mesh, method, precision and middle viscosity
        _case("mixed-schur-48", "solve", 48),
        # Method 2 on an odd mesh (non-nested coarsening), viscous, with a pressure load
        _case("mixed-coupled-33", "solve", 33, method="coupled", mu=0.1, load=True),
        # the coupled augmented-Lagrangian form at the largest configured size
        _case("coupled-al-96", "solve", 96, method="coupled", mu=1e-3, gamma=1.0, block_lu=False),
        # four body forces of one operator in lockstep, Method 2 (the batch's largest instance)
        _case("lockstep4-coupled-40", "solve", 40, method="coupled", rhs=4),
        # six right-hand sides (a full group and a padded one) by Method 1, with pressure loads
        _case("lockstep6-schur-25", "solve", 25, rhs=6, load=True),
        # uneven instances at once, four forces each
        _case("batch-6x4", "batch", 40, method="coupled", rhs=4, instances=6),
        # forward and backward through autograd on the adjoint configuration
        _case("adjoint-64", "adjoint", 64),
        # a changed mesh or time step: setup and one solve
        _case("setup-solve-20", "setup", 20, mu=0.05),
        # the FP64-accurate strain product of the refinement residual, as a building block
        _case("apply-A-df-48", "apply", 48, op="A_DF"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "multi", "multi", "batch", "adjoint", "setup", "apply"])
    mu, dt = _log_uniform(rng, 1e-4, 1.0), _log_uniform(rng, 1e-4, 1e-2)
    method = rng.choice(["schur", "coupled"])
    kw = dict(method=method)
    if kind == "solve":
        n = int(round(_log_uniform(rng, 8, 72)))
        form = rng.choice(["mixed", "mixed", "mixed", "al", "fp64"])
        if form == "al":
            kw.update(gamma=rng.choice([1.0, 10.0]), block_lu=method == "schur", vcycles=1)
            mu = min(mu, 1e-2)
        elif form == "fp64":
            n = min(n, 24)
            kw.update(mixed=False, vcycles=2)
        kw.update(load=rng.random() < 0.3)
    elif kind == "multi":
        n = int(round(_log_uniform(rng, 8, 40)))
        kind = "solve"
        kw.update(rhs=rng.randint(2, 9), load=rng.random() < 0.3)
    elif kind == "batch":
        n = rng.randint(16, 40)
        kw.update(rhs=rng.randint(1, 4), instances=rng.randint(2, 6))
    elif kind == "adjoint":
        n = int(round(_log_uniform(rng, 8, 64)))
        kw.update(method="schur")
    elif kind == "setup":
        n = int(round(_log_uniform(rng, 8, 40)))
    else:
        n = int(round(_log_uniform(rng, 8, 64)))
        op = rng.choice(["A_DF", "A", "VCYCLE_VEL", "SCHUR_PREC", "LOAD"])
        kw.update(op=op, mixed=op == "A_DF")
    # FP64 reaches 1e-12 with room up to here (less with a rough pressure load)
    mu = min(mu, (0.5 if kw.get("load") else 4.0) / (dt * n * n))
    return _case("", kind, n, mu=mu, dt=dt, **kw)


# ---------------------------------------------------------------------------
# inputs and plans
# ---------------------------------------------------------------------------
def _generator(seed, salt):
    return torch.Generator(device=DEVICE).manual_seed(1009 * int(seed) + salt)


def _vertices(n, jitter, seed, salt=0):
    g = np.arange(n + 1) / n
    k, j, i = np.meshgrid(g, g, g, indexing="ij")
    X = np.stack([i, j, k], axis=-1)
    if jitter:
        d = torch.rand(n - 1, n - 1, n - 1, 3, generator=_generator(seed, 11 + salt), device=DEVICE,
                       dtype=torch.float64)
        X[1:-1, 1:-1, 1:-1] += ((2.0 * d - 1.0) * (jitter / n)).cpu().numpy()
    return X.reshape(-1, 3)


def _normal(seed, salt, *shape):
    return torch.randn(*shape, generator=_generator(seed, salt), device=DEVICE, dtype=torch.float64)


def _rhs(case, n, seed, salt=0):
    """Body forces [rhs, (2n+1)^3, 3] and compatible pressure loads [rhs, (n+1)^3] or None."""
    f = _normal(seed, 101 + salt, case["rhs"], (2 * n + 1) ** 3, 3)
    if not case["load"]:
        return f, None
    # scaled so that the velocities it drives are of the size of those that f drives (about dt)
    g = _normal(seed, 201 + salt, case["rhs"], (n + 1) ** 3) * (case["dt"] / n ** 2)
    return f, g - g.mean(dim=1, keepdim=True)


def _weights(case, seed):
    """dJ/du and dJ/dp of a linear functional, each driving adjoint velocities of the same size."""
    n = case["n"]
    return _normal(seed, 302, (2 * n + 1) ** 3, 3), _normal(seed, 303, (n + 1) ** 3) * (case["dt"] * n)


def _options(case):
    return sk.stokes_default_options(
        method=sk.METHOD_SCHUR if case["method"] == "schur" else sk.METHOD_COUPLED,
        precision=sk.PRECISION_MIXED if case["mixed"] else sk.PRECISION_FP64, vcycles=case["vcycles"],
        block_lu=int(case["block_lu"]), max_refine=12)


def _sizes(case):
    """Cubes per side of every instance: from n downwards in equal steps for a batch."""
    m = case["instances"]
    return [case["n"]] if m == 1 else [case["n"] - i * (case["n"] - 12) // (m - 1) for i in range(m)]


def _out(case, n):
    k = case["rhs"]
    return (torch.empty(k, (2 * n + 1) ** 3, 3, dtype=torch.float64, device=DEVICE),
            torch.empty(k, (n + 1) ** 3, dtype=torch.float64, device=DEVICE))


def _apply_lengths(case):
    n, op = case["n"], case["op"]
    vel, pres, every = 3 * (2 * n - 1) ** 3, (n + 1) ** 3, 3 * (2 * n + 1) ** 3
    return {"LOAD": (every, vel), "SCHUR_PREC": (pres, pres)}.get(op, (vel, vel))


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    state = dict(case=case)
    V = _vertices(n, case["jitter"], seed)
    if kind == "batch":
        spec = [(m, _vertices(m, case["jitter"], seed, 1000 + i), case["mu"], case["dt"], case["gamma"])
                for i, m in enumerate(_sizes(case))]
        state["solver"] = sk.StokesBatch(spec, _options(case))
        state["f"] = [_rhs(case, m, seed, 1000 + i)[0] for i, m in enumerate(_sizes(case))]
    elif kind == "setup":
        state.update(vertices=V, f=_rhs(case, n, seed)[0][0])
    else:
        state["solver"] = sk.Stokes(n, V, case["mu"], case["dt"], case["gamma"], _options(case))
        if kind == "apply":
            state["x"] = _normal(seed, 301, _apply_lengths(case)[0])
        else:
            state["f"], state["g"] = _rhs(case, n, seed)
            state["out"] = _out(case, n)
        if kind == "adjoint":
            state["weights"] = _weights(case, seed)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        S, f, g, (u, p) = (state[k] for k in ("solver", "f", "g", "out"))
        if case["rhs"] == 1:
            S.solve(f[0], None if g is None else g[0], TOL, out=(u[0], p[0]))
        else:
            S.solve_multi(f, g, TOL, out=(u, p))
        return u, p
    if kind == "batch":
        outs, _, _ = state["solver"].solve_all(state["f"], TOL)
        return [[u, p] for inst in outs for u, p in inst]
    if kind == "adjoint":
        f = state["f"][0].detach().requires_grad_(True)
        mu = torch.tensor(case["mu"], dtype=torch.float64, device=DEVICE, requires_grad=True)
        u, p = sk.StokesSolve.apply(state["solver"], f, mu, TOL)
        wu, wp = state["weights"]
        ((u * wu).sum() + (p * wp).sum()).backward()
        return u.detach(), p.detach(), f.grad, mu.grad
    if kind == "setup":
        S = sk.Stokes(case["n"], state["vertices"], case["mu"], case["dt"], case["gamma"], _options(case))
        u, p, _ = S.solve(state["f"], None, TOL)
        S.close()
        return u, p
    return state["solver"].apply(case["op"], state["x"], _apply_lengths(case)[1])


def work(case):
    """Inputs read and outputs written once; the flops of one evaluation of the system (strain form, B and B^T) per
    solve, which no method does without, or of the one product."""
    total_b = total_f = 0.0
    for n in _sizes(case):
        velocity, pressure, nodes = 3.0 * (2 * n - 1) ** 3, (n + 1.0) ** 3, 3.0 * (2 * n + 1) ** 3
        a = 2.0 * 9 * 28 * velocity / 3  # about 28 coupled nodes per node, 3x3 blocks
        b = 2.0 * 2 * 3 * 8 * velocity / 3
        if case["kind"] == "apply":
            total_b += 8.0 * sum(_apply_lengths(case)) + 24.0 * pressure
            total_f += b if case["op"] == "SCHUR_PREC" else a
            continue
        solves = case["rhs"] * (2 if case["kind"] == "adjoint" else 1)
        total_b += 8.0 * solves * (2 * nodes + pressure * (2 if case["load"] else 1)) + 24.0 * pressure
        total_f += solves * (a + b)
    return {"bytes": total_b, "flops": total_f}


# ---------------------------------------------------------------------------
# the same results in plain torch, FP64
# ---------------------------------------------------------------------------
class _Reference:
    """The P2-P1 operators element by element on the Kuhn mesh, from the barycentric gradients of each tetrahedron."""

    EDGES = [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)]

    def __init__(self, n, V, mu, dt):
        self.n, self.mu, self.dt = n, mu, dt
        dev = dict(device=DEVICE)
        dev64 = dict(device=DEVICE, dtype=torch.float64)
        paths = []
        for perm in [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]:
            o = [np.zeros(3, int)]
            for a in perm:
                o.append(o[-1] + np.eye(3, dtype=int)[a])
            paths.append(np.stack(o))
        corner = torch.tensor(np.stack(paths), **dev)                                   # [6, 4, 3]
        c = torch.arange(n, **dev)
        K, J, I = torch.meshgrid(c, c, c, indexing="ij")
        cube = torch.stack([I, J, K], dim=-1).reshape(-1, 1, 1, 3)
        vert = (cube + corner).reshape(-1, 4, 3)                                        # [T, 4, 3]
        half = torch.cat([2 * vert, torch.stack([vert[:, i] + vert[:, j] for i, j in self.EDGES], dim=1)], dim=1)
        N, m = 2 * n + 1, 2 * n - 1
        self.np, self.N3, self.m3 = (n + 1) ** 3, N ** 3, m ** 3
        self.pidx = vert[..., 0] + (n + 1) * (vert[..., 1] + (n + 1) * vert[..., 2])
        self.nidx = half[..., 0] + N * (half[..., 1] + N * half[..., 2])
        inner = torch.zeros(N, N, N, dtype=torch.bool, **dev)
        inner[1:-1, 1:-1, 1:-1] = True
        self.inner = inner.reshape(-1).nonzero().reshape(-1)
        X = torch.tensor(V, **dev)[self.pidx]                                           # [T, 4, 3]
        E = X[:, 1:] - X[:, :1]
        G = torch.cross(E[:, [1, 2, 0]], E[:, [2, 0, 1]], dim=2)
        det = (E[:, 0] * G[:, 0]).sum(-1)
        G = G / det[:, None, None]                                                      # rows: gradients 1..3
        self.grad = torch.cat([-G.sum(1, keepdim=True), G], dim=1)                      # [T, 4, 3]
        self.vol = det.abs() / 6.0
        D = torch.zeros(10, 4, 4, dtype=torch.float64)  # d(basis a)/d(lambda_m) at vertex k
        for i in range(4):
            for k in range(4):
                D[i, k, i] = 4.0 * (i == k) - 1.0
        M = torch.full((10, 10), 16.0, dtype=torch.float64)
        for e, (i, j) in enumerate(self.EDGES):
            D[4 + e, j, i] = D[4 + e, i, j] = 4.0
            for q in range(4):
                M[4 + e, q] = M[q, 4 + e] = -4.0 if q in (i, j) else -6.0
            for h, other in enumerate(self.EDGES):
                if not set(other) & {i, j}:
                    M[4 + e, 4 + h] = 8.0
            M[4 + e, 4 + e] = 32.0
        M[:4, :4] = 1.0 + 5.0 * torch.eye(4, dtype=torch.float64)
        self.D, self.M = D.to(DEVICE), (M / 420.0).to(DEVICE)
        self.W = ((torch.ones(4, 4, **dev64) + torch.eye(4, **dev64)) / 20.0)
        # diagonals for Jacobi, and the pressure mass and lumped velocity mass
        g2 = torch.einsum("akm,tmc->takc", self.D, self.grad)
        G2 = torch.einsum("takc,kl,talc->tac", g2, self.W, g2) * self.vol[:, None, None]
        diag = (self.M.diagonal()[None, :, None] * self.vol[:, None, None] / dt
                + mu * (G2.sum(-1, keepdim=True) + G2))
        self.adiag = self.scatter(diag)
        lump = torch.tensor([3.0 / 32.0] * 4 + [0.2] * 6, **dev64)
        self.lumped = self.scatter((lump[None, :, None] * self.vol[:, None, None]).expand(-1, 10, 3).contiguous())
        self.mq1 = torch.zeros(self.np, dtype=torch.float64, **dev).index_add_(
            0, self.pidx.reshape(-1), (self.vol[:, None] / 4).expand(-1, 4).reshape(-1))

    def gather(self, U):
        full = torch.zeros(self.N3, 3, dtype=torch.float64, device=DEVICE)
        full[self.inner] = U
        return full[self.nidx]

    def scatter(self, loc, every=False):
        full = torch.zeros(self.N3, 3, dtype=torch.float64, device=DEVICE)
        full.index_add_(0, self.nidx.reshape(-1), loc.reshape(-1, 3))
        return full if every else full[self.inner]

    def mass_loc(self, loc):
        return torch.einsum("ab,tbc->tac", self.M, loc) * self.vol[:, None, None]

    def A(self, U, mass=True):
        x = self.gather(U)
        H = torch.einsum("tmp,tkmc->tkpc", self.grad, torch.einsum("akm,tac->tkmc", self.D, x))
        S = torch.einsum("kl,tlpc->tkpc", self.W, H + H.transpose(2, 3)) * (self.mu * self.vol)[:, None, None, None]
        y = torch.einsum("akm,tkmc->tac", self.D, torch.einsum("tmp,tkpc->tkmc", self.grad, S))
        return self.scatter(y + self.mass_loc(x) / self.dt if mass else y)

    def load(self, f):
        return self.scatter(self.mass_loc(f[self.nidx]))

    def B(self, U):
        x = self.gather(U)
        div = torch.einsum("tmc,tkmc->tk", self.grad, torch.einsum("akm,tac->tkmc", self.D, x))
        loc = torch.einsum("kl,tl->tk", self.W, div) * self.vol[:, None]
        return torch.zeros(self.np, dtype=torch.float64, device=DEVICE).index_add_(0, self.pidx.reshape(-1),
                                                                                  loc.reshape(-1))

    def BT(self, P):
        s = torch.einsum("kl,tl->tk", self.W, P[self.pidx]) * self.vol[:, None]
        return self.scatter(torch.einsum("akm,tkmc->tac", self.D, torch.einsum("tk,tmc->tkmc", s, self.grad)))

    @staticmethod
    def cg(op, pre, b, rtol, most):
        x, r = torch.zeros_like(b), b.clone()
        z = pre(r)
        d, rz, stop = z.clone(), (r * z).sum(), rtol * b.norm()
        for it in range(most):
            q = op(d)
            a = rz / (d * q).sum()
            x += a * d
            r -= a * q
            if it % 4 == 3 and not bool(r.norm() > stop):
                break
            z = pre(r)
            new = (r * z).sum()
            d = z + (new / rz) * d
            rz = new
        return x

    def ainv(self, b, rtol=1e-12):
        return b.clone() if not bool(b.norm() > 0) else self.cg(self.A, lambda r: r / self.adiag, b, rtol, 2000)

    def solve(self, F, g):
        """A U - B^T P = F, B U = g: CG on the Schur complement, repeated on the residual."""
        def mean_free(r):
            return r - r.mean()

        ones = torch.ones(self.np, dtype=torch.float64, device=DEVICE)
        tdiag = torch.zeros_like(ones)
        b = torch.einsum("kl,alm,tmc->takc", self.W, self.D, self.grad) * self.vol[:, None, None, None]
        tdiag.index_add_(0, self.pidx.reshape(-1),
                         (b.square().sum(-1) / self.lumped_loc()[..., None]).sum(1).reshape(-1))

        def pre(r):
            r = mean_free(r)
            t = self.cg(lambda p: self.B(self.BT(p) / self.lumped), lambda q: mean_free(q / tdiag), r, 1e-8, 400)
            return mean_free(2.5 * self.mu * r / self.mq1 + t / self.dt)

        U, P = torch.zeros_like(F), torch.zeros_like(ones)
        g = torch.zeros_like(ones) if g is None else g
        size = math.sqrt(float(F.square().sum() + g.square().sum()))
        for _ in range(8):
            rF, rg = F - self.A(U) + self.BT(P), g - self.B(U)
            if math.sqrt(float(rF.square().sum() + rg.square().sum())) <= 1e-14 * size:
                break
            w = self.ainv(rF)
            dP = self.cg(lambda p: mean_free(self.B(self.ainv(self.BT(p)))), pre, mean_free(rg - self.B(w)), 1e-7, 60)
            P = P + dP
            U = U + w + self.ainv(self.BT(dP))
        return U, P - (self.mq1 @ P) / self.mq1.sum()

    def lumped_loc(self):
        full = torch.full((self.N3,), math.inf, dtype=torch.float64, device=DEVICE)
        full[self.inner] = self.lumped[:, 0]
        return full[self.nidx]

    def everywhere(self, U):
        full = torch.zeros(self.N3, 3, dtype=torch.float64, device=DEVICE)
        full[self.inner] = U
        return full


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "apply":
        if case["op"] not in ("A", "A_DF", "LOAD"):
            return None  # a V-cycle or an inexact preconditioner: what it returns is defined by its own steps
        R = _Reference(n, _vertices(n, case["jitter"], seed), case["mu"], case["dt"])
        x = _normal(seed, 301, _apply_lengths(case)[0])
        y = R.load(x.reshape(-1, 3)) if case["op"] == "LOAD" else R.A(x.reshape(3, -1).T.contiguous())
        return y.T.contiguous().reshape(-1)
    if kind == "batch" or n > 20 or case["rhs"] * n ** 3 > 8000:
        return None
    R = _Reference(n, _vertices(n, case["jitter"], seed), case["mu"], case["dt"])
    f, g = _rhs(case, n, seed)
    sol = [R.solve(R.load(f[k]), None if g is None else g[k]) for k in range(case["rhs"])]
    u, p = torch.stack([R.everywhere(U) for U, _ in sol]), torch.stack([P for _, P in sol])
    if kind == "solve":
        return u, p
    if kind == "setup":
        return u[0], p[0]
    # adjoint: K^T [lu; lp] = [jU; jP] is the forward system with lp = -P' and the pressure part negated; J sees the
    # normalised pressure, so jP first loses its component along the pressure mass of the constants
    jU, jP = _weights(case, seed)
    jP = jP - R.mq1 * jP.sum() / R.mq1.sum()
    lu, _ = R.solve(jU[R.inner], -jP)
    dmu = -(lu * R.A(sol[0][0], mass=False)).sum() / R.mu
    return u[0], p[0], R.scatter(R.mass_loc(R.gather(lu)), every=True), dmu
