"""Timed cases of the solver's public entry points.

Each case is one call (or one short sequence of calls) that a user of the
library makes, over the sizes of the repository's own configurations:

  assemble   binding.assemble_noalloc: the finest operator alone, no context
  solve      binding.Solver.solve on a hierarchy that is already set up
  step       assemble + setup + solve: the same grid with a new coefficient
  grad       autograd.solve and its backward pass (setup, solve, adjoint solve,
             per-cell gradient)
  gradbatch  autograd.solve_batch over independent members, forward and backward
  batch      binding.Batch.solve: many problems of uneven sizes, four
             right-hand sides each
  aux        binding.AuxSolver.solve: the P1 system of a physical mesh with the
             structured grid as its coarse level

Grids have n = 2^k + 1 nodes per side, the only sizes the solver takes; the
allocation-free assembly and the physical meshes take any size.  Maps:
annulus, bump and identity in 2-D, box (identity) and shell octant in 3-D.
Coefficients: one, lognormal (smooth Gaussian field), rough (independent per
cell, up to 257^2: beyond that point Gauss-Seidel needs ever more iterations
on it) and layers (1 and 1000 on either side of the shell's mid surface).
"""
import math

import numpy as np
import torch

from paper_2509_08109_gb300 import autograd, binding, inputs

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # the smallest call: the operator of a coarse problem for a caller
        # that manages its own memory; an odd size, launch-bound
        dict(name="assemble_2d_129", do="assemble", dim=2, n=129, map="annulus", coef="lognormal"),
        # quarter annulus with kappa = 1 at 65^2: the smallest configuration,
        # bound by latency and launches
        dict(name="solve_2d_65_refine", do="solve", dim=2, n=65, map="annulus", coef="one", outer="refine", tol=1e-12),
        # the constructor's defaults (FP64 V-cycle, plain CG) at an ordinary size
        dict(name="solve_2d_1025_cg", do="solve", dim=2, n=1025, map="annulus", coef="lognormal", outer="cg",
             tol=1e-10),
        # the headline workload: 16.8 M unknowns, FP32 V-cycle with FP64 refinement
        dict(name="solve_2d_4097_refine", do="solve", dim=2, n=4097, map="annulus", coef="lognormal", outer="refine",
             tol=1e-10),
        # 3-D with the constructor's defaults
        dict(name="solve_3d_129_cg", do="solve", dim=3, n=129, map="box", coef="lognormal", outer="cg", tol=1e-10),
        # the spherical-shell octant with a 1/1000 coefficient: hundreds of
        # iterations on one hierarchy
        dict(name="solve_3d_shell_129_refine", do="solve", dim=3, n=129, map="shell", coef="layers", outer="refine",
             tol=1e-12),
        # the largest 3-D grid
        dict(name="solve_3d_257_refine", do="solve", dim=3, n=257, map="box", coef="lognormal", outer="refine",
             tol=1e-10),
        # a time step or an outer iteration with a new coefficient: setup counts
        dict(name="step_3d_129_refine", do="step", dim=3, n=129, map="box", coef="lognormal", outer="refine",
             tol=1e-10),
        # one member of a coefficient inversion: forward and backward at 513^2
        dict(name="grad_2d_513_refine", do="grad", dim=2, n=513, map="annulus", coef="lognormal", outer="refine",
             tol=1e-10),
        # eight inversions at once, each member on its own stream
        dict(name="gradbatch_2d_513x8", do="gradbatch", dim=2, n=513, map="annulus", coef="lognormal",
             outer="refine", members=8, tol=1e-10),
        # uneven problems, four right-hand sides each, solved together
        dict(name="batch_2d_16x4", do="batch", members=16, kmin=6, kmax=10, nrhs=4, tol=1e-10),
        # the physical-mesh solve, flexible CG around the two-grid cycle
        dict(name="aux_423x632_fcg", do="aux", nr=423, nt=632, n=257, krylov=True, tol=1e-10),
    ]


def draw(rng):
    do = rng.choice(["assemble", "solve", "solve", "solve", "step", "step", "grad", "gradbatch", "batch", "aux"])
    if do == "assemble":
        dim = rng.choice([2, 3])
        n = _log_int(rng, 20, 640) if dim == 2 else _log_int(rng, 8, 48)
        return dict(do=do, dim=dim, n=n, map="bump" if dim == 2 else "shell", coef="lognormal")
    if do in ("solve", "step"):
        dim = rng.choice([2, 3])
        outer = rng.choice(["cg", "refine", "flexible"])
        if dim == 2:
            mp = rng.choice(["annulus", "bump"])
            coef = rng.choice(["one", "lognormal", "rough"])
            k = rng.randint(5, 8 if coef == "rough" else 12)
            return dict(do=do, dim=2, n=2 ** k + 1, map=mp, coef=coef, outer=outer,
                        tol=rng.choice([1e-10, 1e-12]) if k <= 10 else 1e-10)
        mp = rng.choice(["box", "shell"])
        if mp == "shell":
            return dict(do=do, dim=3, n=2 ** rng.randint(4, 6) + 1, map=mp, coef="layers", outer=outer, tol=1e-12)
        k = rng.randint(4, 8 if do == "solve" else 7)
        return dict(do=do, dim=3, n=2 ** k + 1, map=mp, coef=rng.choice(["one", "lognormal"]), outer=outer,
                    tol=rng.choice([1e-10, 1e-12]))
    if do == "grad":
        dim = rng.choice([2, 2, 3])
        outer = rng.choice(["cg", "refine"])
        if dim == 2:
            coef = rng.choice(["rough", "lognormal"])
            return dict(do=do, dim=2, n=2 ** rng.randint(5, 8 if coef == "rough" else 9) + 1,
                        map=rng.choice(["annulus", "bump"]), coef=coef, outer=outer, tol=1e-10)
        return dict(do=do, dim=3, n=2 ** rng.randint(4, 6) + 1, map="box", coef="rough", outer=outer, tol=1e-10)
    if do == "gradbatch":
        return dict(do=do, dim=2, n=2 ** rng.randint(6, 9) + 1, map="annulus", coef="lognormal", outer="refine",
                    members=rng.randint(2, 8), tol=1e-10)
    if do == "batch":
        return dict(do=do, members=_log_int(rng, 3, 16), kmin=6, kmax=rng.randint(7, 10), nrhs=rng.randint(1, 4),
                    tol=1e-10)
    nr = _log_int(rng, 60, 423)
    nt = int(nr * rng.uniform(1.2, 1.5))
    return dict(do="aux", nr=nr, nt=nt, n=2 ** max(5, min(8, round(math.log2(0.53 * math.sqrt(nr * nt))))) + 1,
                krylov=rng.random() < 0.75, tol=1e-10)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# ------------------------------------------------------------------ inputs
def _coords(dim, n, mp, gen):
    s = torch.linspace(0.0, 1.0, n, dtype=F64, device=DEV)
    if dim == 2:
        s, t = s[None, :].expand(n, n), s[:, None].expand(n, n)
        if mp == "annulus":
            r, th = 0.5 + 0.5 * s, 0.5 * math.pi * t
            return torch.stack([r * torch.cos(th), r * torch.sin(th)]).contiguous()
        if mp == "bump":
            a, b = gen.uniform(-0.15, 0.15, size=2)
            w = torch.sin(math.pi * s) * torch.sin(math.pi * t)
            return torch.stack([s + a * w, t + b * w]).contiguous()
        return torch.stack([s, t]).contiguous()
    x, y, z = (s[None, None, :].expand(n, n, n), s[None, :, None].expand(n, n, n), s[:, None, None].expand(n, n, n))
    if mp == "shell":
        r, th, ph = 0.5 + 0.5 * x, 0.5 * math.pi * y, 0.5 * math.pi * z
        return torch.stack([r * torch.sin(th) * torch.cos(ph), r * torch.sin(th) * torch.sin(ph),
                            r * torch.cos(th)]).contiguous()
    return torch.stack([x, y, z]).contiguous()


def _corner(c, dim, b):
    """Values of nodal field c (..., n, n[, n]) at corner b of every cell."""
    sl = tuple(slice(1, None) if (b >> a) & 1 else slice(0, -1) for a in reversed(range(dim)))
    return c[(Ellipsis,) + sl]


def _kappa(dim, n, coef, coords, gen):
    shape = (n - 1,) * dim
    if coef == "one":
        return torch.ones(shape, dtype=F64, device=DEV)
    if coef == "layers":
        k = torch.ones(shape, dtype=F64, device=DEV)
        k[..., (n - 1) // 2:] = 1000.0
        return k
    if coef == "rough":
        return torch.exp(0.5 * torch.randn(shape, dtype=F64, device=DEV, generator=_torch_gen(gen)))
    field = inputs.GaussianField.draw(gen, dim)
    centre = sum(_corner(coords, dim, b) for b in range(2 ** dim)) / 2 ** dim
    return torch.exp(field(centre)).contiguous()


def _torch_gen(gen):
    return torch.Generator(DEV).manual_seed(int(gen.integers(1 << 31)))


def _load(dim, n, gen, lead=()):
    """U[-1, 1] per interior node, zero on the boundary."""
    f = torch.rand(lead + (n,) * dim, dtype=F64, device=DEV, generator=_torch_gen(gen)) * 2.0 - 1.0
    for a in range(dim):
        f.select(-1 - a, 0).zero_()
        f.select(-1 - a, n - 1).zero_()
    return f


def _problem(case, seed):
    gen = np.random.default_rng(seed)
    dim, n = case["dim"], case["n"]
    coords = _coords(dim, n, case["map"], gen)
    return gen, coords, _kappa(dim, n, case["coef"], coords, gen)


def _batch_problems(case, seed):
    """(n, coords, kappa, right-hand sides) of every member: the sizes go
    round k = kmax .. kmin so that every size class is present."""
    gen = np.random.default_rng(seed)
    ks = list(range(case["kmax"], case["kmin"] - 1, -1))
    out = []
    for p in range(case["members"]):
        n = 2 ** ks[p % len(ks)] + 1
        coords = _coords(2, n, "bump", gen)
        out.append((n, coords, _kappa(2, n, "lognormal", coords, gen), _load(2, n, gen, (case["nrhs"],))))
    return out


def _solver(case, stream=None):
    return binding.Solver(case["dim"], case["n"], precision="fp64" if case["outer"] == "cg" else "fp32",
                          outer=case["outer"], stream=stream)


def prepare(case, seed):
    do = case["do"]
    if do == "batch":
        probs = _batch_problems(case, seed)
        solvers = [binding.Solver(2, n, precision="fp32", outer="refine").assemble(c, k).setup()
                   for n, c, k, _ in probs]
        return dict(case=case, batch=binding.Batch(solvers), bs=[list(f.unbind(0)) for _, _, _, f in probs],
                    rhs=[f for _, _, _, f in probs])
    if do == "aux":
        mesh = inputs.annulus_mesh(case["nr"], case["nt"], seed=seed)
        coarse = binding.Solver(2, case["n"], precision="fp32")
        n = case["n"]
        coarse.assemble(_coords(2, n, "annulus", None), torch.ones((n - 1, n - 1), dtype=F64, device=DEV)).setup()
        return dict(case=case, aux=binding.AuxSolver(coarse, mesh, krylov=case["krylov"]),
                    f=torch.as_tensor(mesh.f, device=DEV))
    gen, coords, kappa = _problem(case, seed)
    dim, n = case["dim"], case["n"]
    if do == "assemble":
        return dict(case=case, coords=coords, kappa=kappa,
                    out=torch.empty((n,) * dim + (3 ** dim,), dtype=F64, device=DEV))
    if do in ("solve", "step"):
        f = _load(dim, n, gen)
        s = _solver(case)
        if do == "solve":
            s.assemble(coords, kappa).setup()
        return dict(case=case, solver=s, coords=coords, kappa=kappa, f=f)
    members = case.get("members", 1)
    ms = [torch.log(kappa if b == 0 else _kappa(dim, n, case["coef"], coords, gen)).requires_grad_(True)
          for b in range(members)]
    fs = [_load(dim, n, gen).requires_grad_(True) for _ in range(members)]
    obs = [_load(dim, n, gen) for _ in range(members)]
    solvers = [_solver(case, torch.cuda.Stream() if do == "gradbatch" else None) for _ in range(members)]
    return dict(case=case, solvers=solvers, coords=coords, ms=ms, fs=fs, obs=obs)


def run(state):
    case = state["case"]
    do, tol = case["do"], case.get("tol")
    if do == "assemble":
        return binding.assemble_noalloc(case["dim"], case["n"], state["coords"], state["kappa"], state["out"])
    if do == "solve":
        return state["solver"].solve(state["f"], tol=tol, maxit=2000)[0]
    if do == "step":
        state["solver"].assemble(state["coords"], state["kappa"]).setup()
        return state["solver"].solve(state["f"], tol=tol, maxit=2000)[0]
    if do == "batch":
        xs = [torch.zeros_like(f) for f in state["rhs"]]
        state["batch"].solve(state["bs"], [list(x.unbind(0)) for x in xs], tol=tol)
        return xs
    if do == "aux":
        return state["aux"].solve(state["f"], tol=tol)[0]
    if do == "grad":
        us = [autograd.solve(state["ms"][0], state["fs"][0], state["coords"], state["solvers"][0], tol=tol)]
    else:
        us = autograd.solve_batch(state["ms"], state["fs"], state["coords"], state["solvers"], tol=tol)
    loss = sum(0.5 * ((u - o) ** 2).sum() for u, o in zip(us, state["obs"]))
    grads = torch.autograd.grad(loss, state["ms"] + state["fs"])
    k = len(us)
    return {"u": [u.detach() for u in us], "dm": list(grads[:k]), "df": list(grads[k:])}


def work(case):
    """Inputs read once and outputs written once: the symmetric half of the
    operator, right-hand side and solution (FP64); for a setup the map and the
    coefficient instead of the operator.  Operations: one residual per
    solve, and the element matrices where the operator is formed."""
    do = case["do"]
    if do == "aux":
        nv = case["nr"] * case["nt"]
        return {"bytes": nv * (4 * 8 + 4 * 4 + 16), "flops": nv * 14}
    if do == "batch":
        ks = list(range(case["kmax"], case["kmin"] - 1, -1))
        nodes = sum((2 ** ks[p % len(ks)] + 1) ** 2 for p in range(case["members"]))
        return {"bytes": nodes * (40 + 16 * case["nrhs"]), "flops": nodes * 18 * case["nrhs"]}
    dim = case["dim"]
    nodes = float(case["n"]) ** dim
    half, row, elem = (5, 9, 200) if dim == 2 else (14, 27, 1500)
    if do == "assemble":
        return {"bytes": nodes * 8 * (dim + 1 + row), "flops": nodes * elem}
    if do == "solve":
        return {"bytes": nodes * 8 * (half + 2), "flops": nodes * 2 * row}
    if do == "step":
        return {"bytes": nodes * 8 * (dim + 1 + 2), "flops": nodes * (elem + 2 * row)}
    # coords once; m, f, u_obs in; u, dL/dm, dL/df out, per member
    members = case.get("members", 1)
    return {"bytes": nodes * 8 * (dim + 6 * members), "flops": nodes * members * (2 * elem + 4 * row)}


# ------------------------------------------------------------------ 64-bit values
def _element_matrices(coords, dim):
    """K[a][b] per cell at kappa = 1: trilinear (bilinear) elements, two
    Gauss points per direction, isoparametric map."""
    nb = 2 ** dim
    g = [0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)]
    X = [torch.stack([_corner(coords[r], dim, b) for b in range(nb)]) for r in range(dim)]
    K = None
    for q in range(nb):
        xi = [g[(q >> a) & 1] for a in range(dim)]
        grad = np.zeros((nb, dim))
        for b in range(nb):
            for m in range(dim):
                v = 1.0
                for a in range(dim):
                    bit = (b >> a) & 1
                    v *= (1.0 if bit else -1.0) if a == m else (xi[a] if bit else 1.0 - xi[a])
                grad[b, m] = v
        G = torch.as_tensor(grad, device=coords.device)
        J = torch.stack([torch.stack([torch.tensordot(G[:, m], X[r], 1) for m in range(dim)], -1)
                         for r in range(dim)], -2)          # (..., r, m)
        if dim == 2:
            det = J[..., 0, 0] * J[..., 1, 1] - J[..., 0, 1] * J[..., 1, 0]
            adj = torch.stack([torch.stack([J[..., 1, 1], -J[..., 0, 1]], -1),
                               torch.stack([-J[..., 1, 0], J[..., 0, 0]], -1)], -2)
        else:
            c = [torch.linalg.cross(J[..., (r + 1) % 3, :], J[..., (r + 2) % 3, :], dim=-1) for r in range(3)]
            adj = torch.stack(c, -1)                         # adj[m, r]
            det = (J[..., 0, :] * c[0]).sum(-1)
        w = adj @ adj.transpose(-1, -2) / (det * nb)[..., None, None]
        part = torch.einsum("am,...mp,bp->ab...", G, w, G)
        K = part if K is None else K + part
    return K


class _Operator:
    """The assembled operator with the boundary nodes eliminated, as one
    coefficient array per neighbour offset."""

    def __init__(self, coords, kappa):
        dim = self.dim = coords.shape[0]
        n = self.n = coords.shape[-1]
        K = _element_matrices(coords, dim) * kappa
        self.a = torch.zeros((3 ** dim,) + (n,) * dim, dtype=F64, device=coords.device)
        for a in range(2 ** dim):
            for b in range(2 ** dim):
                o = sum((((b >> t) & 1) - ((a >> t) & 1) + 1) * 3 ** t for t in range(dim))
                _corner(self.a[o], dim, a).add_(K[a, b])
        inner = torch.zeros((n,) * dim, dtype=F64, device=coords.device)
        inner[(slice(1, -1),) * dim] = 1.0
        self.shift = []
        for o in range(3 ** dim):
            d = [o // 3 ** t % 3 - 1 for t in range(dim)]
            sl = tuple(slice(1 + d[t], n - 1 + d[t]) for t in reversed(range(dim)))
            self.shift.append((Ellipsis,) + sl)
            core = self.a[o][(slice(1, -1),) * dim] * inner[sl]
            self.a[o].zero_()
            self.a[o][(slice(1, -1),) * dim] = core
        self.core = (Ellipsis,) + (slice(1, -1),) * dim
        self.diag = self.a[3 ** dim // 2]

    def __call__(self, x):
        y = torch.zeros_like(x)
        yc = y[self.core]
        for o, sl in enumerate(self.shift):
            yc.addcmul_(self.a[o][self.core], x[sl])
        return y

    def precondition(self, r):
        z = torch.zeros_like(r)
        z[self.core] = r[self.core] / self.diag[self.core]
        return z


class _Mesh:
    """The P1 stiffness matrix of a triangulation with its boundary vertices
    eliminated."""

    def __init__(self, mesh):
        xy = mesh.xy[mesh.tri]
        e = np.stack([xy[:, (k + 2) % 3] - xy[:, (k + 1) % 3] for k in range(3)], 1)
        area2 = e[:, 0, 0] * e[:, 1, 1] - e[:, 0, 1] * e[:, 1, 0]
        K = np.einsum("tad,tbd->tab", e, e) * (mesh.kappa / (2.0 * area2))[:, None, None]
        inner = ~mesh.dirichlet
        row, col = np.repeat(mesh.tri, 3, 1).reshape(-1), np.tile(mesh.tri, (1, 3)).reshape(-1)
        keep = inner[row] & inner[col]
        nv = len(inner)
        self.inner = torch.as_tensor(inner, device=DEV).to(F64)
        at = torch.as_tensor(np.stack([row[keep], col[keep]]).astype(np.int64), device=DEV)
        A = torch.sparse_coo_tensor(at, torch.as_tensor(K.reshape(-1)[keep], device=DEV), (nv, nv)).coalesce()
        d = torch.zeros(nv, dtype=F64, device=DEV)
        on = A.indices()[0] == A.indices()[1]
        d[A.indices()[0][on]] = A.values()[on]
        self.diag = torch.where(d > 0, d, torch.ones_like(d))
        self.A = A.to_sparse_csr()

    def __call__(self, x):
        return (self.A @ x[0][:, None])[:, 0][None]

    def precondition(self, r):
        return r / self.diag * self.inner


def _solve64(A, b, maxit=30000):
    """A x = b by Jacobi-preconditioned CG for every right-hand side along
    the first axis, restarted from the true residual until it is at the
    rounding level."""
    axes = tuple(range(1, b.dim()))
    dot = lambda u, v: (u * v).sum(axes, keepdim=True)       # noqa: E731
    x = torch.zeros_like(b)
    for goal in (1e-9, 1e-6):
        r = b - A(x)
        d = torch.zeros_like(b)
        z = A.precondition(r)
        p, rz, rr0 = z, dot(r, z), dot(r, r)
        for it in range(maxit):
            q = A(p)
            alpha = rz / dot(p, q).clamp_min(1e-300)
            d.addcmul_(alpha, p)
            r = r - alpha * q
            if it % 50 == 49 and bool((dot(r, r) <= goal ** 2 * rr0).all()):
                break
            z = A.precondition(r)
            rz, old = dot(r, z), rz
            p = z + rz / old.clamp_min(1e-300) * p
        x = x + d
    return x


def exact(case, seed):
    """The same problem assembled and solved by plain torch in 64 bits; None
    where its Jacobi-preconditioned CG would take too long."""
    do = case["do"]
    if do == "aux":
        mesh = inputs.annulus_mesh(case["nr"], case["nt"], seed=seed)
        return _solve64(_Mesh(mesh), torch.as_tensor(mesh.f, device=DEV)[None])[0]
    if do == "batch":
        return [_solve64(_Operator(c, k), f) if n <= 257 else None for n, c, k, f in _batch_problems(case, seed)]
    dim, n = case["dim"], case["n"]
    if n > (1025 if dim == 2 else 257) or n * case.get("members", 1) > 4104:
        return None
    gen, coords, kappa = _problem(case, seed)
    if do == "assemble":
        return torch.movedim(_Operator(coords, kappa).a, 0, -1).contiguous()
    if do in ("solve", "step"):
        return _solve64(_Operator(coords, kappa), _load(dim, n, gen)[None])[0]
    members = case.get("members", 1)
    kappas = [kappa if b == 0 else _kappa(dim, n, case["coef"], coords, gen) for b in range(members)]
    fs = [_load(dim, n, gen) for _ in range(members)]
    obs = [_load(dim, n, gen) for _ in range(members)]
    out = {"u": [], "dm": [], "df": []}
    K = _element_matrices(coords, dim)
    for kap, f, o in zip(kappas, fs, obs):
        A = _Operator(coords, kap)
        u = _solve64(A, f[None])[0]
        lam = _solve64(A, (u - o)[None])[0]
        ue = torch.stack([_corner(u, dim, b) for b in range(2 ** dim)])
        le = torch.stack([_corner(lam, dim, b) for b in range(2 ** dim)])
        out["u"].append(u)
        out["dm"].append(-kap * torch.einsum("a...,ab...,b...->...", le, K, ue))
        out["df"].append(lam)
    return out
