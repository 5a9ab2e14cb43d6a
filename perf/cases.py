"""The work a user of the FETI dual-operator library has it do, as timed cases.

Each case is one pass through the Python binding (`paper_2502_08382_gb300.feti`): applying the explicit or the
implicit dual operator, assembling it, one whole step (assembly and the projected CG solve), or the adjoint.
Meshes are the box meshes of `problems.py`: Q1 quads / Hex8 bricks, heat with lognormal conductivity, elasticity
(constant modulus, or a random density field with E = rho^3), Total FETI gluing.  Subdomain shapes are those of the five named
workloads; the subdomain counts are smaller, so that inputs are quick to make.

A case: kind, physics ("heat2d", "heat3d", "elast3d"), `axis` subdomains per axis, `elems` elements per axis and
subdomain (`hi` > 0: uneven cuts of elems..hi), prec, precond, route, and `spread`, the sigma of the log-conductivity (heat)
or the lowest density (elasticity's adjoint).  The heat cases' conductivities and the adjoint's
densities come from the seed; the other elasticity cases have a constant modulus, as workload 3 has, and a load
density that comes from the seed.
"""
import dataclasses
import functools
import random
import warnings

import numpy as np
import torch

from paper_2502_08382_gb300 import feti
from paper_2502_08382_gb300.problems import make_problem, subdomain_K_values

TOL = 1e-10  # of the solves, the benchmark's


def _case(name, kind, physics, axis, elems, prec, hi=0, precond="none", route="syrk", spread=None):
    if spread is None:  # the named workloads' materials
        spread = {"heat2d": 1.0, "heat3d": 0.5, "elast3d": 0.1}[physics]
    return {"name": name, "kind": kind, "physics": physics, "axis": axis, "elems": elems, "hi": hi, "prec": prec,
            "precond": precond, "route": route, "spread": spread}


def listed():
    return [
        # the smallest call: F.p of workload 1 (16 subdomains of 16x16), all latency
        _case("apply_small_2d_fp64", "apply", "heat2d", 4, 16, "fp64"),
        # one application inside a user's own Krylov loop, workload 3's subdomains, F far larger than L2
        _case("apply_elast3d_mixed", "apply", "elast3d", 5, 12, "split_bf16"),
        # the same with FP64 tiles on workload 4's uneven subdomains: ragged tiles, every size of subdomain
        _case("apply_heat3d_uneven_fp64", "apply", "heat3d", 5, 8, "fp64", hi=24),
        # the implicit operator of a solve's refinement (workload 2's subdomains, many small fronts)
        _case("implicit_heat2d", "implicit", "heat2d", 24, 64, "split_bf16"),
        # assembling for a user's own solver, everything in FP64: 2D, small fronts
        _case("assemble_heat2d_fp64", "assemble", "heat2d", 16, 64, "fp64"),
        # the same in 3D with uneven subdomains: large separators, unequal work
        _case("assemble_heat3d_uneven_fp64", "assemble", "heat3d", 4, 8, "fp64", hi=24),
        # and with workload 3's elasticity subdomains: the largest FP64 assembly
        _case("assemble_elast3d_fp64", "assemble", "elast3d", 3, 12, "fp64"),
        # the smallest whole step (workload 1): assembly, solve and recovery of u in FP64
        _case("step_small_2d_fp64", "step", "heat2d", 4, 16, "fp64"),
        # a time step of a multi-step 2D run: new K values, mixed assembly, solve (workload 2's subdomains)
        _case("step_heat2d_mixed", "new_step", "heat2d", 16, 64, "split_bf16"),
        # the headline step: mixed assembly and solve of 3D elasticity (workload 3's subdomains)
        _case("step_elast3d_mixed", "step", "elast3d", 4, 12, "split_bf16"),
        # uneven 3D heat with the lumped preconditioner and the TF32 SYRK (workload 4's ranges)
        _case("step_heat3d_lumped_tf32", "step", "heat3d", 5, 8, "tf32", hi=24, precond="lumped"),
        # the sensitivity: assembly is done, dL/dtheta of L = sum <W_i, F_i> for every element
        _case("adjoint_elast3d", "adjoint", "elast3d", 2, 10, "fp64"),
    ]


def draw(rng):
    kind = rng.choice(["apply", "apply", "implicit", "assemble", "assemble", "step", "step", "new_step", "new_step", "adjoint"])
    physics = rng.choice(["heat2d", "heat3d", "elast3d"]) if kind != "adjoint" else "elast3d"
    span = {"heat2d": ((2, 20), (5, 80)), "heat3d": ((2, 5), (3, 20)), "elast3d": ((1, 4), (2, 12))}[physics]
    if kind == "adjoint":
        span = ((1, 3), (3, 10))
    log = lambda lo, hi: int(round(lo * (hi / lo) ** rng.random()))  # noqa: E731
    axis, elems = log(*span[0]), log(*span[1])
    # no more elements in all than the largest listed cases have
    axis = max(span[0][0], min(axis, {"heat2d": 1280, "heat3d": 60, "elast3d": 40}[physics] // elems))
    if kind == "adjoint":
        axis = min(axis, max(1, 20 // elems))
    hi = 0
    if physics != "elast3d" and rng.random() < 0.4:
        hi = min(span[1][1], elems + rng.randrange(1, elems + 2))
        hi = 0 if hi <= elems else hi
    prec = "fp64" if kind == "adjoint" else rng.choice(["fp64", "split_bf16", "split_bf16", "tf32"])
    precond = rng.choice(["none", "none", "lumped"]) if "step" in kind else "none"
    route = "schur" if kind != "adjoint" and elems <= 12 and rng.random() < 0.15 else "syrk"
    spread = round(rng.uniform(0.05, 0.3) if physics == "elast3d" else rng.uniform(0.3, 1.1), 3)
    c = _case("", kind, physics, axis, elems, prec, hi, precond, route, spread)
    del c["name"]
    return c


# ---- inputs


@functools.lru_cache(maxsize=4)
def _geometry(physics, axis, elems, hi):
    """The mesh and its gluing (no material): a user's program reads these once."""
    dim = 2 if physics == "heat2d" else 3
    if hi > elems:
        # the same multiset of widths on every axis, in another order: equal element counts per axis
        r = random.Random(1000 * axis + 100 * elems + hi)
        some = [elems, r.randint(elems, hi), hi]
        w = [r.choice(some) for _ in range(axis)]
        cuts = [r.sample(w, axis) for _ in range(dim)]
    else:
        cuts = [[elems] * axis] * dim
    return make_problem(dim=dim, physics="elasticity" if physics == "elast3d" else "heat", cuts=cuts)


class _Values:
    """The problem's geometry with the material of one seed."""

    def __init__(self, case, seed):
        P = _geometry(case["physics"], case["axis"], case["elems"], case["hi"])
        rng = np.random.default_rng([seed, 20])
        ne = int(np.prod(P.elem_global_shape))
        if case["physics"] == "elast3d" and case["kind"] != "adjoint":
            self.coef, self.dcoef = np.ones(ne), np.zeros(ne)
        elif case["physics"] == "elast3d":
            rho = rng.uniform(case["spread"], 1.0, size=ne)
            self.coef, self.dcoef = rho ** 3, 3.0 * rho ** 2
        else:
            self.coef = np.exp(rng.normal(0.0, case["spread"], size=ne))
            self.dcoef = self.coef.copy()
        self.base = P
        if case["physics"] == "elast3d" and case["kind"] != "adjoint":
            self.K = [s.K_val for s in P.subs]
            load = rng.uniform(0.5, 1.5, size=ne)
            # the consistent load of a body force that varies from element to element
            self.f = []
            for s in P.subs:
                ed = s.elem_dofs[:, 2::3]
                w = np.repeat(load[s.elem_global] * (-P.h ** 3 / 8.0), 8)
                self.f.append(np.bincount(ed.ravel(), weights=w, minlength=s.n))
        else:
            self.K = [subdomain_K_values(P, i, self.coef[s.elem_global]) for i, s in enumerate(P.subs)]
            self.f = [s.f for s in P.subs]

    def problem(self):
        subs = [dataclasses.replace(s, K_val=k, f=f, elem_coef=self.coef[s.elem_global],
                                    elem_dcoef=self.dcoef[s.elem_global])
                for s, k, f in zip(self.base.subs, self.K, self.f)]
        return dataclasses.replace(self.base, subs=subs)


def _vector(n, seed):
    return np.random.default_rng([seed, 21]).normal(0.0, 1.0, size=n)


def _weights(P, seed):
    """Symmetric N(0, 1) weights W_i, concatenated (made on the GPU where there is one)."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device=dev).manual_seed(seed + 5)
    out = []
    for s in P.subs:
        a = torch.randn(s.m, s.m, generator=g, device=dev, dtype=torch.float64)
        out.append((torch.tril(a) + torch.tril(a, -1).T).reshape(-1))
    return torch.cat(out)


def prepare(case, seed):
    V = _Values(case, seed)
    kind = case["kind"]
    mixed = case["prec"] != "fp64"
    op = feti.FetiOperator(V.problem(), prec=case["prec"], tol=TOL, maxit=4000, precond=case["precond"],
                           route=case["route"], refine_drop=1e-4 if mixed else 0.0, refine_restart=mixed,
                           with_elements=kind == "adjoint")
    s = {"kind": kind, "op": op}
    # the first assembly (its autotuning and graph) belongs to the handle that a program keeps
    op.assemble()
    if kind in ("apply", "implicit", "assemble"):
        s["p"] = torch.from_numpy(_vector(op.n_lambda, seed)).cuda()
    if kind == "new_step":
        # the next time step's material: other values on the same pattern
        s["K"] = _Values(case, seed + 100_003).K
    if kind == "adjoint":
        s["W"] = _weights(V.base, seed)
    return s


def run(s):
    op, kind = s["op"], s["kind"]
    if kind == "apply":
        return op.apply(s["p"])
    if kind == "implicit":
        return op.apply_implicit(s["p"])
    if kind == "assemble":
        op.assemble()
        return op.apply(s["p"])
    if kind == "adjoint":
        return op.adjoint(s["W"])
    if kind == "new_step":
        for i, v in enumerate(s["K"]):
            op.update_values(i, v)
    op.assemble()
    lam, alpha, u, _ = op.solve()
    return lam, alpha, u


# ---- what a pass cannot do without


@functools.lru_cache(maxsize=64)
def _counts(physics, axis, elems, hi, route):
    """(sum nnz(K), sum nnz(L), assembly flops, sum m(m+1)/2, sum n, sum m, n_lambda, sum n m (n + m))."""
    P = _geometry(physics, axis, elems, hi)
    seen, tot = {}, np.zeros(8)
    for s in P.subs:
        key = (s.shape, s.B_dof.tobytes())
        if key not in seen:
            a = feti.analyse(s, route=route)
            seen[key] = (s.nnz, a["nnzL"], a["chol_flops"] + a["trsm_flops"] + a["syrk_flops"],
                         s.m * (s.m + 1) / 2, s.n, s.m)
        nnz, nl, fl, mm, n, m = seen[key]
        tot += [nnz, nl, fl, mm, n, m, 0, 4.0 * nl * m + 2.0 * n * m * m]
    tot[6] = P.n_lambda
    return tuple(float(x) for x in tot)


def work(case):
    nnz, nl, fl, mm, n, m, nlam, adj = _counts(case["physics"], case["axis"], case["elems"], case["hi"], case["route"])
    e = 8 if case["prec"] == "fp64" else 4
    kind = case["kind"]
    if kind == "apply":
        return {"bytes": e * mm + 20 * m + 16 * nlam, "flops": 4 * mm}
    if kind == "implicit":
        return {"bytes": 8 * nl + 20 * m + 16 * nlam, "flops": 4 * nl}
    if kind == "assemble":
        return {"bytes": 8 * nnz + e * mm + 16 * nlam, "flops": fl}
    if kind == "adjoint":
        return {"bytes": 8 * nl + 16 * mm + 16 * n, "flops": adj}
    # a step: K read once, F written once and read once (the iterations' reads depend on the values)
    return {"bytes": 8 * nnz + 2 * e * mm + 24 * n + 16 * nlam, "flops": fl}


# ---- 64-bit references in plain torch


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _dense_factor(s, K):
    """Cholesky factor of K + rho * (unit penalty on the fixing DOFs), rho = max diag K, dense."""
    A = torch.sparse_csr_tensor(torch.from_numpy(s.K_rowptr), torch.from_numpy(s.K_col.astype(np.int64)),
                                torch.from_numpy(K), size=(s.n, s.n)).to(_dev()).to_dense()
    fix = torch.from_numpy(s.fix_dofs.astype(np.int64)).to(A.device)
    A[fix, fix] += torch.diagonal(A).max()
    return torch.linalg.cholesky(A)


def _exact_apply(case, seed):
    V = _Values(case, seed)
    P = V.base
    if sum(s.n ** 3 / 3.0 for s in P.subs) > 6e12:
        return None  # dense factorisations of that many DOFs take too long
    p = torch.from_numpy(_vector(P.n_lambda, seed)).to(_dev())
    q = torch.zeros_like(p)
    for s, K in zip(P.subs, V.K):
        L = _dense_factor(s, K)
        lam = torch.from_numpy(s.B_lambda.astype(np.int64)).to(p.device)
        dof = torch.from_numpy(s.B_dof.astype(np.int64)).to(p.device)
        sg = torch.from_numpy(s.B_sign).to(p.device)
        b = torch.zeros(s.n, dtype=torch.float64, device=p.device).index_add_(0, dof, sg * p[lam])
        q.index_add_(0, lam, sg * torch.cholesky_solve(b[:, None], L)[dof, 0])
    return q


def _exact_adjoint(case, seed):
    V = _Values(case, seed)
    P = V.base
    if sum(s.n ** 3 / 3.0 for s in P.subs) > 2e12:
        return None
    W = _weights(P, seed)
    Kref = torch.from_numpy(np.array(P.K_ref)).to(W.device)
    out, o = [], 0
    for s, K in zip(P.subs, V.K):
        L = _dense_factor(s, K)
        B = torch.zeros(s.n, s.m, dtype=torch.float64, device=W.device)
        B[torch.from_numpy(s.B_dof.astype(np.int64)), torch.arange(s.m)] = torch.from_numpy(s.B_sign).to(W.device)
        Z = torch.cholesky_solve(B, L)
        H = Z @ W[o:o + s.m * s.m].reshape(s.m, s.m) @ Z.T
        o += s.m * s.m
        ed = torch.from_numpy(s.elem_dofs.astype(np.int64)).to(W.device)
        g = (H[ed[:, :, None], ed[:, None, :]] * Kref).sum((1, 2))
        out.append(-g * torch.from_numpy(V.dcoef[s.elem_global]).to(W.device))
    return torch.cat(out)


def _cg(mul, b, diag, tol, maxit):
    """Jacobi CG, with the residual recomputed between rounds (its accuracy is that of `mul`)."""
    x = torch.zeros_like(b)
    for _ in range(4):
        r = b - mul(x)
        if not bool(r.norm() > tol * b.norm()):
            break
        z = r / diag
        d, rz, stop = z.clone(), torch.dot(r, z), 1e-4 * tol * float(b.norm()) + 1e-11 * float(r.norm())
        e = torch.zeros_like(b)
        for k in range(maxit):
            q = mul(d)
            a = rz / torch.dot(d, q).clamp(min=1e-300)  # 0 / 0 once r is exactly zero
            e += a * d
            r -= a * q
            if k % 50 == 49 and float(r.norm()) <= stop:
                break
            z = r / diag
            new = torch.dot(r, z)
            d = z + (new / rz.clamp(min=1e-300)) * d
            rz = new
        x = x + e
    return x


def _exact_step(case, seed):
    """u from the monolithic system by CG; lambda from the subdomains' residual forces (B^T lambda = f - K u, B of
    full row rank); alpha from u at the fixing DOFs, where K_reg^-1 of a balanced load vanishes."""
    V = _Values(case, seed + 100_003 if case["kind"] == "new_step" else seed)
    P, dev = V.base, _dev()
    if P.n_global_dofs > 1_500_000:
        return None
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    off = np.concatenate([[0], np.cumsum([s.n for s in P.subs])])
    l2g = t(np.concatenate([s.l2g for s in P.subs]))
    rows = t(np.concatenate([np.repeat(np.arange(s.n), np.diff(s.K_rowptr)) + o for s, o in zip(P.subs, off)]))
    cols = t(np.concatenate([s.K_col.astype(np.int64) + o for s, o in zip(P.subs, off)]))
    vals = t(np.concatenate(V.K))
    n = int(off[-1])
    warnings.filterwarnings("ignore", message="Sparse")
    Kb = torch.sparse_coo_tensor(torch.stack([rows, cols]), vals, (n, n)).coalesce().to_sparse_csr()
    f = t(np.concatenate(V.f))
    free = torch.ones(P.n_global_dofs, dtype=torch.float64, device=dev)
    free[t(P.dirichlet_dofs)] = 0.0
    gather = lambda y: torch.zeros(P.n_global_dofs, dtype=torch.float64, device=dev).index_add_(0, l2g, y)  # noqa: E731
    mul = lambda x: free * gather((Kb @ (free * x)[l2g][:, None])[:, 0]) + (1 - free) * x  # noqa: E731
    diag = free * gather(torch.zeros(n, dtype=torch.float64, device=dev).index_add_(
        0, rows, torch.where(rows == cols, vals, torch.zeros_like(vals)))) + (1 - free)
    u = (free * _cg(mul, free * gather(f), diag, 1e-15, 20000))[l2g]
    r = f - (Kb @ u[:, None])[:, 0]
    lam = t(np.concatenate([s.B_lambda.astype(np.int64) for s in P.subs]))
    dof = t(np.concatenate([s.B_dof.astype(np.int64) + o for s, o in zip(P.subs, off)]))
    sg = t(np.concatenate([s.B_sign for s in P.subs]))
    B = lambda x: torch.zeros(P.n_lambda, dtype=torch.float64, device=dev).index_add_(0, lam, sg * x[dof])  # noqa: E731
    Bt = lambda y: torch.zeros(n, dtype=torch.float64, device=dev).index_add_(0, dof, sg * y[lam])  # noqa: E731
    two = torch.zeros(P.n_lambda, dtype=torch.float64, device=dev).index_add_(0, lam, sg * sg)
    lmb = _cg(lambda y: B(Bt(y)), B(r), two, 1e-15, 200)
    alpha = []
    for s, o in zip(P.subs, off):
        fix = s.fix_dofs.astype(np.int64)
        alpha.append(torch.linalg.solve(t(s.R[fix]), u[t(fix + o)]))
    return lmb, torch.cat(alpha), u


def exact(case, seed):
    if case["kind"] in ("apply", "implicit", "assemble"):
        return _exact_apply(case, seed)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    return _exact_step(case, seed)
