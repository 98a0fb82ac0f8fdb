"""What a user of this library has it do, as timed cases.

The library's work is the MVM of a composed operator, the solves built on it
(CG in its precisions, the eigen-structured direct solve, batches of uneven
systems), stochastic Lanczos quadrature and the gradient of a solve.  Each
kind below goes through the package's public calls on operators built the way
the benchmark and the tests build them: RBF kernel factors on points drawn
uniformly from [0, 1], a noise shift or a per-point noise diagonal, N(0, 1)
right-hand sides, Rademacher probes; and the 2-D Poisson operator with a
diagonal and a low-rank term.

Refined solves run to 1e-10 instead of the benchmark's 1e-8: their FP64
solutions are then determined to about 1e-10 whatever the rounding of the
inner recurrence, so that solutions can be compared as FP64 numbers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2309_03060_gb300 as cola
from paper_2309_03060_gb300 import autograd as cola_autograd

_PREC = {"f64": cola.PREC_F64, "f32": cola.PREC_F32, "mixed": cola.PREC_MIXED}


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # one small MVM in the default precision: a call inside a user's own
        # loop, where latency and launches are all there is (the 64 x 64 FP64
        # workload's operator)
        dict(name="mvm_f64_64x64_r1", kind="mvm", prec="f64", n1=64, n2=64, n3=1, rhs=1,
             ell=0.2, shift=0.1),
        # the 128^3 operator on a block of vectors in the default precision:
        # true residuals, FP64 checks of a solution
        dict(name="mvm_f64_128x128x128_r16", kind="mvm", prec="f64", n1=128, n2=128, n3=128,
             rhs=16, ell=0.1, shift=0.01),
        # plain FP32 on factor sides that are no multiple of anything
        dict(name="mvm_f32_97x120x101_r5", kind="mvm", prec="f32", n1=97, n2=120, n3=101, rhs=5,
             ell=0.1, shift=0.01),
        # the headline operator's tensor-core MVM
        dict(name="mvm_mixed_128x128x128_r16", kind="mvm", prec="mixed", n1=128, n2=128, n3=128,
             rhs=16, ell=0.1, shift=0.01),
        # the direct solve of a Kronecker-structured GP (exact inference on a
        # grid), ragged sides
        dict(name="eig_f64_120x97x75_r8", kind="eig", n1=120, n2=97, n3=75, rhs=8, ell=0.1,
             shift=0.1),
        # the plain FP64 single solve: N = 4096, one right-hand side
        dict(name="cg_f64_64x64_r1", kind="cg", prec="f64", precond="none", n1=64, n2=64, n3=1,
             rhs=1, ell=0.2, shift=0.1),
        # the headline solve (16 right-hand sides on the 128^3 operator,
        # tensor-core contractions, FP32 recurrences, FP64 refinement), with
        # unit noise so that one solve takes a fraction of a second
        dict(name="cg_mixed_128x128x128_r16", kind="cg", prec="mixed", precond="none", n1=128,
             n2=128, n3=128, rhs=16, ell=0.1, shift=1.0),
        # per-point noise (heteroscedastic GP): CG with the Kronecker preconditioner
        dict(name="cg_mixed_kronprecond_128x128x128_r16", kind="cg", prec="mixed",
             precond="kron", n1=128, n2=128, n3=128, rhs=16, ell=0.1, shift=0.01),
        # the PDE-style operator in FP32 with the diagonal preconditioner
        dict(name="cg_f32_pde_1024x1024_k32_r8", kind="pde", n=1024, rank=32, rhs=8),
        # many independent uneven systems in one call
        dict(name="cg_batched_mixed_64sys", kind="batched", nsys=64, nmin=16, nmax=256, rmax=8),
        # training through a solve: forward, adjoint solve, leaf gradients
        dict(name="solve_grad_mixed_256x256_r4", kind="grad", n1=256, n2=256, rhs=4, ell=0.1,
             shift=0.1),
        # the log-determinant of the 64 x 64 workload: 16 probes, 50
        # reorthogonalised Lanczos steps
        dict(name="slq_f64_64x64_p16_m50", kind="slq", n1=64, n2=64, probes=16, steps=50,
             ell=0.2, shift=0.1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, nmax_total):
    """Two or three factor sides between 16 and 128 (odd ones among them)."""
    while True:
        d = rng.choice((2, 3, 3))
        n = [rng.choice((128, rng.randint(16, 128))) for _ in range(d)] + [1] * (3 - d)
        if n[0] * n[1] * n[2] <= nmax_total:
            return n


def draw(rng):
    kind = rng.choice(("mvm", "mvm", "mvm", "eig", "cg", "cg", "pde", "batched", "grad", "slq"))
    if kind == "mvm":
        prec = rng.choice(("f64", "f32", "mixed"))
        if rng.random() < 0.25:  # two larger factors
            n1, n2, n3 = rng.randint(129, 400), rng.randint(129, 400), 1
        else:
            n1, n2, n3 = _sides(rng, 128 ** 3)
        return dict(kind=kind, prec=prec, n1=n1, n2=n2, n3=n3, rhs=_log_int(rng, 1, 16),
                    ell=rng.uniform(0.05, 0.3), shift=10.0 ** rng.uniform(-2, 0))
    if kind == "eig":
        n1, n2, n3 = _sides(rng, 128 ** 3)
        return dict(kind=kind, n1=n1, n2=n2, n3=n3, rhs=_log_int(rng, 1, 16),
                    ell=rng.uniform(0.05, 0.3), shift=10.0 ** rng.uniform(-1, 0))
    if kind == "cg":
        prec, precond = rng.choice((("f64", "none"), ("mixed", "none"), ("mixed", "kron")))
        if prec == "f64":
            n1, n2, n3, rhs = rng.randint(16, 96), rng.randint(16, 96), 1, _log_int(rng, 1, 4)
        else:
            n1, n2, n3 = _sides(rng, 128 ** 3)
            rhs = _log_int(rng, 1, 16)
        shift = 10.0 ** (rng.uniform(-1, 0) if precond == "none" and n3 == 1 else
                         rng.uniform(0, 0.5) if precond == "none" else rng.uniform(-2, 0))
        ell = rng.uniform(0.05, 0.1) if n3 > 1 else rng.uniform(0.1, 0.3)
        return dict(kind=kind, prec=prec, precond=precond, n1=n1, n2=n2, n3=n3, rhs=rhs,
                    ell=ell, shift=shift)
    if kind == "pde":
        return dict(kind=kind, n=_log_int(rng, 64, 1024), rank=rng.randint(1, 32),
                    rhs=rng.randint(1, 8))
    if kind == "batched":
        return dict(kind=kind, nsys=_log_int(rng, 4, 64), nmin=16, nmax=rng.randint(64, 256),
                    rmax=rng.randint(1, 8))
    if kind == "grad":
        return dict(kind=kind, n1=rng.randint(32, 256), n2=rng.randint(32, 256),
                    rhs=rng.randint(1, 4), ell=rng.uniform(0.1, 0.3), shift=rng.uniform(0.1, 1.0))
    return dict(kind=kind, n1=rng.randint(16, 96), n2=rng.randint(16, 96),
                probes=rng.randint(2, 16), steps=rng.randint(10, 50), ell=rng.uniform(0.1, 0.3),
                shift=10.0 ** rng.uniform(-1, 0))


# ---------------------------------------------------------------- the inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _randn(g, *shape, dtype=torch.float64):
    return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)


def _rbf(g, n, ell):
    x = _rand(g, n)
    d = x[:, None] - x[None, :]
    return torch.exp(-(d * d) / (2.0 * ell * ell))


def _factors(g, case):
    sides = [case[k] for k in ("n1", "n2", "n3") if case.get(k, 1) > 1]
    return [_rbf(g, n, case["ell"]) for n in sides]


def _inputs(case, seed):
    """Every tensor of a case, from its seed alone."""
    g = _gen(seed)
    kind = case["kind"]
    if kind == "pde":
        n, N = case["n"], case["n"] ** 2
        L = 2.0 * torch.eye(n, device="cuda", dtype=torch.float64)
        i = torch.arange(n - 1, device="cuda")
        L[i, i + 1] = -1.0
        L[i + 1, i] = -1.0
        return dict(L=L.float(), d=(0.5 + _rand(g, N)).float(),
                    U=_randn(g, N, case["rank"], dtype=torch.float32) / math.sqrt(N),
                    B=_randn(g, case["rhs"], N, dtype=torch.float32))
    if kind == "batched":
        # sides uniform, lengthscales in [0.05, 0.5], noise in [1e-1, 1];
        # the sizes are the case's own and do not change with the seed
        sizes = np.random.default_rng([case["nsys"], case["nmax"], case["rmax"]])
        systems = []
        for _ in range(case["nsys"]):
            n1, n2 = (int(v) for v in sizes.integers(case["nmin"], case["nmax"] + 1, 2))
            l1, l2 = sizes.uniform(0.05, 0.5, 2)
            s = 10.0 ** sizes.uniform(-1.0, 0.0)
            r = int(sizes.integers(1, case["rmax"] + 1))
            systems.append(dict(K=[_rbf(g, n1, l1), _rbf(g, n2, l2)],
                                s=torch.tensor([s], device="cuda", dtype=torch.float64),
                                B=_randn(g, r, n1 * n2)))
        return dict(systems=systems)
    K = _factors(g, case)
    N = math.prod(k.shape[0] for k in K)
    t = dict(K=K, N=N)
    if kind == "cg" and case["precond"] == "kron":
        t["d"] = case["shift"] * (0.5 + _rand(g, N))
    else:
        t["s"] = torch.tensor([case["shift"]], device="cuda", dtype=torch.float64)
    if kind == "slq":
        t["Z"] = torch.where(_rand(g, case["probes"], N) < 0.5, -1.0, 1.0).to(torch.float64)
        return t
    dtype = torch.float32 if kind == "mvm" and case["prec"] != "f64" else torch.float64
    t["B"] = _randn(g, case["rhs"], N, dtype=dtype)
    if kind == "grad":
        t["W"] = _randn(g, case["rhs"], N)  # the gradient that arrives from the loss
    return t


def _operator(ctx, K, s=None, d=None):
    """K_1 (x) ... (x) K_d + s I (or + Diag(d))."""
    N = math.prod(k.shape[0] for k in K)
    kron = cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(ctx, k) for k in K])
    noise = cola.cola_linop_diag(ctx, d) if d is not None else cola.cola_linop_diag(ctx, s, n=N)
    return cola.cola_linop_sum(ctx, [kron, noise]).set_spd()


def _refined(**kw):
    return cola.cola_cg_opts_default(precision=cola.PREC_MIXED, refine=1, tol=1e-10,
                                     maxiter=60000, **kw)


def prepare(case, seed):
    t = _inputs(case, seed)
    kind = case["kind"]
    ctx = cola.cola_create(0)
    state = dict(case=case, ctx=ctx, t=t)
    if kind == "pde":
        Ld = cola.cola_linop_dense(ctx, t["L"])
        ks = cola.cola_linop_kronsum(ctx, Ld, Ld)
        state["op"] = cola.cola_linop_sum(ctx, [ks, cola.cola_linop_diag(ctx, t["d"]),
                                                cola.cola_linop_lowrank(ctx, t["U"])]).set_spd()
        state["opts"] = cola.cola_cg_opts_default(precision=cola.PREC_F32, refine=0, tol=1e-6,
                                                  maxiter=5000, jacobi=1)
    elif kind == "batched":
        state["op"] = [_operator(ctx, s["K"], s["s"]) for s in t["systems"]]
        state["opts"] = _refined()
    else:
        state["op"] = _operator(ctx, t["K"], t.get("s"), t.get("d"))
        if kind == "cg":
            if case["prec"] == "f64":
                state["opts"] = cola.cola_cg_opts_default(precision=cola.PREC_F64, refine=0,
                                                          tol=1e-10)
            elif case["precond"] == "kron":
                state["opts"] = _refined(kron_precond=1, graph_chunk=8)
            else:
                state["opts"] = _refined()
        elif kind == "grad":
            state["opts"] = _refined()
            state["leaves"] = [*t["K"], t["s"]]
    return state


# ------------------------------------------------------------------- the call

def run(state):
    case, ctx, t, op = state["case"], state["ctx"], state["t"], state["op"]
    kind = case["kind"]
    if kind == "mvm":
        return cola.cola_matvec(ctx, op, t["B"], _PREC[case["prec"]], split_terms=3)
    if kind == "eig":
        return cola.cola_kron_eig_solve(ctx, op, t["B"])
    if kind in ("cg", "pde"):
        X, _, _ = cola.cola_cg_solve(ctx, op, t["B"], state["opts"])
        return X
    if kind == "batched":
        Xs, _, _ = cola.cola_cg_solve_batched(ctx, op, [s["B"] for s in t["systems"]],
                                              state["opts"])
        return Xs
    if kind == "grad":
        B = t["B"].detach().requires_grad_(True)
        leaves = [l.detach().requires_grad_(True) for l in state["leaves"]]
        X = cola_autograd.solve(ctx, op, B, leaves, state["opts"])
        grads = torch.autograd.grad(X, [B, *leaves], t["W"])
        return [X.detach(), *grads]
    logdet, _, per_probe, _ = cola.cola_slq_logdet(ctx, op, case["probes"], case["steps"],
                                                   probes=t["Z"], precision=cola.PREC_F64,
                                                   reorth=1)
    return [logdet, per_probe]


# --------------------------------------------------------------------- floors

def _kron_flops(sides, rhs):
    return 2.0 * math.prod(sides) * sum(sides) * rhs


def work(case):
    """Bytes: every input read once, every output written once.  Flops: of one
    MVM of the operator (two of a direct or gradient solve); the iterations of
    a solve depend on its data and are not counted."""
    kind = case["kind"]
    if kind == "pde":
        n, k, r = case["n"], case["rank"], case["rhs"]
        N = n * n
        return {"bytes": 4.0 * (N * k + N + n * n + 2 * r * N), "flops": r * N * (4.0 * k + 13.0)}
    if kind == "batched":
        sizes = np.random.default_rng([case["nsys"], case["nmax"], case["rmax"]])
        nbytes = flops = 0.0
        for _ in range(case["nsys"]):
            n1, n2 = (int(v) for v in sizes.integers(case["nmin"], case["nmax"] + 1, 2))
            sizes.uniform(0.05, 0.5, 2)
            sizes.uniform(-1.0, 0.0)
            r = int(sizes.integers(1, case["rmax"] + 1))
            nbytes += 8.0 * (n1 * n1 + n2 * n2 + 1 + 2 * r * n1 * n2)
            flops += _kron_flops([n1, n2], r)
        return {"bytes": nbytes, "flops": flops}
    sides = [case[k] for k in ("n1", "n2", "n3") if case.get(k, 1) > 1]
    N = math.prod(sides)
    facs = 8.0 * sum(n * n for n in sides)
    if kind == "slq":
        return {"bytes": facs + 8.0 * (case["probes"] * N + case["probes"] + 2),
                "flops": case["steps"] * _kron_flops(sides, case["probes"])}
    r = case["rhs"]
    if kind == "grad":  # B, W, X, gradB; the factors and their gradients
        return {"bytes": 2 * facs + 32.0 * r * N, "flops": 4 * _kron_flops(sides, r)}
    if kind == "mvm":
        elem = 8.0 if case["prec"] == "f64" else 4.0
        return {"bytes": facs + 2 * elem * r * N, "flops": _kron_flops(sides, r)}
    extra = 8.0 * N if kind == "cg" and case["precond"] == "kron" else 8.0
    return {"bytes": facs + extra + 16.0 * r * N,
            "flops": _kron_flops(sides, r) * (2 if kind == "eig" else 1)}


# ------------------------------------------------------- the values in 64 bits

def _modes(K, X):
    """((x) K) X for a block X [R][N], one mode at a time."""
    R = X.shape[0]
    Y = X.reshape(R, *[k.shape[1] for k in K])
    for a, k in enumerate(K):
        Y = torch.movedim(torch.tensordot(Y, k, dims=([a + 1], [1])), -1, a + 1)
    return Y.reshape(R, -1)


def _kron_solver(K, s):
    """B -> (K_1 (x) ... + s I)^-1 B from the factors' eigendecompositions."""
    lam, Q = None, []
    for k in K:
        w, V = torch.linalg.eigh(k)
        lam = w if lam is None else (lam[:, None] * w[None, :]).reshape(-1)
        Q.append(V)
    Qt = [q.t().contiguous() for q in Q]
    return lambda B: _modes(Q, _modes(Qt, B) / (lam + s))


def _cg64(mvm, B, precond, tol, maxiter):
    X = torch.zeros_like(B)
    R = B.clone()
    Z = precond(R)
    P = Z.clone()
    rz = (R * Z).sum(1, keepdim=True)
    bn = B.norm(dim=1)
    for _ in range(maxiter):
        AP = mvm(P)
        a = rz / (P * AP).sum(1, keepdim=True)
        X += a * P
        R -= a * AP
        if bool((R.norm(dim=1) <= tol * bn).all()):
            break
        Z = precond(R)
        new = (R * Z).sum(1, keepdim=True)
        P = Z + (new / rz) * P
        rz = new
    return X


def exact(case, seed):
    t = _inputs(case, seed)
    kind = case["kind"]
    if kind == "mvm":
        B = t["B"].double()
        return _modes(t["K"], B) + t["s"] * B
    if kind == "eig":
        return _kron_solver(t["K"], t["s"])(t["B"])
    if kind == "cg":
        if case["precond"] == "none":
            return _kron_solver(t["K"], t["s"])(t["B"])
        M = _kron_solver(t["K"], t["d"].mean())
        return _cg64(lambda X: _modes(t["K"], X) + t["d"] * X, t["B"], M, 1e-13, 60)
    if kind == "pde":
        n, R = case["n"], case["rhs"]
        d, U, B = t["d"].double(), t["U"].double(), t["B"].double()

        def mvm(X):
            G = X.reshape(R, n, n)
            Y = 4.0 * G
            Y[:, 1:] -= G[:, :-1]
            Y[:, :-1] -= G[:, 1:]
            Y[:, :, 1:] -= G[:, :, :-1]
            Y[:, :, :-1] -= G[:, :, 1:]
            return Y.reshape(R, -1) + d * X + (X @ U) @ U.t()

        diag = 4.0 + d + (U * U).sum(1)
        return _cg64(mvm, B, lambda X: X / diag, 1e-13, 500)
    if kind == "batched":
        return [_kron_solver(s["K"], s["s"])(s["B"]) for s in t["systems"]]
    if kind == "grad":
        solve = _kron_solver(t["K"], t["s"])
        X, G = solve(t["B"]), solve(t["W"])
        K1, K2 = t["K"]
        R = X.shape[0]
        x, g = X.reshape(R, case["n1"], case["n2"]), G.reshape(R, case["n1"], case["n2"])
        g1 = -torch.einsum("rij,rkj->ik", g, x @ K2.t())
        g2 = -torch.einsum("rij,ril->jl", g, torch.einsum("ik,rkl->ril", K1, x))
        return [X, G, g1, g2, -(G * X).sum().reshape(1)]
    # slq: Lanczos with full reorthogonalisation, Gauss quadrature of the logarithm
    K, s, Z, m = t["K"], t["s"], t["Z"], case["steps"]
    N = t["N"]
    q = Z / Z.norm(dim=1, keepdim=True)
    Q, alpha, beta = [q], [], []
    for j in range(m):
        w = _modes(K, Q[j]) + s * Q[j]
        alpha.append((w * Q[j]).sum(1))
        S = torch.stack(Q, 1)
        for _ in range(2):
            w = w - torch.einsum("pj,pjn->pn", torch.einsum("pjn,pn->pj", S, w), S)
        b = w.norm(dim=1)
        beta.append(b)
        Q.append(w / b[:, None])
    T = torch.diag_embed(torch.stack(alpha, 1))
    off = torch.stack(beta[:-1], 1) if m > 1 else None
    if off is not None:
        T = T + torch.diag_embed(off, 1) + torch.diag_embed(off, -1)
    theta, V = torch.linalg.eigh(T)
    per_probe = N * (V[:, 0, :] ** 2 * torch.log(theta)).sum(1)
    return [float(per_probe.mean()), per_probe]
