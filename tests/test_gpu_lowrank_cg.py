"""FP32 CG on stencil + diagonal + low rank with U read once per iteration,
against the FP64 oracle's CG, over grid edges (strips, quads, 128-row stages),
ranks below 32, right-hand sides on both sides of 8, term orders, coefficients
and diagonals, with and without Jacobi and FP64 refinement.

kappa(A) <= (8 + max d + ||U U^T||) / min d <= 24, so a solve to tol is within
24 tol of the exact solution (plus FP32 rounding of x, 1e-6)."""
import numpy as np
import pytest

import workloads as wl
from oracle import krylov
from oracle import linop as O

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2,rank,R,diag,order,jacobi,refine", [
    (8, 12, 4, 1, "vector", (0, 1, 2), 1, 0),
    (33, 20, 8, 3, "vector", (2, 0, 1), 1, 0),
    (64, 64, 32, 8, "vector", (0, 1, 2), 0, 0),
    (17, 256, 28, 9, "scalar", (1, 2, 0), 1, 0),
    (130, 100, 32, 2, "vector", (0, 1, 2), 1, 1),
    (1, 36, 12, 5, "scalar", (0, 1, 2), 0, 1),
    (96, 8, 16, 17, "vector", (0, 2, 1), 1, 0),
])
def test_lowrank_cg(n1, n2, rank, R, diag, order, jacobi, refine):
    import paper_2309_03060_gb300 as cola
    r = np.random.default_rng(n1 * 1000 + n2)
    N = n1 * n2
    L = [wl.dirichlet_laplacian(n) for n in (n1, n2)]
    d = np.array([0.8]) if diag == "scalar" else 0.5 + r.random(N)
    U = r.standard_normal((N, rank)) / np.sqrt(N)
    B = r.standard_normal((R, N))
    co = (1.0, 1.5, 2.0)
    U = U.astype(np.float32).astype(np.float64)
    d = d.astype(np.float32).astype(np.float64)
    B = B.astype(np.float32).astype(np.float64)
    ctx = cola.cola_create(0)
    t = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    ks = cola.cola_linop_kronsum(ctx, *[cola.cola_linop_dense(ctx, t(a)) for a in L])
    dg = cola.cola_linop_diag(ctx, t(d), n=N) if diag == "scalar" else cola.cola_linop_diag(ctx, t(d))
    lr = cola.cola_linop_lowrank(ctx, t(U))
    terms = (ks, dg, lr)
    op = cola.cola_linop_sum(ctx, [terms[i] for i in order], [co[i] for i in order]).set_spd()
    tol = 1e-10 if refine else 1e-6
    opts = cola.cola_cg_opts_default(precision=cola.PREC_F32, refine=refine, tol=tol,
                                     maxiter=2000, jacobi=jacobi)
    Bd = torch.tensor(B, dtype=torch.float64 if refine else torch.float32, device="cuda")
    X, info, st = cola.cola_cg_solve(ctx, op, Bd, opts)
    assert st == 0, info
    ref = O.Sum([O.KronSum([O.Dense(a) for a in L]), O.Diag(d if diag == "vector" else 0.8, N),
                 O.LowRank(U)], list(co))
    if diag == "scalar":
        ref = O.Sum([O.KronSum([O.Dense(a) for a in L]), O.Diag(float(d[0]), N), O.LowRank(U)],
                    list(co))
    X = X.double().cpu().numpy()
    for v in range(R):
        x, _ = krylov.cg(ref, B[v], tol=1e-13, maxiter=2000)
        err = np.linalg.norm(X[v] - x) / np.linalg.norm(x)
        assert err <= 24 * tol + (0.0 if refine else 1e-6), (v, err)
        assert info[v]["iterations"] <= 200
    # the stopping rule holds on the true residual
    for v in range(R):
        res = np.linalg.norm(B[v] - ref @ X[v]) / np.linalg.norm(B[v])
        assert res <= (tol if refine else 10 * tol), (v, res)


def test_breakdown_stays_in_its_right_hand_side():
    import paper_2309_03060_gb300 as cola
    r = np.random.default_rng(5)
    n, N = 32, 32 * 32
    ctx = cola.cola_create(0)
    t = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    Ld = cola.cola_linop_dense(ctx, t(wl.dirichlet_laplacian(n)))
    op = cola.cola_linop_sum(ctx, [cola.cola_linop_kronsum(ctx, Ld, Ld),
                                   cola.cola_linop_diag(ctx, t(np.ones(N))),
                                   cola.cola_linop_lowrank(ctx, t(r.standard_normal((N, 8)) / n))])
    op.set_spd()
    B = r.standard_normal((3, N))
    B[1, 17] = np.nan
    opts = cola.cola_cg_opts_default(precision=cola.PREC_F32, refine=0, tol=1e-5, maxiter=500)
    X, info, st = cola.cola_cg_solve(ctx, op, t(B), opts, raise_on_error=False)
    assert st == 4 and info[1]["status"] == 4
    assert info[0]["status"] == 0 and info[2]["status"] == 0
    assert torch.isfinite(X[0]).all() and torch.isfinite(X[2]).all()
