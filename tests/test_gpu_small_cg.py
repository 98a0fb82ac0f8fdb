"""The one-kernel CG loop of small Kronecker operators: sides around the 4 x 8
output tile, one to several right-hand sides and tasks per block, scalar,
per-element and absent diagonals, both precisions, Jacobi, an initial guess, an
iteration cap and a right-hand side that breaks down, against the dense FP64
solution.

||x - x*|| / ||x*|| <= kappa tol (b spans all eigenvectors); kappa is computed."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _problem(cola, n1, n2, diag, dtype, seed=0):
    r = np.random.default_rng(seed + n1 * 100 + n2)
    F = [wl.rbf_factor(r.random(n), 0.3) for n in (n1, n2)]
    N = n1 * n2
    d = None if diag is None else np.array([0.3]) if diag == "scalar" else 0.2 + r.random(N)
    if diag is None:
        F = [f + 0.5 * np.eye(f.shape[0]) for f in F]
    t = lambda a: torch.tensor(a, dtype=dtype, device="cuda")
    F = [t(f).double().cpu().numpy() for f in F]
    A = np.kron(*F)
    if d is not None:
        d = t(d).double().cpu().numpy()
        A = 2.0 * A + 1.5 * np.diag(np.broadcast_to(d, (N,)))
    ctx = cola.cola_create(0)
    op = cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(ctx, t(f)) for f in F])
    if d is not None:
        dg = cola.cola_linop_diag(ctx, t(d), n=N) if diag == "scalar" else \
            cola.cola_linop_diag(ctx, t(d))
        op = cola.cola_linop_sum(ctx, [op, dg], [2.0, 1.5])
    return ctx, op.set_spd(), A, r


@pytest.mark.parametrize("n1,n2,R,diag,jacobi", [
    (1, 1, 1, "scalar", 0), (4, 8, 1, "scalar", 0), (5, 9, 3, "vector", 1),
    (64, 64, 1, "scalar", 0), (33, 17, 4, None, 0), (64, 64, 4, "vector", 0),
    (17, 40, 7, "scalar", 1), (100, 12, 2, "vector", 1), (3, 70, 1, "vector", 0),
])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_small_cg(n1, n2, R, diag, jacobi, prec):
    import paper_2309_03060_gb300 as cola
    f64 = prec == "f64"
    dtype = torch.float64 if f64 else torch.float32
    ctx, op, A, r = _problem(cola, n1, n2, diag, dtype)
    B = r.standard_normal((R, n1 * n2)).astype(np.float64 if f64 else np.float32)
    tol = 1e-10 if f64 else 1e-5
    opts = cola.cola_cg_opts_default(precision=cola.PREC_F64 if f64 else cola.PREC_F32, refine=0,
                                     tol=tol, maxiter=5000, jacobi=jacobi)
    X, info, st = cola.cola_cg_solve(ctx, op, torch.tensor(B, device="cuda"), opts)
    assert st == 0, info
    ref = np.linalg.solve(A, B.T.astype(np.float64)).T
    kappa = np.linalg.cond(A)
    X = X.double().cpu().numpy()
    eps = 1e-15 if f64 else 1e-6
    for v in range(R):
        err = np.linalg.norm(X[v] - ref[v]) / np.linalg.norm(ref[v])
        assert err <= kappa * (tol + 10 * eps), (v, err, kappa)
        # CG in exact arithmetic needs at most N steps; rounding a few more
        assert info[v]["iterations"] <= 4 * n1 * n2 + 50


def test_initial_guess_and_iteration_cap():
    import paper_2309_03060_gb300 as cola
    ctx, op, A, r = _problem(cola, 40, 24, "scalar", torch.float64)
    B = r.standard_normal((2, 960))
    opts = cola.cola_cg_opts_default(precision=cola.PREC_F64, refine=0, tol=1e-10)
    X, info, st = cola.cola_cg_solve(ctx, op, torch.tensor(B, device="cuda"), opts)
    assert st == 0
    X2, info2, st2 = cola.cola_cg_solve(ctx, op, torch.tensor(B, device="cuda"), opts, X0=X)
    assert st2 == 0 and max(i["iterations"] for i in info2) <= 2
    few = cola.cola_cg_opts_default(precision=cola.PREC_F64, refine=0, tol=1e-10, maxiter=1)
    _, info3, st3 = cola.cola_cg_solve(ctx, op, torch.tensor(B, device="cuda"), few)
    assert st3 == 5 and all(i["iterations"] == 1 and i["status"] == 5 for i in info3)


def test_breakdown_stays_in_its_right_hand_side():
    import paper_2309_03060_gb300 as cola
    ctx, op, A, r = _problem(cola, 32, 32, "scalar", torch.float64)
    B = r.standard_normal((3, 1024))
    B[1, 5] = np.inf
    opts = cola.cola_cg_opts_default(precision=cola.PREC_F64, refine=0, tol=1e-9)
    X, info, st = cola.cola_cg_solve(ctx, op, torch.tensor(B, device="cuda"), opts,
                                     raise_on_error=False)
    assert st == 4 and info[1]["status"] == 4
    ref = np.linalg.solve(A, B[[0, 2]].T).T
    assert np.abs(X.cpu().numpy()[[0, 2]] - ref).max() < 1e-6 * np.abs(ref).max()
    # an operator annotated spd that is not: p . A p < 0 in the first iteration
    K = cola.cola_linop_dense(ctx, torch.eye(32, dtype=torch.float64, device="cuda"))
    s = torch.tensor([-2.0], dtype=torch.float64, device="cuda")
    neg = cola.cola_linop_sum(ctx, [cola.cola_linop_kron(ctx, K, K),
                                    cola.cola_linop_diag(ctx, s, n=1024)]).set_spd()
    X, info, st = cola.cola_cg_solve(ctx, neg, torch.tensor(B[:1], device="cuda"), opts,
                                     raise_on_error=False)
    assert st == 4 and info[0]["status"] == 4 and info[0]["iterations"] == 0
