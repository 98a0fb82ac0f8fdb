"""The slab kernel's per-element and transposed forms: CG on K_1 (x) K_2 (x) K_3 +
Diag(d) with 128 x 128 last factors (diagonal per element in the epilogue), and
its Kronecker preconditioner (the scaling in the epilogue of Q^T, the transposed
product for Q).  A wrong preconditioner would still converge, but not within
kappa(M^-1 A) <= 3 iterations' count: 2 sqrt(3) ln(2 / tol) / 2 < 40 plus
restarts; the true residual is formed in FP64 on the host."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _mvm(F, d, X):
    R = X.shape[0]
    Y = X
    for f in F:
        Y = np.ascontiguousarray(np.swapaxes(np.matmul(f, Y.reshape(R, f.shape[1], -1)), 1, 2))
    return Y.reshape(R, -1) + d * X


@pytest.mark.parametrize("n1,R", [(1, 1), (3, 2), (8, 5)])
@pytest.mark.parametrize("precond", [0, 1])
def test_kron_diag_slab_cg(n1, R, precond):
    import paper_2309_03060_gb300 as cola
    r = np.random.default_rng(n1)
    sides = (n1, 128, 128)
    F = [wl.rbf_factor(r.random(n), 0.2) for n in sides]
    N = int(np.prod(sides))
    shift = 1.0 if precond else 200.0  # without M: kappa ~ 50
    d = shift * (0.5 + r.random(N))
    B = r.standard_normal((R, N))
    ctx = cola.cola_create(0)
    kron = cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(ctx, torch.tensor(f, device="cuda"))
                                       for f in F])
    op = cola.cola_linop_sum(ctx, [kron, cola.cola_linop_diag(ctx, torch.tensor(d, device="cuda"))])
    op.set_spd()
    opts = cola.cola_cg_opts_default(precision=cola.PREC_MIXED, refine=1, tol=1e-9, maxiter=3000,
                                     kron_precond=precond)
    X, info, st = cola.cola_cg_solve(ctx, op, torch.tensor(B, device="cuda"), opts)
    assert st == 0, info
    X = X.cpu().numpy()
    res = np.linalg.norm(B - _mvm(F, d, X), axis=1) / np.linalg.norm(B, axis=1)
    assert (res <= 1.01e-9).all(), res
    if precond:
        assert max(i["iterations"] for i in info) <= 80, info
