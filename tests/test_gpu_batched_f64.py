"""Batched solves whose FP64 residuals run as digit products over a problem table:
uneven sides around the 64-vector, 128-output and 128-k steps, several right-hand
sides, and systems that retire at different times, against the exact solution
(within kappa tol) and on the true FP64 residual."""
import numpy as np
import pytest

import workloads as wl
from oracle import exact

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sides", [
    [(130, 200), (64, 65), (129, 17), (256, 255), (128, 128), (33, 240)] * 4,
    [(200, 200)] * 12,
])
def test_batched_refined(sides):
    import paper_2309_03060_gb300 as cola
    r = np.random.default_rng(len(sides))
    ctx = cola.cola_create(0)
    ops, Bs, raw = [], [], []
    for k, (n1, n2) in enumerate(sides):
        F = [wl.rbf_factor(r.random(n), 0.1 + 0.3 * r.random()) for n in (n1, n2)]
        s = 10.0 ** r.uniform(-2, -1)
        B = r.standard_normal((1 + k % 5, n1 * n2))
        kron = cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(ctx, torch.tensor(f, device="cuda"))
                                           for f in F])
        st = torch.tensor([s], dtype=torch.float64, device="cuda")
        ops.append(cola.cola_linop_sum(ctx, [kron, cola.cola_linop_diag(ctx, st, n=n1 * n2)],
                                       [1.0, 2.0]).set_spd())
        Bs.append(torch.tensor(B, device="cuda"))
        raw.append((F, 2.0 * s, B))
    opts = cola.cola_cg_opts_default(precision=cola.PREC_MIXED, refine=1, tol=1e-9)
    Xs, info, status = cola.cola_cg_solve_batched(ctx, ops, Bs, opts)
    assert status == 0, info
    for X, (F, s, B) in zip(Xs, raw):
        X = X.cpu().numpy()
        R = B.shape[0]
        Y = np.einsum("ij,rjk,lk->ril", F[0], X.reshape(R, F[0].shape[0], -1), F[1],
                      optimize=True).reshape(R, -1) + s * X
        res = np.linalg.norm(B - Y, axis=1) / np.linalg.norm(B, axis=1)
        assert (res <= 1.01e-9).all(), res
        ref = exact.kron_shift_solve(F, s, B)
        kappa = 1.0 + np.prod([np.linalg.eigvalsh(f)[-1] for f in F]) / s
        err = np.linalg.norm(X - ref, axis=1) / np.linalg.norm(ref, axis=1)
        assert (err <= kappa * 1e-9).all(), err
