"""Split GEMM steps with 128, 64 and 32 rows per tile (sides above 128): MVMs with
and without a diagonal, one and two wide factors (chained steps write the next
step's image, whose columns past the end must be zero), rests around the tile
heights, and the fused CG step.

Per entry within 2e-5 of sum |K| |x| (3 x 3 BF16 terms, at most 400 entries a
mode); the solve to its tolerance times the condition number."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _kron(F, X):
    R = X.shape[0]
    for f in F:
        X = np.ascontiguousarray(np.swapaxes(np.matmul(f, X.reshape(R, f.shape[1], -1)), 1, 2))
    return X.reshape(R, -1)


@pytest.mark.parametrize("sides,R", [
    ((256, 256), 1), ((256, 256), 4), ((256, 256), 40),   # 32, 32 and 128 rows
    ((200, 300), 12), ((129, 131), 3), ((160, 24), 5), ((24, 160), 5), ((33, 400), 2),
    ((400, 20), 9), ((130, 65), 30), ((150, 9, 17), 4),
])
@pytest.mark.parametrize("diag", [None, "scalar", "vector"])
def test_mvm(sides, R, diag):
    import paper_2309_03060_gb300 as cola
    r = np.random.default_rng(sum(sides) + R)
    F = [r.standard_normal((n, n)) for n in sides]
    N = int(np.prod(sides))
    X = r.standard_normal((R, N))
    ctx = cola.cola_create(0)
    op = cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(ctx, torch.tensor(f, device="cuda"))
                                     for f in F])
    ref, bound = _kron(F, X), _kron([np.abs(f) for f in F], np.abs(X))
    if diag:
        d = r.standard_normal(1 if diag == "scalar" else N)
        dt = torch.tensor(d, device="cuda")
        dg = cola.cola_linop_diag(ctx, dt, n=N) if diag == "scalar" else \
            cola.cola_linop_diag(ctx, dt)
        op = cola.cola_linop_sum(ctx, [op, dg])
        ref, bound = ref + d * X, bound + np.abs(d * X)
    Xd = torch.tensor(X, dtype=torch.float32, device="cuda")
    for _ in range(2):  # the workspace (images) of the first call is reused by the second
        Y = cola.cola_matvec(ctx, op, Xd, cola.PREC_MIXED, split_terms=3).double().cpu().numpy()
        assert (np.abs(Y - ref) <= 2e-5 * bound).all(), float((np.abs(Y - ref) / bound).max())


@pytest.mark.parametrize("sides,R", [((200, 140), 1), ((256, 130), 5), ((40, 150), 3)])
def test_fused_cg(sides, R):
    import paper_2309_03060_gb300 as cola
    from oracle import exact
    r = np.random.default_rng(7)
    F = [wl.rbf_factor(r.random(n), 0.2) for n in sides]
    B = r.standard_normal((R, sides[0] * sides[1]))
    ctx = cola.cola_create(0)
    s = torch.tensor([0.5], dtype=torch.float64, device="cuda")
    op = cola.cola_linop_sum(ctx, [cola.cola_linop_kron(
        ctx, *[cola.cola_linop_dense(ctx, torch.tensor(f, device="cuda")) for f in F]),
        cola.cola_linop_diag(ctx, s, n=B.shape[1])]).set_spd()
    opts = cola.cola_cg_opts_default(precision=cola.PREC_MIXED, refine=1, tol=1e-9)
    X, info, st = cola.cola_cg_solve(ctx, op, torch.tensor(B, device="cuda"), opts)
    assert st == 0, info
    ref = exact.kron_shift_solve(F, 0.5, B)
    kappa = 1.0 + np.prod([np.linalg.eigvalsh(f)[-1] for f in F]) / 0.5
    err = np.linalg.norm(X.cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert (err <= kappa * 1e-9).all(), err
