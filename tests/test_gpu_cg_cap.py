"""The iteration count of unrefined CG solves, which is kept in whole chunks of
graph_chunk iterations after the first one: a solve that does not converge
stops at 1 + ceil((maxiter - 1) / graph_chunk) graph_chunk iterations, and one
that converges is taken to have used its whole chunk, so that the verification
of the true residual and its restarts come at the same iterations whatever the
host's timing.  On every path of the loop: general, one kernel, stencil + low
rank, fused tensor-core."""
import os

import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _kron(cola, ctx, sides, shift, dtype):
    r = np.random.default_rng(sum(sides))
    t = lambda a: torch.tensor(a, dtype=dtype, device="cuda")
    F = [cola.cola_linop_dense(ctx, t(wl.rbf_factor(r.random(n), 0.3))) for n in sides]
    N = int(np.prod(sides))
    dg = cola.cola_linop_diag(ctx, t(np.array([shift])), n=N)
    return cola.cola_linop_sum(ctx, [cola.cola_linop_kron(ctx, *F), dg]).set_spd(), N


def _pde(cola, ctx, n):
    r = np.random.default_rng(n)
    t = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    L = cola.cola_linop_dense(ctx, t(wl.dirichlet_laplacian(n)))
    op = cola.cola_linop_sum(ctx, [cola.cola_linop_kronsum(ctx, L, L),
                                   cola.cola_linop_diag(ctx, t(1e-4 * (1 + r.random(n * n)))),
                                   cola.cola_linop_lowrank(ctx, t(r.standard_normal((n * n, 4)) / 8))])
    return op.set_spd(), n * n


# path: operator, precision, right-hand sides
PATHS = {"general_f64": ("f64", (64, 64), 8), "small_f64": ("f64", (64, 64), 1),
         "small_f32": ("f32", (40, 24), 2), "fused_mixed": ("mixed", (64, 48, 32), 2),
         "lowrank_f32": ("f32", None, 3)}


def _setup(cola, path, shift=0.1):
    prec, sides, R = PATHS[path]
    ctx = cola.cola_create(0)
    dtype = torch.float64 if prec == "f64" else torch.float32
    op, N = _pde(cola, ctx, 64) if sides is None else _kron(cola, ctx, sides, shift, dtype)
    B = torch.tensor(np.random.default_rng(1).standard_normal((R, N)), dtype=dtype, device="cuda")
    P = {"f64": cola.PREC_F64, "f32": cola.PREC_F32, "mixed": cola.PREC_MIXED}[prec]
    return ctx, op, B, P


@pytest.mark.parametrize("path", list(PATHS))
@pytest.mark.parametrize("maxiter,chunk", [(100, 64), (100, 5), (33, 40), (2, 16), (150, 24)])
def test_capped_solve_stops_at_the_chunk_of_maxiter(path, maxiter, chunk):
    import paper_2309_03060_gb300 as cola
    ctx, op, B, P = _setup(cola, path)
    # the fused path's chunk is a multiple of its ring of 8 directions
    c = (chunk + 7) // 8 * 8 if path == "fused_mixed" else chunk
    want = 1 + -(-(maxiter - 1) // c) * c
    opts = cola.cola_cg_opts_default(precision=P, refine=0, tol=0.0, maxiter=maxiter,
                                     graph_chunk=chunk)
    first = None
    for _ in range(3):  # captures graphs, then replays them
        X, info, _ = cola.cola_cg_solve(ctx, op, B, opts, raise_on_error=False)
        assert [i["iterations"] for i in info] == [want] * B.shape[0]
        first = X.clone() if first is None else first
        assert torch.equal(X, first)


@pytest.mark.parametrize("path", ["general_f64", "small_f32"])
def test_converged_solve_counts_its_whole_chunk(path, capfd, monkeypatch):
    """maxiter within the chunk that the solve converges in: no iterations are left
    for a verification; one more: a single verification."""
    import paper_2309_03060_gb300 as cola
    ctx, op, B, P = _setup(cola, path, shift=10.0)
    tol = 1e-8 if P == cola.PREC_F64 else 1e-9  # FP32: the true residual never meets it
    monkeypatch.setitem(os.environ, "COLA_TRACE", "1")
    for maxiter, n in ((65, 0), (66, 1)):
        opts = cola.cola_cg_opts_default(precision=P, refine=0, tol=tol, maxiter=maxiter,
                                         graph_chunk=64)
        for _ in range(2):
            capfd.readouterr()
            _, info, _ = cola.cola_cg_solve(ctx, op, B, opts, raise_on_error=False)
            assert max(i["iterations"] for i in info) < 129
            assert capfd.readouterr().err.count("] verify iter 65 ") == n
