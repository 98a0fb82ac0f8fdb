"""A call that returns host results reports a tensor-core time-out of its own
products itself: the stochastic diagonal estimate, the split product solve and
SLQ, with FP64 products large enough for the tensor cores (and MIXED SLQ).  The
launch made to wait takes its ordinary time-out path (20 ms); the call after it
gives the result of an undisturbed one, bit for bit."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TIMEOUT = 6


def _setup(cola):
    ctx = cola.cola_create(0)
    r = np.random.default_rng(5)
    F = [cola.cola_linop_dense(ctx, torch.tensor(wl.rbf_factor(r.random(128), 0.2), device="cuda"))
         for _ in range(2)]
    s = torch.tensor([0.5], dtype=torch.float64, device="cuda")
    op = cola.cola_linop_sum(ctx, [cola.cola_linop_kron(ctx, *F),
                                   cola.cola_linop_diag(ctx, s, n=128 * 128)]).set_spd()
    return ctx, op


def _product(cola, ctx, op):
    B = torch.tensor(np.random.default_rng(6).standard_normal((16, 128 * 128)), device="cuda")
    A = cola.cola_linop_product(ctx, [op, op])
    o = cola.cola_cg_opts_default(precision=cola.PREC_F64, refine=0, tol=1e-8)
    X, info, _ = cola.cola_product_solve(ctx, A, B, o)
    return X.cpu(), [i["rel_residual"] for i in info]


CALLS = {
    "estimate_f64": lambda cola, ctx, op: cola.cola_diag_estimate(ctx, op, 16)[1],
    "product_f64": _product,
    "slq_f64": lambda cola, ctx, op: cola.cola_slq_logdet(
        ctx, op, 16, 10, precision=cola.PREC_F64, reorth=1)[0],
    "slq_mixed": lambda cola, ctx, op: cola.cola_slq_logdet(
        ctx, op, 16, 10, precision=cola.PREC_MIXED)[0],
}


@pytest.mark.parametrize("call", list(CALLS))
def test_time_out_is_reported_by_the_call_itself(call):
    import paper_2309_03060_gb300 as cola
    ctx, op = _setup(cola)
    first = CALLS[call](cola, ctx, op)
    torch.cuda.synchronize()
    ctx.test_stall_next_launch(20_000_000)
    with pytest.raises(cola.ColaError) as e:
        CALLS[call](cola, ctx, op)
    assert e.value.status == TIMEOUT
    after = CALLS[call](cola, ctx, op)
    if call.startswith("product"):
        assert torch.equal(after[0], first[0]) and after[1] == first[1]
    else:
        assert after == first
