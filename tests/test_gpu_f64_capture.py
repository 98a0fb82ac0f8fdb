"""An FP64 product that a caller captured into a graph of their own, replayed
after a product whose vectors are smaller but whose factors are larger: the
captured kernels still have their digit images."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_captured_product_outlives_a_larger_factor():
    import paper_2309_03060_gb300 as cola
    r = np.random.default_rng(7)
    ctx = cola.cola_create(0)
    op = lambda n: cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(
        ctx, torch.tensor(r.standard_normal((n, n)), device="cuda")) for _ in range(2)])
    small, large = op(128), op(300)
    X = torch.tensor(r.standard_normal((6, 128 * 128)), device="cuda")
    Z = torch.tensor(r.standard_normal((1, 300 * 300)), device="cuda")
    first = cola.cola_matvec(ctx, small, X, cola.PREC_F64)
    Y = torch.empty_like(first)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        cola.cola_matvec(ctx, small, X, cola.PREC_F64, out=Y)
    W = cola.cola_matvec(ctx, large, Z, cola.PREC_F64)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y, first)
    assert torch.equal(cola.cola_matvec(ctx, large, Z, cola.PREC_F64), W)
