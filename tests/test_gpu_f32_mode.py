"""FP32 Kronecker products large enough for the 128 x 16 TN register-tiled
kernel: sides around its 16-wide output and k steps, several output chunks, no
alignment to four; against FP64, within 2e-5 of sum |K| |x| per entry (at most
300 contracted entries a mode: 300 x 2^-24 = 1.8e-5 for both modes' worst case
half)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _kron(F, X):
    R = X.shape[0]
    for f in F:
        X = np.ascontiguousarray(np.swapaxes(np.matmul(f, X.reshape(R, f.shape[1], -1)), 1, 2))
    return X.reshape(R, -1)


@pytest.mark.parametrize("shapes,R", [
    (((97, 97), (50, 50)), 60), (((130, 130), (9, 9)), 50), (((5, 300), (300, 5)), 70),
    (((16, 16), (17, 17)), 90), (((128, 128), (112, 112)), 48), (((129, 129), (15, 15)), 50),
])
@pytest.mark.parametrize("diag", [None, "scalar", "vector"])
def test_f32_mode_products(shapes, R, diag):
    import paper_2309_03060_gb300 as cola
    r = np.random.default_rng(R)
    F = [r.standard_normal(s) for s in shapes]
    rows, cols = (int(np.prod([s[i] for s in shapes])) for i in (0, 1))
    if diag and rows != cols:
        pytest.skip("a diagonal term needs a square operator")
    X = r.standard_normal((R, cols))
    ctx = cola.cola_create(0)
    op = cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(
        ctx, torch.tensor(f, dtype=torch.float32, device="cuda")) for f in F])
    ref, bound = _kron(F, X), _kron([np.abs(f) for f in F], np.abs(X))
    if diag:
        d = r.standard_normal(1 if diag == "scalar" else rows)
        dt = torch.tensor(d, dtype=torch.float32, device="cuda")
        dg = cola.cola_linop_diag(ctx, dt, n=rows) if diag == "scalar" else \
            cola.cola_linop_diag(ctx, dt)
        op = cola.cola_linop_sum(ctx, [op, dg], [0.5, -2.0])
        ref, bound = 0.5 * ref - 2.0 * d * X, 0.5 * bound + np.abs(2.0 * d * X)
    Y = cola.cola_matvec(ctx, op, torch.tensor(X, dtype=torch.float32, device="cuda"),
                         cola.PREC_F32).double().cpu().numpy()
    assert (np.abs(Y - ref) <= 2e-5 * bound).all(), float((np.abs(Y - ref) / bound).max())
