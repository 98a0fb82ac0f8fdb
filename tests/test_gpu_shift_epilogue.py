"""MVMs of Kron + Diag with the diagonal term in the last product's epilogue, in
every precision, for scalar and per-element diagonals, either order of the
terms and coefficients other than 1, against the FP64 oracle-style product.

Tolerances: FP64 1e-12 and FP32 / MIXED (3 x 3 terms) 2e-5 of sum |K| |x| + |d x|
per entry (at most 257 contracted entries a mode, three modes)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _kron(F, X):
    R = X.shape[0]
    for f in F:
        X = np.ascontiguousarray(np.swapaxes(np.matmul(f, X.reshape(R, f.shape[1], -1)), 1, 2))
    return X.reshape(R, -1)


@pytest.mark.parametrize("prec", ["f64", "f32", "mixed"])
@pytest.mark.parametrize("scalar", [True, False])
@pytest.mark.parametrize("sides,R", [
    ((5, 7), 1), ((64, 64), 1), ((33, 17), 3),          # one output per thread
    ((128, 128), 6), ((65, 130), 9), ((257, 64), 5),    # digit products, several chunks
    ((4, 128, 128), 2), ((24, 20, 36), 4), ((31, 8, 45), 9), ((16, 16), 200),
])
def test_kron_plus_diag(prec, scalar, sides, R):
    import paper_2309_03060_gb300 as cola
    r = np.random.default_rng(sum(sides) + R)
    F = [r.standard_normal((n, n)) for n in sides]
    N = int(np.prod(sides))
    d = r.standard_normal(1 if scalar else N)
    X = r.standard_normal((R, N))
    ctx = cola.cola_create(0)
    kron = cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(ctx, torch.tensor(f, device="cuda"))
                                       for f in F])
    dt = torch.tensor(d, device="cuda")
    dg = cola.cola_linop_diag(ctx, dt, n=N) if scalar else cola.cola_linop_diag(ctx, dt)
    code = {"f64": cola.PREC_F64, "f32": cola.PREC_F32, "mixed": cola.PREC_MIXED}[prec]
    Xd = torch.tensor(X, dtype=torch.float64 if prec == "f64" else torch.float32, device="cuda")
    bound = _kron([np.abs(f) for f in F], np.abs(X))
    for terms, co in (((kron, dg), (1.0, 1.0)), ((dg, kron), (-0.5, 2.0))):
        op = cola.cola_linop_sum(ctx, list(terms), list(co))
        ck, cd = (co[0], co[1]) if terms[0] is kron else (co[1], co[0])
        Y = cola.cola_matvec(ctx, op, Xd, code, split_terms=3).double().cpu().numpy()
        ref = ck * _kron(F, X) + cd * d * X
        tol = (1e-12 if prec == "f64" else 2e-5) * (abs(ck) * bound + abs(cd * d * X))
        assert (np.abs(Y - ref) <= tol).all(), float((np.abs(Y - ref) / tol).max())
