"""FP64 Kronecker products computed as digit products on the tensor cores,
against extended precision (numpy longdouble).

Bound of one mode step with K contracted entries, per output: inputs are kept
to 2^-55 (vector) and 2^-56 (factor row) of their largest entry, the dropped
digit pairs are at most 2^-52.4 K fmax xmax, the result is rounded once
(2^-53) per chunk of 128 k and once per sum of chunks; together below
2^-51 K fmax xmax.  A second step applies |F| to the first step's bound.  Sizes: one
and several k chunks and output chunks, edges of the 64-vector, 128-output and
16-wide k tiles, and products just above the size from which this path runs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cola():
    import paper_2309_03060_gb300 as m
    return m


def _steps(F, X):
    """Cyclic mode steps in longdouble with the error bound above."""
    L = np.longdouble
    R = X.shape[0]
    cur = X.astype(L)
    bound = np.zeros_like(cur)
    for f in F:
        K = f.shape[1]
        c = cur.reshape(R, K, -1)
        b = bound.reshape(R, K, -1)
        fl = f.astype(L)
        y = np.matmul(fl, c)
        fmax, xmax = np.abs(fl).max(1), np.abs(c).max(1)
        nb = np.matmul(np.abs(fl), b) + L(2.0) ** -51 * K * fmax[None, :, None] * xmax[:, None, :]
        cur = np.ascontiguousarray(np.swapaxes(y, 1, 2)).reshape(R, -1)
        bound = np.ascontiguousarray(np.swapaxes(nb, 1, 2)).reshape(R, -1)
    return cur, bound


def _gpu(cola, F, X):
    ctx = cola.cola_create(0)
    op = cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(ctx, torch.tensor(f, device="cuda"))
                                     for f in F])
    return cola.cola_matvec(ctx, op, torch.tensor(X, device="cuda"), cola.PREC_F64).cpu().numpy()


@pytest.mark.parametrize("shapes,R", [
    (((128, 128), (128, 128)), 5),     # full tiles
    (((64, 64), (65, 65)), 33),        # one vector past a 64-vector tile
    (((63, 63), (129, 129)), 17),      # one entry past a k chunk and an output chunk
    (((130, 130), (67, 67)), 9),
    (((257, 257), (33, 33)), 6),       # three k chunks
    (((16, 16), (17, 17), (200, 200)), 3),
    (((40, 200), (150, 48)), 9),       # rectangular factors
    (((5, 300), (300, 7)), 120),
])
def test_f64_products_match_extended_precision(cola, shapes, R):
    r = np.random.default_rng(R)
    F = [r.standard_normal(s) * np.exp(r.uniform(-3, 3, (s[0], 1))) for s in shapes]
    X = r.standard_normal((R, int(np.prod([s[1] for s in shapes]))))
    X *= np.exp(3.0 * r.standard_normal(X.shape))  # entries over several orders
    X[0, ::7] = 0.0
    Y = _gpu(cola, F, X)
    ref, bound = _steps(F, X)
    err = np.abs(Y.astype(np.longdouble) - ref)
    assert (err <= bound).all(), float((err / np.maximum(bound, 1e-300)).max())


def test_f64_products_extreme_scales(cola):
    """Rows and vectors near the ends of the exponent range, zero rows and
    vectors, and negative powers that leave denormal results."""
    r = np.random.default_rng(1)
    F = [r.standard_normal((128, 128)), r.standard_normal((96, 96))]
    F[0][3] = 0.0
    F[0][5] *= 2.0 ** 500
    F[0][6] *= 2.0 ** -500
    X = r.standard_normal((9, 128 * 96))
    X[1] = 0.0
    X[2] *= 2.0 ** 400
    X[3] *= 2.0 ** -560
    X[4] *= 2.0 ** -1040  # denormal inputs
    Y = _gpu(cola, F, X)
    ref, bound = _steps(F, X)
    err = np.abs(Y.astype(np.longdouble) - ref)
    tiny = np.longdouble(2.0) ** -1074 * 400  # denormal intermediates round absolutely
    assert (err <= bound + tiny * (1 + np.abs(F[1]).sum(1).max())).all()
    assert (Y[1] == 0).all()


def test_f64_products_non_finite(cola):
    """A NaN or Inf entry reaches exactly the outputs a plain product gives it."""
    r = np.random.default_rng(2)
    F = [r.standard_normal((128, 128)), r.standard_normal((128, 128))]
    X = r.standard_normal((6, 128 * 128))
    X[1, 700] = np.nan
    X[2, 300] = np.inf
    F[0][9, 4] = np.inf
    Y = _gpu(cola, F, X)
    with np.errstate(invalid="ignore"):
        T = np.swapaxes(np.matmul(F[0], X.reshape(6, 128, 128)), 1, 2)
        ref = np.swapaxes(np.matmul(F[1], np.ascontiguousarray(T)), 1, 2).reshape(6, -1)
    assert (np.isnan(Y) == np.isnan(ref)).all()
    assert (np.isinf(Y) == np.isinf(ref)).all() and (Y[np.isinf(Y)] == ref[np.isinf(ref)]).all()
    fin = np.isfinite(ref)
    assert np.abs(Y[fin] - ref[fin]).max() < 1e-9 * np.abs(ref[fin]).max()


def test_f64_product_time_out_is_reported_and_context_recovers(cola):
    r = np.random.default_rng(4)
    ctx = cola.cola_create(0)
    op = cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(
        ctx, torch.tensor(r.standard_normal((128, 128)), device="cuda")) for _ in range(2)])
    X = torch.tensor(r.standard_normal((6, 128 * 128)), device="cuda")
    first = cola.cola_matvec(ctx, op, X, cola.PREC_F64)
    ctx.test_stall_next_launch(20_000_000)
    cola.cola_matvec(ctx, op, X, cola.PREC_F64)
    torch.cuda.synchronize()
    with pytest.raises(cola.ColaError):
        for _ in range(3):  # reported once the queued copy of the flag has arrived
            cola.cola_matvec(ctx, op, X, cola.PREC_F64)
            torch.cuda.synchronize()
    assert torch.equal(cola.cola_matvec(ctx, op, X, cola.PREC_F64), first)
