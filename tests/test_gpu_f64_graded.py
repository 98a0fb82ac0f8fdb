"""FP64 products on the tensor cores are accurate entry by entry: every output of
a mode step is within a bound of its own sum |f| |x|, whatever the other entries
of its factor row and vector are.

Bound of one mode step with K contracted entries.  An output keeps its digit
product only where the sum of leading magnitudes is at least 2560.  A leading
magnitude is at most twice |f| 2^(7 - Ef) or |x| 2^(6 - Ex), so there sum |f| |x| >=
2560 / 4 2^-13 2^(Ef + Ex) = 2^-3.68 2^(Ef + Ex).  Dropped digit pairs (6 2^-55), x kept
to 2^-55 and f to 2^-56 of 2^Ex and 2^Ef are at most 1.14 2^-52 K 2^(Ef + Ex), hence at
most 0.92 2^-48 K sum |f| |x|; with the roundings, 2^-48 K sum |f| |x|.  Plain FP64
products stay within 2^-53 K sum |f| |x|.  Contributions of a later k chunk may
also be hidden by the sum so far: 1.14 2^-52 K 2^-4 of it, and that sum is at most
sum |f| |x| of its chunks."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _apply(F, X):
    import paper_2309_03060_gb300 as cola
    ctx = cola.cola_create(0)
    op = cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(ctx, torch.tensor(f, device="cuda"))
                                     for f in F])
    return cola.cola_matvec(ctx, op, torch.tensor(X, device="cuda"), cola.PREC_F64).cpu().numpy()


def _check(F, X):
    L = np.longdouble
    R = X.shape[0]
    cur, mag, c = X.astype(L), np.abs(X).astype(L), L(0)
    for f in F:
        y = np.matmul(f.astype(L), cur.reshape(R, f.shape[1], -1))
        s = np.matmul(np.abs(f).astype(L), mag.reshape(R, f.shape[1], -1))
        cur = np.ascontiguousarray(np.swapaxes(y, 1, 2)).reshape(R, -1)
        mag = np.ascontiguousarray(np.swapaxes(s, 1, 2)).reshape(R, -1)
        c += f.shape[1] * L(2.0) ** -48
    err = np.abs(_apply(F, X).astype(L) - cur)
    assert (err <= c * mag).all(), float((err / np.maximum(c * mag, L(1e-4900))).max())


def _rbf(r, n, ell, ordered=False):
    x = np.sort(r.random(n)) if ordered else r.random(n)
    return np.exp(-(x[:, None] - x[None]) ** 2 / (2 * ell * ell))


def test_identity_factors_return_graded_vectors():
    """Entries of one fibre 18 and 100 orders apart come back exactly: 0 and 1 times
    them are exact, in FP64 multiply-adds and in digits, which an output of a row with
    one entry takes only from an entry within a binade of its vector's largest."""
    r = np.random.default_rng(1)
    X = r.standard_normal((8, 128 * 128))
    X[:, ::3] *= 1e-18
    X[1, ::7] = 0.0
    X[2, 1:] *= 1e-100
    Y = _apply([np.eye(128), np.eye(128)], X)
    assert (Y == X).all()


@pytest.mark.parametrize("sides,R", [((128, 128), 6), ((65, 128), 16), ((130, 64), 9),
                                     ((257, 40), 9), ((33, 129), 17)])
@pytest.mark.parametrize("kind", ["rbf_unit_vectors", "rbf_graded", "blocks", "ordered_rbf"])
def test_outputs_are_accurate_entry_by_entry(sides, R, kind):
    r = np.random.default_rng(R)
    N = sides[0] * sides[1]
    if kind == "rbf_unit_vectors":  # columns of a covariance: entries down to 1e-87
        F = [_rbf(r, n, 0.05) for n in sides]
        X = np.zeros((R, N))
        X[np.arange(R), r.integers(0, N, R)] = 1.0
    elif kind == "rbf_graded":
        F = [_rbf(r, n, 0.1) for n in sides]
        X = r.standard_normal((R, N)) * np.exp(12.0 * r.standard_normal((R, N)))
    elif kind == "blocks":  # independent blocks of very different sizes
        F = []
        for n in sides:
            f = np.zeros((n, n))
            for b in range(0, n, 20):
                m = min(20, n - b)
                f[b:b + m, b:b + m] = r.standard_normal((m, m)) * 10.0 ** (-b / 5.0)
            F.append(f)
        X = r.standard_normal((R, N)) * 10.0 ** r.uniform(-30, 30, (R, N))
    else:  # a grid: k chunks far from the diagonal are tiny
        F = [_rbf(r, n, 0.05, ordered=True) for n in sides]
        X = r.standard_normal((R, N))
        X[0, : N // 2] = 0.0
    _check(F, X)


@pytest.mark.parametrize("n,R", [(128, 6), (64, 64), (200, 5)])
def test_residuals_of_identity_factors_are_exact(n, R):
    """Old values and a factor of -1: b - A x of a solve that starts from its solution,
    with entries of one fibre 18 orders apart, is 0 (the products are exact)."""
    import paper_2309_03060_gb300 as cola
    r = np.random.default_rng(n)
    X = r.standard_normal((R, n * n))
    X[:, ::3] *= 1e-18
    X[1, : n // 2] = 0.0
    ctx = cola.cola_create(0)
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    op = cola.cola_linop_kron(ctx, *[cola.cola_linop_dense(ctx, eye) for _ in range(2)]).set_spd()
    B = torch.tensor(X, device="cuda")
    opts = cola.cola_cg_opts_default(precision=cola.PREC_MIXED, refine=1, tol=1e-10, maxiter=0)
    Y, info, st = cola.cola_cg_solve(ctx, op, B, opts, X0=B)
    assert st == 0 and [i["rel_residual"] for i in info] == [0.0] * R
    assert torch.equal(Y, B)
