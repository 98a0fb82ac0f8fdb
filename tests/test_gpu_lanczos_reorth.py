"""Full reorthogonalisation of the Lanczos basis (reorth=1): block-chunked
Gram-Schmidt passes, at vector lengths around the 512-entry chunk and with
more stored vectors than one 256-entry coefficient tile.

The operator is diagonal with distinct entries, so its eigenvalues are known.
With the basis kept orthogonal, T_m has no repeated (ghost) Ritz values and its
extreme ones converge to the extreme entries; the first coefficients equal a
plain FP64 recurrence's with the same two projections."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cola():
    import paper_2309_03060_gb300 as m
    return m


def _lanczos_ref(d, z, m):
    q = z / np.linalg.norm(z)
    Q, a, b = [q], [], []
    for j in range(m):
        w = d * Q[j] - (b[-1] * Q[j - 1] if j else 0.0)
        a.append(w @ Q[j])
        w = w - a[-1] * Q[j]
        S = np.stack(Q)
        for _ in range(2):
            w = w - S.T @ (S @ w)
        b.append(np.linalg.norm(w))
        Q.append(w / b[-1])
    return np.array(a), np.array(b)


@pytest.mark.parametrize("N,m,nv", [(7, 5, 1), (511, 40, 2), (512, 40, 1), (513, 40, 3),
                                    (700, 300, 2), (40000, 30, 2)])
def test_reorthogonalised_lanczos_f64(cola, N, m, nv):
    r = np.random.default_rng(N + m)
    d = np.sort(0.5 + r.random(N))
    Z = r.choice([-1.0, 1.0], (nv, N))
    ctx = cola.cola_create(0)
    op = cola.cola_linop_diag(ctx, torch.tensor(d, device="cuda")).set_spd()
    al, be, me = cola.cola_lanczos(ctx, op, torch.tensor(Z, device="cuda"), m, cola.PREC_F64,
                                   reorth=1)
    al, be = al.cpu().numpy(), be.cpu().numpy()
    assert (me.cpu().numpy() == m).all()
    k = min(m, 20)
    for v in range(nv):
        a_ref, b_ref = _lanczos_ref(d, Z[v], k)
        # 20 steps amplify FP64 rounding (1e-16) by far less than 1e6
        assert np.abs(al[v, :k] - a_ref).max() < 1e-10
        assert np.abs(be[v, :k - 1] - b_ref[:k - 1]).max() < 1e-10
        T = np.diag(al[v]) + np.diag(be[v, :m - 1], 1) + np.diag(be[v, :m - 1], -1)
        th = np.linalg.eigvalsh(T)
        assert d[0] - 1e-12 < th[0] and th[-1] < d[-1] + 1e-12
        assert np.diff(th).min() > 1e-9  # no ghost copies
        if 2 * m >= N // 2:
            assert np.abs(th[-3:] - d[-3:]).max() < (1e-8 if m > 100 else 1.0)


def test_reorthogonalised_lanczos_f32(cola):
    """FP32 vectors: extreme Ritz values of 300 steps on 700 entries without
    ghosts, to FP32 accuracy (the matrix norm is 1.5; 1e-5 is ~80 ulp)."""
    r = np.random.default_rng(3)
    d = np.sort(0.5 + r.random(700))
    ctx = cola.cola_create(0)
    op = cola.cola_linop_diag(ctx, torch.tensor(d, dtype=torch.float32, device="cuda")).set_spd()
    Z = torch.tensor(r.choice([-1.0, 1.0], (1, 700)), dtype=torch.float32, device="cuda")
    al, be, me = cola.cola_lanczos(ctx, op, Z, 300, cola.PREC_F32, reorth=1)
    al, be = al.cpu().numpy()[0], be.cpu().numpy()[0]
    th = np.linalg.eigvalsh(np.diag(al) + np.diag(be[:299], 1) + np.diag(be[:299], -1))
    assert np.abs(th[-3:] - d[-3:]).max() < 1e-5 and np.abs(th[:3] - d[:3]).max() < 1e-5
    assert np.diff(th)[-5:].min() > 1e-5 or np.diff(d)[-5:].min() < 2e-5
