"""The hand-written FP64 dense generalised Hermitian eigensolver (the Rayleigh-Ritz subspace problem,
§5.1) through the C ABI, against the oracle's dense LAPACK eigensolve.

Bars: eigenvalues within 1e-11 of the largest |eigenvalue| of the oracle's (a backward-stable
solver's error on these well-conditioned B); eigenvectors checked by their own invariants, since
degenerate and clustered eigenvalues make individual vectors gauge-dependent: the residual
|A X - B X diag(w)| <= 1e-11 |A| and B-orthonormality |X^H B X - I| <= 1e-11.  Real symmetric
pencils run in real arithmetic and are checked the same way (and for exactly real outputs); the
returned Cholesky factor is checked against LAPACK's.
"""
import numpy as np
import pytest

import oracle as O
import paper_2507_08578_gb300.kss as K
from tests.kss_helpers import ensure_built, make_ctx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    ensure_built()
    c = make_ctx()
    yield c
    torch.cuda.synchronize()
    K.kss_destroy(c)


def pencil(n, seed, real=False, cond=1e3):
    rng = np.random.default_rng(seed)
    def rnd():
        m = rng.standard_normal((n, n))
        return m if real else m + 1j * rng.standard_normal((n, n))
    a = rnd()
    A = (a + a.conj().T) / 2
    m = rnd()
    B = m @ m.conj().T / n + np.eye(n) / cond
    return A.astype(np.complex128), B.astype(np.complex128)


def to_dev(M, ld=None):
    """Column-major device copy: a (ncols, ld) tensor whose row j holds column j (rows past n are
    filled with a marker value that must stay untouched by the lower-triangle reads)."""
    import torch
    n = M.shape[0]
    ld = ld or n
    T = np.full((n, ld), 5.0 + 5.0j)
    T[:, :n] = M.T
    # poison the strictly upper triangle: the solver reads the lower triangles only
    for j in range(n):
        T[j, :j] = np.nan + 1j * np.nan
    return torch.from_numpy(T).cuda()


def check(A, B, w, X, tol=1e-11):
    wr, _ = O.lowest_generalized_eigenpairs(A, B, A.shape[0])
    scale = max(1.0, np.max(np.abs(wr)))
    assert np.max(np.abs(w - wr)) <= tol * scale, np.max(np.abs(w - wr))
    R = A @ X - (B @ X) * w[None, :]
    assert np.max(np.abs(R)) <= tol * max(1.0, np.max(np.abs(A))) * max(1.0, np.max(np.abs(X))), np.max(np.abs(R))
    G = X.conj().T @ B @ X
    assert np.max(np.abs(G - np.eye(A.shape[0]))) <= tol * max(1.0, np.linalg.norm(B, 2))


def run(ctx, pencils, real=False, lds=None):
    import torch
    As = [to_dev(A, None if lds is None else lds[i]) for i, (A, _) in enumerate(pencils)]
    Bs = [to_dev(B) for _, B in pencils]
    ws = [torch.zeros(max(1, A.shape[0]), dtype=torch.float64, device="cuda") for A, _ in pencils]
    info = K.kss_dense_hegv(ctx, As, Bs, ws, real=real)
    out = []
    for i, (A, B) in enumerate(pencils):
        n = A.shape[0]
        T = As[i].cpu().numpy()
        if lds is not None:
            assert np.all(T[:, n:] == 5.0 + 5.0j)  # rows past n untouched
        out.append((ws[i].cpu().numpy()[:n], T[:, :n].T.copy()))
    return info, out


@pytest.mark.parametrize("n", [1, 2, 3, 17, 31, 32, 64, 159, 160, 301, 564])
def test_single_pencil(ctx, n):
    A, B = pencil(n, seed=n)
    info, [(w, X)] = run(ctx, [(A, B)])
    assert info[0] == 0
    check(A, B, w, X)


def test_batched_pencils_of_uneven_order_with_padding(ctx):
    ps = [pencil(n, seed=100 + n) for n in (5, 33, 96, 141, 7, 120)]
    lds = [p[0].shape[0] + 3 for p in ps]
    info, out = run(ctx, ps, lds=lds)
    assert np.all(info == 0)
    for (A, B), (w, X) in zip(ps, out):
        check(A, B, w, X)


@pytest.mark.parametrize("n", [40, 200])
def test_degenerate_clusters(ctx, n):
    """Exactly degenerate eigenvalues (shells of 1, 6, 12 and the rest, as in the free-electron
    spectrum) in a random unitary frame, B = I: the cluster's vectors must come out orthonormal."""
    rng = np.random.default_rng(7)
    lam = np.concatenate([np.zeros(1), np.full(6, 0.2), np.full(12, 0.4), np.linspace(0.5, 2.0, n - 19)])
    q, _ = np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    A = (q * lam[None, :]) @ q.conj().T
    A = (A + A.conj().T) / 2
    B = np.eye(n, dtype=np.complex128)
    info, [(w, X)] = run(ctx, [(A, B)])
    assert info[0] == 0
    check(A, B, w, X)


@pytest.mark.parametrize("n", [1, 2, 24, 31, 32, 159, 300, 700])
def test_real_symmetric(ctx, n):
    """Real symmetric pencils (solved in real arithmetic): a single pencil runs on one CTA below
    order 32 and on the cooperative grid from 32; imaginary parts planted in the inputs are
    ignored."""
    A, B = pencil(n, seed=3 * n, real=True)
    rng = np.random.default_rng(n)
    junk = 1j * rng.standard_normal((n, n))
    info, [(w, X)] = run(ctx, [(A + junk, B + junk.T)], real=True)
    assert info[0] == 0
    assert np.all(X.imag == 0)
    check(A.real.astype(np.complex128), B.real.astype(np.complex128), w, X)


def test_real_batched_pencils_of_uneven_order_with_padding(ctx):
    ps = [pencil(n, seed=200 + n, real=True) for n in (3, 40, 97, 150, 8)]
    lds = [p[0].shape[0] + 5 for p in ps]
    info, out = run(ctx, ps, real=True, lds=lds)
    assert np.all(info == 0)
    for (A, B), (w, X) in zip(ps, out):
        assert np.all(X.imag == 0)
        check(A, B, w, X)


@pytest.mark.parametrize("n", [40, 200])
def test_real_degenerate_clusters(ctx, n):
    """Exactly degenerate shells in a random orthogonal frame, B = I, in real arithmetic."""
    rng = np.random.default_rng(9)
    lam = np.concatenate([np.zeros(1), np.full(6, 0.2), np.full(12, 0.4), np.linspace(0.5, 2.0, n - 19)])
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    A = (q * lam[None, :]) @ q.T
    A = ((A + A.T) / 2).astype(np.complex128)
    B = np.eye(n, dtype=np.complex128)
    info, [(w, X)] = run(ctx, [(A, B)], real=True)
    assert info[0] == 0
    check(A, B, w, X)


@pytest.mark.parametrize("n,real", [(50, False), (50, True), (260, False), (260, True)])
def test_cholesky_factor_returned(ctx, n, real):
    """On return the lower triangle of B holds L with B = L L^H (LAPACK's factor: positive real
    diagonal), the strictly upper triangle is untouched."""
    import torch
    A, B = pencil(n, seed=11 * n, real=real)
    Bd = to_dev(B)
    Ad = to_dev(A)
    w = torch.zeros(n, dtype=torch.float64, device="cuda")
    info = K.kss_dense_hegv(ctx, [Ad], [Bd], [w], real=real)
    assert info[0] == 0
    T = Bd.cpu().numpy().T  # column-major back to (row, col)
    L = np.tril(T)
    ref = np.linalg.cholesky(B)
    assert np.max(np.abs(L - ref)) <= 1e-12 * np.max(np.abs(ref))
    assert np.all(np.isnan(T[np.triu_indices(n, 1)]))
    if real:
        assert np.all(L.imag == 0)


@pytest.mark.parametrize("n", [12, 200])
def test_not_positive_definite(ctx, n):
    """B with a negative eigenvalue: the Cholesky stops with info = j + 1 > 0 (LAPACK convention)."""
    A, B = pencil(n, seed=5)
    B = B - 2.0 * np.linalg.norm(B, 2) * np.outer(np.eye(n)[n // 2], np.eye(n)[n // 2])
    info, _ = run(ctx, [(A, B)])
    assert 0 < info[0] <= n


@pytest.mark.parametrize("name", ["graded", "split", "tight", "scaled_down", "scaled_up", "wilkinson", "zero"])
@pytest.mark.parametrize("n", [21, 67])
def test_tridiagonal_spectra(ctx, name, n):
    """Tridiagonal pencils (B = 1) whose Sturm sequences and pivots leave the ordinary range: sizes
    graded over 1e-28, off-diagonals exactly zero, pairs closer than the bracket of one count,
    norms near the ends of the exponent range, Wilkinson's near-equal pairs, the zero matrix."""
    d = np.linspace(-1.0, 1.0, n) ** 3
    e = np.full(n - 1, 0.1)
    s = 1.0
    if name == "graded":
        d, e = 10.0 ** -np.linspace(0, 28, n), 0.3 * 10.0 ** -np.linspace(0, 28, n - 1)
    elif name == "split":
        e[::3] = 0.0
    elif name == "tight":
        e[:] = 1e-9
        d = np.round(d * 4) / 4 + 1e-8 * np.arange(n)
    elif name == "scaled_down":
        s = 1e-120
    elif name == "scaled_up":
        s = 1e120
    elif name == "wilkinson":
        d, e = np.abs(np.arange(n) - n // 2).astype(float), np.ones(n - 1)
    elif name == "zero":
        d, e = 0 * d, 0 * e
    A = (np.diag(d) + np.diag(e, 1) + np.diag(e, -1)).astype(np.complex128)
    info, [(w, X)] = run(ctx, [(A * s, np.eye(n, dtype=np.complex128))], real=True)
    assert info[0] == 0
    check(A, np.eye(n, dtype=np.complex128), w / s, X)


@pytest.mark.parametrize("count,n,real", [(3, 33, False), (150, 21, True), (150, 18, False), (400, 9, False), (1000, 5, True)])
def test_batches_on_clusters(ctx, count, n, real):
    """Batches whose pencils run on 8, 4, 2 and 1 CTAs each, one of them not positive definite: it
    stops alone, the others are solved."""
    ps = [pencil(n - i % 3, seed=300 + i % 7, real=real) for i in range(count)]
    bad = count // 2
    A, B = ps[bad]
    ps[bad] = (A, B - 3.0 * np.linalg.norm(B, 2) * np.eye(B.shape[0]))
    info, out = run(ctx, ps, real=real)
    assert info[bad] == 1 and np.all(np.delete(info, bad) == 0)
    for i in list(range(0, count, max(1, count // 12))) + [count - 1]:
        if i != bad:
            check(*ps[i], *out[i])


@pytest.mark.parametrize("n,real", [(1300, False), (1216, False), (1217, False), (1830, True)])
def test_orders_whose_columns_stay_in_memory(ctx, n, real):
    """Single pencils around and above the order up to which a CTA of the grid holds its columns in
    shared memory during the tridiagonalisation (1216 complex, 1824 real).  B as well conditioned as a
    filtered block's Gram matrix: at these orders the spread of levels that a badly conditioned B gives
    leaves hundreds of them closer than 1e-5 |T|, which one thread orthogonalises."""
    A, B = pencil(n, seed=n, real=real, cond=1.0)
    info, [(w, X)] = run(ctx, [(A, B)], real=real)
    assert info[0] == 0
    check(A, B, w, X)


@pytest.mark.parametrize("count,n,real", [(3, 300, False), (2, 420, True), (130, 170, False), (470, 122, True)])
def test_batches_whose_columns_stay_in_memory(ctx, count, n, real):
    """Batches above the order at which a CTA holds its columns, on clusters of 8 (two forms) and 4 and
    on single CTAs, unevenly: the smaller pencils of a batch take the form of the largest."""
    ps = [pencil(n - (i % 5) * (n // 9), seed=400 + i % 11, real=real, cond=1.0) for i in range(count)]
    info, out = run(ctx, ps, real=real)
    assert np.all(info == 0)
    for i in list(range(0, count, max(1, count // 6))) + [count - 1]:
        check(*ps[i], *out[i])


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("count", [20, 60, 76, 152])
def test_batches_of_equal_order(ctx, count, real):
    """Batches that fill the chip once with clusters of 8, 4 and 2, and with single CTAs (order 64)."""
    ps = [pencil(64, seed=500 + i % 5, real=real) for i in range(count)]
    info, out = run(ctx, ps, real=real)
    assert np.all(info == 0)
    for i in (0, 1, count // 2, count - 1):
        check(*ps[i], *out[i])
