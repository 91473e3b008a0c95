"""The eigensolver and the FP64-accurate product in the fixed order of operations of
the mixed iteration's Rayleigh-Ritz: against LAPACK at the orders, spectra and
special matrices (and tolerances) of tests/test_gpu_dense.py and
tests/test_gpu_house_cols.py, the product exactly on integers, and the bits of the
results, which are what the fixed order keeps."""
import hashlib

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rand(n):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return A + A.conj().T


def _matrix(n, kind):
    from test_gpu_dense import _herm
    G = _rand(n)
    if kind in ("rand", "degenerate", "cluster"):
        return _herm(n, n + 7, kind)
    if kind == "diag":
        return np.diag(np.diag(G))
    if kind == "tri":
        return np.triu(np.tril(G, 1), -1)
    if kind == "rank1":
        A = np.outer(G[0], G[0].conj())
        return 0.5 * (A + A.conj().T)
    if kind == "rank3":
        A = G[:, :3] @ G[:, :3].conj().T
        return 0.5 * (A + A.conj().T)
    if kind == "block":
        A = G.copy()
        A[n // 2:, :n // 2] = 0
        A[:n // 2, n // 2:] = 0
        return A
    if kind == "range":
        d = 10.0 ** np.random.default_rng(n).uniform(-3, 3, n)
        return G * np.sqrt(np.outer(d, d)) * 1e-6 + np.diag(d)
    raise ValueError(kind)


ORDERS = [(1, 1, "rand"), (2, 1, "rand"), (3, 3, "rand"), (33, 11, "rand"), (72, 24, "rand"), (97, 30, "diag"),
          (130, 40, "degenerate"), (200, 64, "cluster"), (515, 170, "rand")]
PANELS = [(n, 64, "rand") for n in (258, 290, 321, 511, 1024, 1025, 1064, 1066)]
SPECTRA = [(1100, 300, "degenerate"), (1200, 333, "cluster"), (1150, 250, "range"), (1700, 600, "rand")]
SPECIAL = [(n, 32, k) for n in (300, 1030) for k in ("diag", "tri", "rank1", "rank3", "block")]


@pytest.mark.parametrize("n,nb,kind", ORDERS + PANELS + SPECTRA + SPECIAL)
def test_matches_lapack(n, nb, kind):
    import paper_2406_10765_gb300 as pw
    A = _matrix(n, kind)
    w, Y = pw.pw_heev_fixed(torch.from_numpy(A).cuda(), nb)
    w, Y = w.cpu().numpy(), Y.cpu().numpy()
    ref = np.linalg.eigvalsh(A)
    scale = max(1.0, np.abs(ref).max())
    assert np.abs(w - ref).max() < 1e-13 * scale * n ** 0.5
    assert np.abs(A @ Y - Y * w[:nb]).max() < 1e-12 * scale
    assert np.abs(Y.conj().T @ Y - np.eye(nb)).max() < 1e-12


@pytest.mark.parametrize("k", [1, 8, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 129, 1000])
@pytest.mark.parametrize("m,n", [(128, 32), (33, 65), (130, 3), (1300, 1000), (129, 4900)])
def test_integer_products_exact(m, n, k):
    """Tiles, chunks of 32 complex K, several tiles per CTA for every K, K split."""
    import paper_2406_10765_gb300 as pw
    from gpu_util import to_dev
    rng = np.random.default_rng(1000 * k + m + n)
    top = 2 ** 18 - 1
    A = rng.integers(-top, top + 1, (m, k)) + 1j * rng.integers(-top, top + 1, (m, k))
    B = rng.integers(-top, top + 1, (k, n)) + 1j * rng.integers(-top, top + 1, (k, n))
    A[0], B[:, 0] = top - 1j * top, -top + 1j * top            # the largest digits, one sign
    C = rng.integers(-top, top + 1, (m, n)) + 1j * rng.integers(-top, top + 1, (m, n))
    c = to_dev(C)
    pw.pw_zgemm_f64tc_fixed("N", "N", to_dev(A), to_dev(B), alpha=-1, beta=1, C=c)
    # |Re|, |Im| < 2 k 2^36 + 2^18 < 2^53: the reference is exact in FP64 too
    assert np.array_equal(c.cpu().numpy(), C - A @ B)


def _bits(n):
    """Hermitian, entries in multiples of 2^-30: the same on every machine."""
    u = synth.uniform01(n, np.arange(2 * n * n)).reshape(2, n, n) - 0.5
    u = np.round(u * 2.0 ** 30) * 2.0 ** -30
    A = np.tril(u[0], -1) + 1j * np.tril(u[1], -1)
    return A + A.conj().T + np.diag(np.diag(u[0]))


def _digest(t):
    return hashlib.sha256(np.ascontiguousarray(t.cpu().numpy()).tobytes()).hexdigest()[:16]


# recorded with the kernels that the fixed order is the order of (35378f1)
@pytest.mark.parametrize("n,nb,w_bits,y_bits", [
    (54, 18, "d44916d543e2135e", "97cf3e8622292719"), (300, 100, "5ae215caf2b51805", "2206a4f48b41c7c8"),
    (640, 200, "6192231036178e35", "12cbc7ffbf0ee23e"), (1100, 300, "394b67f05c47887a", "a3bb15b255787817"),
    (1458, 486, "870a3fa9aea8146d", "7138195134cb32a1")])
def test_bits_of_the_eigenpairs(n, nb, w_bits, y_bits):
    import paper_2406_10765_gb300 as pw
    w, Y = pw.pw_heev_fixed(torch.from_numpy(_bits(n)).cuda(), nb)
    assert (_digest(w), _digest(Y)) == (w_bits, y_bits)


@pytest.mark.parametrize("m,n,k,c_bits", [(300, 200, 700, "b25edf7647e027e3"), (1000, 1000, 64, "c4548a3b2cc2f2e7"),
                                          (700, 90, 1500, "0bd9760a63353101")])
def test_bits_of_the_product(m, n, k, c_bits):
    import paper_2406_10765_gb300 as pw

    def op(rows, cols, seed):
        u = synth.uniform01(seed, np.arange(2 * rows * cols)).reshape(2, rows, cols) - 0.5
        return torch.from_numpy((u[0] + 1j * u[1]).T.copy()).cuda().T

    assert _digest(pw.pw_zgemm_f64tc_fixed("N", "N", op(m, k, 1), op(k, n, 2))) == c_bits


@pytest.mark.parametrize("n", [257, 520, 1060])
@pytest.mark.parametrize("e", [-400, -100, 9, 100, 400])
def test_scaled(n, e):
    """Matrices far from 1 in size, as tests/test_gpu_heev_scale.py has them for pw_heev."""
    import paper_2406_10765_gb300 as pw
    A = _rand(n)
    w, Y = pw.pw_heev_fixed(torch.from_numpy(A * 2.0 ** e).cuda(), 24)
    w, Y = w.cpu().numpy() * 2.0 ** -e, Y.cpu().numpy()
    ref = np.linalg.eigvalsh(A)
    scale = np.abs(ref).max()
    assert np.abs(w - ref).max() <= 1e-13 * scale * n ** 0.5
    assert np.abs(A @ Y - Y * w[:24]).max() <= 1e-12 * scale
    assert np.abs(Y.conj().T @ Y - np.eye(24)).max() <= 1e-12
