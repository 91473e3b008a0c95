"""The chained column kernels of the Householder reduction at the orders where
their shapes change: rows per CTA (152 x 7 and 152 x 15 rows below the column),
the tensor-core products' threshold, ragged last tiles and panels, and columns
whose products nearly cancel, against LAPACK (tolerances of
tests/test_gpu_dense.py) and against the all-FP64 products."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(A, nb, panels=0):
    import paper_2406_10765_gb300 as pw
    n = A.shape[0]
    pw.pw_householder_panels(panels)
    try:
        w, y = pw.pw_heev(torch.from_numpy(A).cuda(), nb)
    finally:
        pw.pw_householder_panels(0)
    w, y = w.cpu().numpy(), y.cpu().numpy()
    ref = np.linalg.eigvalsh(A)
    scale = np.abs(ref).max()
    assert np.abs(w - ref).max() <= 1e-13 * scale * n ** 0.5
    assert np.abs(A @ y - y * w[:nb]).max() <= 1e-12 * scale
    assert np.abs(y.conj().T @ y - np.eye(nb)).max() <= 1e-12


def _rand(n):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return A + A.conj().T


@pytest.mark.parametrize("n", [258, 290, 321, 511, 1024, 1025, 1064, 1066, 1100])
@pytest.mark.parametrize("panels", [0, 2])
def test_orders(n, panels):
    _check(_rand(n), 64, panels)


def test_largest_row_blocks():
    _check(_rand(2300), 32)


@pytest.mark.parametrize("n", [300, 1030])
@pytest.mark.parametrize("kind", ["diag", "tri", "rank1", "rank3", "block", "arrow"])
def test_special_columns(n, kind):
    G = _rand(n)
    if kind == "diag":
        A = np.diag(np.diag(G))
    elif kind == "tri":
        A = np.triu(np.tril(G, 1), -1)
    elif kind == "rank1":              # every column after the first cancels to rounding
        A = np.outer(G[0], G[0].conj())
        A = 0.5 * (A + A.conj().T)
    elif kind == "rank3":
        A = G[:, :3] @ G[:, :3].conj().T
        A = 0.5 * (A + A.conj().T)
    elif kind == "block":
        A = G.copy()
        A[n // 2:, :n // 2] = 0
        A[:n // 2, n // 2:] = 0
    else:
        A = np.diag(np.diag(G)) * 100
        A[:, 0] = G[:, 0]
        A[0, :] = G[:, 0].conj()
        A[0, 0] = 1.0
    _check(A, 32)
