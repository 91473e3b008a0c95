"""The Householder reduction of the last columns in one thread-block cluster:
orders around its own largest (all of the matrix, or the end of a larger one),
the CTA count and the warps, degenerate columns and extreme scales, against
LAPACK (tolerances of tests/test_gpu_dense.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(A, nb):
    import paper_2406_10765_gb300 as pw
    n = A.shape[0]
    w, y = pw.pw_heev(torch.from_numpy(A).cuda(), nb)
    w, y = w.cpu().numpy(), y.cpu().numpy()
    ref = np.linalg.eigvalsh(A)
    scale = np.abs(ref).max()
    assert np.abs(w - ref).max() <= 1e-13 * scale * n ** 0.5
    assert np.abs(A @ y - y * w[:nb]).max() <= 1e-12 * scale
    assert np.abs(y.conj().T @ y - np.eye(nb)).max() <= 1e-12


@pytest.mark.parametrize("n", [1, 2, 3, 4, 15, 16, 17, 18, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 272, 288,
                               289, 300])
def test_orders(n):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    _check(A + A.conj().T, n)


@pytest.mark.parametrize("n", [5, 40, 200])
@pytest.mark.parametrize("kind", ["diag", "tri", "real", "rank1", "block", "tiny", "huge"])
def test_degenerate_columns_and_scales(n, kind):
    rng = np.random.default_rng(7 * n)
    G = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    G = G + G.conj().T
    if kind == "diag":
        A = np.diag(np.diag(G))
    elif kind == "tri":
        A = np.triu(np.tril(G, 1), -1)
    elif kind == "real":
        A = G.real.astype(complex)
    elif kind == "rank1":
        A = np.outer(G[0], G[0].conj())
        A = 0.5 * (A + A.conj().T)
    elif kind == "block":              # zero columns below the diagonal in the middle of the reduction
        A = G.copy()
        A[n // 2:, :n // 2] = 0
        A[:n // 2, n // 2:] = 0
    else:
        # the squares of a column leave the range in which approximate reciprocals are refined
        A = G * (2.0 ** -468 if kind == "tiny" else 2.0 ** 480)
    _check(A, max(1, n // 2))


def test_several_streams():
    """Clusters of concurrent solves on different streams."""
    import paper_2406_10765_gb300 as pw
    from concurrent.futures import ThreadPoolExecutor
    rng = np.random.default_rng(5)
    mats = []
    for n in (54, 72, 200, 256, 300, 54, 130, 90):
        A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        mats.append(A + A.conj().T)

    def solve(A):
        st = torch.cuda.Stream()
        a = torch.from_numpy(A).cuda()
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            w, _ = pw.pw_heev(a, 10, stream=st.cuda_stream)
        st.synchronize()
        return w.cpu().numpy()

    with ThreadPoolExecutor(4) as ex:
        got = list(ex.map(solve, mats * 3))
    for A, w in zip(mats * 3, got):
        ref = np.linalg.eigvalsh(A)
        assert np.abs(w - ref).max() <= 1e-13 * np.abs(ref).max() * len(ref) ** 0.5
