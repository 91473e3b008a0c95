"""FP64-accurate tensor-core product where a CTA takes several tiles: more tiles
than SMs, ragged last rows and columns, K of less than a chunk to several, alpha
and beta of the plain epilogue (+-1; 0 or 1) and of the general one.  (Hermitian
outputs, whole ranges of tiles skipped: the eigensolver's tests.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [5, 33, 100])
@pytest.mark.parametrize("m,n", [(1300, 1000), (129, 4900), (20000, 33)])
@pytest.mark.parametrize("alpha,beta", [(1, 0), (-1, 1), (2j, 1 - 1j)])
def test_integer_products_exact(m, n, k, alpha, beta):
    import paper_2406_10765_gb300 as pw
    from gpu_util import to_dev
    rng = np.random.default_rng(m + n + k)
    top = 2 ** 18 - 1
    A = rng.integers(-top, top + 1, (m, k)) + 1j * rng.integers(-top, top + 1, (m, k))
    B = rng.integers(-top, top + 1, (k, n)) + 1j * rng.integers(-top, top + 1, (k, n))
    C = rng.integers(-top, top + 1, (m, n)) + 1j * rng.integers(-top, top + 1, (m, n))
    c = to_dev(C)
    pw.pw_zgemm_f64tc("N", "N", to_dev(A), to_dev(B), alpha=alpha, beta=beta, C=c)
    # every term is an integer below 2^53
    assert np.array_equal(c.cpu().numpy(), alpha * (A @ B) + beta * C)
