"""Eigenproblems of matrices far from 1 in size (the digit products of the
reduction's updates scale v and w together): the decomposition of 2^e A is that of
A scaled, up to the tolerances of tests/test_gpu_dense.py, on either side of the
order from which the reduction's updates are products and its column products use
the tensor cores."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [257, 520, 1060])
@pytest.mark.parametrize("e", [-400, -100, -9, 9, 100, 400])
def test_scaled(n, e):
    import paper_2406_10765_gb300 as pw
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    A = A + A.conj().T
    w, y = pw.pw_heev(torch.from_numpy(A * 2.0 ** e).cuda(), 24)
    w, y = w.cpu().numpy() * 2.0 ** -e, y.cpu().numpy()
    ref = np.linalg.eigvalsh(A)
    scale = np.abs(ref).max()
    assert np.abs(w - ref).max() <= 1e-13 * scale * n ** 0.5
    assert np.abs(A @ y - y * w[:24]).max() <= 1e-12 * scale
    assert np.abs(y.conj().T @ y - np.eye(24)).max() <= 1e-12
