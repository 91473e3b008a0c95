"""The digit slices of the Householder products on the tensor cores (five 12-bit
digits of the matrix, fourteen 4-bit digits of the vector, 128 products of up to
five pairs per FP32 sum): entries whose digits are all as large as they get and of
one sign, so that every group's sum is, and orders at which a tile's slices are
dealt to several CTAs, against LAPACK (tolerances of tests/test_gpu_dense.py; one
unit lost in a group's sum would show at 1e-7)."""
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


@pytest.mark.parametrize("digits", [(2047, 2047, 2047, 2047), (2047, -2048, -2048, -2048), (1024, -2048, -2048, -2048),
                                    (1025, 1, -1, 2047)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -300])
def test_extreme_digits(digits, scale):
    n = 1160
    a = scale * sum(d * 2.0 ** (-12 * (p + 1)) for p, d in enumerate(digits))
    s = np.sign(np.arange(n)[:, None] - np.arange(n)[None, :])
    _check(a * (1.0 + 1j * s), 16)


@pytest.mark.parametrize("n", [1153, 1408, 1537, 1700])
def test_pieces(n):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    # rows over twelve orders of magnitude: the vector's blocks differ in scale
    d = 10.0 ** (-12 * np.arange(n) / n)
    _check(d[:, None] * (A + A.conj().T) * d[None, :], 32)
