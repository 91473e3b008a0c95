"""FP64-accurate tensor-core product at the edges of its inner-dimension
handling: K around the 16-wide MMA steps, the half chunks (48 real K) after
which each half of the digit groups is emptied, and the whole chunks (96), in
one part and split over several, with rows and columns around the tile."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")


def test_chunk_bound():
    """Two pairs |d_1 d_8| <= 2^13 and six |d_p d_q| <= 2^12 per real K over a chunk
    of 96 stay below 2^22, the range of the accumulator-to-integer conversion."""
    per_k = max(sum((2 ** 7 if p == 1 else 2 ** 6) * (2 ** 7 if g - p == 1 else 2 ** 6)
                    for p in range(max(1, g - 8), min(8, g - 1) + 1)) for g in range(2, 10))
    assert per_k * 96 < 2 ** 22


@pytest.mark.gpu
@pytest.mark.parametrize("k", [1, 7, 8, 9, 15, 16, 17, 23, 24, 25, 47, 48, 49, 71, 72, 73, 96, 97, 143, 145, 1000])
@pytest.mark.parametrize("m,n", [(128, 32), (33, 65), (130, 3)])
def test_integer_products_exact(m, n, k):
    """Integers of up to 18 bits (three digits, every digit sign): the product is exact."""
    import paper_2406_10765_gb300 as pw
    from gpu_util import to_dev
    rng = np.random.default_rng(1000 * k + m + n)
    top = 2 ** 18 - 1
    A = rng.integers(-top, top + 1, (m, k)) + 1j * rng.integers(-top, top + 1, (m, k))
    B = rng.integers(-top, top + 1, (k, n)) + 1j * rng.integers(-top, top + 1, (k, n))
    A[0], B[:, 0] = top - 1j * top, -top + 1j * top            # the largest digits, one sign
    got = pw.pw_zgemm_f64tc("N", "N", to_dev(A), to_dev(B)).cpu().numpy()
    # |Re|, |Im| <= 2 k 2^36 < 2^53: the reference is exact in FP64 too
    assert np.array_equal(got, A @ B)
