"""Eigenproblems with NaN or infinite entries: the divide and conquer's indices stay
indices.  A merge of two sorted halves places each value by its rank in the other
half; with doubles compared as doubles NaNs collide and leave places unwritten, with
their order-preserving integers the places are a permutation."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")


def _ordered_bits(x):
    b = np.asarray(x, dtype=np.float64).view(np.int64)
    return np.where(b < 0, np.int64(-2 ** 63) - b, b)


def _places(left, right):
    """Binary searches as k_dc_deflate runs them."""
    def search(half, go_right):
        l, r = 0, len(half)
        while l < r:
            m = (l + r) >> 1
            if go_right(half[m]):
                l = m + 1
            else:
                r = m
        return l
    return ([p + search(right, lambda w, v=v: w < v) for p, v in enumerate(left)]
            + [q + search(left, lambda w, v=v: w <= v) for q, v in enumerate(right)])


def test_places_of_a_merge_are_a_permutation():
    rng = np.random.default_rng(0)
    pool = np.array([np.nan, -np.nan, np.inf, -np.inf, 0.0, -0.0, 1.0, 1.0, -2.5, 5e-324])
    lost = 0
    for _ in range(500):
        n, m = rng.integers(1, 9, 2)
        left, right = (np.sort(_ordered_bits(rng.choice(pool, k))) for k in (n, m))
        assert sorted(_places(left, right)) == list(range(n + m))
        vals = [np.where(h < 0, np.int64(-2 ** 63) - h, h).view(np.float64) for h in (left, right)]
        lost += sorted(_places(*vals)) != list(range(n + m))
    assert lost > 0                        # doubles compared as doubles do lose places


@pytest.mark.gpu
@pytest.mark.parametrize("n", [2, 3, 54, 300, 1100])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("whole", [False, True])
def test_nonfinite_matrices_leave_the_library_usable(n, bad, whole):
    import paper_2406_10765_gb300 as pw
    rng = np.random.default_rng(n)
    G = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    G = G + G.conj().T
    ref = np.linalg.eigvalsh(G)
    B = np.full((n, n), bad, dtype=complex) if whole else G.copy()
    B[n - 1, 0] = B[0, n - 1] = bad
    good, broken = torch.from_numpy(G).cuda(), torch.from_numpy(B).cuda()
    for heev in (pw.pw_heev, pw.pw_heev_fixed):
        for _ in range(2):                 # a workspace that an earlier call has written
            w, _y = heev(good, 1 + n // 3)
            assert np.abs(w.cpu().numpy() - ref).max() < 1e-13 * np.abs(ref).max() * n ** 0.5
            w, _y = heev(broken, 1 + n // 3)
            assert not torch.isfinite(w).all()
