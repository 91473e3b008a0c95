"""The eigensolver's reciprocal, quotient and reflector scalars, formed from the
hardware's approximate reciprocal and reciprocal square root, against CUDA's rounded
operations and exact arithmetic.  The bounds are derived, not measured: see the
comments at each."""
from decimal import Decimal, getcontext

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 1 << 20
U = 2.0 ** -53


def _values(rng, n, lo, hi):
    """Mantissas dense in [1, 2), at its ends and at the 20th bit, where the
    hardware's approximations stop looking; exponents lo..hi; both signs."""
    m = 1.0 + rng.random(n)
    edge = rng.integers(0, 8, n)
    k = rng.integers(0, 1 << 20, n) * 2.0 ** -20
    m = np.where(edge == 0, 1.0, m)
    m = np.where(edge == 1, 1.0 + 2.0 ** -52 * rng.integers(0, 4, n), m)
    m = np.where(edge == 2, 2.0 - 2.0 ** -52 * rng.integers(1, 4, n), m)
    m = np.where(edge == 3, 1.0 + k, m)
    m = np.where(edge == 4, np.minimum(1.0 + k + (2.0 ** -20 - 2.0 ** -52), 2.0 - 2.0 ** -52), m)
    return np.ldexp(m * rng.choice([-1.0, 1.0], n), rng.integers(lo, hi + 1, n))


def _ulps(got, ref):
    return (got.view(torch.int64) - ref.view(torch.int64)).abs().max().item()


def test_reciprocal_within_an_ulp_of_the_rounded_one():
    # |e| < 2^-18 of the instruction: e^3 < 2^-54, half an ulp at most, and half an
    # ulp of the last rounding
    import paper_2406_10765_gb300 as pw
    x = _values(np.random.default_rng(0), N, -1021, 1020)
    a = torch.from_numpy(x).cuda()
    assert _ulps(pw.pw_selftest_fp64_ops(0, a), 1.0 / a) <= 1


def test_quotient_within_an_ulp_of_the_rounded_one():
    # the first quotient is within a few ulps and its remainder off by 2^-53 of itself
    # at most, so the corrected one is off by little more than its rounding
    import paper_2406_10765_gb300 as pw
    rng = np.random.default_rng(1)
    a = torch.from_numpy(_values(rng, N, -500, 500)).cuda()
    x = torch.from_numpy(_values(rng, N, -500, 500)).cuda()
    assert _ulps(pw.pw_selftest_fp64_ops(1, a, x), a / x) <= 1


def _reflector(xn2, ax, ay):
    """beta, tau, s of reflector_scalars in 60 digits."""
    xn2, ax, ay = Decimal(xn2), Decimal(ax), Decimal(ay)
    b = (ax * ax + ay * ay + xn2).sqrt()
    if ax >= 0 and not ax.is_signed():
        b = -b
    dx = ax - b
    dd = dx * dx + ay * ay
    return b, (b - ax) / b, -ay / b, dx / dd, -ay / dd


def _reflector_cases():
    rng = np.random.default_rng(2)
    n = 6000
    ax, ay, x = (_values(rng, n, -40, 40) for _ in range(3))
    e = rng.integers(-460, 461, n)
    # around both ends of the range of the fast form, sums of squares of 1e+-280
    e[:1500] = rng.choice([-466, -465, -464, -463, 463, 464, 465, 466], 1500)
    ax[:1500], ay[:1500], x[:1500] = (_values(rng, 1500, -2, 2) for _ in range(3))
    kind = rng.integers(0, 8, n)
    ax = np.where(kind == 0, 0.0, np.where(kind == 1, -0.0, ax))
    ay = np.where(kind == 2, 0.0, ay)
    x = np.where(kind == 3, 0.0, x)
    ax, ay, x = np.ldexp(ax, e), np.ldexp(ay, e), np.ldexp(x, e)
    keep = ~((ay == 0) & (x == 0))
    return (x * x)[keep], ax[keep], ay[keep]


def test_reflector_scalars_against_exact_arithmetic():
    # roundings, in units of 2^-53: the sum of squares 2 and its root's half of that,
    # 1/sqrt 2.7 with its own, beta 2.1; alpha - beta 3.1 (no cancellation); tau 6.7;
    # |alpha - beta|^2 7.2, its inverse 8.3, s 12.3.  The rounded form outside the
    # range: beta 2.5, tau 7, s 14.5.
    import paper_2406_10765_gb300 as pw
    getcontext().prec = 60
    xn2, ax, ay = _reflector_cases()
    got = pw.pw_selftest_fp64_ops(2, *(torch.from_numpy(v).cuda() for v in (xn2, ax, ay))).cpu().numpy()
    worst = np.zeros(5)
    for i in range(xn2.size):
        for k, r in enumerate(_reflector(*(float(v[i]) for v in (xn2, ax, ay)))):
            g = Decimal(float(got[k, i]))
            if abs(r) < Decimal(2) ** -1022:      # below the normal numbers
                assert abs(g - r) <= Decimal(2) ** -1022
            else:
                worst[k] = max(worst[k], float(abs(g - r) / abs(r)) / U)
    assert np.all(worst <= [4, 8, 8, 16, 16]), worst


def test_reflector_of_a_finished_column():
    import paper_2406_10765_gb300 as pw
    ax = torch.tensor([0.0, -0.0, 3.0, -3.0], dtype=torch.float64, device="cuda")
    z = torch.zeros_like(ax)
    got = pw.pw_selftest_fp64_ops(2, z, ax, z).cpu().numpy()
    assert np.array_equal(got[0], ax.cpu().numpy()) and not got[1:].any()


def test_argument_errors():
    import paper_2406_10765_gb300 as pw
    a = torch.ones(4, dtype=torch.float64, device="cuda")
    for bad in [(3, a), (-1, a), (1, a), (2, a, a)]:
        with pytest.raises(pw.PwError):
            pw.pw_selftest_fp64_ops(*bad)
