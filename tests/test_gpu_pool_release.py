"""Device memory that the library keeps after a call: at most the pool's bound as
soon as the call has returned, nothing once it is asked for or a serving run has
started."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KEEP = 2 << 30               # pool.cu
SLACK = 256 << 20            # modules loaded meanwhile, the driver's own blocks


def _held():
    """Device memory in use besides torch's."""
    free, total = torch.cuda.mem_get_info()
    return total - free - torch.cuda.memory_reserved()


def _tc():
    # split operands 8 (2 m + n) k bytes: 9.8 GB
    import paper_2406_10765_gb300 as pw
    A = torch.randn(1024, 400000, dtype=torch.complex128, device="cuda").T
    C = torch.zeros(1024, 1024, dtype=torch.complex128, device="cuda").T
    return lambda: pw.pw_zgemm_tc("C", A, A, C)


def _heev():
    # 88 n^2 bytes of matrices and 0.6 GB of slices: 3.8 GB at least
    import paper_2406_10765_gb300 as pw
    A = torch.diag(torch.arange(6000, dtype=torch.float64, device="cuda")).to(torch.complex128)
    A[0, 1] = A[1, 0] = 1.0
    return lambda: pw.pw_heev(A, 8)


@pytest.mark.parametrize("make", [_tc, _heev])
def test_bounded_on_return(make):
    call = make()
    torch.cuda.synchronize()
    before = _held()
    for _ in range(2):
        call()
        assert _held() - before <= KEEP + SLACK


@pytest.mark.parametrize("budget", [0, 64 << 30])
def test_serving_run_starts_with_an_empty_pool(budget):
    import paper_2406_10765_gb300 as pw
    req = dict(synth.serving_requests(1, rate_per_s=20.0, seed=77)[0], n=1, nbands=18, t_arrival=0.0)
    pw.pw_serve([req], max_slots=1)
    call = _tc()
    before = _held()
    call()
    assert _held() - before > KEEP // 2
    assert pw.pw_serve([req], max_slots=1, hbm_budget=budget)[0]["status"] == 0
    assert _held() - before <= SLACK


@pytest.mark.parametrize("make", [_tc, _heev])
def test_release_memory(make):
    import paper_2406_10765_gb300 as pw
    call = make()
    call()
    pw.pw_release_memory()
    before = _held()
    call()
    assert _held() - before > KEEP // 2
    pw.pw_release_memory()
    assert _held() - before <= SLACK
    call()                                       # and takes new memory
