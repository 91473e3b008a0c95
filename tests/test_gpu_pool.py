"""The library's memory pool for transient workspaces: calls on several streams
and threads share it without touching each other's data, sizes that outgrow it
work, and a repeated call keeps no more than the bound."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_concurrent_streams_share_the_pool():
    import paper_2406_10765_gb300 as pw

    def work(seed):
        rng = np.random.default_rng(seed)
        m, n, k = (int(v) for v in rng.integers(20, 300, 3))
        A = torch.from_numpy(rng.standard_normal((k, m)) + 1j * rng.standard_normal((k, m))).cuda().T
        B = torch.from_numpy(rng.standard_normal((n, k)) + 1j * rng.standard_normal((n, k))).cuda().T
        H = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
        H = torch.from_numpy(H + H.conj().T).cuda()
        torch.cuda.synchronize()
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            c = pw.pw_zgemm_f64tc("N", "N", A, B, stream=st.cuda_stream)
            t = pw.pw_zgemm_tc("N", A, B, stream=st.cuda_stream)
            w, _ = pw.pw_heev(H, 1, stream=st.cuda_stream)
        st.synchronize()
        ref = A @ B
        scale = ref.abs().max().item()
        return ((c - ref).abs().max().item() / scale, (t - ref).abs().max().item() / scale,
                np.abs(w.cpu().numpy() - np.linalg.eigvalsh(H.cpu().numpy())).max() / (2 * m) ** 0.5)

    with ThreadPoolExecutor(6) as ex:
        got = np.array(list(ex.map(work, range(24))))
    # the products' stated accuracies, 11 K 2^-55 max max and ~1e-6, and the
    # eigenvalue tolerance of tests/test_gpu_dense.py
    assert got[:, 0].max() < 1e-13 and got[:, 1].max() < 1e-5 and got[:, 2].max() < 1e-12


def test_bounded_between_calls():
    import paper_2406_10765_gb300 as pw
    A = torch.randn(1500, 60000, dtype=torch.complex128, device="cuda").T
    pw.pw_zgemm_tc("C", A[:, :8], A[:, :8])          # modules loaded, pool created
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        pw.pw_zgemm_tc("C", A, A)                    # ~3 GB of split operands
    pw.pw_zgemm_tc("C", A[:, :8], A[:, :8])
    torch.cuda.synchronize()
    C = 1500 * 1500 * 16
    assert free0 - torch.cuda.mem_get_info()[0] <= (2 << 30) + 16 * C + (256 << 20)
