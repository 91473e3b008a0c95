"""The FP64 products on 8 x 8 and 64 x 64 tiles through their callers, at sizes
around the tiles, the 32-wide K slab and the rule that picks between them: H
psi without allocation (both products, K split, ragged bands) against the
oracle, and the eigensolver with every product on the FP64 pipe (herm and
triangular modes, batched inverse pairs) against LAPACK."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [1, 7, 8, 9, 31, 33, 64, 65, 100])
def test_projector_products(nb):
    import paper_2406_10765_gb300 as pw
    import synth
    from gpu_util import to_dev
    from oracle import pw_oracle as o
    ci = synth.cell_inputs("C", 1, 3)
    oc = o.make_cell(ci["L"], ci["tau"], ci["depth"], ci["dkb"], 8.0)
    cell = pw.Cell(ci["L"], ci["tau"], ci["depth"], ci["dkb"], 8.0)
    x = synth.draw_x0(nb, 8, cell.npw, nb)
    out = pw.new_block(cell.npw, nb)
    pw.pw_apply_H_noalloc(cell.h, to_dev(x), out)
    ref = o.apply_H(oc, x)
    # the stated FP64 tolerance of H psi
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [7, 8, 9, 31, 32, 33, 63, 64, 65, 95, 127, 129, 160, 193])
def test_solve_fp64_pipe(n):
    import paper_2406_10765_gb300 as pw
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    A = A + A.conj().T
    pw.pw_dense_products(0)
    try:
        w, y = pw.pw_heev(torch.from_numpy(A).cuda(), n)
    finally:
        pw.pw_dense_products(1)
    w, y = w.cpu().numpy(), y.cpu().numpy()
    ref = np.linalg.eigvalsh(A)
    scale = np.abs(ref).max()
    # as tests/test_gpu_dense.py
    assert np.abs(w - ref).max() < 1e-13 * scale * n ** 0.5
    assert np.abs(A @ y - y * w).max() < 1e-12 * scale
    assert np.abs(y.conj().T @ y - np.eye(n)).max() < 1e-12
