"""The work that programs have this library do, as measurable cases.

Each case goes through the public entry points of paper_2406_10765_gb300, on
the sizes of the repository's workloads: Si and C diamond supercells of 8 to
512 atoms, cutoffs of 8 to 12 Ha, 1.125 bands per occupied one, and the dense
problems that a block eigensolver step of those cells poses.
"""
import math

import numpy as np
import torch

import paper_2406_10765_gb300 as pw

LATTICE = {"Si": 10.26, "C": 6.74}          # bohr
WIDTH = 1.2                                 # bohr: Gaussian wells and projectors
BASIS = np.array([[0, 0, 0], [0, 2, 2], [2, 0, 2], [2, 2, 0],
                  [1, 1, 1], [1, 3, 3], [3, 1, 3], [3, 3, 1]]) / 4.0


def listed():
    def cell(kind, name, species, n, ecut, nb, precision, **more):
        return dict(name=name, kind=kind, species=species, n=n, ecut=ecut, nb=nb, precision=precision, **more)

    return [
        # H psi, the call that every iterative solver makes most often.  The smallest served
        # request (8 C atoms, 18 bands): a handful of short launches.
        cell("apply", "apply_c8_mixed", "C", 1, 8.0, 18, "mixed", onthefly=False),
        # A 64-atom cell in plain FP64, all bands at once.
        cell("apply", "apply_si64_fp64", "Si", 2, 9.3, 144, "fp64", onthefly=False),
        # The largest served request in mixed precision, with an odd number of active bands
        # (converged bands leave the block).
        cell("apply", "apply_si216_mixed", "Si", 3, 11.3, 457, "mixed", onthefly=False),
        # The benchmark's cell: 512 atoms, 1,152 bands.
        cell("apply", "apply_si512_mixed", "Si", 4, 10.0, 1152, "mixed", onthefly=False),
        # S^H S of the 216-atom cell's basis [X W P] in split FP16 (mixed precision).
        dict(name="gram_si216", kind="zgemm_tc", op="C", m=1458, n=1458, k=43819),
        # The eigenvector product M Y of the 512-atom Rayleigh-Ritz, FP64-accurate.
        dict(name="f64tc_si512", kind="zgemm_f64tc", op="NN", m=3456, n=1152, k=3456),
        # The dense eigenproblem of a Rayleigh-Ritz step, order 3 x bands: 8, 216 and 512 atoms.
        dict(name="heev_54", kind="heev", n=54, nb=18),
        dict(name="heev_1458", kind="heev", n=1458, nb=486),
        dict(name="heev_3456", kind="heev", n=3456, nb=1152),
        # A short solve from a given block and the density of its bands, as one iteration of a
        # self-consistent loop makes them, on the 8-atom cell: latency and launches.
        cell("solve", "solve_si8_fp64", "Si", 1, 10.0, 24, "fp64", steps=8),
        # One LOBPCG step, FP64, of the 216-atom cell.
        cell("step", "step_si216_fp64", "Si", 3, 10.0, 486, "fp64"),
        # One LOBPCG step, mixed precision, of the 512-atom cell: the benchmark's unit of work.
        cell("step", "step_si512_mixed", "Si", 4, 10.0, 1152, "mixed"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["apply", "apply", "apply", "zgemm_tc", "zgemm_f64tc", "heev", "heev", "solve", "step"])
    if kind == "zgemm_tc":
        if rng.random() < 0.5:      # Gram-type: basis columns against each other over the plane waves
            return dict(kind=kind, op="C", m=log_int(18, 3456), n=log_int(18, 1458), k=log_int(341, 60000))
        return dict(kind=kind, op="N", m=log_int(341, 60000), n=log_int(18, 1458), k=log_int(18, 3456))
    if kind == "zgemm_f64tc":
        return dict(kind=kind, op=rng.choice(["NN", "CN", "NC"]), m=log_int(54, 3456), n=log_int(18, 3456),
                    k=log_int(54, 3456))
    if kind == "heev":
        n = log_int(40, 3456)
        return dict(kind=kind, n=n, nb=max(1, round(n * rng.uniform(0.3, 0.5))))
    species = rng.choice(["Si", "C"])
    n = {"apply": rng.choice([1, 2, 2, 3, 3, 4]), "solve": rng.choice([1, 1, 2]), "step": 3}[kind]
    ecut = round(rng.uniform(8.0, 12.0 if n < 4 else 10.0), 3)
    nb = 18 * n ** 3                # 1.125 bands per occupied one; fewer once some have converged
    if species == "Si" and kind == "apply":
        nb = max(1, log_int(nb // 12, nb))
    elif kind != "apply":
        nb -= rng.randrange(0, 4 * n)
    precision = rng.choice(["fp64", "mixed"]) if kind != "solve" and n < 4 else "mixed" if n == 4 else "fp64"
    more = dict(onthefly=rng.random() < 0.15) if kind == "apply" else dict(steps=rng.randint(3, 8)) if kind == "solve" else {}
    return dict(kind=kind, species=species, n=n, ecut=ecut, nb=nb, precision=precision, **more)


# --------------------------------------------------------------- inputs

def _cell_inputs(case, seed):
    """Positions, well depths and projector coefficients of a diamond supercell."""
    n, a = case["n"], LATTICE[case["species"]]
    corner = np.array([(i, j, k) for i in range(n) for j in range(n) for k in range(n)], float)
    tau = (corner[:, None, :] + BASIS[None]).reshape(-1, 3) * a
    r = np.random.default_rng(seed)
    return dict(L=n * a, tau=tau, depth=-1.0 + 0.1 * r.uniform(-1, 1, len(tau)),
                dkb=r.uniform(0.5, 1.5, (len(tau), 4)))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _randn(rows, cols, seed):
    """Column-major complex Gaussian matrix."""
    return torch.randn(cols, rows, dtype=torch.complex128, device="cuda", generator=_gen(seed)).T


def _kinetic(m, L):
    g = torch.as_tensor(m, device="cuda").double() * (2 * math.pi / L)
    return 0.5 * (g * g).sum(1)


def _block(kin, nb, seed):
    """Unit columns whose coefficients fall off with the kinetic energy, as wavefunctions' do."""
    x = _randn(len(kin), nb, seed).T.mul_(1.0 / (1.0 + kin * kin))
    return x.div_(torch.linalg.vector_norm(x, dim=1, keepdim=True)).T


def _start(npw, nb, seed):
    """Uniform random start block of a solve, not normalised."""
    x = torch.rand(nb, npw, 2, dtype=torch.float64, device="cuda", generator=_gen(seed)) - 0.5
    return torch.view_as_complex(x).T


def _hermitian(n, seed):
    """A Rayleigh-Ritz matrix: the energies of the basis on the diagonal (the bands' low ones first,
    kinetic ones up to twice the cutoff after them), coupled by small Hermitian entries."""
    a = _randn(n, n, seed) / math.sqrt(n)
    a = 0.5 * (a + a.mH)
    d = torch.sort(torch.rand(n, dtype=torch.float64, device="cuda", generator=_gen(seed + 1)) * 21.0 - 1.0)[0]
    a.diagonal().add_(d)
    return a.T.contiguous().T


class _Solver:
    """A cell and a solver on it, given back together."""

    def __init__(self, cell, case, x0):
        self.cell, self.nb = cell, case["nb"]
        self.h = pw.pw_solver_create(cell.h, case["nb"], tol=0.0, x0=x0, precision=case["precision"])

    def __del__(self):
        if getattr(self, "h", None):
            pw.pw_solver_destroy(self.h)


def _cell(case, seed):
    c = _cell_inputs(case, seed)
    return pw.Cell(c["L"], c["tau"], c["depth"], c["dkb"], case["ecut"], vwidth=WIDTH, pwidth=WIDTH,
                   precision=case["precision"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "zgemm_tc":
        rows = case["k"] if case["op"] == "C" else case["m"]
        cols = case["m"] if case["op"] == "C" else case["k"]
        return dict(case=case, A=_randn(rows, cols, seed).div_(math.sqrt(rows)), B=_randn(case["k"], case["n"], seed + 1),
                    C=pw.new_block(case["m"], case["n"]))
    if kind == "zgemm_f64tc":
        a, b = ((p, q) if o == "N" else (q, p) for o, p, q in
                zip(case["op"], (case["m"], case["k"]), (case["k"], case["n"])))
        return dict(case=case, A=_randn(*a, seed), B=_randn(*b, seed + 1), C=pw.new_block(case["m"], case["n"]))
    if kind == "heev":
        return dict(case=case, A=_hermitian(case["n"], seed))
    cell = _cell(case, seed)
    if kind == "apply":
        if case["onthefly"]:
            pw.pw_cell_set_projectors(cell.h, True)
        psi = _block(_kinetic(cell.m, case["n"] * LATTICE[case["species"]]), case["nb"], seed)
        return dict(case=case, cell=cell, psi=psi, out=pw.new_block(cell.npw, case["nb"]))
    x0 = _start(cell.npw, case["nb"], seed)
    if kind == "solve":
        return dict(case=case, cell=cell, x0=x0, psi=pw.new_block(cell.npw, case["nb"]))
    return dict(case=case, solver=_Solver(cell, case, x0),
                block=pw.new_block(cell.npw, case["nb"]) if case["precision"] == "fp64" else None)


def _phased(y):
    """Eigenvector columns with their arbitrary phase fixed: the largest entry is made positive."""
    p = y.gather(0, y.abs().argmax(0, keepdim=True))
    return y * (p.conj() / p.abs())


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "apply":
        return state["cell"].apply_H(state["psi"], state["out"])
    if kind == "zgemm_tc":
        return pw.pw_zgemm_tc(case["op"], state["A"], state["B"], C=state["C"])
    if kind == "zgemm_f64tc":
        return pw.pw_zgemm_f64tc(case["op"][0], case["op"][1], state["A"], state["B"], C=state["C"])
    if kind == "heev":
        w, y = pw.pw_heev(state["A"], case["nb"])
        return dict(w=w, y=_phased(y))
    if kind == "solve":
        eig, _, _ = pw.pw_eigsolve(state["cell"].h, case["nb"], tol=0.0, maxit=case["steps"], x0=state["x0"],
                                   precision=case["precision"], psi_out=state["psi"], raise_noconv=False)
        return dict(eig=eig, psi=_phased(state["psi"]), rho=pw.pw_density(state["cell"].h, state["psi"]))
    s = state["solver"]
    pw.pw_subspace_step(s.cell.h, s.h)
    eig, resid = pw.pw_solver_eigs(s.h, s.nb)
    out = dict(eig=eig, resid=resid)
    if state["block"] is not None:
        # The new block.  In mixed precision it stays in the solver: a step's single-precision
        # rounding moves its columns within clusters of bands, and a program reads it once, at the end.
        pw.pw_solver_block(s.h, state["block"])
        out["block"] = _phased(state["block"])
    return out


# --------------------------------------------------------------- least work

def _sizes(case):
    """Plane waves (the sphere's volume) and grid points per axis of a cell."""
    L = case["n"] * LATTICE[case["species"]]
    npw = L ** 3 * (2 * case["ecut"]) ** 1.5 / (6 * math.pi ** 2)
    return npw, _grid(case["ecut"], L)


def _grid(ecut, L):
    least = 1.5 * math.sqrt(2 * ecut) * L / math.pi
    return min(2 ** a * 3 ** b for a in range(12) for b in range(8) if 2 ** a * 3 ** b >= least)


def _apply_work(case, nb):
    npw, N = _sizes(case)
    nproj = 32 * case["n"] ** 3
    beta = 0 if case.get("onthefly") else 16 * npw * nproj
    return 32 * npw * nb + 8 * N ** 3 + beta, nb * (10 * N ** 3 * math.log2(N ** 3) + 16 * npw * nproj)


def _heev_work(n, nb):
    return 16 * n * n + 8 * n + 16 * n * nb, 8 * (4 / 3 * n ** 3 + n * n * nb) + 4 / 3 * n ** 3


def _step_work(case):
    """Residual and W from X and H X; H W; the Gram pair of [X W P]; the dense problem; X', P' and
    their H blocks.  The blocks X, P, H X, H P are read and written once."""
    npw, _ = _sizes(case)
    nb = case["nb"]
    hb, hf = _apply_work(case, nb)
    db, df = _heev_work(3 * nb, nb)
    return 8 * 16 * npw * nb + hb + db, hf + 8 * npw * nb * nb * (9 + 10) + df + 8 * 27 * nb ** 3


def work(case):
    kind = case["kind"]
    if kind.startswith("zgemm"):
        m, n, k = case["m"], case["n"], case["k"]
        b, f = 16 * (m * k + k * n + m * n), 8 * m * n * k
    elif kind == "heev":
        b, f = _heev_work(case["n"], case["nb"])
    elif kind == "apply":
        b, f = _apply_work(case, case["nb"])
    elif kind == "step":
        b, f = _step_work(case)
    else:
        npw, N = _sizes(case)
        b, f = (case["steps"] * v for v in _step_work(case))
        b, f = b + 16 * npw * case["nb"] + 8 * N ** 3, f + case["nb"] * 5 * N ** 3 * math.log2(N ** 3)
    return dict(bytes=float(b), flops=float(f))


# --------------------------------------------------------------- 64-bit values

class _Exact:
    """The plane-wave Hamiltonian of a case, written out with torch in complex128."""

    def __init__(self, case, seed):
        c = _cell_inputs(case, seed)
        L, N = c["L"], _grid(case["ecut"], c["L"])
        top = int(math.sqrt(2 * case["ecut"]) * L / (2 * math.pi)) + 1
        axis = torch.arange(-top, top + 1, device="cuda")
        m = torch.cartesian_prod(axis, axis, axis)
        m = m[_kinetic(m, L) <= case["ecut"]]
        self.m, self.N, self.kin = m, N, _kinetic(m, L)
        self.at = ((m[:, 0] % N) * N + m[:, 1] % N) * N + m[:, 2] % N
        tau = torch.as_tensor(c["tau"], device="cuda")
        r = torch.arange(N, device="cuda").double() * (L / N)
        image = torch.arange(-3, 4, device="cuda").double() * L
        d = r[None, None, :, None] - tau[:, :, None, None] - image
        well = torch.exp(-d * d / (2 * WIDTH ** 2)).sum(3)                  # atom, axis, point
        self.V = torch.einsum("ai,aj,ak->ijk", well[:, 0] * torch.as_tensor(c["depth"], device="cuda")[:, None],
                              well[:, 1], well[:, 2])
        g = m.double() * (2 * math.pi / L)
        radial = torch.exp(-self.kin * WIDTH ** 2) / math.sqrt(L ** 3)
        ph = g @ tau.T
        ph = torch.polar(radial[:, None].expand_as(ph).contiguous(), -ph)
        ns = math.sqrt(8 * math.pi ** 1.5 * WIDTH ** 3)
        np_ = math.sqrt(16 * math.pi ** 1.5 * WIDTH ** 5)
        self.beta = torch.stack([ns * ph] + [np_ * -1j * g[:, k:k + 1] * ph for k in range(3)], 2).flatten(1)
        self.D = torch.as_tensor(c["dkb"], device="cuda").reshape(-1, 1)

    def real_space(self, x):
        f = torch.zeros(x.shape[1], self.N ** 3, dtype=torch.complex128, device="cuda")
        f[:, self.at] = x.T
        return torch.fft.ifftn(f.view(-1, self.N, self.N, self.N), dim=(1, 2, 3), norm="forward")

    def apply(self, x):
        y = self.beta @ (self.D * (self.beta.mH @ x)) + self.kin[:, None] * x
        for j in range(0, x.shape[1], 32):
            f = torch.fft.fftn(self.real_space(x[:, j:j + 32]) * self.V, dim=(1, 2, 3), norm="forward")
            y[:, j:j + 32] += f.flatten(1)[:, self.at].T
        return y

    def density(self, x):
        rho = sum((self.real_space(x[:, j:j + 32]).abs() ** 2).sum(0) for j in range(0, x.shape[1], 32))
        return rho.permute(2, 1, 0).contiguous()

    def solve(self, x0, steps):
        """`steps` LOBPCG steps from the Ritz vectors of x0: eigenvalues, block and residual norms."""
        nb = x0.shape[1]

        def ritz(s, hs):
            g, a = s.mH @ s, s.mH @ hs
            d = g.diagonal().real.rsqrt()
            l = torch.linalg.cholesky(d[:, None] * g * d)
            t = torch.linalg.solve_triangular(l, d[:, None] * a * d, upper=False)
            t = torch.linalg.solve_triangular(l, t.mH, upper=False)
            w, y = torch.linalg.eigh(0.5 * (t + t.mH))
            return w[:nb], d[:, None] * torch.linalg.solve_triangular(l.mH, y[:, :nb].contiguous(), upper=True)

        hx = self.apply(x0)
        w, c = ritz(x0, hx)
        x, hx, p, hp = x0 @ c, hx @ c, None, None
        for _ in range(steps):
            ek = (self.kin[:, None] * x.abs() ** 2).sum(0) / (x.abs() ** 2).sum(0)
            q = self.kin[:, None] / ek
            poly = 27 + q * (18 + q * (12 + 8 * q))
            r = (hx - x * w) * (poly / (poly + 16 * q ** 4))
            s = torch.cat([x, r] + ([p] if p is not None else []), 1)
            hs = torch.cat([hx, self.apply(r)] + ([hp] if p is not None else []), 1)
            w, c = ritz(s, hs)
            p, hp = s[:, nb:] @ c[nb:], hs[:, nb:] @ c[nb:]
            x, hx = s @ c, hs @ c
        return w, x, torch.linalg.vector_norm(hx - x * w, dim=0)


def exact(case, seed):
    kind = case["kind"]
    if kind.startswith("zgemm"):
        s = prepare(case, seed)
        a, b = s["A"], s["B"]
        op = case["op"] if kind == "zgemm_f64tc" else case["op"] + "N"
        return (a.mH if op[0] == "C" else a) @ (b.mH if op[1] == "C" else b)
    if kind == "heev":
        w, y = torch.linalg.eigh(_hermitian(case["n"], seed))
        return dict(w=w, y=_phased(y[:, :case["nb"]]))
    if kind == "step" and case["precision"] == "mixed":
        return None         # a mixed step's values depend on single-precision rounding
    h = _Exact(case, seed)
    if kind == "apply":
        return h.apply(_block(h.kin, case["nb"], seed))
    w, x, r = h.solve(_start(len(h.kin), case["nb"], seed), case.get("steps", 1))
    if kind == "solve":
        return dict(eig=w, psi=_phased(x), rho=h.density(x))
    return dict(eig=w, resid=r, block=_phased(x))
