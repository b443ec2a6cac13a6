"""Products of stored factors whose columns are graded against each other (column k of Y1 by s_k, of Y2 by
1/s_k): |out - Y1 op(Y2)| <= r 2^-48 |Y1| |Y2| per entry, the bound of float-float products, which such
a grading does not change.  Both sides of the 128 columns at which the digits take over."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_01457_gb300 as mod

    mod.build.build()
    return mod


@pytest.mark.parametrize("pseudo", [False, True])
@pytest.mark.parametrize("binades", [4, 16, 60, 250])
@pytest.mark.parametrize("n,r", [(9, 128), (12, 127), (30, 129), (130, 300), (600, 161)])
def test_factors_graded_against_each_other(F, n, r, binades, pseudo):
    rng = np.random.default_rng(n + r + binades)
    binades = binades if r >= 128 else min(binades, 60)  # (float-float has the range of FP32)
    s = 2.0 ** rng.integers(-binades, binades + 1, r)
    draw = lambda *q: rng.integers(-(2**19), 2**19, q) + 1j * rng.integers(-(2**19), 2**19, q)
    P, Q = draw(n, r), draw(n, r)
    P[1], Q[:, 3], Q[2, 5:] = 0, 0, 0  # a zero row, a zero k and a row with few entries
    out = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
    F.lowrank_combine(torch.tensor(P * s, device="cuda"), torch.tensor(Q / s, device="cuda"), out, pseudo=pseudo, prec=F.MIXED)
    ref = P @ (Q.T if pseudo else Q.conj().T)  # integers, exact in FP64
    assert (np.abs(out.cpu().numpy() - ref) <= r * 2.0**-48 * (np.abs(P) @ np.abs(Q).T)).all()


def test_infinities_and_nan_stay_in_their_rows_and_columns(F):
    rng = np.random.default_rng(4)
    n, r = 140, 200
    draw = lambda: rng.standard_normal((n, r)) + 1j * rng.standard_normal((n, r))
    P, Q, s = draw(), draw(), 10.0 ** rng.uniform(-6, 6, r)
    ref = P @ Q.T
    P, Q = P * s, Q / s
    P[3, 7], P[130, 0], Q[65, 5] = np.inf, complex(0, np.nan), -np.inf
    out = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
    F.lowrank_combine(torch.tensor(P, device="cuda"), torch.tensor(Q, device="cuda"), out, pseudo=True, prec=F.MIXED)
    C = out.cpu().numpy()
    bad = np.zeros((n, n), dtype=bool)
    bad[[3, 130], :] = bad[:, 65] = True
    assert np.isnan(C[bad].real).all() and np.isnan(C[bad].imag).all()
    assert (np.abs(C - ref)[~bad] <= 1e-12 * np.abs(ref).max()).all()


def test_gradient_of_many_directions_is_the_sum_of_its_parts(F):
    """The transposed product A^T C has 3 n_inc values of k: 144 in digits, 72 in float-float."""
    import fosb_synth as S

    sm = S.icosphere(1)
    m = F.mesh_create(sm.verts, sm.tris, sm.vnormals)
    rng = np.random.default_rng(7)
    d = rng.standard_normal((48, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    p = np.cross(d, rng.standard_normal((48, 3)))
    p /= np.linalg.norm(p, axis=1, keepdims=True)
    inc = F.incidence(d, p)
    Z = torch.empty((m.n_edges,) * 2, dtype=torch.complex128, device="cuda")
    b = torch.empty((m.n_edges, 48), dtype=torch.complex128, device="cuda")
    F.assemble_efie(m, 2.0, Z, inc=inc, b=b)
    lu = F.factor(Z, prec=F.MIXED)
    F.solve(lu, b)
    w = rng.uniform(0.5, 1.5, 48)

    def grad(q):
        g = torch.empty((sm.verts.shape[0], 3), dtype=torch.float64, device="cuda")
        F.rcs_monostatic(m, 2.0, inc[q], b[:, q].contiguous(), lu=lu, weights=w[q], grad=g)
        return g.cpu().numpy()

    whole, parts = grad(slice(0, 48)), grad(slice(0, 24)) + grad(slice(24, 48))
    # each solve's relative residual is below 1e-13 and the system's condition below 1e3
    assert np.abs(whole - parts).max() <= 1e-10 * np.abs(whole).max()
