"""complex64 factorisations of matrices whose rows differ in scale, at sizes with one to four trailing
updates of 256 columns: |B - Z X| <= c (|Z| |X| + |B|) per entry.  Row scalings do not change the
bound of partial pivoting without growth, c = 3 n u with u = 2^-24 for a solve without refinement;
refinement (the first solve and at least two corrections) gains three digits per step at least."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [257, 300, 384, 513, 640, 1000]


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_01457_gb300 as mod

    mod.build.build()
    return mod


def _system(n, rows, columns):
    rng = np.random.default_rng(n + rows)
    draw = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    Z = draw(n, n) * (10.0 ** rng.uniform(-rows, rows, n))[:, None] * 10.0 ** rng.uniform(-columns, columns, n)
    Z = Z.astype(np.complex64).astype(np.complex128)
    return Z, (Z @ draw(n, 6)).astype(np.complex64).astype(np.complex128)


def _componentwise(Z, X, B):
    l1 = lambda t: np.abs(t.real) + np.abs(t.imag)
    return (l1(B - Z @ X) / (l1(Z) @ l1(X) + l1(B))).max()


@pytest.mark.parametrize("rows,columns", [(3, 0), (6, 0), (8, 0), (8, 6)])
@pytest.mark.parametrize("n", SIZES)
def test_without_refinement(F, n, rows, columns):
    Z, B = _system(n, rows, columns)
    X = torch.empty((n, 6), dtype=torch.complex64, device="cuda")
    F.solve(F.factor(torch.tensor(Z, device="cuda").to(torch.complex64)), torch.tensor(B, device="cuda").to(torch.complex64), X)
    assert _componentwise(Z, X.cpu().numpy().astype(np.complex128), B) <= 3 * n * 2.0**-24


@pytest.mark.parametrize("rows", [3, 6, 8])
@pytest.mark.parametrize("n", SIZES)
def test_refined(F, n, rows):
    Z, B = _system(n, rows, 0)
    Zd = torch.tensor(Z, device="cuda")
    lu = F.factor(Zd, prec=F.MIXED)
    for r in (2, 6):
        X = torch.empty((n, r), dtype=torch.complex128, device="cuda")
        _, steps, _ = F.solve(lu, torch.tensor(B[:, :r].copy(), device="cuda"), X)
        assert steps <= 4
        assert _componentwise(Z, X.cpu().numpy(), B[:, :r]) <= 3 * n * 2.0**-24 * 1e-6
