"""Factorisations of matrices with few entries in many of their columns, or banded, whose rows (and columns)
differ in scale, so that the columns of a block row of U see different parts of the rows' scales:
|B - Z X| <= c (|L| |U| |X| + |Z| |X| + |B|) per entry with the factors of the same pivoting rule on the CPU,
c = n 2^-52 for FP64 where the pivoting grows, 32 2^-52 where it does not (errors of rounding add up as
random signs), and 3 n 2^-24 for complex64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
scipy_linalg = pytest.importorskip("scipy.linalg")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_01457_gb300 as mod

    mod.build.build()
    return mod


def _l1(t):
    return np.abs(t.real) + np.abs(t.imag)


def _matrix(n, kind, columns):
    rng = np.random.default_rng(n)
    Z = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    Z = Z * (10.0 ** rng.uniform(-8, 8, n))[:, None] * 10.0 ** rng.uniform(-columns, columns, n)
    if kind == "band":
        return Z * (np.abs(np.arange(n)[:, None] - np.arange(n)) < 100)
    keep = rng.random((n, n)) < 10.0 / n  # half of the columns keep about ten entries and the diagonal
    keep[:, ::2] = True
    keep[np.arange(n), np.arange(n)] = True
    return Z * keep


def _errors(F, Z, dtype, prec):
    rng = np.random.default_rng(1)
    B = Z @ (rng.standard_normal((len(Z), 3)) + 1j * rng.standard_normal((len(Z), 3)))
    X = torch.empty(B.shape, dtype=dtype, device="cuda")
    F.solve(F.factor(torch.tensor(Z, device="cuda").to(dtype), prec=prec), torch.tensor(B, device="cuda").to(dtype), X)
    X = X.cpu().numpy().astype(np.complex128)
    PL, U = scipy_linalg.lu(Z, permute_l=True)
    return (_l1(B - Z @ X) / (_l1(PL) @ (_l1(U) @ _l1(X)) + _l1(Z) @ _l1(X) + _l1(B))).max()


@pytest.mark.parametrize("columns", [0, 6])
@pytest.mark.parametrize("n", [193, 330, 640])
@pytest.mark.parametrize("kind", ["sparse", "band"])
def test_fp64(F, kind, n, columns):
    c = 32 if kind == "sparse" else n
    assert _errors(F, _matrix(n, kind, columns), torch.complex128, F.FP64) <= c * 2.0**-52


@pytest.mark.parametrize("columns", [0, 6])
@pytest.mark.parametrize("n", [330, 640])
@pytest.mark.parametrize("kind", ["sparse", "band"])
def test_complex64(F, kind, n, columns):
    Z = _matrix(n, kind, columns).astype(np.complex64).astype(np.complex128)
    assert _errors(F, Z, torch.complex64, F.FP32) <= 3 * n * 2.0**-24
