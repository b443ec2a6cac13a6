"""Refined solves report the backward error of the solution they return, also where the last correction was
taken from an iterate that met the default tolerance already, and return that iterate where the
correction is none.  The reported value is compared with a residual in extended precision: both are sums of n products
and a rounding of x, 2 sqrt(n) 2^-53 of the norms apart, and where digits were left out 2^-48."""
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


def _l1(t):
    return np.abs(t.real) + np.abs(t.imag)


def _backward_error(Z, X, B):
    Zl, Xl, Bl = (t.astype(np.clongdouble) for t in (Z, X, B))
    return float((_l1(Bl - Zl @ Xl).max(0) / (_l1(Zl).sum(1).max() * _l1(Xl).max(0) + _l1(Bl).max(0))).max())


@pytest.mark.parametrize("r", [1, 4, 5, 17])
@pytest.mark.parametrize("n", [100, 256, 320, 360, 480, 520, 600, 700])
def test_reported_backward_error_is_that_of_the_solution(F, n, r):
    rng = np.random.default_rng(n)
    draw = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    Z, B = draw(n, n), draw(n, r)
    X = torch.empty((n, r), dtype=torch.complex128, device="cuda")
    _, steps, reported = F.solve(F.factor(torch.tensor(Z, device="cuda"), prec=F.MIXED), torch.tensor(B, device="cuda"), X)
    true = _backward_error(Z, X.cpu().numpy(), B)
    floor = 2 * np.sqrt(n) * 2.0**-53 + (2.0**-48 if r > 4 and n >= 256 else 0.0)
    assert abs(reported - true) <= floor
    assert true <= max(64, 8 * np.sqrt(n)) * 2.0**-52
