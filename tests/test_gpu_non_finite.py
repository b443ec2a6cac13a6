"""A right-hand side with NaN or an infinity is not a converged solve: FOSB_ERR_NOT_CONVERGED, with the other
columns refined as without it (backward error at the default tolerance)."""
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


@pytest.mark.parametrize("solver", ["REFINE_AUTO", "REFINE_IR", "REFINE_GMRES"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("r", [1, 3, 6])
def test_non_finite_right_hand_side(F, r, bad, solver):
    n, rng = 300, np.random.default_rng(r)
    Z = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    B = rng.standard_normal((n, r)) + 1j * rng.standard_normal((n, r))
    B[7, r - 1] = bad
    Zd, Bd = torch.tensor(Z, device="cuda"), torch.tensor(B, device="cuda")
    X = torch.zeros_like(Bd)
    lu = F.factor(Zd, prec=F.MIXED)
    with pytest.raises(F.FosbError) as e:
        F.solve(lu, Bd, X, solver=getattr(F, solver))
    assert e.value.status == F.FOSB_ERR_NOT_CONVERGED
    assert not torch.isfinite(X[:, r - 1].abs()).all()
    l1 = lambda t: t.real.abs() + t.imag.abs()
    for c in range(r - 1):
        err = l1(Bd[:, c] - Zd @ X[:, c]).max() / (l1(Zd).sum(1).max() * l1(X[:, c]).max() + l1(Bd[:, c]).max())
        assert err <= 8 * np.sqrt(n) * 2.0**-52
    B[7, r - 1] = 1.0
    F.solve(lu, torch.tensor(B, device="cuda"), X, solver=getattr(F, solver))
