"""Complex64 factors at the sizes where the tournament's levels change: one CTA (up to 128 and
256 rows), one cluster (up to 1024 and 2048), two levels above, ragged widths among them.
Tolerance: the normwise backward error of LU without growth, n u with u = 2^-24, plus four units
for the smallest systems."""
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


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 128, 129, 255, 257, 513, 1023, 1025, 1500, 2047, 2049, 3001])
def test_unrefined_factors_backward_error(F, n):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    b = rng.standard_normal((n, 2)) + 1j * rng.standard_normal((n, 2))
    Z = torch.tensor(A, dtype=torch.complex64, device="cuda")
    x = torch.tensor(b, dtype=torch.complex64, device="cuda")
    r0 = x.clone()
    F.solve(F.factor(Z), x)
    Zd, xd = Z.to(torch.complex128), x.to(torch.complex128)
    r = (r0.to(torch.complex128) - Zd @ xd).abs().max(0).values
    be = r / (Zd.abs().sum(1).max() * xd.abs().max(0).values + r0.abs().max(0).values)
    assert be.max().item() <= (n + 4) * 2.0**-24


@pytest.mark.parametrize("n,col", [(100, 70), (300, 5), (1500, 1300), (2500, 64)])
def test_zero_column_is_reported_by_every_level(F, n, col):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    A[:, col] = 0
    with pytest.raises(F.FosbError) as e:
        F.factor(torch.tensor(A, dtype=torch.complex64, device="cuda"))
    assert e.value.status == F.FOSB_ERR_SINGULAR
