"""FP64 factorisations around the size where the trailing updates change from FP64 products to digits,
with rows and columns of very different scale: |B - Z X| <= n 2^-52 (|Z| |X| + |B|) per entry, the
bound of partial pivoting without growth, which row and column scalings do not change."""
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


@pytest.mark.parametrize("scaled", ["none", "rows", "columns", "both"])
@pytest.mark.parametrize("n", [64, 128, 129, 193, 321, 1000])
def test_componentwise_backward_error(F, n, scaled):
    rng = np.random.default_rng(n)
    Z = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    if scaled in ("rows", "both"):
        Z = Z * 10.0 ** rng.uniform(-6, 6, n)[:, None]
    if scaled in ("columns", "both"):
        Z = Z * 10.0 ** rng.uniform(-6, 6, n)
    B = Z @ (rng.standard_normal((n, 2)) + 1j * rng.standard_normal((n, 2)))
    X = torch.empty((n, 2), dtype=torch.complex128, device="cuda")
    F.solve(F.factor(torch.tensor(Z, device="cuda"), prec=F.FP64), torch.tensor(B, device="cuda"), X)
    X = X.cpu().numpy()
    l1 = lambda t: np.abs(t.real) + np.abs(t.imag)
    assert (l1(B - Z @ X) <= n * 2.0**-52 * (l1(Z) @ l1(X) + l1(B))).all()


def test_tiny_and_huge_scales(F):
    """Row scales whose products with the column scales leave the range of one power of two."""
    n = 300
    rng = np.random.default_rng(2)
    Z = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    r = 2.0 ** rng.integers(-450, 450, n)
    b = Z @ np.ones((n, 1))
    x, y = (torch.empty((n, 1), dtype=torch.complex128, device="cuda") for _ in range(2))
    F.solve(F.factor(torch.tensor(Z, device="cuda"), prec=F.FP64), torch.tensor(b, device="cuda"), x)
    F.solve(F.factor(torch.tensor(Z / r, device="cuda"), prec=F.FP64), torch.tensor(b, device="cuda"), y)
    # columns scaled by powers of two: the same pivots and, digit by digit, the same factors
    assert torch.equal(x[:, 0], y[:, 0] / torch.tensor(r, device="cuda"))
