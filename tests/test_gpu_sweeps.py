"""Triangular sweeps of complex64 factors: every chunk width, ragged blocks, and the exactness of
power-of-two scalings.  Backward errors against n u, u = 2^-24 (LU without growth), plus four
units for the smallest systems."""
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


def _system(n, seed):
    rng = np.random.default_rng(seed)
    return torch.tensor(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)), dtype=torch.complex64, device="cuda")


def _backward_error(Z, X, B):
    Zd, Xd, Bd = (t.to(torch.complex128) for t in (Z, X, B))
    r = (Bd - Zd @ Xd).abs().max(0).values
    return (r / (Zd.abs().sum(1).max() * Xd.abs().max(0).values + Bd.abs().max(0).values)).max().item()


@pytest.mark.parametrize("n", [1, 63, 64, 65, 130, 333])
def test_every_chunk_width(F, n):
    Z = _system(n, n)
    lu = F.factor(Z)
    rng = np.random.default_rng(n + 1)
    for r in (1, 2, 3, 4, 5, 6, 7, 8, 9, 16, 17, 33):
        B = torch.tensor(rng.standard_normal((n, r)) + 1j * rng.standard_normal((n, r)), dtype=torch.complex64, device="cuda")
        X = torch.empty_like(B)
        F.solve(lu, B, X)
        assert _backward_error(Z, X, B) <= (n + 4) * 2.0**-24, r


def test_power_of_two_column_scaling_is_exact(F):
    """Z D with D a power of two per column has the same pivots and the same factors up to exact
    scalings (the trailing update scales its columns itself), so x comes out as D^-1 x bit by bit."""
    n = 900
    Z = _system(n, 5)
    rng = np.random.default_rng(6)
    e = torch.tensor(rng.integers(-20, 21, n), device="cuda")
    d = torch.pow(2.0, e.to(torch.float64)).to(torch.float32)
    b = torch.tensor(rng.standard_normal((n, 3)) + 1j * rng.standard_normal((n, 3)), dtype=torch.complex64, device="cuda")
    x, y = torch.empty_like(b), torch.empty_like(b)
    F.solve(F.factor(Z), b, x)
    F.solve(F.factor(Z * d), b, y)
    assert torch.equal(x, y * d[:, None])


@pytest.mark.parametrize("n,r", [(513, 2600), (1000, 1088), (1000, 1101), (5121, 209)])
def test_superblocks(F, n, r):
    """Both sides of the size where the sweeps go 512 rows at a time (1000 x 1088 is one kernel),
    with one row in the last superblock and with odd numbers of columns."""
    Z = _system(n, n)
    rng = np.random.default_rng(n + 1)
    B = torch.tensor(rng.standard_normal((n, r)) + 1j * rng.standard_normal((n, r)), dtype=torch.complex64, device="cuda")
    X = torch.empty_like(B)
    F.solve(F.factor(Z), B, X)
    assert _backward_error(Z, X, B) <= (n + 4) * 2.0**-24
