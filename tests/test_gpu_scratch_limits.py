"""Calls whose optional scratch memory cannot be had do without it: the allocation fails at each place in turn."""
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
    yield mod
    mod.debug_fail_allocation(-1)


def _system(n, r, dtype=torch.complex128):
    rng = np.random.default_rng(n)
    draw = lambda *s: torch.tensor(rng.standard_normal(s) + 1j * rng.standard_normal(s), device="cuda").to(dtype)
    return draw(n, n), draw(n, r)


def _backward_error(Z, X, B):
    Z, X, B = (t.to(torch.complex128) for t in (Z, X, B))
    l1 = lambda t: t.real.abs() + t.imag.abs()
    return (l1(B - Z @ X) / (l1(Z) @ l1(X) + l1(B))).max().item()


@pytest.mark.parametrize("after", [1, 2, 3, 4, 7])
def test_fp64_factorisation_without_digits(F, after):
    """The first allocation is the panels' scratch; everything else is for the digits."""
    n = 400
    Z, B = _system(n, 2)
    F.debug_fail_allocation(after)
    lu = F.factor(Z, prec=F.FP64)
    F.debug_fail_allocation(-1)
    X = torch.empty_like(B)
    F.solve(lu, B, X)
    assert _backward_error(Z, X, B) <= n * 2.0**-52


@pytest.mark.parametrize("n,r", [(200, 1), (200, 7), (130, 1100), (700, 1501)])
def test_complex64_sweeps_in_parts(F, n, r):
    """The sweeps' copies of the right-hand sides do not fit at the first attempt."""
    Z, B = _system(n, r, torch.complex64)
    lu = F.factor(Z, prec=F.FP32)
    X = torch.empty_like(B)
    F.debug_fail_allocation(0)
    if r == 1:  # one column cannot be halved
        with pytest.raises(F.FosbError) as e:
            F.solve(lu, B, X)
        assert e.value.status == F.FOSB_ERR_OOM
    F.solve(lu, B, X)
    F.debug_fail_allocation(-1)
    assert _backward_error(Z, X, B) <= 3 * n * 2.0**-24
