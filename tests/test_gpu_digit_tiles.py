"""The digit-split product where its work is cut differently: tiles along k in pieces, one and
several chunks of 128, ragged edges of the 128 x 64 tiles, and digits at the ends of their range.
Integer operands make the FP64 reference exact; the bound is the 4e-15 of sum |Z||X| per entry that
seven digits give for any K."""
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


def _product(F, Z, X):
    C = torch.empty((Z.shape[0], X.shape[1]), dtype=torch.complex128, device="cuda")
    F.zgemm_fp64class(torch.tensor(Z, device="cuda"), torch.tensor(X, device="cuda"), C, 0)
    return C.cpu().numpy()


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (128, 64, 16), (129, 65, 128), (127, 63, 129), (130, 70, 2100),
                                   (300, 5, 4097), (2560, 193, 2048), (10000, 65, 130)])
def test_integer_products(F, M, N, K):
    rng = np.random.default_rng(M + N + K)
    draw = lambda *s: (rng.integers(-(2**19), 2**19, s) + 1j * rng.integers(-(2**19), 2**19, s)).astype(np.complex128)
    Z, X = draw(M, K), draw(K, N)
    err = np.abs(_product(F, Z, X) - Z @ X)
    assert (err <= 4e-15 * (np.abs(Z) @ np.abs(X))).all()


@pytest.mark.parametrize("digit", [-128, 127])
def test_digits_at_the_ends_of_their_range(F, digit):
    """All digits but the first and the last are -128 (or 127) in every entry: the order sums of Im
    are at their bounds, those of Re cancel to zero."""
    F_int = -127 * 2**48 + sum(digit * 256**j for j in range(1, 6)) if digit < 0 else 127 * sum(256**j for j in range(1, 7))
    x, K = float(F_int) * 2.0**-55, 1000
    assert int(x * 2.0**55) == F_int
    Z = np.full((5, K), complex(x, x))
    X = np.full((K, 3), complex(x, x))
    C = _product(F, Z, X)
    exact = 2 * K * F_int * F_int  # Im, in units of 2^-110
    assert np.abs(C.real).max() <= 4e-15 * 2 * K * x * x
    assert np.abs(C.imag - float(exact) * 2.0**-110).max() <= 4e-15 * 2 * K * x * x
