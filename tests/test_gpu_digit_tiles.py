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


def test_refinement_with_columns_of_different_convergence(F):
    """Blocks of columns whose corrections shrink at different rates, so that a CTA meets tiles with
    different numbers of digit orders (192 and more tiles over 152 SMs); backward error at the
    default tolerance of the refinement, 8 sqrt(n) 2^-52, in the norms it is defined in."""
    n, r = 3000, 320
    rng = np.random.default_rng(8)
    h = n // 2
    gauss = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    Z = np.zeros((n, n), dtype=np.complex128)
    Z[:h, :h] = gauss(h, h) + 2 * np.sqrt(h) * np.eye(h) * 10
    Z[h:, h:] = gauss(h, h)
    Z[h:, h] *= 1e-3  # a badly scaled column: slower convergence of the right-hand sides that meet it
    B = np.zeros((n, r), dtype=np.complex128)
    for c in range(0, r, 64):
        rows = slice(0, h) if (c // 64) % 2 else slice(h, n)
        B[rows, c : c + 64] = gauss(h, 64)
    Zd, Bd = torch.tensor(Z, device="cuda"), torch.tensor(B, device="cuda")
    X = torch.empty_like(Bd)
    F.solve(F.factor(Zd, prec=F.MIXED), Bd, X)
    l1 = lambda t: t.real.abs() + t.imag.abs()
    R = l1(Bd - Zd @ X).max(0).values
    den = l1(Zd).sum(1).max() * l1(X).max(0).values + l1(Bd).max(0).values
    assert (R / den).max().item() <= 8 * np.sqrt(n) * 2.0**-52


@pytest.mark.parametrize("pseudo", [False, True])
@pytest.mark.parametrize("n,r", [(3, 128), (9, 300), (12, 127), (12, 128), (130, 129), (195, 500)])
def test_products_of_stored_factors(F, n, r, pseudo):
    """out <- out + w Y1 op(Y2) on rows longer than the factors, on both sides of the 128 columns at
    which the digits take over from float-float (whose bound is r 2^-48); integers, exact in FP64."""
    rng = np.random.default_rng(n * r + pseudo)
    draw = lambda *s: (rng.integers(-(2**19), 2**19, s) + 1j * rng.integers(-(2**19), 2**19, s)).astype(np.complex128)
    Y1, Y2, out = draw(n, r + 5), draw(n, r + 2), draw(n, n + 3)
    o = torch.tensor(out, device="cuda")
    F.lowrank_combine(torch.tensor(Y1, device="cuda")[:, :r], torch.tensor(Y2, device="cuda")[:, 1 : r + 1], o[:, :n],
                      weight=2.0, pseudo=pseudo, accumulate=True, prec=F.MIXED)
    a, b = Y1[:, :r], Y2[:, 1 : r + 1]
    ref = out[:, :n] + 2 * a @ (b.T if pseudo else b.conj().T)
    mag = 2 * np.abs(a) @ np.abs(b).T
    assert (np.abs(o.cpu().numpy()[:, :n] - ref) <= max(4e-15, r * 2.0**-48) * mag + 2.0**-52 * np.abs(ref)).all()
    assert (o.cpu().numpy()[:, n:] == out[:, n:]).all()


def test_infinities_and_nan_stay_in_their_rows_and_columns(F):
    rng = np.random.default_rng(4)
    Z = rng.standard_normal((140, 200)) + 1j * rng.standard_normal((140, 200))
    X = rng.standard_normal((200, 70)) + 1j * rng.standard_normal((200, 70))
    ref = Z @ X
    Z[3, 7], Z[130, 0], X[5, 65] = np.inf, complex(0, np.nan), -np.inf
    C = _product(F, Z, X)
    bad = np.zeros((140, 70), dtype=bool)
    bad[[3, 130], :] = bad[:, 65] = True
    assert np.isnan(C[bad].real).all() and np.isnan(C[bad].imag).all()
    assert (np.abs(C - ref)[~bad] <= 1e-13 * (np.abs(ref).max())).all()
