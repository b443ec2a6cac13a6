"""Failure detection of the digit products on the GPU without a fault: the kernel's bounded waits are made
to run out by a tiny poll limit (fosb_debug_set_wait_limit); the call reports FOSB_ERR_TIMEOUT and the same
call works once the limit is restored.  Sizes with one tile and one chunk of 128, with tiles cut along k,
and with several tiles per SM."""
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


def _draw(*shape):
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    return torch.randn(shape, dtype=torch.complex128, device="cuda", generator=g)


def _times_out_then_works(F, call):
    try:
        F.debug_set_wait_limit(1)
        with pytest.raises(F.FosbError) as e:
            call()
        assert e.value.status == F.FOSB_ERR_TIMEOUT
    finally:
        F.debug_set_wait_limit(0)
    call()


@pytest.mark.parametrize("M,N,K", [(100, 20, 100), (130, 70, 2100), (5000, 300, 400)])
def test_product(F, M, N, K):
    Z, X = _draw(M, K), _draw(K, N)
    C = torch.empty((M, N), dtype=torch.complex128, device="cuda")
    _times_out_then_works(F, lambda: F.zgemm_fp64class(Z, X, C, 0))
    assert (C - Z @ X).abs().max() <= 1e-13 * (Z.abs() @ X.abs()).max()
