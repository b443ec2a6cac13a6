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


@pytest.mark.parametrize("mirror", [False, True])
def test_lowrank_combine(F, mirror):
    Y1, Y2 = _draw(150, 200), _draw(150, 200)
    out = torch.empty((150, 150), dtype=torch.complex128, device="cuda")
    _times_out_then_works(F, lambda: F.lowrank_combine(Y1, Y2, out, mirror=mirror, prec=F.MIXED))
    ref = Y1 @ Y2.conj().T
    assert (out - (ref + ref.conj().T if mirror else ref)).abs().max() <= 1e-13 * (Y1.abs() @ Y2.abs().T).max()


def test_far_field_and_rcs(F):
    import fosb_synth as S

    sm = S.icosphere(2)
    m = F.mesh_create(sm.verts, sm.tris, sm.vnormals)
    dirs = S.hplane_directions(61)
    X, Sigma = _draw(m.n_edges, 12), _draw(m.n_edges, m.n_edges)
    mean = torch.empty((183, 12), dtype=torch.complex128, device="cuda")
    cov = torch.empty((183, 183), dtype=torch.complex128, device="cuda")
    _times_out_then_works(F, lambda: F.farfield_moments(m, 2.0, dirs, X, mean, prec=F.MIXED))
    _times_out_then_works(F, lambda: F.farfield_moments(m, 2.0, dirs, Sigma, cov, m2=m, mirror=True, prec=F.MIXED))
    for got, X0, kw in ((mean, X, {}), (cov, Sigma, dict(m2=m, mirror=True))):
        ref = torch.empty_like(got)
        F.farfield_moments(m, 2.0, dirs, X0, ref, prec=F.FP64, **kw)
        assert (got - ref).abs().max() <= 1e-12 * ref.abs().max()
    inc = F.incidence(S.hplane_directions(12), [[0.0, 1.0, 0.0]] * 12)
    _times_out_then_works(F, lambda: F.rcs_monostatic(m, 2.0, inc, X))


def test_capture(F):
    """A captured combination has no host to report to: float-float products, which have no waits."""
    Y1, Y2 = _draw(150, 200), _draw(150, 200)
    out = torch.zeros((150, 150), dtype=torch.complex128, device="cuda")
    call = lambda: F.lowrank_combine(Y1, Y2, out, prec=F.MIXED)
    call()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    Y1.copy_(_draw(200, 150).T)
    graph.replay()
    torch.cuda.synchronize()
    assert (out - Y1 @ Y2.conj().T).abs().max() <= 200 * 2.0**-48 * (Y1.abs() @ Y2.abs().T).max()
