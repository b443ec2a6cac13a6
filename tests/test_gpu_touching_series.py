"""Touching pairs through the phase series: every number of series terms up to the largest
phase, the per-point path above it, and the smallest and largest n_ss, against the oracle.
The series truncates below 2^-56 and its rounding stays within a few units of 2^-52 of the
moments, so the 1e-12 of max|Z| of the FP64 assembly holds unchanged."""
import numpy as np
import pytest

import fosb_synth as S
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,n_ss", [(1e-3, 5), (0.1, 5), (1.0, 1), (1.0, 12), (1.9, 5), (2.6, 2), (2.7, 5), (3.2, 5),
                                    (9.0, 3), (9.0, 12)])
def test_touching_pairs_match_oracle_at_every_phase(k, n_ss):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_01457_gb300 as F

    F.build.build()
    sm = S.ellipsoid(0, (1.0, 0.7, 1.2))  # 20 triangles with edges near 1: k |x - y| up to about 1.3 k
    m, om = F.mesh_create(sm.verts, sm.tris, sm.vnormals), O.from_synth(sm)
    N = m.n_edges
    Z = torch.empty((N, N), dtype=torch.complex128, device="cuda:0")
    F.assemble_efie(m, k, Z, n_ss=n_ss)
    Zo = O.assemble_z(om, k, n_ss)
    assert np.abs(Z.cpu().numpy() - Zo).max() <= 1e-12 * np.abs(Zo).max()


@pytest.mark.parametrize("k0,n_ss", [(0.05, 5), (1.0, 12), (2.0, 1), (2.4, 5), (8.0, 3)])
def test_pmchwt_touching_pairs_match_oracle_at_every_phase(k0, n_ss):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_01457_gb300 as F

    F.build.build()
    sm = S.ellipsoid(0, (1.0, 0.7, 1.2))
    m, om = F.mesh_create(sm.verts, sm.tris, sm.vnormals), O.from_synth(sm)
    N = m.n_edges
    Z = torch.empty((2 * N, 2 * N), dtype=torch.complex128, device="cuda:0")
    F.assemble_pmchwt(m, k0, 1.7, 1.0, Z, n_ss=n_ss)
    Zo = O.assemble_pmchwt(om, k0, 1.7, 1.0, n_ss)
    for r in range(2):
        for c in range(2):
            zo = Zo[r * N:(r + 1) * N, c * N:(c + 1) * N]
            zg = Z[r * N:(r + 1) * N, c * N:(c + 1) * N].cpu().numpy()
            assert np.abs(zg - zo).max() <= 1e-12 * np.abs(zo).max()


@pytest.mark.parametrize("shape,k,n_inc", [("ellipsoid", 0.4, 1), ("ellipsoid", 2.4, 3), ("ellipsoid", 9.0, 2),
                                           ("torus", 2.0, 5)])
def test_adjoint_gradient_matches_oracle_at_every_phase(shape, k, n_inc):
    """The series (and the per-point path above phase 3) of the adjoint's touching pairs, and its
    unordered regular pairs on a mesh that fills no tile (90 triangles): 1e-8, as the refined
    solves and the oracle's LAPACK ones agree to."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_01457_gb300 as F

    F.build.build()
    sm = S.ellipsoid(0, (1.0, 0.7, 1.2)) if shape == "ellipsoid" else S.torus(9, 5)
    d, p, _ = S.monostatic_directions(n_inc)
    m, inc = F.mesh_create(sm.verts, sm.tris, sm.vnormals), F.incidence(d, p)
    Z = torch.empty((m.n_edges, m.n_edges), dtype=torch.complex128, device="cuda:0")
    U = torch.empty((m.n_edges, n_inc), dtype=torch.complex128, device="cuda:0")
    F.assemble_efie(m, k, Z, inc=inc, b=U)
    lu = F.factor(Z, prec=F.FP64)
    F.solve(lu, U)
    rng = np.random.default_rng(3)
    w = rng.uniform(0.5, 1.5, n_inc)
    grad = torch.zeros((sm.nv, 3), dtype=torch.float64, device="cuda:0")
    F.rcs_monostatic(m, k, inc, U, lu=lu, weights=w, grad=grad)
    sel = rng.choice(3 * sm.nv, size=12, replace=False)
    _, J = O.rcs_monostatic_jacobian(O.from_synth(sm), k, d, p, [(int(s // 3), int(s % 3)) for s in sel])
    g, go = grad.cpu().numpy().reshape(-1)[sel], w @ J
    assert np.linalg.norm(g - go) <= 1e-8 * np.linalg.norm(go)
