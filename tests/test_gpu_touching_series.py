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
