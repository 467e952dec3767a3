"""Prefix sums over the Euler tour at the edges of their 4096-slot chunks: branch
currents A^T x (post-processing, FP64 sums) against the exported loop matrix, and
the mixed and double-float products against FP64 (their sums run in
double-float), on bars whose tours end just before, at and after one, two and
three chunks."""
import numpy as np
import pytest
import scipy.sparse as sp

import synth
from synth.meshes import box_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_04891_gb300 import api, SPACE_LOOP, PREC_FP64, PREC_MIXED, PREC_DF  # noqa: E402


@pytest.mark.parametrize("nx", [169, 170, 171, 340, 341, 342, 511, 512, 513])
def test_tour_sums_at_chunk_edges(nx):
    m = box_mesh(nx * 8e-6, 20e-6, 10e-6, nx, 2, 1, jitter=0.1, seed=nx)
    M = api.Mesh.from_synth(m)
    L = api.Loops(M, m.ports)
    assert abs(2 * L.stats["n_nodes"] - 4096 * round(nx / 170.0)) < 100
    P = api.Plan(M, L, dict(grid=(64, 8, 8), n_touch=4))
    x = synth.complex_gaussian(L.nl, 3, seed=nx)
    xt = torch.from_numpy(x).cuda()
    om = 2 * np.pi * np.array([1e8, 1e9, 1e10])
    row_ptr, col, val, _ = L.export()
    A = sp.csr_matrix((val.astype(np.float64), col, row_ptr), shape=(L.nl, L.nb + L.np))
    ref = (A.T @ x.T).T[:, :L.nb]
    a, _, _ = api.postprocess(P, xt, om, voltages=False, potentials=False)
    assert np.abs(a.cpu().numpy() - ref).max() < 1e-12 * np.abs(ref).max()
    y = api.pfft_matvec(P, xt, om, SPACE_LOOP, PREC_FP64)
    # FP64 loop voltages: A times the branch voltages of those currents
    yb = api.pfft_matvec(P, a, om, 1, PREC_FP64).cpu().numpy()
    ref = (A[:, :L.nb] @ yb.T).T
    assert np.linalg.norm(y.cpu().numpy() - ref) < 1e-11 * np.linalg.norm(ref)
    for prec, tol in ((PREC_MIXED, 1e-5), (PREC_DF, 1e-11)):
        d = api.pfft_matvec(P, xt, om, SPACE_LOOP, prec) - y
        assert (torch.linalg.norm(d, dim=1) / torch.linalg.norm(y, dim=1)).max().item() < tol
