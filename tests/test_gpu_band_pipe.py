"""The pipelined band sweeps (bands 32 to about 180 in FP64, 400 in FP32) and the
kernel of wider bands, against nested dissection of the same Laplacian (another
factorisation, another order: 1e-10, the bar of those two routes) and FP32
against FP64 (1e-4, the bar of the FP32 sweeps), on plates whose bands lie on
both sides of the limits and whose unknowns are no multiple of the 32-pivot chunk."""
import numpy as np
import pytest

import synth
from synth.meshes import box_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_04891_gb300 import api, native as N, PREC_FP64, PREC_MIXED  # noqa: E402

bands = {}


@pytest.mark.parametrize("nx,ny", [(14, 12), (20, 17), (31, 30), (45, 43), (64, 62), (70, 69), (101, 97), (154, 152)])
def test_band_sweeps_match_nested_dissection(nx, ny):
    h = 40e-6
    m = box_mesh(nx * h, ny * h, 35e-6, nx, ny, 1, jitter=0.1, seed=nx)
    M = api.Mesh.from_synth(m)
    L = api.Loops(M, m.ports)
    P = api.Plan(M, L, dict(grid=(16, 16, 8), n_touch=4, near_factor=1.0, near_min_diam=1.0))
    api.precond_set_method(P, N.PC_BAND)
    bands[nx] = api.precond_info(P)["band_width"]
    assert 31 < bands[nx] < 1024
    R = 3
    y = torch.from_numpy(synth.complex_gaussian(L.nl, R, seed=ny)).cuda()
    om = 2 * np.pi * np.array([1e7, 1e9, 1e9])
    z = api.pfft_precond_apply(P, y, om)
    f = api.pfft_precond_apply(P, y, om, prec=PREC_MIXED)
    api.precond_set_method(P, N.PC_ND)
    ref = api.pfft_precond_apply(P, y, om)
    nrm = torch.linalg.norm(ref, dim=1)
    assert (torch.linalg.norm(z - ref, dim=1) / nrm).max().item() < 1e-10
    assert (torch.linalg.norm(f - ref, dim=1) / nrm).max().item() < 1e-4


def test_bands_cover_the_limits():
    if len(bands) < 8:
        pytest.skip("needs every size above")
    w = sorted(bands.values())
    assert w[0] < 64 and any(140 < v < 178 for v in w) and any(180 < v < 390 for v in w) and w[-1] > 400


@pytest.mark.parametrize("nx,ny,band,R,prec", [(16, 15, (37, 64), 400, PREC_FP64), (30, 29, (76, 97), 320, PREC_FP64), (38, 37, (97, 113), 400, PREC_FP64),
                                               (74, 73, (179, 240), 770, PREC_MIXED)])
def test_many_chains_of_wide_panels(nx, ny, band, R, prec):
    """Bands whose panels fill an SM, with more chains than the pipeline takes, against a
    few chains of the same: FP32 takes the same order bit for bit, FP64 fused products
    in one of them (1e-11, the bar of two orders of one FP64 solve)."""
    h = 40e-6
    m = box_mesh(nx * h, ny * h, 35e-6, nx, ny, 1, jitter=0.1, seed=nx)
    M = api.Mesh.from_synth(m)
    L = api.Loops(M, m.ports)
    P = api.Plan(M, L, dict(grid=(16, 16, 8), n_touch=4, near_factor=1.0, near_min_diam=1.0))
    api.precond_set_method(P, N.PC_BAND)
    assert band[0] <= api.precond_info(P)["band_width"] < band[1]
    few = [0, 1, R // 2, R - 1]
    g = torch.Generator(device="cuda").manual_seed(3)
    y = torch.randn(R, L.nl, dtype=torch.complex128, device="cuda", generator=g)
    z = api.pfft_precond_apply(P, y, 2e9, prec=prec)[few]
    ref = api.pfft_precond_apply(P, y[few].contiguous(), 2e9, prec=prec)
    if prec == PREC_MIXED:
        assert torch.equal(z, ref)
    else:
        assert (torch.linalg.norm(z - ref, dim=1) / torch.linalg.norm(ref, dim=1)).max().item() < 1e-11


def test_these_sizes_lie_on_both_sides_of_the_limits():
    """Alone, from the plans themselves: a band each for the first tiles above a warp, the
    FP64 pipeline's last, the FP32 pipeline's and the wider kernel's."""
    h = 40e-6
    for nx, ny, lo, hi in ((14, 12, 32, 64), (64, 62, 140, 178), (101, 97, 180, 390), (154, 152, 400, 1024)):
        m = box_mesh(nx * h, ny * h, 35e-6, nx, ny, 1, jitter=0.1, seed=nx)
        M = api.Mesh.from_synth(m)
        P = api.Plan(M, api.Loops(M, m.ports), dict(grid=(16, 16, 8), n_touch=4, near_factor=1.0, near_min_diam=1.0))
        api.precond_set_method(P, N.PC_BAND)
        assert lo <= api.precond_info(P)["band_width"] < hi, (nx, ny)
