"""The gathers by real columns (projection, near field, interpolation) at every
team shape: FP64 and double-float with groups of lanes per row for up to 8
right-hand sides, one to four column sets per lane above, ragged last slabs;
FP32 with several rows per warp for up to 16 right-hand sides, one row above.

Every right-hand side is compared with the oracle pFFT (1e-10 for FP64 and
double-float, 1e-5 for the mixed form: their parity bars), and must equal, bit
for bit, the product of that right-hand side alone: the order of a row's sum
does not depend on how many right-hand sides share the call (mixed form: below
the 96 at which the near field changes to the tensor cores).
"""
import numpy as np
import pytest

import synth
from synth.meshes import wire_array_mesh
from oracle.graph import build_loops
from oracle.pfft import PfftSystem, PfftParams

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_04891_gb300 import api, SPACE_LOOP, PREC_FP64, PREC_MIXED, PREC_DF  # noqa: E402


@pytest.fixture(scope="module")
def system():
    m = synth.tiny_wires()
    O = build_loops(m)
    prm = dict(grid=(16, 8, 4), order=3, near_factor=4.0, near_min_diam=2.0, n_touch=8)
    S = PfftSystem(m, O, PfftParams(**prm))
    M = api.Mesh.from_synth(m)
    P = api.Plan(M, api.Loops(M, m.ports), dict(prm, h0=0.0))
    om = 2 * np.pi * np.logspace(7, 10, 130)
    x = synth.complex_gaussian(O.nl, 130, seed=21)
    ref = np.stack([S.matvec(x[r], om[r]) for r in range(130)])
    xt = torch.from_numpy(x).cuda()
    alone = {prec: torch.cat([api.pfft_matvec(P, xt[r:r + 1], om[r:r + 1], SPACE_LOOP, prec) for r in range(130)])
             for prec in (PREC_FP64, PREC_DF, PREC_MIXED)}
    return P, om, xt, ref, alone


@pytest.mark.parametrize("prec", [PREC_FP64, PREC_DF], ids=["fp64", "df"])
@pytest.mark.parametrize("R", [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 32, 33, 48, 49, 64, 65, 97, 130])
def test_columns_match_oracle_and_single_right_hand_side(system, R, prec):
    P, om, xt, ref, alone = system
    y = api.pfft_matvec(P, xt[:R].contiguous(), om[:R], SPACE_LOOP, prec)
    assert torch.equal(y, alone[prec][:R])
    check(y, ref[:R], 1e-10)


@pytest.mark.parametrize("R", [1, 2, 3, 4, 5, 6, 8, 10, 11, 15, 16, 17, 31, 32, 33, 48, 65, 95])
def test_mixed_columns_match_oracle_and_single_right_hand_side(system, R):
    P, om, xt, ref, alone = system
    y = api.pfft_matvec(P, xt[:R].contiguous(), om[:R], SPACE_LOOP, PREC_MIXED)
    assert torch.equal(y, alone[PREC_MIXED][:R])
    check(y, ref[:R], 1e-5)


def check(y, ref, tol):
    err = np.linalg.norm(y.cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() < tol


def test_empty_grid_rows_are_skipped_without_a_trace():
    """Wires far apart leave most y rows of the grid without stencil nodes; the
    products skip them (32 rows and more) and must not see what another product, here
    of NaN currents, left in the buffers.  Against the oracle at the parity bars."""
    m = synth.wire_array_mesh(2, 10e-6, 60e-6, 900e-6, n_sides=6, n_seg=4, jitter=0.1, seed=9)
    O = build_loops(m)
    prm = dict(grid=(8, 64, 4), order=2, near_factor=1.0, near_min_diam=2.0, n_touch=8)
    S = PfftSystem(m, O, PfftParams(**prm))
    P = api.Plan(api.Mesh.from_synth(m), api.Loops(api.Mesh.from_synth(m), m.ports), dict(prm, h0=0.0))
    om = 2 * np.pi * np.logspace(8, 9, 20)
    x = synth.complex_gaussian(O.nl, 20, seed=4)
    ref = np.stack([S.matvec(x[r], om[r]) for r in range(20)])
    xt = torch.from_numpy(x).cuda()
    for prec, tol in ((PREC_FP64, 1e-10), (PREC_DF, 1e-10), (PREC_MIXED, 1e-5)):
        for R in (1, 20):
            g = torch.full((3 * R, 8, 64, 4), float("nan"), device="cuda",
                           dtype=torch.complex64 if prec == PREC_MIXED else torch.complex128)
            api.pfft_convolve(P, g, PREC_MIXED if prec == PREC_MIXED else PREC_FP64)
            api.pfft_matvec(P, torch.full_like(xt[:R], float("nan")), om[:R], SPACE_LOOP, prec)
            check(api.pfft_matvec(P, xt[:R].contiguous(), om[:R], SPACE_LOOP, prec), ref[:R], tol)


@pytest.fixture(scope="module", params=[(386, (32, 8, 16)), (930, (64, 16, 16))], ids=["5418", "13034"])
def long_wire(request):
    """A seven-sided wire: 5,418 triangles (component form, two rows per warp) and 13,034
    (column form, up to five), ragged in the last warp and block; 4,096 and 16,384 nodes
    (one row per warp, up to six)."""
    seg, grid = request.param
    m = wire_array_mesh(1, 10e-6, seg * 1e-5, 4e-5, n_sides=7, n_seg=seg, jitter=0.1, seed=seg)
    assert m.nt == 14 * (seg + 1)
    M = api.Mesh.from_synth(m)
    P = api.Plan(M, api.Loops(M, m.ports), dict(grid=grid, n_touch=8))
    om = 2 * np.pi * np.logspace(7, 10, 17)
    x = torch.from_numpy(synth.complex_gaussian(P.nl, 17, seed=22)).cuda()
    alone = torch.cat([api.pfft_matvec(P, x[r:r + 1], om[r:r + 1], SPACE_LOOP, PREC_MIXED) for r in range(17)])
    return P, om, x, alone, api.pfft_matvec(P, x, om, SPACE_LOOP, PREC_FP64).cpu().numpy()


@pytest.mark.parametrize("R", range(1, 18))
def test_mixed_columns_of_several_rows_per_warp(long_wire, R):
    P, om, x, alone, ref = long_wire
    y = api.pfft_matvec(P, x[:R].contiguous(), om[:R], SPACE_LOOP, PREC_MIXED)
    assert torch.equal(y, alone[:R])
    check(y, ref[:R], 1e-5)
