"""The FP64 and double-float gathers by real columns (projection, near field,
interpolation) at every team shape: groups of lanes per row for up to 8
right-hand sides, one to four column sets per lane above, ragged last slabs.

Every right-hand side is compared with the oracle pFFT (FP64 1e-10, the parity
bar of both forms), and must equal, bit for bit, the product of that
right-hand side alone: the order of a row's sum does not depend on how many
right-hand sides share the call.
"""
import numpy as np
import pytest

import synth
from oracle.graph import build_loops
from oracle.pfft import PfftSystem, PfftParams

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_04891_gb300 import api, SPACE_LOOP, PREC_FP64, PREC_DF  # noqa: E402


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
             for prec in (PREC_FP64, PREC_DF)}
    return P, om, xt, ref, alone


@pytest.mark.parametrize("prec", [PREC_FP64, PREC_DF], ids=["fp64", "df"])
@pytest.mark.parametrize("R", [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 32, 33, 48, 49, 64, 65, 97, 130])
def test_columns_match_oracle_and_single_right_hand_side(system, R, prec):
    P, om, xt, ref, alone = system
    y = api.pfft_matvec(P, xt[:R].contiguous(), om[:R], SPACE_LOOP, prec)
    assert torch.equal(y, alone[prec][:R])
    err = np.linalg.norm(y.cpu().numpy() - ref[:R], axis=1) / np.linalg.norm(ref[:R], axis=1)
    assert err.max() < 1e-10
