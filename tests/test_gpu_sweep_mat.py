"""The matrix sweeps of narrow bands (few right-hand sides x blocks) against the
stepped sweeps of the same factor, which more right-hand sides take: the same
solve in another order, so FP64 to 1e-11 and double-float to 1e-10 (the bars of
those sweeps against FP64 and the oracle), one block and several, lengths around
multiples of the 32-pivot chunk, one and several frequencies."""
import numpy as np
import pytest

import synth
from synth.meshes import box_mesh, wire_array_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_04891_gb300 import api, PREC_FP64, PREC_DF  # noqa: E402


def meshes():
    for nx in (1, 5, 20, 21, 22, 60):
        yield "bar%d" % nx, lambda nx=nx: box_mesh(nx * 8e-6, 20e-6, 10e-6, nx, 2, 1, jitter=0.1, seed=nx)
    for n, seg, sides in ((1, 9, 5), (3, 21, 8), (2, 30, 16)):
        yield "wires%d_%d" % (n, sides), lambda n=n, seg=seg, sides=sides: wire_array_mesh(
            n, 10e-6, seg * 1e-5, 4e-5, n_sides=sides, n_seg=seg, jitter=0.1, seed=seg)


@pytest.mark.parametrize("make", [m[1] for m in meshes()], ids=[m[0] for m in meshes()])
def test_matrix_sweeps_match_stepped(make):
    m = make()
    M = api.Mesh.from_synth(m)
    L = api.Loops(M, m.ports)
    P = api.Plan(M, L, dict(grid=(16, 8, 8), n_touch=4))
    info = api.precond_info(P)
    assert info["band_width"] <= 31
    many = 64 // info["blocks"] + 1               # more chains than the matrix sweeps take
    om = 2 * np.pi * np.array([1e7, 1e9, 1e10])[np.arange(many) % 3]
    y = torch.from_numpy(synth.complex_gaussian(L.nl, many, seed=5)).cuda()
    for prec, tol in ((PREC_FP64, 1e-11), (PREC_DF, 1e-10)):
        ref = api.pfft_precond_apply(P, y, om, prec=prec)
        for R in (1, 3, min(8, many - 1)):
            z = api.pfft_precond_apply(P, y[:R].contiguous(), om[:R], prec=prec)
            err = torch.linalg.norm(z - ref[:R], dim=1) / torch.linalg.norm(ref[:R], dim=1)
            assert err.max().item() < tol, (prec, R)


@pytest.mark.parametrize("make", [m[1] for m in meshes()], ids=[m[0] for m in meshes()])
def test_matrix_sweeps_within_the_bars(make):
    """The second application with the same factors (matrices whatever their build costs)
    against many more chains (steps): FP64 to 1e-11, and double-float to FP64's result
    at 1e-11, the bar of the stepped double-float sweeps."""
    m = make()
    M = api.Mesh.from_synth(m)
    L = api.Loops(M, m.ports)
    P = api.Plan(M, L, dict(grid=(16, 8, 8), n_touch=4))
    blocks = api.precond_info(P)["blocks"]
    om = 2 * np.pi * np.array([1e7, 1e9, 1e10])[np.arange(64 // blocks + 1) % 3]
    y = torch.from_numpy(synth.complex_gaussian(L.nl, om.size, seed=6)).cuda()
    ref = api.pfft_precond_apply(P, y, om)
    nrm = torch.linalg.norm(ref, dim=1)
    for prec in (PREC_FP64, PREC_DF):
        for R in (1, 3, min(8, om.size - 1)):
            api.pfft_precond_apply(P, y[:R].contiguous(), om[:R], prec=prec)
            z = api.pfft_precond_apply(P, y[:R].contiguous(), om[:R], prec=prec)
            assert (torch.linalg.norm(z - ref[:R], dim=1) / nrm[:R]).max().item() < 1e-11, (prec, R)


def test_one_application_does_not_pay_for_many_matrices():
    """64 frequencies, one application: the steps, as 65 take them, bit for bit and with
    no more launches; a second one with the same factors takes the matrices."""
    m = box_mesh(60 * 8e-6, 20e-6, 10e-6, 60, 2, 1, jitter=0.1, seed=2)
    M = api.Mesh.from_synth(m)
    L = api.Loops(M, m.ports)
    om = 2 * np.pi * np.logspace(7, 10, 65)
    y = torch.from_numpy(synth.complex_gaussian(L.nl, 65, seed=7)).cuda()
    for prec in (PREC_FP64, PREC_DF):
        P = api.Plan(M, L, dict(grid=(16, 8, 8), n_touch=4))
        count = []

        def apply(R):
            before = P.launches()
            z = api.pfft_precond_apply(P, y[:R].contiguous(), om[:R], prec=prec)
            count.append(P.launches() - before)
            return z
        ref = apply(65)
        assert torch.equal(apply(64), ref[:64]) and count[1] == count[0], prec
        z = apply(64)
        assert not torch.equal(z, ref[:64])
        assert (torch.linalg.norm(z - ref[:64], dim=1) / torch.linalg.norm(ref[:64], dim=1)).max().item() < 1e-11
        assert torch.equal(apply(64), z)
        apply(65)                                    # other factors
        assert torch.equal(apply(64), ref[:64]), prec
