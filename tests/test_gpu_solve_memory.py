"""Solves near the end of device memory: what only speeds the preconditioner up (the
chunk matrices of the narrow band's sweeps) leaves a solve its memory.  The free
memory is set to what the same solve took before, less a part of the matrices (pools
grow in steps of tens of MB: a third leaves the solve room and the matrices none)."""
import contextlib

import numpy as np
import pytest

import synth
from synth.meshes import box_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_04891_gb300 import api, native, PREC_FP64  # noqa: E402

NF = 64
FREQS = np.logspace(8.5, 9.5, NF)


def bar():
    m = box_mesh(400 * 8e-6, 20e-6, 10e-6, 400, 2, 1, jitter=0.1, seed=4)
    M = api.Mesh.from_synth(m)
    return M, api.Loops(M, m.ports)


def plan(M, L):
    return api.Plan(M, L, dict(grid=(64, 8, 8), n_touch=4))


def matrix_bytes(P):
    i = api.precond_info(P)
    assert i["blocks"] == 1 and i["band_width"] <= 31
    return NF * 2 * -(-i["unknowns"] // 32) * (i["band_width"] + 32) * 32 * 16


def free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


@contextlib.contextmanager
def only(left):
    """Holds all device memory but `left` bytes."""
    hold = torch.empty(free() - left, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del hold
        torch.cuda.empty_cache()


def solve(P, restart):
    return api.sie_solve(P, FREQS, tol=1e-6, restart=restart, prec=PREC_FP64)


def test_workspace_goes_before_the_matrices():
    M, L = bar()
    solve(plan(M, L), 40)                         # kernels loaded
    P = plan(M, L)
    f0 = free()
    Z, st = solve(P, 40)
    need, mats = f0 - free(), matrix_bytes(P)
    assert st["converged"] and mats > 200 << 20
    del P
    P = plan(M, L)
    with only(need - mats // 3):
        Z2, st = solve(P, 40)
    assert st["converged"] and np.abs(Z2 - Z).max() < 1e-5 * np.abs(Z).max()


def test_matrices_give_way_to_a_larger_workspace():
    M, L = bar()
    P = plan(M, L)
    Z, _ = solve(P, 40)
    mats = matrix_bytes(P)
    per_vector = NF * L.nl * 16
    restart = 40 + int(1.5 * mats) // per_vector
    larger = (restart + 1) * per_vector + NF * restart * (restart + 1) * 16   # basis and Hessenberg
    with only(larger - mats // 2):
        Z2, st = solve(P, restart)
    assert st["converged"] and np.abs(Z2 - Z).max() < 1e-5 * np.abs(Z).max()


def test_preconditioner_after_a_growth_that_failed():
    M, L = bar()
    P = plan(M, L)
    om = 2 * np.pi * 1e9
    y = torch.from_numpy(synth.complex_gaussian(L.nl, 2, seed=5)).cuda()
    z = api.pfft_precond_apply(P, y, om)
    many = torch.zeros(8000, L.nl, dtype=torch.complex128, device="cuda")
    out = torch.empty_like(many)
    with only(200 << 20), pytest.raises(native.SieError):
        api.pfft_precond_apply(P, many, om, out=out)
    assert torch.equal(api.pfft_precond_apply(P, y, om), z)


def test_batch_solve_gives_the_matrices_back():
    M, L = bar()
    P = [plan(M, L), plan(M, L)]
    B = api.Batch(P)
    B.solve([FREQS[:2]] * 2, restart=4, graph=True)
    f0 = free()
    ref = B.solve([FREQS, FREQS], restart=40, graph=True)
    need, mats = f0 - free(), matrix_bytes(P[0])
    del B, P
    P = [plan(M, L), plan(M, L)]
    B = api.Batch(P)
    B.solve([FREQS[:2]] * 2, restart=4, graph=True)
    with only(need - mats - mats // 3):
        out = B.solve([FREQS, FREQS], restart=40, graph=True)
    for (Z, _), (Z2, st) in zip(ref, out):
        assert st["converged"] and np.abs(Z2 - Z).max() < 1e-5 * np.abs(Z).max()
