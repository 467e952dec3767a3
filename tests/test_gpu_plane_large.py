"""The FP32 convolution of planes larger than one CTA's padded form, every size it
is built for, with one grid, an odd number and several per CTA, against the same
zero-padded convolution by torch.fft in FP64: 2e-6 relative 2-norm per grid, the
mixed convolution's bar, and element by element within 2e-5 of the largest."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_04891_gb300 import api, PREC_MIXED  # noqa: E402


@pytest.mark.parametrize("grid", [(8, 256, 8), (32, 256, 16), (8, 256, 32), (16, 128, 32)],
                         ids=lambda g: "x".join(map(str, g)))
def test_large_plane_convolution(grid):
    m = synth.tiny_bar()
    M = api.Mesh.from_synth(m)
    P = api.Plan(M, api.Loops(M, m.ports), dict(grid=grid, n_touch=4))
    h = (m.xyz.max(0) - m.xyz.min(0)) / (np.array(grid) - 1)
    ax = [torch.from_numpy(np.minimum(np.arange(2 * n), 2 * n - np.arange(2 * n)) * s).cuda() for n, s in zip(grid, h)]
    r = torch.sqrt(ax[0][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[2][None, None, :] ** 2)
    r[0, 0, 0] = np.inf
    H = torch.fft.fftn(1.0 / r)
    for nb in (1, 5, 3 * 152 * 8 * 3 // (2 * grid[0])):   # the last: several grids per CTA
        g = torch.Generator(device="cuda").manual_seed(nb)
        q = torch.randn(nb, *grid, dtype=torch.complex64, device="cuda", generator=g)
        y = api.pfft_convolve(P, q.clone(), PREC_MIXED)
        for b in sorted({0, nb // 2, nb - 1}):
            ref = torch.fft.ifftn(torch.fft.fftn(q[b].to(torch.complex128), s=H.shape) * H)
            ref = ref[:grid[0], :grid[1], :grid[2]]
            d = y[b].to(torch.complex128) - ref
            assert (torch.linalg.norm(d) / torch.linalg.norm(ref)).item() < 2e-6, (nb, b)
            assert (d.abs().max() / ref.abs().max()).item() < 2e-5, (nb, b)
