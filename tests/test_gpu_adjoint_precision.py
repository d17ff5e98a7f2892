"""The adjoint image of a fit (grid_correct, IMAGE_PER_POL_RAW) is as accurate as a complex FP32 transform of the same grid:
on the grid of a smooth sky's visibilities, peaked at its centre, its distance from the 64-bit image is at most a tenth
more than that of torch's complex64 FFT of that grid (one transform of the same length and precision; the products by
the taper round once more)."""
import numpy as np
import pytest
import torch

import paper_1403_4209_gb300 as wg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [1, 2])
@pytest.mark.parametrize("N", [512, 1024, 1500])
def test_adjoint_image_of_a_smooth_sky(N, P):
    dev, rng, du = "cuda", np.random.default_rng(N), 60.0
    tab = wg.ConvTable.build(du, 1, 0.0, 8, 7, supports=[9])
    # tracks: 300 baselines, denser towards short ones, 60 steps of an arc each, in cells
    r, a0 = np.abs(rng.normal(0, N / 10, 300)).clip(2, N / 2 - 12), rng.uniform(0, 2 * np.pi, 300)
    arc = a0[:, None] + np.linspace(0, 0.8, 60)[None]
    uvw = np.zeros((300 * 60, 3))
    uvw[:, 0], uvw[:, 1] = (r[:, None] * np.cos(arc)).ravel(), 0.7 * (r[:, None] * np.sin(arc)).ravel()
    uvw *= du * 299792458.0 / 1e8
    shape = (len(uvw), 1, P)
    weight, flag = torch.ones(shape, device=dev), torch.zeros(shape, dtype=torch.uint8, device=dev)
    model = wg.SkyModel(tab, torch.as_tensor(uvw, device=dev), torch.tensor([1e8], dtype=torch.float64, device=dev),
                        weight, flag, N, du)
    x = torch.arange(N, device=dev, dtype=torch.float64) - N / 2
    # one cell of a delta grid images the inverse of the taper alone, in FP32
    one = wg.Grid(N, du, 1, 1)
    one.data[0, N // 2, N // 2] = 1.0
    corr = 1.0 / wg.grid_correct(one, tab, mode=wg.IMAGE_PER_POL_RAW)[0, 0].double()
    sky = torch.exp(-(x[:, None] ** 2 + (x[None] + N / 16) ** 2) / (2 * (N / 24) ** 2))
    at = torch.as_tensor(rng.integers(N // 4, 3 * N // 4, (2, 40)), device=dev)
    sky[at[0], at[1]] += 100 * torch.as_tensor(rng.uniform(0, 1, 40), device=dev)
    image = (sky * corr).float().expand(1, P, N, N).contiguous()
    got = model.adjoint_image(model.forward_vis(image)).double() * corr
    sign = (-1.0) ** torch.arange(N, device=dev, dtype=torch.float64)
    sign = sign[:, None] * sign[None]
    grid = model.grid_adj.data.permute(0, 3, 1, 2)
    exact = torch.fft.ifft2(grid.to(torch.complex128) * sign, norm="forward").real * sign
    single = torch.fft.ifft2(grid * sign.to(torch.complex64), norm="forward").real.double() * sign
    err, ref = (got - exact).norm() / exact.norm(), (single - exact).norm() / exact.norm()
    assert err <= 1.1 * ref, (float(err), float(ref))
