"""The image finaliser's half-plane transforms against plain FP64 FFTs of the same grids: every mode and
polarisation count at the smallest and odd-factored grid sides (Hermitian partners at index 0 and N/2),
a polarisation without data, the transpose, the w-stacking sum when a channel's planes
span transform groups, and an image buffer that is only float-aligned.  Images are compared after multiplying
taper x sinc back (towards the edges it divides by values down to 1e-4), within 1e-5 of their
peak: FP32 transforms of n points err by a few 6e-8 sqrt(log2 n)."""
import numpy as np
import pytest
import torch

import paper_1403_4209_gb300 as wg

pytestmark = pytest.mark.gpu

MODES = {"per_pol": wg.IMAGE_PER_POL, "raw": wg.IMAGE_PER_POL_RAW, "stokes_i": wg.IMAGE_STOKES_I,
         "linear": wg.IMAGE_STOKES_LINEAR, "circular": wg.IMAGE_STOKES_CIRCULAR}


def _table(du=0.02, K=1, stacking=False):
    return wg.ConvTable.build(du, K, 30.0 if K > 1 else 0.0, 8, 7, supports=[7] * K, stacking=stacking)


def _fft(x, inverse):
    x = torch.fft.ifftshift(x, dim=(-2, -1))
    return torch.fft.fftshift(torch.fft.ifft2(x, norm="forward") if inverse else torch.fft.fft2(x), dim=(-2, -1))


def _corr(tab, N):
    # taper x sinc from the library's own transpose of one bright pixel is circular; take it from a delta
    # grid instead: a constant image is 1 / (taper sinc) in the raw mode
    g = wg.Grid(N, tab.du, 1, 1)
    g.data[0, N // 2, N // 2, 0] = 1.0
    return 1.0 / wg.grid_correct(g, tab, mode=wg.IMAGE_PER_POL_RAW)[0, 0].double()


def _grid(tab, N, P, C, seed):
    g = wg.Grid(N, tab.du, P, C)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    torch.view_as_real(g.data).normal_(generator=gen)
    g.normaliser().copy_(torch.rand((C, P), generator=gen, device="cuda", dtype=torch.float64) + 0.5)
    return g


def _expected(g, mode):
    z = _fft(g.data.to(torch.complex128).permute(0, 3, 1, 2), True)
    P, n = g.n_pol, g.normaliser()
    if mode == "raw":
        return z.real
    z = z * torch.where(n != 0, 1 / n, torch.zeros_like(n))[:, :, None, None]
    if mode == "stokes_i":
        return 0.5 * (z[:, 0] + z[:, P - 1]).real
    if mode == "per_pol" or P == 1:
        return z.real
    if P == 2:
        return 0.5 * torch.stack([z[:, 0] + z[:, 1], z[:, 0] - z[:, 1]], 1).real
    par_s, par_d, crs_s, crs_d = z[:, 0] + z[:, 3], z[:, 0] - z[:, 3], z[:, 1] + z[:, 2], -1j * (z[:, 1] - z[:, 2])
    out = [par_s, par_d, crs_s, crs_d] if mode == "linear" else [par_s, crs_s, crs_d, par_d]
    return 0.5 * torch.stack(out, 1).real


@pytest.mark.parametrize("N", [8, 10, 54, 250])
@pytest.mark.parametrize("P", [1, 2, 4])
@pytest.mark.parametrize("mode", list(MODES))
def test_image_modes(mode, P, N):
    tab = _table()
    g = _grid(tab, N, P, 3, N + P)
    if P > 1:
        g.normaliser()[1, 0] = 0.0
    want = _expected(g, mode)
    got = wg.grid_correct(g, tab, mode=MODES[mode])
    flat = torch.empty(got.numel() + 1, device="cuda")
    odd = wg.grid_correct(g, tab, mode=MODES[mode], out=flat[1:].view(got.shape))
    assert torch.equal(odd, got)
    err = (got.double() * _corr(tab, N) - want).abs().max()
    assert float(err) < 1e-5 * float(want.abs().max())


@pytest.mark.parametrize("N", [8, 10, 54, 250])
@pytest.mark.parametrize("P", [1, 2, 4])
def test_transpose_also_when_first_called_under_capture(P, N):
    tab = _table()
    g = _grid(tab, N, P, 2, N)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(P)
    img = torch.randn((2, P, N, N), generator=gen, device="cuda")
    wg.grid_correct(g, tab, mode=wg.IMAGE_PER_POL)           # prepares the scratch, not the transpose's plan
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        wg.image_to_grid(g, tab, img)
    graph.replay()
    torch.cuda.synchronize()
    want = _fft((img.double() / _corr(tab, N)).to(torch.complex128), False).permute(0, 2, 3, 1)
    assert float((g.data - want).abs().max()) < 1e-5 * float(want.abs().max())


@pytest.mark.parametrize("N,P,K,C", [(54, 1, 5, 2), (54, 2, 3, 3), (1024, 4, 48, 1)])
def test_wstack_sum_over_groups(N, P, K, C):
    # the last case's 48 planes of 1024^2 x 4 take two transform groups of 24
    du = 0.6
    tab = _table(du=du, K=K, stacking=True)
    g = _grid(tab, N, P, C * K, K)
    got = wg.grid_correct(g, tab, mode=wg.IMAGE_WSTACK).double() * _corr(_table(du=du), N)
    lm = (torch.arange(N, device="cuda", dtype=torch.float64) - N // 2) / (N * du)
    r2 = lm[:, None] ** 2 + lm[None, :] ** 2
    nm1 = -r2 / (1 + torch.sqrt((1 - r2).clamp(min=0)))
    want = torch.zeros((C, P, N, N), dtype=torch.float64, device="cuda")
    for c in range(C):
        for k in range(K):
            z = _fft(g.data[c * K + k].to(torch.complex128).permute(2, 0, 1), True)
            w = 30.0 * (k / (K - 1)) ** 2
            want[c] += (z * torch.polar((r2 < 1).double(), 2 * np.pi * w * nm1)).real
        want[c] /= g.normaliser()[c * K][:, None, None]
    assert float((got - want).abs().max()) < 1e-5 * float(want.abs().max())
