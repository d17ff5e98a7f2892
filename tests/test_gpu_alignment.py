"""Buffers aligned to their elements and no further, as views into a program's larger arrays are: every
entry point that takes one answers as it does for an aligned copy."""
import pytest
import torch

import paper_1403_4209_gb300 as wg
from test_gpu_pairs import _case, _grid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [wg.DEGRID_PREDICT, wg.DEGRID_ADJOINT])
@pytest.mark.parametrize("P", [1, 2, 4])
def test_degridding_into_an_odd_element(P, mode):
    N, C = 48, 3
    ref, tab, pl, batch, vis, wt, fl = _case([7, 9], P, N, 301, P, C=C)
    g, work = _grid(tab, batch, P, N, C, None)
    want = wg.degrid_vis(g, tab, batch, work, mode)
    flat = torch.full((vis.size + 2,), 7.0 + 7.0j, dtype=torch.complex64, device="cuda")
    out = flat[1:-1].view(vis.shape)
    assert out.data_ptr() % 16 == 8
    wg.degrid_vis(g, tab, batch, work, mode, out=out)
    # the entries' sums come from atomics, whose order varies by an ulp or two of the largest sum
    assert (out - want).abs().max() <= 1e-6 * want.abs().max()
    assert flat[0] == 7.0 + 7.0j and flat[-1] == 7.0 + 7.0j
