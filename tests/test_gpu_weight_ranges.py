"""vis_weight over polarisation counts, weights from 1e-28 to 1e22 (the robust quotient's FP32 form and
its FP64 form on either side of its range), and weight and flag arrays that are only aligned to their
elements.  Reference: oracle/weighting.py, FP64; every new weight within 1e-6 relative, for cells of a few
records each (FP32 sums of a few terms, one rounding of the quotient)."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
import paper_1403_4209_gb300 as wg
import synth
from gpu_common import gpu_table, oracle_table
from oracle.weighting import reweight

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme,robust", [("uniform", 0.0), ("robust", -2.0), ("robust", 0.5)])
@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("P", [1, 2, 4])
@pytest.mark.parametrize("scale", [1e-28, 1.0, 1e22])
def test_weights_over_their_range(P, scale, aligned, scheme, robust):
    base = synth.make("degrid_1k", n_times=5, n_chan=3, n_baselines=200, flag_frac=0.05)
    sel = {1: [0], 2: [0, 3], 4: [0, 1, 2, 3]}[P]
    wl = dataclasses.replace(base, vis=base.vis[..., sel].contiguous(), weight=base.weight[..., sel].contiguous(),
                             flag=base.flag[..., sel].contiguous())
    rng = np.random.default_rng(P)
    w = (scale * rng.uniform(0.5, 2.0, wl.weight.shape)).astype(np.float32)

    def dev(a):
        t = torch.as_tensor(a, device="cuda")
        if aligned:
            return t
        flat = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")
        flat[1:] = t.reshape(-1)
        return flat[1:].view(t.shape)

    t = gpu_table(wl)
    g = wg.Grid(wl.n_grid, wl.du, P, wl.n_chan)
    b = wg.VisBatch(torch.as_tensor(wl.uvw, device="cuda"), torch.as_tensor(wl.freq, device="cuda"), wl.vis.cuda(), dev(w),
                    dev(wl.flag.numpy()))
    assert (b.weight.data_ptr() % 16 == 0) == aligned
    got = wg.vis_weight(g, t, b, scheme=scheme, robust=robust).cpu().numpy().reshape(-1, P).astype(np.float64)
    pl = oracle.place(wl.uvw, wl.freq, wl.du, wl.n_grid, oracle_table(wl), flag=wl.flag.numpy())
    exp = reweight(pl, w, wl.flag.numpy(), wl.n_grid, scheme, robust=robust)
    ok = pl.griddable
    assert ok.sum() > 1000
    assert np.max(np.abs(got[ok] - exp[ok]) / np.abs(exp[ok]).clip(1e-45)) < 1e-6
    assert np.array_equal(got[~ok], w.reshape(-1, P)[~ok].astype(np.float64))
