"""Moves of the footprint at the ends of their range: supports of one point and of the largest, rows and columns up
to the far corner of the largest grid, and moves by every small step.  Against the FP64 oracle, within the bars of
test_gpu_pairs.py (sums of FP32 products, 6e-8 each)."""
import numpy as np
import pytest
import torch

import oracle
import paper_1403_4209_gb300 as wg
from gpu_common import max_rel
from test_gpu_pairs import C0, _grid, _tables

pytestmark = pytest.mark.gpu


def _walk(N, h, rows, rng):
    """every move of up to three columns and rows in turn, back from the far corner, then jumps"""
    lim = N // 2 - h - 1
    steps = [(dx, dy) for dx in range(-3, 4) for dy in range(-3, 4)] * 2
    rng.shuffle(steps)
    pos, out = np.array([lim, lim]), []
    for r in range(rows):
        d = steps[r] if r < len(steps) else rng.integers(-min(lim, 60), min(lim, 60) + 1, 2)
        pos = np.clip(pos + d, max(-lim, lim - 70), lim)
        out.append([*(pos + rng.uniform(-0.3, 0.3, 2)), 0.0])
    return np.array(out)


@pytest.mark.parametrize("P", [1, 2, 4])
@pytest.mark.parametrize("S,N,rows", [(1, 64, 150), (3, 64, 150), (13, 128, 150), (27, 160, 150), (1023, 1200, 16)])
def test_every_small_move(S, N, rows, P):
    rng = np.random.default_rng(S + P)
    ref, tab = _tables([S], 1 if S > 500 else 2, S)
    uvw, freq = _walk(N, S // 2, rows, rng), np.array([C0])
    vis = (rng.normal(size=(rows, 1, P)) + 1j * rng.normal(size=(rows, 1, P))).astype(np.complex64)
    wt, fl = np.ones((rows, 1, P), np.float32), np.zeros((rows, 1, P), np.uint8)
    pl = oracle.place(uvw, freq, 1.0, N, ref, flag=fl)
    assert pl.griddable.all()
    batch = wg.VisBatch(*(torch.as_tensor(a, device="cuda") for a in (uvw, freq, vis, wt, fl)))
    y = (rng.normal(size=(1, N, N, P)) + 1j * rng.normal(size=(1, N, N, P))).astype(np.complex64)
    want, pred = oracle.grid_plain(pl, ref, vis, wt, fl, N), oracle.degrid(pl, ref, y.astype(np.complex128), wt, fl)
    for plan in (None, (32, 64, False), (256, 256, False)):
        g, work = _grid(tab, batch, P, N, 1, plan)
        assert max_rel(g.data.cpu().numpy(), want) < 1e-5
        g.data.copy_(torch.as_tensor(y))
        assert max_rel(wg.degrid_vis(g, tab, batch, work).cpu().numpy().reshape(-1, P), pred) < 1e-5


def test_far_corner_of_the_largest_grid():
    # rows and columns up to 32767: footprints are compared with those of a small grid, whose last 200 cells a side
    # hold the same numbers
    N, n, S, P, rows = 32768, 200, 9, 1, 300
    rng = np.random.default_rng(3)
    ref, tab = _tables([S], 2, 3)
    small = _walk(n, S // 2, rows, rng)
    big = small.copy()
    big[:, :2] += N // 2 - n // 2
    vis = (rng.normal(size=(rows, 1, P)) + 1j * rng.normal(size=(rows, 1, P))).astype(np.complex64)
    wt, fl, freq = np.ones((rows, 1, P), np.float32), np.zeros((rows, 1, P), np.uint8), np.array([C0])
    y = torch.randn((n, n, P), dtype=torch.complex64, device="cuda")
    out = []
    for uvw, side in ((small, n), (big, N)):
        batch = wg.VisBatch(*(torch.as_tensor(a, device="cuda") for a in (uvw, freq, vis, wt, fl)))
        g, work = _grid(tab, batch, P, side, 1, None)
        gridded = g.data[0, side - n:, side - n:].clone()
        assert g.data[0, :side - n].abs().max() == 0 if side > n else True
        g.data[0, side - n:, side - n:] = y
        out.append((gridded, wg.degrid_vis(g, tab, batch, work), work.stats()["griddable"]))
        del g, work
    assert out[0][2] == out[1][2] == rows
    for a, b in zip(out[0][:2], out[1][:2]):
        assert (a - b).abs().max() <= 1e-6 * a.abs().max()
