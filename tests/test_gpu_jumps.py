"""Gridding of lists whose footprints jump about (k_grid_jumps), alone and beside smooth stretches in one list: moves of a
few columns and rows (which leave part of a footprint where it was), by exactly half a footprint's rows, and anywhere;
supports from one point to several task blocks and passes, plans, compensated flushes, non-finite visibilities.
Against the FP64 oracle, within the bars of test_gpu_pairs.py."""
import numpy as np
import pytest
import torch

import oracle
import paper_1403_4209_gb300 as wg
from gpu_common import max_rel, rel_l2
from test_gpu_pairs import _case as _walk_case
from test_gpu_pairs import _grid, _tables

pytestmark = pytest.mark.gpu


def _case(kind, supports, P, rows, seed):
    rng = np.random.default_rng(seed)
    h, H = max(supports) // 2, (max(supports) + 1) // 2
    N = 2 * (max(supports) + 30)
    lim = N // 2 - h - 1
    ref, tab = _tables(supports, 3, seed)
    step = {"few": lambda: rng.integers(-3, 4, 2), "half": lambda: np.array([rng.integers(-1, 2), rng.choice([-H, H])]),
            "any": lambda: rng.integers(-lim, lim + 1, 2)}
    uvw = np.empty((rows, 3))
    pos = np.zeros(2)
    for r in range(rows):
        smooth = kind == "mixed" and (r // 150) % 2 == 0
        d = rng.normal(0, 0.1, 2) if smooth else step[kind if kind != "mixed" else "few"]()
        pos = pos + d
        pos = np.where(np.abs(pos) > lim, -np.sign(pos) * lim * rng.random(2), pos)      # back from the edge
        uvw[r, :2] = pos + rng.uniform(-0.3, 0.3, 2)
    uvw[:, 2] = np.repeat(rng.uniform(-100, 100, -(-rows // 90)), 90)[:rows]
    vis = (rng.normal(size=(rows, 1, P)) + 1j * rng.normal(size=(rows, 1, P))).astype(np.complex64)
    wt = rng.uniform(0.5, 1.5, (rows, 1, P)).astype(np.float32)
    fl = (rng.random((rows, 1, P)) < 0.05).astype(np.uint8)
    freq = np.array([299792458.0])
    pl = oracle.place(uvw, freq, 1.0, N, ref, flag=fl)
    batch = wg.VisBatch(*(torch.as_tensor(a, device="cuda") for a in (uvw, freq, vis, wt, fl)))
    return ref, tab, pl, batch, vis, wt, fl, N


@pytest.mark.parametrize("kind", ["few", "half", "any", "mixed"])
@pytest.mark.parametrize("P", [1, 2, 4])
@pytest.mark.parametrize("supports", [[1], [7], [9, 15], [31, 45], [129]], ids=str)
def test_lists_of_jumps(supports, P, kind):
    ref, tab, pl, batch, vis, wt, fl, N = _case(kind, supports, P, 900, 11 * P + len(kind))
    want = oracle.grid_plain(pl, ref, vis, wt, fl, N)
    assert pl.griddable.sum() > 700
    for plan, comp in ((None, False), ((32, 64, False), False), ((256, 256, True), False), (None, True)):
        g, work = _grid(tab, batch, P, N, 1, plan, comp)
        got = g.data.cpu().numpy()
        assert rel_l2(got, want) < 1e-5 and max_rel(got, want) < 1e-5
        assert g.normaliser().cpu().numpy() == pytest.approx(oracle.normaliser(pl, ref, wt, fl), rel=1e-5)


@pytest.mark.parametrize("P", [1, 4])
def test_nonfinite_among_jumps(P):
    ref, tab, pl, batch, vis, wt, fl, N = _case("few", [9, 11], P, 400, 5)
    bad = np.nonzero(pl.griddable)[0][[3, 57, 58, 200]]
    hit = np.zeros((N, N), bool)
    for r, v in zip(bad, (np.inf, np.nan, -np.inf, np.nan)):
        batch.vis[int(r), 0, 0] = complex(v, 1.0)
        batch.flag[int(r), 0, 0] = 0
        batch.weight[int(r), 0, 0] = 1.0
        fl[r] = 1
        hit[pl.y0[r]:pl.y0[r] + pl.S[r], pl.x0[r]:pl.x0[r] + pl.S[r]] = True
    g = _grid(tab, batch, P, N, 1, None)[0].data.cpu().numpy()[0]
    assert not np.isfinite(g[..., 0][hit]).any() and np.isfinite(g[~hit]).all()
    pl0 = oracle.place(batch.uvw.cpu().numpy(), batch.freq.cpu().numpy(), 1.0, N, ref, flag=fl)
    want = oracle.grid_plain(pl0, ref, vis, wt, fl, N)[0, ..., 0]
    assert np.abs(g[..., 0][~hit] - want[~hit]).max() < 1e-5 * np.abs(want).max()


@pytest.mark.parametrize("supports", [[9], [1, 5, 9]], ids=str)
def test_tables_of_two_units(supports):
    # P = 4 with every support at most 9: the two-unit kernel, at its largest support (45 pairs)
    N = 60
    ref, tab, pl, batch, vis, wt, fl = _walk_case(supports, 4, N, 3000, 21, C=2)
    want = oracle.grid_plain(pl, ref, vis, wt, fl, N)
    for plan, comp in ((None, False), ((32, 64, False), False), ((256, 256, True), True)):
        got = _grid(tab, batch, 4, N, 2, plan, comp)[0].data.cpu().numpy()
        assert rel_l2(got, want) < 1e-5 and max_rel(got, want) < 1e-5


@pytest.mark.parametrize("kind", ["few", "half", "any", "mixed"])
@pytest.mark.parametrize("P", [1, 2, 4])
@pytest.mark.parametrize("supports", [[1], [7], [9, 15], [31, 45]], ids=str)
def test_degridding_lists_of_jumps(supports, P, kind):
    ref, tab, pl, batch, vis, wt, fl, N = _case(kind, supports, P, 900, 13 * P + len(kind))
    rng = np.random.default_rng(P)
    y = (rng.normal(size=(1, N, N, P)) + 1j * rng.normal(size=(1, N, N, P))).astype(np.complex64)
    want = oracle.degrid(pl, ref, y.astype(np.complex128), wt, fl)
    for plan in (None, (32, 64, False), (256, 256, True)):
        g, work = _grid(tab, batch, P, N, 1, plan)
        g.data.copy_(torch.as_tensor(y))
        got = wg.degrid_vis(g, tab, batch, work).cpu().numpy().reshape(-1, P)
        assert max_rel(got, want) < 1e-5
