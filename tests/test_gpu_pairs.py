"""The paired-point kernels at the sizes where their bookkeeping can go wrong: supports from one point
to several task blocks (ragged last units, supports whose blocks need a second pass), footprints on
every edge of the grid, walks that move by one column, one row, both, or jump, and segments shorter
than a warp's 32 entries.  Random kernel tables (no symmetry), so that a transposed, shifted or
mirrored sample shows.  Reference: the FP64 oracle on the same table and coordinates, held to
the parity tests' FP32 bar (1e-5 of the norm: sums of a few hundred FP32 products, 6e-8 each).

An infinite or NaN visibility reaches the pixels of its own footprint and no others; an infinite or
NaN pixel reaches the visibilities whose footprints hold it and no others."""
import numpy as np
import pytest
import torch

import oracle
import paper_1403_4209_gb300 as wg
from gpu_common import max_rel, rel_l2
from oracle.table import Table

pytestmark = pytest.mark.gpu

C0 = 299792458.0


def _tables(supports, beta, seed):
    rng = np.random.default_rng(seed)
    K = len(supports)
    n = beta * beta * np.asarray(supports, dtype=np.int64) ** 2
    off = np.concatenate([[0], np.cumsum(n)[:-1]])
    data = (rng.normal(size=n.sum()) + 1j * rng.normal(size=n.sum())).astype(np.complex64).astype(np.complex128)
    zeta = rng.uniform(0.5, 1.0, K * beta * beta)
    w_max = 100.0 if K > 1 else 0.0
    wp = w_max * (np.arange(K) / max(1, K - 1)) ** 2
    ref = Table(beta, np.asarray(supports, np.int32), off, data, zeta, wp, w_max)
    return ref, wg.ConvTable.from_host(K, beta, w_max, 1.0, 7, supports, data, zeta)


def _walk(rows, N, supports, rng):
    """cell coordinates that walk by small steps, sit on the grid's edges and jump"""
    h = max(supports) // 2
    lim = N // 2 - h - 1
    pos = rng.uniform(-lim, lim, 2)
    out = np.empty((rows, 3))
    for r in range(rows):
        kind = rng.random()
        if kind < 0.05:
            pos = rng.uniform(-lim, lim, 2)                       # a jump
        elif kind < 0.10:
            pos = rng.choice([-1.0, 1.0], 2) * (N // 2 - h)       # a corner, or just off the grid
        elif kind < 0.3:
            pos = pos + rng.choice([-1.0, 1.0]) * np.eye(2)[rng.integers(2)]
        else:
            pos = pos + rng.normal(0, 0.15, 2)                    # sub-cells
        pos = np.clip(pos, -(N // 2), N // 2)
        out[r, :2] = pos
    out[:, 2] = np.repeat(rng.uniform(-100, 100, -(-rows // 40)), 40)[:rows]
    return out


def _case(supports, P, N, rows, seed, beta=3, C=1):
    rng = np.random.default_rng(seed)
    ref, tab = _tables(supports, beta, seed)
    uvw, freq = _walk(rows, N, supports, rng), C0 * (1.0 - 0.01 * np.arange(C))
    vis = (rng.normal(size=(rows, C, P)) + 1j * rng.normal(size=(rows, C, P))).astype(np.complex64)
    wt = rng.uniform(0.5, 1.5, (rows, C, P)).astype(np.float32)
    fl = (rng.random((rows, C, P)) < 0.05).astype(np.uint8)
    pl = oracle.place(uvw, freq, 1.0, N, ref, flag=fl)
    dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    batch = wg.VisBatch(dev(uvw), dev(freq), dev(vis), dev(wt), dev(fl))
    return ref, tab, pl, batch, vis, wt, fl


def _grid(tab, batch, P, N, C, plan, comp=False):
    g = wg.Grid(N, 1.0, P, C, compensated=comp)
    work = wg.WorkList(batch.rows * C, C, P)
    if plan:
        work.plan(tab, *plan)
    wg.vis_compress(g, tab, batch, work)
    wg.grid_vis(g, tab, work)
    assert work.stats()["dropped"] == 0
    return g, work


SUPPORTS = [[1], [3], [5, 7], [9, 15, 17], [11, 39, 45], [65, 63], [129]]


@pytest.mark.parametrize("P", [1, 2, 4])
@pytest.mark.parametrize("supports", SUPPORTS, ids=str)
def test_gridding_of_edges_walks_and_jumps(supports, P):
    N, C = 2 * (max(supports) + 20), 2
    ref, tab, pl, batch, vis, wt, fl = _case(supports, P, N, 700, 5 * P + len(supports), C=C)
    want = oracle.grid_plain(pl, ref, vis, wt, fl, N)
    assert pl.griddable.sum() > 500
    for plan in (None, (32, 64, False), (256, 256, True)):
        g, _ = _grid(tab, batch, P, N, C, plan)
        got = g.data.cpu().numpy()
        assert rel_l2(got, want) < 1e-5 and max_rel(got, want) < 1e-5
    got = _grid(tab, batch, P, N, C, None, comp=True)[0].data.cpu().numpy()
    assert rel_l2(got, want) < 1e-5


@pytest.mark.parametrize("rows", [1, 31, 33, 5000])
def test_gridding_of_short_and_long_lists(rows):
    # from less than one warp's entries to more tasks than the device has warps
    supports, P, N = [33, 35], 4, 160
    ref, tab, pl, batch, vis, wt, fl = _case(supports, P, N, rows, rows)
    got = _grid(tab, batch, P, N, 1, None)[0].data.cpu().numpy()
    want = oracle.grid_plain(pl, ref, vis, wt, fl, N)
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)


@pytest.mark.parametrize("comp", [False, True])
@pytest.mark.parametrize("P", [1, 4])
def test_nonfinite_visibilities_stay_in_their_footprints(P, comp):
    supports, N = [9, 11], 96
    ref, tab, pl, batch, vis, wt, fl = _case(supports, P, N, 400, 77)
    bad = np.nonzero(pl.griddable)[0][[3, 57, 58, 200]]
    keep = np.ones(400, bool)
    keep[bad] = False
    hit = np.zeros((N, N), bool)
    for r, v in zip(bad, (np.inf, np.nan, -np.inf, np.nan)):
        batch.vis[int(r), 0, 0] = complex(v, 1.0)
        fl[r] = 1
        batch.flag[int(r), 0, 0] = 0
        batch.weight[int(r), 0, 0] = 1.0
        hit[pl.y0[r]:pl.y0[r] + pl.S[r], pl.x0[r]:pl.x0[r] + pl.S[r]] = True
    g = _grid(tab, batch, P, N, 1, None, comp)[0].data.cpu().numpy()[0]
    assert not np.isfinite(g[..., 0][hit]).any() and np.isfinite(g[~hit]).all()
    # polarisation 0 outside the footprints: the other records alone
    pl0 = oracle.place(batch.uvw.cpu().numpy(), batch.freq.cpu().numpy(), 1.0, N, ref, flag=fl)
    want = oracle.grid_plain(pl0, ref, vis, wt, fl, N)[0, ..., 0]
    assert np.abs(g[..., 0][~hit] - want[~hit]).max() < 1e-5 * np.abs(want).max()


@pytest.mark.parametrize("P", [1, 2, 4])
@pytest.mark.parametrize("supports", SUPPORTS, ids=str)
def test_degridding_of_edges_walks_and_jumps(supports, P):
    N, C = 2 * (max(supports) + 20), 2
    ref, tab, pl, batch, vis, wt, fl = _case(supports, P, N, 700, 9 * P + len(supports), C=C)
    rng = np.random.default_rng(P)
    y = (rng.normal(size=(C, N, N, P)) + 1j * rng.normal(size=(C, N, N, P))).astype(np.complex64)
    want = oracle.degrid(pl, ref, y.astype(np.complex128), wt, fl)
    for plan in (None, (32, 64, False), (256, 256, True)):
        g, work = _grid(tab, batch, P, N, C, plan)
        g.data.copy_(torch.as_tensor(y))
        got = wg.degrid_vis(g, tab, batch, work).cpu().numpy().reshape(-1, P)
        assert max_rel(got, want) < 1e-5


@pytest.mark.parametrize("P", [1, 4])
def test_nonfinite_pixels_stay_in_their_footprints(P):
    # one bad row of pixels: the records whose footprint touches it are not finite, the others are exact
    # (a footprint that ends on the row above it has that row in its pairs, with zero samples)
    supports, N = [9, 11], 96
    ref, tab, pl, batch, vis, wt, fl = _case(supports, P, N, 900, 31)
    rng = np.random.default_rng(5)
    y = (rng.normal(size=(1, N, N, P)) + 1j * rng.normal(size=(1, N, N, P))).astype(np.complex64)
    clean = oracle.degrid(pl, ref, y.astype(np.complex128), wt, fl)
    row = 50
    bad = y.copy()
    bad[0, row] = np.nan
    bad[0, row, ::2] = np.inf
    g, work = _grid(tab, batch, P, N, 1, None)
    g.data.copy_(torch.as_tensor(bad))
    got = wg.degrid_vis(g, tab, batch, work).cpu().numpy().reshape(-1, P)
    hit = pl.griddable & (pl.y0 <= row) & (pl.y0 + pl.S > row)
    assert hit.any() and (pl.griddable & (pl.y0 + pl.S == row)).any()
    assert not np.isfinite(got[hit]).any() and np.isfinite(got[~hit]).all()
    assert np.abs(got[~hit] - clean[~hit]).max() < 1e-5 * np.abs(clean).max()


def test_degridding_again_with_an_odd_number_of_entries():
    # the per-entry sums start at zero in every call, also the last entry's when the list's length is
    # odd at one polarisation
    supports, P, N = [9], 1, 64
    ref, tab, pl, batch, vis, wt, fl = _case(supports, P, N, 300, 3)
    g = wg.Grid(N, 1.0, P, 1)
    work = wg.WorkList(300, 1, P)
    for rows in (299, 300):              # one of the two lists has an odd length
        b = wg.VisBatch(batch.uvw[:rows], batch.freq, batch.vis[:rows], batch.weight[:rows], batch.flag[:rows])
        wg.vis_compress(g, tab, b, work, compress=False)
        g.data.fill_(1.0)
        first = wg.degrid_vis(g, tab, b, work).clone()
        assert torch.equal(wg.degrid_vis(g, tab, b, work), first)
