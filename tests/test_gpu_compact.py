"""The work list over the shapes of a preparation tile: one to thousands of channels (tiles of 2048 rows down to one),
row counts that leave a ragged last tile, one to four polarisations, with and without compression.
Everything integer exact against the FP64 oracle, the sums within the bars of test_gpu_parity.py."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_parity import _check

pytestmark = pytest.mark.gpu


def _track(rows, C, P):
    """One baseline's smooth track on a 64 x 64 grid, every channel crossing cells and planes at its own rows."""
    rng = np.random.default_rng(rows * 7919 + C)
    th = 0.3 + 5e-4 * np.arange(rows)
    uvw = np.stack([900 * np.cos(th), 700 * np.sin(th), 1500 * np.sin(2 * th)], 1)
    shape = (rows, C, P)
    vis = torch.as_tensor((rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64))
    return synth.Workload("track", uvw, np.linspace(1.0e8, 2.0e8, C), vis,
                          torch.as_tensor(rng.uniform(0.5, 2.0, shape).astype(np.float32)),
                          torch.as_tensor((rng.random(shape) < 0.03).astype(np.uint8)), 64, 20.0, 4, 2000.0, 8, [5, 7, 9, 11], 5,
                          1, rows)


@pytest.mark.parametrize("compress", [False, True])
@pytest.mark.parametrize("P", [1, 2, 4])
@pytest.mark.parametrize("C,rows", [(1, 2050), (2, 1037), (3, 700), (5, 411), (16, 261), (33, 125), (130, 47), (513, 9), (700, 5),
                                    (1030, 3), (2100, 2)])
def test_tile_shapes(C, rows, P, compress):
    gp, _ = _check(_track(rows, C, P), compress=compress)
    assert len(np.unique(gp["entries"][:, 3] >> 16)) > 0.9 * C     # (the highest channels' w can pass the last plane)
