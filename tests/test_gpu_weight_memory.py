"""vis_weight where memory for the density grid is all there is: the device's memory pool is limited to less than the
records' cells would take.  Weights of 1, so that densities are whole numbers and results equal bit for bit."""
import contextlib
import ctypes

import numpy as np
import pytest
import torch

import paper_1403_4209_gb300 as wg

pytestmark = pytest.mark.gpu


class _PoolProps(ctypes.Structure):                        # CUmemPoolProps
    _fields_ = [("allocType", ctypes.c_int), ("handleTypes", ctypes.c_int), ("locType", ctypes.c_int), ("locId", ctypes.c_int),
                ("security", ctypes.c_void_p), ("maxSize", ctypes.c_size_t), ("usage", ctypes.c_ushort),
                ("reserved", ctypes.c_ubyte * 54)]


@contextlib.contextmanager
def _pool_of(max_bytes):
    cu = ctypes.CDLL("libcuda.so.1")
    dev, old, pool = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_void_p()
    assert cu.cuDeviceGet(ctypes.byref(dev), torch.cuda.current_device()) == 0
    assert cu.cuDeviceGetMemPool(ctypes.byref(old), dev) == 0
    props = _PoolProps(allocType=1, locType=1, locId=dev.value, maxSize=max_bytes)
    assert cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert cu.cuDeviceSetMemPool(dev, pool) == 0
    try:
        yield
    finally:
        torch.cuda.synchronize()
        assert cu.cuDeviceSetMemPool(dev, old) == 0
        assert cu.cuMemPoolDestroy(pool) == 0


@pytest.mark.parametrize("scheme", ["uniform", "robust"])
@pytest.mark.parametrize("P,in_place", [(1, False), (2, True), (4, False)])
def test_weights_without_room_for_the_cells(P, in_place, scheme):
    N, rows, C = 512, 1500000, 32                          # densities 4 P MB a channel, cells 192 MB
    gen = torch.Generator(device="cuda")
    gen.manual_seed(P)
    tab = wg.ConvTable.build(1.0, 1, 0.0, 8, 7, supports=[7])
    uvw = torch.zeros((rows, 3), dtype=torch.float64, device="cuda")
    uvw[:, :2].uniform_(-N / 2, N / 2, generator=gen)      # some footprints leave the grid
    freq = torch.full((C,), 299792458.0, dtype=torch.float64, device="cuda")
    shape = (rows, C, P)
    batch = wg.VisBatch(uvw, freq, torch.zeros(shape, dtype=torch.complex64, device="cuda"), torch.ones(shape, device="cuda"),
                        (torch.rand(shape, generator=gen, device="cuda") < 0.05).to(torch.uint8))
    grid = wg.Grid(N, 1.0, P, 1)
    want = wg.vis_weight(grid, tab, batch, scheme=scheme, interleave=True)
    with _pool_of(96 << 20):
        got = wg.vis_weight(grid, tab, batch, scheme=scheme, interleave=True, out=batch.weight if in_place else None)
        torch.cuda.synchronize()
    assert torch.equal(got, want) and not torch.equal(want, torch.ones_like(want))
