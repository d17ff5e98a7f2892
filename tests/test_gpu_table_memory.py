"""The kernel table on the device: its memory, the order in which table_info gives its samples, and the samples that the
gridder reads, bit for bit.  A visibility of 1 of weight 1 alone on the grid leaves its sub-kernel there: 1 x sample + 0."""
import ctypes

import numpy as np
import pytest
import torch

import paper_1403_4209_gb300 as wg
from paper_1403_4209_gb300 import _lib
from test_gpu_pairs import C0, _tables

pytestmark = pytest.mark.gpu


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_table_memory_is_one_copy():
    sup = [251] * 40
    wg.ConvTable.build(0.01, 1, 0.0, 8, 7, supports=[7])                 # (the context's own allocations)
    before = _free()
    t = wg.ConvTable.build(0.01, len(sup), 50.0, 8, 7, supports=sup)     # 161 M samples, 1.29 GB
    one = 8 * t.n_samples
    used = before - _free()
    assert used <= 1.05 * one, (used, one)
    t.set_store("f16")
    assert before - _free() <= 1.05 * 1.5 * one
    t.set_store("f32")
    assert before - _free() <= 1.05 * one
    del t
    assert before - _free() <= 0.05 * one


def test_samples_in_their_order():
    ref, t = _tables([1, 5, 9, 33], 3, 4)
    assert np.array_equal(t.to_host()[0], ref.data.astype(np.complex64))
    for store, dtype in (("f32", None), ("bf16", torch.bfloat16), ("f16", torch.float16)):
        t.set_store(store)
        info = _lib.TableInfo()
        assert wg.lib.table_info(t.handle, ctypes.byref(info)) == 0
        assert (info.data_lp is None) == (store == "f32")
        got = torch.as_tensor(wg.api._DeviceBuffer(info.data, (t.n_samples, 2), "<f4"), device="cuda").cpu()
        want = torch.view_as_real(torch.as_tensor(ref.data.astype(np.complex64)))
        assert torch.equal(got, want)
        if dtype:
            lp = t.lp_samples().cpu().view(dtype).reshape(-1, 2)
            assert torch.equal(lp.view(torch.int16), want.to(dtype).view(torch.int16))


@pytest.mark.parametrize("store", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("supports", [[1], [3, 7], [9, 15, 33]], ids=str)
def test_gridded_samples_bit_for_bit(supports, store):
    beta, N = 3, 40 * len(supports) + 8 * max(supports)
    ref, t = _tables(supports, beta, 9)
    t.set_store(store)
    want = torch.view_as_real(torch.as_tensor(ref.data.astype(np.complex64)))
    if store != "f32":
        want = want.to(torch.bfloat16 if store == "bf16" else torch.float16).float()
    want = want.numpy()
    rng, S = np.random.default_rng(1), max(supports)
    for _ in range(12):
        k = int(rng.integers(len(supports)))
        uvw = np.array([[*rng.uniform(-3, 3, 2), ref.w_planes[k]]])
        batch = wg.VisBatch(*(torch.as_tensor(a, device="cuda") for a in
                              (uvw, np.array([C0]), np.ones((1, 1, 2), np.complex64), np.ones((1, 1, 2), np.float32),
                               np.zeros((1, 1, 2), np.uint8))))
        g, work = wg.Grid(N, 1.0, 2, 1), wg.WorkList(1, 1, 2)
        wg.vis_compress(g, t, batch, work)
        wg.grid_vis(g, t, work)
        x, _, z, w = work.view(1)[0][0].tolist()
        s = supports[w & 0xFFF]
        x0, y0 = x & 0xFFFF, x >> 16
        exp = np.zeros((N, N, 2), np.float32)
        exp[y0:y0 + s, x0:x0 + s] = want[z:z + s * s].reshape(s, s, 2)
        got = torch.view_as_real(g.data[0]).cpu().numpy()
        for p in range(2):
            assert np.array_equal(got[:, :, p], exp)


def test_table_info_while_a_stream_is_captured():
    # its first call makes the samples: neither the capture nor what it holds is disturbed
    ref, t = _tables([5, 9], 3, 6)
    t.set_store("f16")
    x = torch.zeros(4, device="cuda")
    graph = torch.cuda.CUDAGraph()
    info = _lib.TableInfo()
    with torch.cuda.graph(graph):
        x += 1
        rc = wg.lib.table_info(t.handle, ctypes.byref(info))
        x += 1
    assert rc == 0 and info.data and info.data_lp
    graph.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [2.0] * 4
    got = torch.as_tensor(wg.api._DeviceBuffer(info.data, (t.n_samples, 2), "<f4"), device="cuda").cpu()
    assert torch.equal(got, torch.view_as_real(torch.as_tensor(ref.data.astype(np.complex64))))
