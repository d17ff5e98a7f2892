"""grid_autotune's default list times each plan once: plans that differ only in a flag without effect are one plan."""
import pytest
import torch

import paper_1403_4209_gb300 as wg
import synth
from gpu_common import run_gpu

pytestmark = pytest.mark.gpu


def test_default_list_times_each_plan_once():
    wl = synth.make("w0_small", n_times=8)
    g, t, batch, work = run_gpu(wl)["objects"]
    launches = []
    for f in (lambda: work.plan(t, 64, 128), lambda: wg.grid_vis(g, t, work)):
        n = wg.launch_count()
        f()
        launches.append(wg.launch_count() - n)
    n = wg.launch_count()
    seg, slots, fixed_r, ms = wg.grid_autotune(g, t, work, repeats=1)
    torch.cuda.synchronize()
    # three segment lengths by two task sizes, each planned, warmed up and timed; then the best is planned
    assert wg.launch_count() - n == 6 * (launches[0] + 2 * launches[1]) + launches[0]
    assert seg in (64, 128, 256) and slots in (128, 256) and not fixed_r and ms > 0
