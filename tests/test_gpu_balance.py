"""A call whose work items are about as many as the SMs takes the same time from launch
to launch: no SM holds two of them while another has none (claimed ahead, a third of the
launches took twice as long).
"""
import numpy as np
import pytest

import synth
import paper_2009_00735_gb300 as apt

from test_gpu_plain import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level,nroi", [(4, 150), (5, 38), (6, 20)])
def test_launches_take_the_same_time(torch_cuda, level, nroi):
    torch = torch_cuda
    rng = np.random.default_rng(level)
    xyz = torch.from_numpy((24 * rng.random((470000, 3))).astype(np.float32)).cuda()
    u = synth.icosphere(level).astype(np.float32)
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_load_positions(h, xyz)
    apt.aptidx_set_directions(h, u)
    apt.aptidx_set_binning(h, 10, 20, 23)
    apt.aptidx_set_rois(h, 3.0 + 18.0 * rng.random((nroi, 3)), np.full(nroi, 2.6))
    S = torch.empty(nroi, len(u), device="cuda")
    e = [torch.cuda.Event(enable_timing=True) for _ in range(81)]
    for _ in range(3):
        apt.aptidx_compute_signatures(h, apt.APTIDX_PATH_TC_FP16, 0, S, None, None)
    torch.cuda.synchronize()
    e[0].record()
    for i in range(80):
        apt.aptidx_compute_signatures(h, apt.APTIDX_PATH_TC_FP16, 0, S, None, None)
        e[i + 1].record()
    torch.cuda.synchronize()
    t = np.sort([e[i].elapsed_time(e[i + 1]) for i in range(80)])
    assert t[71] < 1.4 * t[0], t      # nine in ten
    ctx.close()
