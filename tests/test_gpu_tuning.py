"""A launch configuration picked by APTIDX_AUTOTUNE serves the calls of the shape it was
timed on: other ROI sets, bin counts and bands of the same context run as in a context
that never tuned, and the tuned shape has it again when it returns.
"""
import numpy as np
import pytest

import synth
import paper_2009_00735_gb300 as apt

from test_gpu_plain import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

TC, PLAIN = apt.APTIDX_PATH_TC_FP16, apt.APTIDX_PATH_PLAIN_FP32


def test_tuned_configuration_keeps_to_its_shape(torch_cuda, monkeypatch):
    torch = torch_cuda
    monkeypatch.delenv("APTIDX_TUNE_CACHE", raising=False)
    rng = np.random.default_rng(1)
    xyz = torch.from_numpy((20 * rng.random((272000, 3))).astype(np.float32)).cuda()
    u = synth.icosphere(5).astype(np.float32)
    many = 2.0 + 16.0 * rng.random((1500, 3))
    few = many[:16]

    def open_context():
        ctx = apt.Context(0)
        apt.aptidx_load_positions(ctx.handle, xyz)
        apt.aptidx_set_directions(ctx.handle, u)
        apt.aptidx_set_binning(ctx.handle, 8, 9, 11)
        return ctx

    def place(h, c):
        apt.aptidx_set_rois(h, c, np.full(len(c), 1.0))

    def compute(h, c, path, flags=0):
        S = torch.empty(len(c), len(u), device="cuda")
        apt.aptidx_compute_signatures(h, path, flags, S, None, None)
        apt.aptidx_sync(h)
        return S

    fresh, tuned = open_context(), open_context()
    place(fresh.handle, few)
    place(tuned.handle, many)
    for path in (TC, PLAIN):
        compute(tuned.handle, many, path, apt.APTIDX_AUTOTUNE)
    best = [apt.aptidx_get_tuning(tuned.handle, p) for p in (TC, PLAIN)]
    assert best[0][0] in (4, 8, 16, 32, 64) and best[0][1] in (2, 4)
    place(tuned.handle, few)
    for path in (TC, PLAIN):
        want = compute(fresh.handle, few, path)
        got = compute(tuned.handle, few, path)
        assert apt.aptidx_get_tuning(tuned.handle, path) == apt.aptidx_get_tuning(fresh.handle, path)
        assert torch.equal(got, want)
    # 16 ROIs of 81 tiles: 9 tiles per item give one wave over 152 SMs, as no candidate does
    assert apt.aptidx_get_tuning(tuned.handle, TC)[0] not in (4, 8, 16, 32, 64)
    place(tuned.handle, many)
    assert [apt.aptidx_get_tuning(tuned.handle, p) for p in (TC, PLAIN)] == best
    apt.aptidx_set_binning(tuned.handle, 9, 9, 11)
    place(tuned.handle, many)
    assert apt.aptidx_get_tuning(tuned.handle, PLAIN)[0] == 16
    fresh.close()
    tuned.close()
