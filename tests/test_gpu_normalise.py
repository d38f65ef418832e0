"""Normalised signatures are the unnormalised ones times 1 / max (FP32, bit for bit),
for row lengths around a warp's share and what a CTA holds (1280 and 49152 values)
and beyond; a ROI without atoms stays zero."""
import numpy as np
import pytest

import paper_2009_00735_gb300 as apt

from test_gpu_plain import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [1, 31, 33, 1280, 1281, 10242, 40962, 49152, 49153, 51000])
def test_normalise_row_lengths(torch_cuda, nv):
    torch = torch_cuda
    rng = np.random.default_rng(nv)
    xyz = rng.uniform(-3, 3, (4000, 3)).astype(np.float32)
    i = np.arange(nv) + 0.5
    z, a = 1.0 - 2.0 * i / nv, i * np.pi * (3.0 - np.sqrt(5.0))
    dirs = np.stack([np.sqrt(1 - z * z) * np.cos(a), np.sqrt(1 - z * z) * np.sin(a), z], 1).astype(np.float32)
    centres, radii = np.array([[0, 0, 0], [1, 1, 1], [40, 0, 0]], float), np.array([1.0, 1.3, 1.0])
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_load_positions(h, torch.from_numpy(xyz).cuda())
    apt.aptidx_set_directions(h, dirs)
    apt.aptidx_set_binning(h, 8, 5, 8)
    apt.aptidx_set_rois(h, centres, radii)
    out = []
    for flags in (0, apt.APTIDX_NORMALISE_MAX):
        S = torch.full((3, nv), -1.0, device="cuda")
        apt.aptidx_compute_signatures(h, apt.APTIDX_PATH_PLAIN_FP32, flags, S)
        apt.aptidx_sync(h)
        out.append(S.cpu().numpy())
    ctx.close()
    raw, norm = out
    mx = raw.max(1)
    assert mx[0] > 0 and mx[1] > 0 and mx[2] == 0
    assert np.array_equal(norm[:2], raw[:2] * (np.float32(1) / mx[:2])[:, None])
    assert np.array_equal(norm[2], np.zeros(nv, np.float32))
