"""ROIs above 65535 atoms on the FP32 path run in passes, also when they pass that size
only with the atom types of a multi-signature call; smaller ones of the same call in one.
"""
import numpy as np
import pytest

import synth
import paper_2009_00735_gb300 as apt

from test_gpu_plain import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [8, 10, 11])
def test_large_only_with_more_types(torch_cuda, m):
    torch = torch_cuda
    rng = np.random.default_rng(m)
    n = 400000
    xyz = torch.from_numpy((20 * rng.random((n, 3))).astype(np.float32)).cuda()
    types = torch.from_numpy((rng.random(n) < 0.7).astype(np.uint8)).cuda()
    centres = np.array([[10.0, 10.0, 10.0], [6.0, 9.0, 12.0]])
    radii = np.array([7.5, 2.0])            # 88000 atoms, 26500 of type 0; 1700
    u = synth.icosphere(1).astype(np.float32)
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_load_positions(h, xyz, types)
    apt.aptidx_set_directions(h, u)
    apt.aptidx_set_binning(h, m, 5, 9)
    apt.aptidx_set_rois(h, centres, radii, type_mask=1)
    S = torch.empty(2, 2, len(u), device="cuda")
    N = torch.empty(2, 2, dtype=torch.int32, device="cuda")
    apt.aptidx_compute_signatures_multi(h, apt.APTIDX_PATH_PLAIN_FP32, 0, [1, 3], [5, 5], [9, 9], S, None, N)
    assert int(N[1, 0]) > 65535 > int(N[0, 0])
    for s, mask in ((0, 1), (1, 3)):
        apt.aptidx_set_rois(h, centres, radii, type_mask=mask)
        want = torch.empty(2, len(u), device="cuda")
        apt.aptidx_compute_signatures(h, apt.APTIDX_PATH_PLAIN_FP32, 0, want, None, None)
        # the ROI's band alone and a set of bands: the same sums (other passes where the
        # larger ROI is not in the call: FP32 rounding of 1e5 terms of either order)
        assert torch.allclose(S[s], want, rtol=2e-6, atol=1e-2)
    ctx.close()
