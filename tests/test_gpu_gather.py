"""GPU parity of the ROI gather (step a1) where its FP32 decision is at its
limit: atoms on the sphere and one unit in the last place off it, coordinates far
from the origin (FP32 spacing comparable with the shell), ROIs larger than the
kept member masks, ROIs partly and wholly outside the box, and slots laid out for
a wider type mask.  Membership and centred coordinates are exact: no tolerance.
"""
import numpy as np
import pytest

import oracle
import synth
import paper_2009_00735_gb300 as apt

from test_gpu_plain import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def rows(a):
    return a[np.lexsort(a.T[::-1])] if len(a) else a


def shell_case(offset, R, n, seed):
    """Atoms in a ball around offset; a third of them at distance R of the first
    centre up to a few units in the last place."""
    rng = np.random.default_rng(seed)
    c = np.asarray(offset, float)
    d = rng.standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    rad = 1.6 * R * rng.random(n) ** (1 / 3)
    rad[::3] = R
    xyz = (c + d * rad[:, None]).astype(np.float32)
    k = np.arange(0, n, 6)
    xyz[k] = np.nextafter(xyz[k], np.float32(np.inf) * np.sign(d[k]).astype(np.float32))
    centres = np.stack([c, c + 0.3 * R, c + np.array([1.5 * R, 0, 0]), c + 10.0 * R, xyz[0].astype(float)])
    return xyz, np.ascontiguousarray(centres), np.array([R, 0.5 * R, R, R, 0.9 * R])


@pytest.mark.parametrize("offset,R,n", [((0, 0, 0), 1.0, 3000), ((1000.0, -2000.0, 3.0), 2.0, 20000),
                                        ((3.0e5, 3.0e5, -3.0e5), 1.0, 5000), ((0.1, 0.2, 0.3), 1e-4, 500),
                                        ((5, 5, 5), 40.0, 400000), ((5, 5, 5), 1.0, 1)])
def test_members_and_centred_coordinates(torch_cuda, offset, R, n):
    torch = torch_cuda
    xyz, centres, radii = shell_case(offset, R, n, 7)
    types = (np.arange(n) % 3).astype(np.uint8)
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_load_positions(h, torch.from_numpy(xyz).cuda(), torch.from_numpy(types).cuda())
    apt.aptidx_set_directions(h, synth.icosphere(0))
    apt.aptidx_set_binning(h, 8, 3, 9)
    for mask in (0xFFFFFFFF, 0b101):
        apt.aptidx_set_rois(h, centres, radii, type_mask=mask)
        for r in range(len(radii)):
            got = apt.aptidx_get_roi_atoms(h, r)
            _, want = oracle.gather(xyz, centres[r], radii[r], types=types, type_mask=mask)
            assert np.array_equal(rows(got), rows(np.asarray(want, np.float32)))
    # a call over wider masks lays the slots out for their union; the
    # narrower selection of the context still comes back unchanged
    S0 = torch.empty((len(radii), 12), device="cuda")
    S1 = torch.empty_like(S0)
    Sm = torch.empty((2, len(radii), 12), device="cuda")
    apt.aptidx_compute_signatures(h, apt.APTIDX_PATH_PLAIN_FP32, 0, S0)
    apt.aptidx_compute_signatures_multi(h, apt.APTIDX_PATH_PLAIN_FP32, 0, [0b111, 0b101], [3, 3], [9, 9], Sm)
    apt.aptidx_compute_signatures(h, apt.APTIDX_PATH_PLAIN_FP32, 0, S1)
    apt.aptidx_sync(h)
    assert torch.equal(S0, S1) and torch.equal(Sm[1], S0)
    _, want = oracle.gather(xyz, centres[0], radii[0], types=types, type_mask=0b101)
    assert len(apt.aptidx_get_roi_atoms(h, 0)) == len(want)
    ctx.close()


def test_order_is_largest_first_for_any_count(torch_cuda):
    """Uneven counts, empty ROIs among them: every ROI is computed once."""
    torch = torch_cuda
    rng = np.random.default_rng(3)
    xyz = (rng.random((40000, 3)) * 12).astype(np.float32)
    n = 2500
    centres = rng.random((n, 3)) * 14 - 1
    radii = 0.05 + 1.2 * rng.random(n) ** 3
    dirs = synth.icosphere(1)
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_load_positions(h, torch.from_numpy(xyz).cuda())
    apt.aptidx_set_directions(h, dirs)
    apt.aptidx_set_binning(h, 8, 0, 0)      # X(0) = N_w
    apt.aptidx_set_rois(h, centres, radii)
    S = torch.full((n, len(dirs)), -1.0, device="cuda")
    N = torch.empty(n, dtype=torch.int32, device="cuda")
    for path in (apt.APTIDX_PATH_PLAIN_FP32, apt.APTIDX_PATH_TC_FP16):
        apt.aptidx_compute_signatures(h, path, 0, S, None, N)
        apt.aptidx_sync(h)
        assert torch.equal(S, N[:, None].float().expand_as(S))
        S.fill_(-1.0)
    ctx.close()
