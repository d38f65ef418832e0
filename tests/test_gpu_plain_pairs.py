"""The FP32 path projects one direction of an antipodal pair and folds its
spectrum about the middle of the histogram, where a histogram and its mirror
image give the same value bit for bit: pairs and APTIDX_DIRECT agree exactly,
also where atoms force a partner pass (projections that are exactly zero or an
exact whole number of bins), for every band parity, several bins counts, ROIs
above one staged block and above 65535 atoms, and the values match the oracle.
"""
import numpy as np
import pytest

import oracle
import synth
import paper_2009_00735_gb300 as apt

from test_gpu_plain import TOL_PLAIN, roi_error, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

PLAIN = apt.APTIDX_PATH_PLAIN_FP32


def box(n_big=0):
    rng = np.random.default_rng(5)
    q = synth.random_quaternions(rng, 1)[0]
    xyz, _ = synth.lattice_box("fcc", 0.404, (-2.5,) * 3, (2.5,) * 3, rot=synth.quat_to_matrix(q), origin=np.zeros(3))
    xyz = xyz + rng.normal(0, 0.02, xyz.shape)
    # at the first centre: its own position (every projection zero), atoms on the
    # axes at whole numbers of bins of R = 1 at 2^8 bins (scale 127)
    planted = np.array([[0, 0, 0], [0.5, 0, 0], [0, -1.0, 0], [0, 0, 0.25]])
    xyz = np.concatenate([xyz, planted])
    if n_big:
        xyz = np.concatenate([xyz, rng.uniform(-0.9, 0.9, (n_big, 3))])
    centres = np.array([[0.0, 0, 0], [0.31, -0.2, 0.11], [9.0, 9.0, 9.0]])
    return np.ascontiguousarray(xyz.astype(np.float32)), centres, np.array([1.0, 1.7, 1.0])


@pytest.mark.parametrize("m,band,n_big", [(8, (10, 11), 0), (8, (0, 3), 0), (8, (125, 128), 0), (9, (13, 13), 0),
                                          (10, (5, 90), 0), (10, (18, 21), 5000), (8, (7, 12), 70000), (11, (21, 24), 0),
                                          (12, (40, 47), 5000)])
def test_pairs_equal_direct(torch_cuda, m, band, n_big):
    torch = torch_cuda
    xyz, centres, radii = box(n_big)
    dirs = np.concatenate([synth.icosphere(2), [[1, 0, 0], [0, -1, 0], [0.6, 0.8, 0.0]]]).astype(np.float32)
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_load_positions(h, torch.from_numpy(xyz).cuda())
    apt.aptidx_set_directions(h, dirs)
    apt.aptidx_set_binning(h, m, band[0], band[1])
    apt.aptidx_set_rois(h, centres, radii)
    out = []
    for flags in (0, apt.APTIDX_DIRECT):
        S = torch.full((3, len(dirs)), -1.0, device="cuda")
        A = torch.zeros((3, len(dirs)), dtype=torch.uint16, device="cuda")
        apt.aptidx_compute_signatures(h, PLAIN, flags, S, A)
        apt.aptidx_sync(h)
        out.append((S.cpu().numpy(), A.cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    So, _, No = oracle.signatures(xyz, centres, radii, band[0], band[1], dirs, m)
    assert np.array_equal(out[0][0][2], np.zeros(len(dirs)))          # the empty ROI
    assert roi_error(out[0][0][:2], So[:2]).max() <= TOL_PLAIN
    ctx.close()
