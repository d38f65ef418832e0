"""Wide bands on the tensor cores against the FP64 oracle: odd and even numbers of
frequency groups up to the largest, 2^8 to 2^12 bins (one chunk of bins and several),
ROIs of one atom block and of several, per-ROI bands of uneven width in one call,
several bands per contraction, directions with and without antipodes, empty ROIs,
atoms that force partner passes."""
import numpy as np
import pytest

import oracle
import synth
import paper_2009_00735_gb300 as apt

from test_gpu_plain import roi_error, torch_cuda  # noqa: F401
from test_gpu_plain_pairs import box

pytestmark = pytest.mark.gpu

TC = apt.APTIDX_PATH_TC_FP16
TOL = 5e-3      # the path's stated tolerance


def run(torch, xyz, centres, radii, dirs, m, lo, hi):
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_load_positions(h, torch.from_numpy(xyz).cuda())
    apt.aptidx_set_directions(h, dirs)
    apt.aptidx_set_binning(h, m, int(np.min(lo)), int(np.max(hi)))
    apt.aptidx_set_rois(h, centres, radii, lo, hi)
    S = torch.full((len(radii), len(dirs)), -1.0, device="cuda")
    A = torch.zeros((len(radii), len(dirs)), dtype=torch.uint16, device="cuda")
    apt.aptidx_compute_signatures(h, TC, 0, S, A)
    apt.aptidx_sync(h)
    S, A = S.cpu().numpy(), A.cpu().numpy()
    ctx.close()
    return S, A


@pytest.mark.parametrize("m,n_big", [(8, 0), (10, 0), (11, 0), (12, 0), (10, 5000), (12, 5000)])
def test_group_counts(torch_cuda, m, n_big):
    xyz, centres, radii = box(n_big)
    dirs = np.concatenate([synth.icosphere(2), [[0.6, 0.8, 0.0]]]).astype(np.float32)
    for k_lo, width in [(3, 4 * 9 - 1), (8, 4 * 15), (2, 4 * 16 + 1), (5, 4 * 17 - 2), (0, 4 * 24), (8, 120)]:
        lo, hi = np.full(3, k_lo, np.int32), np.full(3, min(k_lo + width, 1 << (m - 1)), np.int32)
        S, A = run(torch_cuda, xyz, centres, radii, dirs, m, lo, hi)
        So, Ao, _ = oracle.signatures(xyz, centres, radii, lo, hi, dirs, m)
        assert np.array_equal(S[2], np.zeros(len(dirs)))
        assert roi_error(S[:2], So[:2]).max() <= TOL
        assert (A[:2] == Ao[:2]).mean() > 0.99
        assert np.all((A >= lo[0]) & (A <= hi[0]))


@pytest.mark.parametrize("m", [9, 10, 11])
def test_uneven_bands_and_repeat(torch_cuda, m):
    """Bands of 1 to 31 groups in one call, many tiles per CTA; the same call
    twice gives the same bits."""
    rng = np.random.default_rng(m)
    xyz, _, _ = box()
    n = 400
    centres, radii = rng.uniform(-1.2, 1.2, (n, 3)), rng.uniform(0.5, 1.2, n)
    lo = rng.integers(0, 60, n).astype(np.int32)
    hi = (lo + rng.integers(0, 4 * 31 - 60, n)).astype(np.int32)
    dirs = synth.icosphere(3)
    S, A = run(torch_cuda, xyz, centres, radii, dirs, m, lo, hi)
    S2, A2 = run(torch_cuda, xyz, centres, radii, dirs, m, lo, hi)
    assert np.array_equal(S, S2) and np.array_equal(A, A2)
    So, Ao, _ = oracle.signatures(xyz, centres, radii, lo, hi, dirs, m)
    assert roi_error(S, So).max() <= TOL
    assert (A == Ao).mean() > 0.99


@pytest.mark.parametrize("m", [10, 12])
def test_several_bands(torch_cuda, m):
    torch = torch_cuda
    xyz, centres, radii = box()
    dirs = synth.icosphere(2)
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_load_positions(h, torch.from_numpy(xyz).cuda())
    apt.aptidx_set_directions(h, dirs)
    apt.aptidx_set_binning(h, m, 10, 20)
    apt.aptidx_set_rois(h, centres, radii)
    lo, hi = [2, 40, 77, 10], [9, 90, 77, 100]
    S = torch.empty((4, 3, len(dirs)), device="cuda")
    apt.aptidx_compute_signatures_multi(h, TC, 0, [0xFFFFFFFF] * 4, lo, hi, S)
    apt.aptidx_sync(h)
    for b in range(4):
        So, _, _ = oracle.signatures(xyz, centres, radii, lo[b], hi[b], dirs, m)
        assert roi_error(S[b, :2].cpu().numpy(), So[:2]).max() <= TOL
    ctx.close()
