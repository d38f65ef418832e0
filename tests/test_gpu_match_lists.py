"""Eq. 3 of many ROIs runs on estimates from per-tile lists and decides by sums
in k order; of one ROI it runs the kernel that sums in k order throughout.  Both
give the same orientations and scores bit for bit: random and smooth rows,
constant rows (every orientation ties), zero rows, rows with infinities and NaN,
ROI counts around the groups of 32, table sizes off every multiple, direction
counts of one and several tiles.
"""
import numpy as np
import pytest

import synth
import paper_2009_00735_gb300 as apt

from test_gpu_lut import spiral
from test_gpu_plain import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def rows(u, sig, n, seed):
    rng = np.random.default_rng(seed)
    S = (sig[None] * rng.random((n, 1)) + 0.2 * rng.random((n, len(u)))).astype(np.float32)
    S[1] = 0.25                        # every orientation ties
    S[2] = 0.0
    S[3] = np.round(S[3] * 4) / 4      # few distinct terms: many near ties
    S[4, ::3] = np.inf
    S[5, 7] = np.nan
    S[6] = np.nan
    S[7] = 1e-25                       # squares underflow
    S[8] = 3e18                        # sums overflow
    return S


@pytest.mark.parametrize("nv,ng,n_hat,nroi", [(2562, 1001, 299, 170), (1752, 777, 33, 3000), (1753, 2500, 130, 161),
                                              (10242, 3301, 101, 193), (40962, 999, 301, 160),
                                              # large enough that the lists serve match and the shorter topk
                                              (2562, 2501, 299, 3000), (1753, 2500, 330, 2900),
                                              (10242, 3301, 401, 1500), (40962, 3301, 501, 700)])
def test_lists_equal_single(torch_cuda, nv, ng, n_hat, nroi):
    torch = torch_cuda
    u = spiral(nv)
    sig = synth.bump_values(synth.family_100(), 12.0, u)
    sig = (sig / sig.max()).astype(np.float32)
    S = torch.from_numpy(rows(u, sig, nroi, ng)).cuda()
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_set_directions(h, u)
    apt.aptidx_set_reference(h, 0, sig, n_hat)
    apt.aptidx_build_lut(h, 0, synth.random_quaternions(np.random.default_rng(2), ng))
    best = torch.full((nroi,), -9, dtype=torch.int32, device="cuda")
    score = torch.full((nroi,), -9.0, device="cuda")
    apt.aptidx_match(h, 0, S, best, score)
    pick = sorted(set(list(range(12)) + list(range(nroi - 40, nroi))))
    b1 = torch.empty(1, dtype=torch.int32, device="cuda")
    s1 = torch.empty(1, device="cuda")
    for r in pick:
        apt.aptidx_match(h, 0, S[r:r + 1], b1, s1)
        apt.aptidx_sync(h)
        assert int(b1) == int(best[r]), r
        assert np.array_equal(s1.cpu().numpy().view(np.int32), score[r:r + 1].cpu().numpy().view(np.int32)), r
    for k in (2, 31, min(ng, 1000)):
        bk = torch.empty((nroi, k), dtype=torch.int32, device="cuda")
        sk = torch.empty((nroi, k), device="cuda")
        apt.aptidx_match_topk(h, 0, S, k, bk, sk)
        b1 = torch.empty((1, k), dtype=torch.int32, device="cuda")
        s1 = torch.empty((1, k), device="cuda")
        for r in pick[:20]:
            apt.aptidx_match_topk(h, 0, S[r:r + 1], k, b1, s1)
            apt.aptidx_sync(h)
            assert torch.equal(b1[0], bk[r]), (k, r)
            assert np.array_equal(s1.cpu().numpy().view(np.int32), sk[r:r + 1].cpu().numpy().view(np.int32)), (k, r)
    ctx.close()
