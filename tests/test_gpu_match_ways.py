"""Eq. 3 by lists and by one CTA per ROI, each where the library chooses it (told by
the launch counter), against sums in k order by plain torch: the same orientations
and scores bit for bit.  Rows of one value, whose orientations all tie (ROIs without
atoms), rows a hair off one value, whose orientations all lie within the error of the
estimates, and rows with infinities and NaN, alone and next to each other.
"""
import numpy as np
import pytest

import oracle
import synth
import paper_2009_00735_gb300 as apt

from test_gpu_lut import spiral
from test_gpu_match_lists import rows
from test_gpu_plain import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

NONE = 0x7FFFFFFF


def reference(nv):
    u = spiral(nv)
    sig = synth.bump_values(synth.family_100(), 12.0, u)
    return u, (sig / sig.max()).astype(np.float32)


def open_context(u, sig, ng, n_hat):
    ctx = apt.Context(0)
    apt.aptidx_set_directions(ctx.handle, u)
    apt.aptidx_set_reference(ctx.handle, 0, sig, n_hat)
    apt.aptidx_build_lut(ctx.handle, 0, synth.random_quaternions(np.random.default_rng(2), ng))
    return ctx


def launched(h, call):
    apt.aptidx_set_profiling(h, True)
    call()
    n = apt.aptidx_get_profile(h)[1]
    apt.aptidx_set_profiling(h, False)
    return n


def k_order_scores(torch, S, lut, ref):
    """Delta [rows, ng]: fma(d, d, acc) in FP32 over k, each fma as one rounding of the
    FP64 sum (a double rounding needs a tie at 53 bits)."""
    acc = torch.zeros(len(S), lut.shape[0], device="cuda")
    for k in range(lut.shape[1]):
        d = S[:, lut[:, k]] - ref[k]
        acc = (d.double() * d.double() + acc.double()).float()
    return acc


def check(torch, S, lut, ref, pick, best, score, bk, sk):
    for i in range(0, len(pick), 16):
        p = pick[i:i + 16]
        acc = k_order_scores(torch, S[p], lut, ref).cpu().numpy()
        for a, r in zip(acc, p):
            a = np.where(np.isnan(a), np.float32(np.nan), a)   # one NaN pattern
            finite = a < np.inf
            g = int(np.argmin(np.where(finite, a, np.inf))) if finite.any() else NONE
            assert int(best[r]) == g, r
            want = a[g] if g != NONE else np.float32(np.inf)
            assert score[r].view(np.int32) == np.float32(want).view(np.int32), r
            order = np.lexsort((np.arange(len(a)), a.view(np.uint32)))[:bk.shape[1]]
            same = ~np.isnan(a[order])   # NaN scores sort last, by their own bits
            assert np.array_equal(bk[r][same], order[same]), r
            assert np.array_equal(sk[r][same].view(np.int32), a[order][same].view(np.int32)), r


def uneven_rows(u, sig, nroi, seed):
    """Bright rows, the special ones of `rows`, a run of 70 rows of zeros, 40 of other
    single values, 40 a hair off a single value."""
    S = rows(u, sig, nroi, seed)
    S[20:90] = 0.0
    S[90:130] = np.linspace(0.1, 2.0, 40, dtype=np.float32)[:, None]
    S[130:170] = 0.5
    S[np.arange(130, 170), np.arange(40) * 7 + 3] = np.float32(0.5 + 1e-6)
    S[-3] = 0.0
    return S


# (launches of match, launches of topk): one CTA per ROI 1 and 2, lists 3 and 4.  The
# last sets: parts of a ROI's orientations summed by several CTAs, their candidate lists
# flushed on the way
@pytest.mark.parametrize("nv,ng,n_hat,nroi,topk,match_l,topk_l", [
    (300, 9, 40, 200, 5, 1, 2), (2562, 777, 33, 200, 100, 1, 2),
    (1753, 2500, 330, 2900, 31, 3, 4), (10242, 3419, 500, 1500, 100, 3, 4),
    (1753, 9000, 1700, 170, 1000, 3, 4), (10242, 20001, 300, 190, 1000, 3, 4)])
def test_flat_and_near_flat_rows(torch_cuda, nv, ng, n_hat, nroi, topk, match_l, topk_l):
    torch = torch_cuda
    u, sig = reference(nv)
    ctx = open_context(u, sig, ng, n_hat)
    h = ctx.handle
    lut = torch.from_numpy(apt.aptidx_get_lut(h, 0, ng=ng).astype(np.int64)).cuda()
    ref = torch.from_numpy(sig[oracle.top_nodes(sig, n_hat)]).cuda()
    S = torch.from_numpy(uneven_rows(u, sig, nroi, ng)).cuda()
    best = torch.full((nroi,), -9, dtype=torch.int32, device="cuda")
    score = torch.full((nroi,), -9.0, device="cuda")
    bk = torch.full((nroi, topk), -9, dtype=torch.int32, device="cuda")
    sk = torch.full((nroi, topk), -9.0, device="cuda")
    assert launched(h, lambda: apt.aptidx_match(h, 0, S, best, score)) == match_l
    assert launched(h, lambda: apt.aptidx_match_topk(h, 0, S, topk, bk, sk)) == topk_l
    pick = sorted(set(range(0, 12)) | {20, 63, 64, 89, 90, 129, 130, 131, 169} | set(range(nroi - 6, nroi)))
    check(torch, S, lut, ref, pick, best.cpu().numpy(), score.cpu().numpy(), bk.cpu().numpy(), sk.cpu().numpy())
    # every row equal
    S[:] = 0.0
    apt.aptidx_match(h, 0, S, best, score)
    apt.aptidx_match_topk(h, 0, S, topk, bk, sk)
    check(torch, S, lut, ref, [0, 65, nroi - 1], best.cpu().numpy(), score.cpu().numpy(), bk.cpu().numpy(),
          sk.cpu().numpy())
    assert bool((best == best[0]).all()) and bool((score == score[0]).all()) and bool((bk == bk[0]).all())
    ctx.close()


@pytest.mark.parametrize("nv,ng,n_hat,nroi,launches", [
    (2562, 30000, 50, 16, 1), (40962, 50000, 100, 64, 1), (40962, 3419, 200, 64, 1), (2562, 100000, 50, 256, 1),
    (40962, 3419, 1000, 64, 3), (40962, 999, 200, 300, 3)])
def test_way_of_few_rois(torch_cuda, nv, ng, n_hat, nroi, launches):
    """Few ROIs against many orientations with short node lists are faster one CTA per
    ROI, long node lists and few orientations by lists (timed both ways)."""
    torch = torch_cuda
    u, sig = reference(nv)
    ctx = open_context(u, sig, ng, n_hat)
    h = ctx.handle
    S = torch.from_numpy(rows(u, sig, nroi, ng)).cuda()
    best = torch.full((nroi,), -9, dtype=torch.int32, device="cuda")
    score = torch.full((nroi,), -9.0, device="cuda")
    assert launched(h, lambda: apt.aptidx_match(h, 0, S, best, score)) == launches
    lut = torch.from_numpy(apt.aptidx_get_lut(h, 0, ng=ng).astype(np.int64)).cuda()
    ref = torch.from_numpy(sig[oracle.top_nodes(sig, n_hat)]).cuda()
    none = np.empty((nroi, 0), np.int32)
    check(torch, S, lut, ref, [0, 1, 4, 9, nroi - 1], best.cpu().numpy(), score.cpu().numpy(), none,
          none.astype(np.float32))
    ctx.close()


def test_flat_rows_take_no_longer(torch_cuda):
    """ROIs without atoms do not slow a call down: at most twice the time of the same
    call on bright rows (summed orientation by orientation they took 14 times as long)."""
    torch = torch_cuda
    u, sig = reference(10242)
    ctx = open_context(u, sig, 3419, 1000)
    h = ctx.handle
    nroi = 4096
    best = torch.empty(nroi, dtype=torch.int32, device="cuda")
    score = torch.empty(nroi, device="cuda")
    S = torch.from_numpy(rows(u, sig, nroi, 1)).cuda()
    S[:9] = S[9:18]   # without the special rows

    def ms():
        t = []
        for _ in range(4):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            apt.aptidx_match(h, 0, S, best, score)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1))
        return min(t[1:])

    bright = ms()
    for empty in (1, 200, nroi):
        S[:empty] = 0.0
        assert ms() < 2.0 * bright, empty
    ctx.close()
