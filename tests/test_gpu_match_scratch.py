"""Scratch of the matching calls: at most 1 GiB whatever the orientation set, none
needed by a call that finds no memory for it or that is captured in a CUDA graph;
those take one CTA per ROI, with the same results.
"""
import numpy as np
import pytest

import synth
import paper_2009_00735_gb300 as apt

from test_gpu_match_lists import rows
from test_gpu_match_ways import launched, open_context, reference
from test_gpu_plain import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

GIB = 1 << 30


def outputs(torch, n, k=None):
    shape = (n,) if k is None else (n, k)
    return torch.full(shape, -9, dtype=torch.int32, device="cuda"), torch.full(shape, -9.0, device="cuda")


def same(a, b):
    return bool((a[0] == b[0]).all()) and np.array_equal(a[1].cpu().numpy().view(np.int32), b[1].cpu().numpy().view(np.int32))


@pytest.mark.parametrize("ng,lists", [(1000000, True), (5000000, False)])
def test_scratch_stays_within_a_gib(torch_cuda, ng, lists):
    """42 directions lie in one tile, so that the lists allow millions of orientations;
    the estimates of 64 ROIs at 5 000 000 would take 1.28 GB."""
    torch = torch_cuda
    u = synth.icosphere(1).astype(np.float32)
    sig = np.random.default_rng(1).random(len(u)).astype(np.float32)
    n = 2432
    S = torch.from_numpy(np.random.default_rng(2).random((n, len(u))).astype(np.float32)).cuda()
    ctx = open_context(u, sig, ng, 40)
    h = ctx.handle
    out = outputs(torch, n)
    one = outputs(torch, 1)
    apt.aptidx_match(h, 0, S[:1], *one)      # one CTA per ROI: no scratch
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ways = launched(h, lambda: apt.aptidx_match(h, 0, S, *out))
    torch.cuda.synchronize()
    # (the first call that takes the lists of this table builds them: 256 MB and 22 of
    # temporaries)
    assert before - torch.cuda.mem_get_info()[0] <= GIB + (4 << 20) + (lists * 320 << 20)
    assert (ways > 1) == lists
    for r in (0, 1, 63, 64, n - 1):
        apt.aptidx_match(h, 0, S[r:r + 1], *one)
        assert same(one, (out[0][r:r + 1], out[1][r:r + 1])), r
    ctx.close()


def test_without_memory(torch_cuda):
    torch = torch_cuda
    u, sig = reference(2562)
    n, ng, k = 2048, 30000, 20
    ctx = open_context(u, sig, ng, 300)
    h = ctx.handle
    S = torch.from_numpy(rows(u, sig, n, 5)).cuda()
    one, out, want = outputs(torch, 1), outputs(torch, n), outputs(torch, n)
    apt.aptidx_match(h, 0, S[:1], *one)      # every kernel the call takes is loaded
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (96 << 20), dtype=torch.uint8, device="cuda")
    assert launched(h, lambda: apt.aptidx_match(h, 0, S, *out)) == 1     # 246 MB of estimates do not fit
    torch.cuda.synchronize()
    del fill
    torch.cuda.empty_cache()
    assert launched(h, lambda: apt.aptidx_match(h, 0, S, *want)) == 3
    assert same(out, want)
    ctx.close()


def test_under_capture(torch_cuda):
    """A captured match is replayed on new signatures after a larger call of the same
    context has replaced the scratch."""
    torch = torch_cuda
    u, sig = reference(2562)
    n, ng = 2048, 3001
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = apt.Context(0)
        h = ctx.handle
        apt.aptidx_set_directions(h, u)
        apt.aptidx_set_reference(h, 0, sig, 300)
        apt.aptidx_build_lut(h, 0, synth.random_quaternions(np.random.default_rng(2), ng))
        S = torch.from_numpy(rows(u, sig, n, 5)).cuda()
        big = torch.from_numpy(rows(u, sig, 2 * n, 6)).cuda()
        out, want, wide = outputs(torch, n), outputs(torch, n), outputs(torch, 2 * n)
        stream.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            apt.aptidx_match(h, 0, S, *out)
        apt.aptidx_match(h, 0, S, *want)
        apt.aptidx_match(h, 0, big, *wide)
        S.copy_(big[n:])
        g.replay()
        apt.aptidx_match(h, 0, S, *want)
        stream.synchronize()
        assert same(out, want)
        assert same(out, (wide[0][n:], wide[1][n:]))
        ctx.close()


def test_lists_are_given_back(torch_cuda):
    """The lists that a table keeps (150 MB beside a table of 50) yield to a call that
    needs memory, and are built again by the next call that takes them."""
    torch = torch_cuda
    u, sig = reference(2562)
    n, ng = 12000, 50000
    ctx = open_context(u, sig, ng, 500)
    h = ctx.handle
    host = rows(u, sig, n, 5)                 # 123 MB, copied to the device by the call
    S = torch.from_numpy(host[:2000]).cuda()
    want, again = outputs(torch, 2000), outputs(torch, 2000)
    assert launched(h, lambda: apt.aptidx_match(h, 0, S, *want)) == 3
    one = outputs(torch, 1)
    apt.aptidx_match(h, 0, torch.zeros(1, len(u), device="cuda"), *one)
    best, score = np.empty(n, np.int32), np.empty(n, np.float32)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (64 << 20), dtype=torch.uint8, device="cuda")
    apt.aptidx_match(h, 0, host, best, score)
    del fill
    torch.cuda.empty_cache()
    assert np.array_equal(best[:2000], want[0].cpu().numpy())
    assert np.array_equal(score[:2000].view(np.int32), want[1].cpu().numpy().view(np.int32))
    assert launched(h, lambda: apt.aptidx_match(h, 0, S, *again)) == 3
    assert same(again, want)
    ctx.close()


def test_lists_only_where_a_call_takes_them(torch_cuda):
    """A signature row of 60000 directions does not fit shared memory and its table is
    not matched: it holds no lists.  A small table gets them from the first call that is
    large enough, with the same results."""
    torch = torch_cuda
    u, sig = reference(60000)
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_set_directions(h, u)
    apt.aptidx_set_reference(h, 0, sig, 500)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    apt.aptidx_build_lut(h, 0, synth.random_quaternions(np.random.default_rng(2), 20000))   # a table of 20 MB
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= 100 << 20
    ctx.close()

    u, sig = reference(162)
    n = 60000
    ctx = open_context(u, sig, 500, 100)
    h = ctx.handle
    S = torch.from_numpy(rows(u, sig, n, 5)).cuda()
    out, one = outputs(torch, n), outputs(torch, 1)
    assert launched(h, lambda: apt.aptidx_match(h, 0, S, *out)) == 3
    for r in list(range(9)) + [63, 64, n - 1]:
        assert launched(h, lambda: apt.aptidx_match(h, 0, S[r:r + 1], *one)) == 1
        assert same(one, (out[0][r:r + 1], out[1][r:r + 1])), r
    ctx.close()
