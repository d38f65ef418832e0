"""The look-up table by the node grid against the table by scans over all nodes (the
same table in pieces small enough that the library scans them, which test_gpu_lut.py
holds to the oracle): direction sets with gaps, uneven norms, duplicates, and clusters
of thousands of directions in one cell of the grid.  Index work: exact.
"""
import numpy as np
import pytest

import synth
import paper_2009_00735_gb300 as apt

from test_gpu_lut import direction_set, spiral
from test_gpu_plain import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def cap(n, degrees):
    """n directions within `degrees` of the z axis"""
    i = np.arange(n) + 0.5
    z = 1 - (1 - np.cos(np.radians(degrees))) * i / n
    a = i * np.pi * (3 - 5 ** 0.5)
    return np.stack([np.sqrt(1 - z * z) * np.cos(a), np.sqrt(1 - z * z) * np.sin(a), z], 1).astype(np.float32)


def near(n, degrees, seed):
    """orientations within a few times `degrees` of the identity"""
    w = np.radians(degrees) * np.random.default_rng(seed).standard_normal((n, 3))
    th = np.linalg.norm(w, axis=1, keepdims=True)
    return np.concatenate([np.cos(th / 2), np.sin(th / 2) * w / th], 1)


def sets(kind):
    if kind == "cluster":
        return np.concatenate([cap(20000, 1.0), spiral(3001)])
    if kind == "clusters":
        return np.concatenate([cap(8000, 0.3), -cap(7001, 2.0), spiral(500)])
    if kind == "even":
        return spiral(40001)
    return direction_set(kind)


@pytest.mark.parametrize("kind", ["cluster", "clusters", "even", "cap", "holes", "norms", "double", "dense"])
def test_grid_equals_scan(torch_cuda, kind):
    u = sets(kind)
    nv = len(u)
    sig = np.random.default_rng(3).random(nv).astype(np.float32)
    sig[::7] = sig[0]
    n_hat = min(nv, 300)
    step = max(1, int(1.9e8 / (nv * n_hat)))           # orientations of a table that is scanned
    ng = min(2000, max(3 * step, int(4.1e8 / (nv * n_hat)) + 2))
    rng = np.random.default_rng(5)
    Q = np.concatenate([[[1.0, 0, 0, 0]], near(ng // 2, 0.5, 7), synth.random_quaternions(rng, ng - ng // 2 - 1)])
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_set_directions(h, u)
    apt.aptidx_set_reference(h, 0, sig, n_hat)
    apt.aptidx_build_lut(h, 0, Q)
    got = apt.aptidx_get_lut(h, 0, ng=ng)
    for g in range(0, ng, step):
        q = Q[g:g + step]
        apt.aptidx_build_lut(h, 0, q)
        assert np.array_equal(apt.aptidx_get_lut(h, 0, ng=len(q)), got[g:g + step]), g
    # other directions in the same context: their own grid
    v = np.ascontiguousarray(u[::2])
    apt.aptidx_set_directions(h, v)
    apt.aptidx_set_reference(h, 0, sig[::2].copy(), min(n_hat, len(v)))
    apt.aptidx_build_lut(h, 0, Q)
    again = apt.aptidx_get_lut(h, 0, ng=ng)
    other = apt.Context(0)
    apt.aptidx_set_directions(other.handle, v)
    apt.aptidx_set_reference(other.handle, 0, sig[::2].copy(), min(n_hat, len(v)))
    apt.aptidx_build_lut(other.handle, 0, Q[:step])
    assert np.array_equal(apt.aptidx_get_lut(other.handle, 0, ng=min(step, ng)), again[:step])
    other.close()
    ctx.close()


def test_clustered_directions_take_no_longer(torch_cuda):
    """40000 directions within one degree: queries among them take no longer than queries
    away from them, which are scanned (a thread that walked its cells took six times as
    long)."""
    torch = torch_cuda
    u = cap(40000, 1.0)
    ctx = apt.Context(0)
    h = ctx.handle
    apt.aptidx_set_directions(h, u)
    apt.aptidx_set_reference(h, 0, np.random.default_rng(1).random(len(u)).astype(np.float32), 500)
    flip = near(400, 0.3, 1)[:, [1, 0, 3, 2]] * [-1, 1, -1, 1]   # the same after half a turn about x

    def ms(Q):
        t = []
        for _ in range(4):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            apt.aptidx_build_lut(h, 0, Q)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1))
        return min(t[1:])

    assert ms(near(400, 0.3, 1)) < 2.0 * ms(np.ascontiguousarray(flip))
    ctx.close()


@pytest.mark.parametrize("nv", [1, 2, 3, 162, 1023, 1024, 1025, 2049, 4096])
def test_strongest_of_few_directions(torch_cuda, nv):
    """Few directions are sorted, more are selected unless about all are asked for: values with
    ties and zeros of both signs, the identity maps every strongest node onto itself."""
    u = spiral(nv)
    sig = (np.random.default_rng(nv).integers(-6, 6, nv) / 4.0).astype(np.float32)
    sig[5::11] = -0.0
    key = np.where(sig.view(np.int32) < 0, ~sig.view(np.uint32), sig.view(np.uint32) | np.uint32(1 << 31))
    want = np.lexsort((np.arange(nv), ~key))
    ctx = apt.Context(0)
    apt.aptidx_set_directions(ctx.handle, u)
    for n_hat in sorted({1, (nv + 1) // 2, nv}):
        apt.aptidx_set_reference(ctx.handle, 0, sig, n_hat)
        apt.aptidx_build_lut(ctx.handle, 0, np.array([[1.0, 0, 0, 0]]))
        assert np.array_equal(apt.aptidx_get_lut(ctx.handle, 0, ng=1)[0], want[:n_hat])
    ctx.close()
