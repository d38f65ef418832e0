"""GPU parity of the look-up table and the strongest nodes on direction sets
where the nearest-node grid is at its limit: a handful of directions, sets with
gaps (whose open queries are scanned), uneven norms inside the accepted 1e-5,
duplicated directions (ties), and dense sets.  Index work: exact.
"""
import numpy as np
import pytest

import oracle
import synth
import paper_2009_00735_gb300 as apt

from test_gpu_plain import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def spiral(n):
    i = np.arange(n) + 0.5
    z = 1 - 2 * i / n
    a = i * np.pi * (3 - 5 ** 0.5)
    return np.stack([np.sqrt(1 - z * z) * np.cos(a), np.sqrt(1 - z * z) * np.sin(a), z], 1).astype(np.float32)


def direction_set(kind):
    rng = np.random.default_rng(11)
    if kind == "one":
        return np.array([[0.0, 0.0, 1.0]], np.float32)
    if kind == "five":
        return spiral(5)
    if kind == "odd":
        return spiral(1999)
    if kind == "cap":
        u = spiral(9000)
        return np.ascontiguousarray(u[u[:, 2] > 0.7])
    if kind == "holes":
        u = synth.icosphere(4)
        return np.ascontiguousarray(u[np.abs(u @ np.array([0.6, 0.0, 0.8], np.float32)) < 0.5])
    if kind == "norms":
        u = synth.icosphere(4).astype(np.float64)
        return (u * (1 + 9e-6 * (2 * rng.random((len(u), 1)) - 1))).astype(np.float32)
    if kind == "double":
        u = synth.icosphere(3)
        return np.ascontiguousarray(np.concatenate([u, u[::-1]]))
    return spiral(70001)          # above 65536: 32-bit table entries


@pytest.mark.parametrize("kind", ["one", "five", "odd", "cap", "holes", "norms", "double", "dense"])
def test_lut_exact(torch_cuda, kind):
    u = direction_set(kind)
    nv = len(u)
    rng = np.random.default_rng(3)
    sig = rng.random(nv).astype(np.float32)
    sig[::7] = sig[0]                                  # ties among the values
    for n_hat in sorted({1, min(nv, 37), min(nv, 300)}):
        Q = np.concatenate([[[1.0, 0, 0, 0]], synth.random_quaternions(rng, 1 if kind == "dense" else 40)])
        ctx = apt.Context(0)
        apt.aptidx_set_directions(ctx.handle, u)
        apt.aptidx_set_reference(ctx.handle, 0, sig, n_hat)
        apt.aptidx_build_lut(ctx.handle, 0, Q)
        got = apt.aptidx_get_lut(ctx.handle, 0, ng=len(Q))
        top = oracle.top_nodes(sig, n_hat)
        assert np.array_equal(got, oracle.lut(u, top, Q))
        ctx.close()


@pytest.mark.parametrize("n_hat", [1, 2, 1023, 1025, 4096, 4097, 10242])
def test_strongest_nodes_exact(torch_cuda, n_hat):
    """Values with many ties, zeros of both signs and negative values; identity
    orientation maps every strongest node onto itself."""
    u = synth.icosphere(5)
    rng = np.random.default_rng(n_hat)
    sig = (rng.integers(-40, 40, len(u)) / 8.0).astype(np.float32)
    sig[5::11] = -0.0
    ctx = apt.Context(0)
    apt.aptidx_set_directions(ctx.handle, u)
    apt.aptidx_set_reference(ctx.handle, 0, sig, n_hat)
    apt.aptidx_build_lut(ctx.handle, 0, np.array([[1.0, 0, 0, 0]]))
    got = apt.aptidx_get_lut(ctx.handle, 0, ng=1)[0]
    # keys order by the bit pattern, in which -0 follows +0
    key = np.where(sig.view(np.int32) < 0, ~sig.view(np.uint32), sig.view(np.uint32) | np.uint32(1 << 31))
    want = np.lexsort((np.arange(len(u)), ~key))[:n_hat]
    assert np.array_equal(got, want)
    ctx.close()
