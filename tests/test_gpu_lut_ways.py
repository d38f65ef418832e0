"""The look-up table by the node grid against the table by scans over all nodes (the
same table in pieces small enough that the library scans them, which test_gpu_lut.py
holds to the oracle): direction sets with gaps, uneven norms, duplicates.  Index
work: exact.
"""
import numpy as np
import pytest

import synth
import paper_2009_00735_gb300 as apt

from test_gpu_lut import direction_set, spiral
from test_gpu_plain import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def near(n, degrees, seed):
    """orientations within a few times `degrees` of the identity"""
    w = np.radians(degrees) * np.random.default_rng(seed).standard_normal((n, 3))
    th = np.linalg.norm(w, axis=1, keepdims=True)
    return np.concatenate([np.cos(th / 2), np.sin(th / 2) * w / th], 1)


def sets(kind):
    if kind == "even":
        return spiral(40001)
    return direction_set(kind)


@pytest.mark.parametrize("kind", ["even", "cap", "holes", "norms", "double", "dense"])
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

