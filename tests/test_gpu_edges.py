"""Kernels that share a warp's or a block's work among their lanes, at the
sizes where a share ends, against the oracle bit for bit: the Lepp primitive
(128 triangles a warp, 1,024 a block; paths that all go on) and the
convexification's corner search (512 triangles a block, at most one corner
each)."""
import numpy as np
import pytest

import oracle
from paper_2403_14723_gb300 import meshgen
from tests.test_gpu_convex import assert_convex_parity, gpu_convex
from tests.test_gpu_lepp import _run
from tests.test_gpu_output import fan

pytestmark = pytest.mark.gpu


def strip(n: int, seed: int = 1):
    """n triangles in a row between two uneven sides (reflex corners on both)."""
    rng = np.random.default_rng(seed)
    k = np.arange(n + 2)
    xy = np.stack([0.5 * k + 0.2 * rng.random(n + 2), (k % 2) + 0.35 * rng.random(n + 2)], axis=1)
    i = np.arange(n)
    odd = (i % 2).astype(bool)
    tri = np.stack([i, np.where(odd, i + 2, i + 1), np.where(odd, i + 1, i + 2)], axis=1)[:, [0, 2, 1]]
    a, b, c = xy[tri[:, 0]], xy[tri[:, 1]], xy[tri[:, 2]]
    turn = (b[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1]) - (b[:, 1] - a[:, 1]) * (c[:, 0] - a[:, 0])
    tri[turn < 0] = tri[turn < 0][:, [0, 2, 1]]
    return meshgen.from_triangles(tri, xy, name=f"strip_{n}")


SIZES = [1, 31, 32, 33, 127, 128, 129, 511, 512, 513, 1023, 1024, 1025, 4099]


@pytest.mark.parametrize("n", SIZES)
def test_lepp_share_edges(n):
    for mesh in (strip(n), fan(min(n, 1025))):    # the fan: every path runs to its far end
        want_t, want_l = oracle.lepp(mesh, oracle.run_mesh(mesh).longest)
        g = _run(mesh)
        assert g["status"] == 0
        assert np.array_equal(g["terminal"], want_t)
        assert np.array_equal(g["length"], want_l)


@pytest.mark.parametrize("n", SIZES)
def test_convex_share_edges(n):
    mesh = strip(n, seed=2)
    c = assert_convex_parity(mesh, gpu_convex(mesh))
    assert n < 511 or len(c.chords) > 0
