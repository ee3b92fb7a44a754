"""The output stage where its bookkeeping can go wrong, against the oracle:
walks that all leave their tile (more than a tile gathers, more than a listing
warp gathers), walks over several chunks, a chunk pool used up, polygons longer
than a record or a staging buffer holds, ragged last tiles."""
import numpy as np
import pytest

import oracle
from paper_2403_14723_gb300 import meshgen
from tests.gpu_helpers import assert_parity, gpu_run
from tests.test_gpu_batch import assert_batch_parity, batch_run

pytestmark = pytest.mark.gpu


def fan(n: int):
    """n triangles around an apex, radii growing slightly: every triangle's
    longest edge is shared with the next one, so all are one polygon of n + 2
    half-edges."""
    a = np.linspace(0.0, 0.9 * np.pi, n + 1)
    r = 1.0 + 1e-7 * np.arange(n + 1)
    xy = np.concatenate([[[0.0, 0.0]], np.stack([r * np.cos(a), r * np.sin(a)], axis=1)])
    i = np.arange(1, n + 1)
    return meshgen.from_triangles(np.stack([np.zeros_like(i), i, i + 1], axis=1), xy, name=f"fan_{n}")


def shuffled(mesh, seed: int):
    """The same triangles in random order: no polygon stays in its tile."""
    p = np.random.default_rng(seed).permutation(mesh.n_triangles)
    return meshgen.from_triangles(mesh.triangles()[p], mesh.coords, name=mesh.name + "_shuffled")


MESHES = [
    (lambda: shuffled(meshgen.exact_grid(60), 1), 0),                  # every walk crosses, ties everywhere
    (lambda: shuffled(meshgen.random_delaunay(9000, seed=12), 2), 0),  # long crossing walks, barrier tips
    (lambda: meshgen.random_delaunay(4000, seed=31), 0),               # long polygons along the hull
    (lambda: fan(5000), 8000),                                         # longer than a staging buffer
    (lambda: fan(20_000), 30_000),                                     # longer than a record holds
    (lambda: shuffled(fan(20_000), 3), 30_000),                        # and with the chunk pool used up
]


@pytest.mark.parametrize("tile,items", [(1024, 2), (1024, 4), (2048, 4), (4096, 4)])
@pytest.mark.parametrize("make,rotation", MESHES, ids=["grid", "delaunay", "hull", "fan5k", "fan20k", "fan20k_shuffled"])
def test_output_bookkeeping(make, rotation, tile, items):
    mesh = make()
    g = gpu_run(mesh, generate_times=2, max_rotation=rotation, tuning={"output_tile": tile, "output_items": items})
    r = oracle.run_mesh(mesh)
    if mesh.name.startswith("fan_"):
        assert r.n_polygons == 1
    assert_parity(mesh, g, r)


def test_output_bookkeeping_batch():
    meshes = [shuffled(meshgen.exact_grid(40), 4), fan(3000), meshgen.two_triangle_square(),
              shuffled(fan(2500), 5), shuffled(meshgen.random_delaunay(3000, seed=13), 6)]
    meshes += [meshgen.exact_grid(2) for _ in range(300)] + [meshgen.random_delaunay(4000, seed=31)]
    for unaligned in (False, True):
        db, g = batch_run(meshes, unaligned=unaligned)
        assert_batch_parity(meshes, db, g)
