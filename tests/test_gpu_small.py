"""The one-kernel generate of small meshes against the oracle, bit for bit: the
sizes where its rounds of threads end and where the staged kernels take over,
long fans (one polygon, deep rotations), barrier tips, exact ties, triangles in
random order; twice in a row, from a graph, and followed by a convexification."""
import numpy as np
import pytest

import oracle
from paper_2403_14723_gb300 import meshgen, polylla
from tests.gpu_helpers import assert_parity, gpu_run
from tests.test_gpu_convex import assert_convex_parity, gpu_convex
from tests.test_gpu_edges import strip
from tests.test_gpu_output import fan, shuffled

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 32, 33, 1023, 1024, 1025, 2047, 2048, 2049]


@pytest.mark.parametrize("n", SIZES)
def test_small_sizes(n):
    for mesh in (strip(n), fan(n), shuffled(strip(n, 3), 4)):
        assert_parity(mesh, gpu_run(mesh, generate_times=2), oracle.run_mesh(mesh))


@pytest.mark.parametrize("make", [
    meshgen.two_triangle_square,
    lambda: meshgen.exact_grid(30),
    lambda: meshgen.perturbed_grid(24, 0.3, seed=5),
    lambda: meshgen.random_delaunay(60, seed=1),
    lambda: meshgen.random_delaunay(1000, seed=2),
    lambda: shuffled(meshgen.random_delaunay(1000, seed=2), 7),
    lambda: meshgen.lattice_delaunay(700, 40, seed=3),
    lambda: meshgen.near_tie_delaunay(700, 40, seed=4),
])
def test_small_meshes(make):
    mesh = make()
    assert mesh.n_triangles <= 2048
    r = oracle.run_mesh(mesh)
    assert_parity(mesh, gpu_run(mesh, generate_times=2), r)
    assert_convex_parity(mesh, gpu_convex(mesh, times=2), chords_too=False)


def test_small_meshes_with_tips_twice_and_from_a_graph():
    import torch

    tips = 0
    for seed in range(12):
        mesh = meshgen.random_delaunay(900, seed=100 + seed)
        r = oracle.run_mesh(mesh)
        tips += int(r.stats["tips"])
        assert_parity(mesh, gpu_run(mesh, generate_times=2), r)
        dm = polylla.DeviceMesh.from_host(mesh)
        stream = torch.cuda.Stream()
        with polylla.Polylla(dm) as p:
            polylla.polylla_capture_graph(p.ctx, stream)
            p.generate(stream)
            out = p.polygons(stream)
            stream.synchronize()
            assert polylla.polylla_launch_count(p.ctx) == 1
            for k in ("seeds", "offsets", "he_list", "v_list"):
                assert np.array_equal(out[k].cpu().numpy(), getattr(r, k))
            assert np.array_equal(dm.next.cpu().numpy(), r.next_out)
    assert tips > 20


def test_small_rotation_cap_is_reported():
    with pytest.raises(polylla.PolyllaError):
        gpu_run(fan(300), max_rotation=40)
