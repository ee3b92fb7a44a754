"""The staged kernels on single meshes small enough for the one-kernel generate
(host-buffer calls, stage times and launch settings set by hand run them): the
same sizes and meshes as that kernel's tests, against the oracle."""
import pytest

import oracle
from paper_2403_14723_gb300 import build, meshgen, polylla
from tests.gpu_helpers import assert_parity, gpu_run
from tests.test_gpu_edges import strip
from tests.test_gpu_output import fan, shuffled
from tests.test_gpu_small import SIZES

pytestmark = pytest.mark.gpu

STAGED = {"output_items": 4}   # the default: setting it selects the staged kernels


@pytest.mark.parametrize("n", SIZES)
def test_small_sizes_staged(n):
    for mesh in (strip(n), fan(n), shuffled(strip(n, 3), 4)):
        assert_parity(mesh, gpu_run(mesh, generate_times=2, tuning=STAGED), oracle.run_mesh(mesh))


@pytest.mark.parametrize("make", [
    meshgen.two_triangle_square,
    lambda: meshgen.exact_grid(30),
    lambda: meshgen.perturbed_grid(24, 0.3, seed=5),
    lambda: meshgen.random_delaunay(60, seed=1),
    lambda: shuffled(meshgen.random_delaunay(1000, seed=2), 7),
    lambda: meshgen.lattice_delaunay(700, 40, seed=3),
    lambda: meshgen.near_tie_delaunay(700, 40, seed=4),
])
def test_small_meshes_staged(make):
    mesh = make()
    assert_parity(mesh, gpu_run(mesh, generate_times=2, tuning=STAGED), oracle.run_mesh(mesh))


def test_small_meshes_with_tips_staged():
    for seed in range(12):
        mesh = meshgen.random_delaunay(900, seed=100 + seed)
        assert_parity(mesh, gpu_run(mesh, tuning=STAGED), oracle.run_mesh(mesh))


def test_launch_counts_of_the_two_routes():
    build.build_library()
    for n, one in ((2048, 1), (2049, 7)):
        with polylla.Polylla(polylla.DeviceMesh.from_host(strip(n))) as p:
            p.generate()
            assert polylla.polylla_launch_count(p.ctx) == one
            polylla.polylla_set_tuning(p.ctx, dict(polylla.polylla_get_tuning(p.ctx), **STAGED))
            p.generate()
            p.polygons()
            assert polylla.polylla_launch_count(p.ctx) == 7
