"""The crossing walks' pool of a batch, which has the memory of the union origin
and prev: unions of few triangles in every tile size, triangles in random order
so that walks leave their tile and use its chunks up, validated (the layout
check fills that memory first) and twice, against the oracle; and a server whose
slot is full."""
import numpy as np
import pytest

import oracle
from paper_2403_14723_gb300 import build, meshgen, polylla
from tests.test_gpu_batch import assert_batch_parity, batch_run
from tests.test_gpu_edges import strip
from tests.test_gpu_output import fan, shuffled

pytestmark = pytest.mark.gpu

BATCHES = [
    lambda: [strip(1)],
    lambda: [shuffled(strip(200), 1), strip(55)],                            # 255 triangles
    lambda: [shuffled(meshgen.exact_grid(20), 2), strip(302)],               # 1,024: a whole tile
    lambda: [shuffled(meshgen.exact_grid(20), 3), strip(303)],               # and one more
    lambda: [shuffled(fan(700), 4), shuffled(meshgen.exact_grid(28), 5)],    # 2,158
    lambda: [shuffled(meshgen.random_delaunay(2200, seed=14), 6), shuffled(meshgen.exact_grid(46), 7)],
]


@pytest.mark.parametrize("tile,items", [(1024, 2), (1024, 4), (2048, 2), (2048, 4), (4096, 4)])
@pytest.mark.parametrize("make", BATCHES, ids=["1", "255", "1024", "1025", "2158", "8k"])
def test_pool_of_small_unions(make, tile, items):
    meshes = make()
    db, g = batch_run(meshes, generate_times=2, tuning={"output_tile": tile, "output_items": items})
    assert_batch_parity(meshes, db, g)


def test_server_slot_filled_to_its_capacity():
    build.build_library()
    with polylla.Server(memory_budget=4 << 20, n_slots=2, max_batch_meshes=4, lane_triangles=-1) as srv:
        st = srv.stats()
        assert st["device_bytes"] <= 4 << 20
        n = st["slot_triangles"]
        for mesh in (shuffled(strip(n, 8), 9), strip(n, 8)):
            r = oracle.run_mesh(mesh)
            hr = polylla.HostRequest(mesh)
            info = srv.wait(srv.submit(hr))
            assert info["status"] == 0
            res = hr.result(info)
            for k, want in (("seeds", r.seeds), ("offsets", r.offsets), ("he_list", r.he_list),
                            ("v_list", r.v_list), ("next", r.next_out), ("prev", r.prev_out)):
                assert np.array_equal(res[k], want), k
