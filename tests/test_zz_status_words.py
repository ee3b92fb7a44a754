"""The no-allocation entry's status words at any address: a caller's packed
buffer need not align them (copies of bytes always took it)."""
import numpy as np
import pytest

import oracle
from paper_2403_14723_gb300 import build, meshgen, polylla
from tests.test_zz_no_alloc import _noalloc_call

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh", [meshgen.exact_grid(20), meshgen.random_delaunay(4000, seed=31)],
                         ids=["one_kernel", "staged"])
def test_status_words_at_any_address(mesh):
    import torch

    build.build_library()
    lib = polylla.load_library()
    T = mesh.n_triangles
    r = oracle.run_mesh(mesh)
    for shift in range(5):
        dm = polylla.DeviceMesh.from_host(mesh)
        outs = {k: torch.zeros(n, dtype=torch.int32, device="cuda")
                for k, n in (("seeds", T), ("offsets", T + 1), ("he_list", 3 * T), ("v_list", 3 * T))}
        words = torch.full((20,), 0xA5, dtype=torch.uint8, device="cuda")
        outs["status"] = words[shift:]
        assert _noalloc_call(lib, mesh, dm, outs, torch.cuda.current_stream()) == 0
        got = words.cpu().numpy()
        assert list(np.frombuffer(got[shift:shift + 12].tobytes(), np.int32)) == [r.n_polygons, len(r.he_list), 0]
        assert np.all(got[:shift] == 0xA5) and np.all(got[shift + 12:] == 0xA5)
        assert np.array_equal(outs["he_list"].cpu().numpy()[:len(r.he_list)], r.he_list)
