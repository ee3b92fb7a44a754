"""Results are read on the context's own stream whichever device is current."""
import numpy as np
import pytest

import oracle
from paper_2403_14723_gb300 import build, meshgen, polylla

pytestmark = pytest.mark.gpu


def test_results_while_another_device_is_current():
    import torch

    if torch.cuda.device_count() < 2:
        pytest.skip("needs two devices")
    build.build_library()
    mesh = meshgen.random_delaunay(4000, seed=31)
    r = oracle.run_mesh(mesh)
    dm = polylla.DeviceMesh.from_host(mesh, device="cuda:0")
    stream = torch.cuda.Stream(device=0)
    with torch.cuda.device(0), torch.cuda.stream(stream):
        p = polylla.Polylla(dm, stream=stream)
        p.generate(stream)
    with torch.cuda.device(1):
        out = p.polygons(stream)
        assert out["seeds"].device.index == 0
        assert np.array_equal(out["seeds"].cpu().numpy(), r.seeds)
        assert polylla.load_library().polylla_last_error(p.ctx) == 0
    with torch.cuda.device(0):
        p.close()
