"""Meshes that were not validated, with a border half-edge as the twin of a
barrier tip's frontier half-edge: the edge stays frontier, so the tip is found,
and the walk to its chord must end there with an error (chord -1) instead of
leaving the mesh.  Everything else is as on the sound mesh."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2403_14723_gb300 import build, meshgen, polylla

pytestmark = pytest.mark.gpu

INVALID_MESH, NONTERMINATING = -2, -5


def _tip_mesh():
    mesh = meshgen.random_delaunay(300, seed=13)
    r = oracle.run_mesh(mesh)
    assert len(r.tip_out) >= 5
    return mesh, r


def _bad_twins(mesh):
    """(twin, status): past the mesh, negative, its first and last border half-edge."""
    return [(10 ** 9, INVALID_MESH), (-7, INVALID_MESH), (3 * mesh.n_triangles, NONTERMINATING),
            (mesh.n_halfedges - 1, NONTERMINATING)]


def _labels_of_failed_run(ctx, status):
    """The tips and chords of a run that ends with status (the call gives them beside it)."""
    import torch

    out = polylla.polylla_labels()
    assert polylla.load_library().polylla_get_labels(ctypes.c_void_p(ctx), ctypes.byref(out),
                                                     polylla._stream_ptr(None)) == status
    return [polylla._view(p, out.n_tips, 32, torch.int32).cpu().numpy() for p in (out.tips, out.chords)]


def _expect(tips, chords, r, shift, bad):
    want = {int(f) + shift: int(c) + shift for f, c in zip(r.tip_out, r.chord)}
    want[bad + shift] = -1
    assert dict(zip(tips.tolist(), chords.tolist())) == want


@pytest.mark.parametrize("which", [0, 4, -1])
@pytest.mark.parametrize("kind", range(4))
def test_batch_tip_with_a_border_twin(kind, which):
    build.build_library()
    mesh, r = _tip_mesh()
    grid = meshgen.exact_grid(12)
    db = polylla.DeviceBatch.from_host([grid, mesh, grid])
    value, status = _bad_twins(mesh)[kind]
    bad = int(r.tip_out[which])
    at = grid.n_halfedges + bad
    ctx = polylla.polylla_batch_create(db, validate=False)
    try:
        db.twin[at] = value
        polylla.polylla_generate(ctx)
        tips, chords = _labels_of_failed_run(ctx, status)
        _expect(tips, chords, r, 3 * grid.n_triangles, bad)
        ho, g = db.halfedge_offset, oracle.run_mesh(grid)
        nxt, prv = db.next.cpu().numpy(), db.prev.cpu().numpy()
        for i in (0, 2):
            assert np.array_equal(nxt[ho[i]:ho[i + 1]], g.next_out) and np.array_equal(prv[ho[i]:ho[i + 1]], g.prev_out)
        for a in (nxt, prv):
            assert a[ho[1]:ho[2]].min() >= 0 and a[ho[1]:ho[2]].max() < mesh.n_halfedges
        db.twin[at] = int(mesh.twin[bad])             # sound again: so are the results
        polylla.polylla_generate(ctx)
        polylla.polylla_get_polygons(ctx)
        assert np.array_equal(db.next.cpu().numpy()[ho[1]:ho[2]], r.next_out)
        assert np.array_equal(db.prev.cpu().numpy()[ho[1]:ho[2]], r.prev_out)
    finally:
        polylla.polylla_destroy(ctx)


@pytest.mark.parametrize("kind", [2, 3])
def test_staged_mesh_tip_with_a_border_twin(kind):
    build.build_library()
    mesh, r = _tip_mesh()
    dm = polylla.DeviceMesh.from_host(mesh)
    value, status = _bad_twins(mesh)[kind]
    bad = int(r.tip_out[1])
    with polylla.Polylla(dm, validate=False) as p:
        polylla.polylla_set_tuning(p.ctx, polylla.polylla_get_tuning(p.ctx))   # the staged kernels
        dm.twin[bad] = value
        p.generate()
        assert polylla.polylla_launch_count(p.ctx) == 7
        _expect(*_labels_of_failed_run(p.ctx, status), r, 0, bad)


@pytest.mark.parametrize("pinned", [True, False])
def test_served_tip_with_a_border_twin(pinned):
    build.build_library()
    mesh, r = _tip_mesh()
    with polylla.Server(memory_budget=1 << 30, n_slots=2) as srv:
        for kind in range(4):
            value, status = _bad_twins(mesh)[kind]
            hr = polylla.HostRequest(mesh, pinned=pinned)
            hr.inp["twin"][int(r.tip_out[kind])] = value
            assert srv.wait(srv.submit(hr))["status"] == status
        hr = polylla.HostRequest(mesh, pinned=pinned)
        info = srv.wait(srv.submit(hr))
        assert info["status"] == 0
        assert np.array_equal(hr.result(info)["next"], r.next_out)


@pytest.mark.parametrize("which", [0, 4, -1])
@pytest.mark.parametrize("kind", [2, 3])
def test_small_mesh_tip_with_a_border_twin(kind, which):
    build.build_library()
    mesh, r = _tip_mesh()
    dm = polylla.DeviceMesh.from_host(mesh)
    value, status = _bad_twins(mesh)[kind]
    bad = int(r.tip_out[which])
    with polylla.Polylla(dm, validate=False) as p:
        dm.twin[bad] = value
        p.generate()
        assert polylla.polylla_launch_count(p.ctx) == 1
        _expect(*_labels_of_failed_run(p.ctx, status), r, 0, bad)
        dm.twin[bad] = int(mesh.twin[bad])
        p.generate()
        p.polygons()
        assert np.array_equal(dm.next.cpu().numpy(), r.next_out) and np.array_equal(dm.prev.cpu().numpy(), r.prev_out)
