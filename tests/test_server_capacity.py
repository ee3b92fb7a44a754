"""What a server of a given budget takes: the slot and lane capacities (in
triangles) that its memory layout has given, on the CPU.  A layout that needs
more memory per triangle would turn requests away that were served."""
import pytest

from paper_2403_14723_gb300 import build, polylla

MiB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build_library()


@pytest.mark.parametrize("budget,n_slots,lane,slot,lane_slot", [
    (64 * MiB, 3, -1, 111_825, 0), (64 * MiB, 3, 0, 83_024, 83_024), (64 * MiB, 3, 4000, 89_365, 64_000),
    (1024 * MiB, 3, -1, 1_839_904, 0), (1024 * MiB, 3, 0, 1_489_252, 1_048_576),
    (1024 * MiB, 3, 4000, 1_817_444, 64_000), (40960 * MiB, 3, -1, 73_727_981, 0),
    (40960 * MiB, 3, 0, 73_377_329, 1_048_576), (40960 * MiB, 3, 4000, 73_705_520, 64_000),
])
def test_capacity_of_a_budget(budget, n_slots, lane, slot, lane_slot):
    p = polylla.server_plan(budget, n_slots=n_slots, lane_triangles=lane)
    assert p["slot_triangles"] >= slot and p["lane_slot_triangles"] >= lane_slot
    assert p["device_bytes"] <= budget
