"""The kernels of a generate are chained (a kernel is resident while those
before it still write), so the read-only load path is only for what no kernel of
a chain writes: the caller's coords, origin and twin, and a batch's tables.  A
batch's union twins are written by its first kernel; kernels that run on both
take ordinary loads of twins unless the batch is told apart at compile time."""
import os
import re

import pytest

from paper_2403_14723_gb300 import build

TABLES = {"w.loc_origin", "w.loc_twin", "w.loc_t_off", "w.loc_h_off", "w.loc_v_off", "w.loc_seg"}
INPUTS = {"m.xy", "xy", "m.origin", "origin"}
ALLOWED = {
    "kernels_label.cu": INPUTS | TABLES | {"m.twin", "twin"},
    "kernels_output.cu": INPUTS | TABLES,
    "kernels_repair.cu": TABLES,
    "kernels_small.cu": INPUTS | {"m.twin"},
    "kernels_convex.cu": INPUTS | {"m.twin"},    # single meshes only
    "kernels_batch.cu": INPUTS,
    "kernels_serve.cu": set(),
    "polylla_noalloc.cu": set(),
}


def _code(name):
    with open(os.path.join(build.CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


@pytest.mark.parametrize("name", sorted(ALLOWED))
def test_read_only_loads_of_inputs_alone(name):
    src = _code(name)
    bases = re.findall(r"__ldg\(\s*([\w.]+)", src)
    assert len(bases) == len(re.findall(r"__ldg\b", src))
    assert set(bases) <= ALLOWED[name], sorted(set(bases) - ALLOWED[name])


def test_twins_in_kernels_of_batches_too():
    # one place, which a batch does not compile
    src = _code("kernels_label.cu")
    assert re.findall(r"[^\n]*__ldg\(m\.twin[^\n]*", src) == ["    return BATCH ? ld_chain(m.twin + e) : __ldg(m.twin + e);"]
    # and the single-mesh longest-edge kernel's lambda over the caller's array
    assert len(re.findall(r"__ldg\(twin\b", src)) == 1


@pytest.mark.parametrize("name", sorted(ALLOWED))
def test_no_restrict_on_what_a_chain_writes(name):
    for decl in re.findall(r"const (\w+) \*\s*__restrict__ (\w+)", _code(name)):
        assert decl in {("double2", "xy"), ("int32_t", "twin")}, decl
