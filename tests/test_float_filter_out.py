"""The second certified decision of the longest-edge filter, restated in numpy
like the first (test_float_filter_longest): on the float64 path the shortest edge
is left out where the filter proves it shorter than the longest, and the other
two are compared from the vertex after it on.  The edge left out must be shorter
in binary64, and the ties found must be those of all three lengths."""
import numpy as np
import pytest

from tests.test_float_filter_longest import shared_bound_filter
from tests.test_float_filters import U, _triangle_sets, fma32, longest_f64, trunc_to_f32


@np.errstate(over="ignore", invalid="ignore")
def edge_left_out(p):
    """p [n, 3, 2] float64 -> out [n]: 0..2, or 3 where all three are compared."""
    t, bad = trunc_to_f32(p.reshape(-1))
    t = t.reshape(p.shape)
    e = np.roll(t, -1, axis=1) - t
    d = fma32(e[..., 0], e[..., 0], e[..., 1] * e[..., 1])
    dm, least = d.max(axis=1), d.min(axis=1)
    X, Y = np.abs(t).max(axis=1).T
    DX, DY = np.abs(e).max(axis=1).T

    def full(c):
        return np.full_like(dm, c)

    b2 = fma32(full(np.float32(24.6) * U), fma32(X, DX, Y * DY),
               fma32(full(np.float32(73.0) * U * U), fma32(X, X, Y * Y),
                     fma32(full(np.float32(9.0) * U), dm, full(np.float32(6.0e-36)))))
    out = np.where(least == d[:, 2], 2, np.where(least == d[:, 0], 0, 1))
    return np.where(~bad.reshape(p.shape).any(axis=(1, 2)) & (dm - least > b2), out, 3)


def ties_without(p, out):
    """The mask of the longest edges as the float64 path finds it: edges a and b
    after the one left out (0 and 1 if none), then the third if none is."""
    d = longest_f64(p)
    n = np.arange(len(p))
    a = np.where(out == 0, 1, np.where(out == 1, 2, 0))
    b = np.where(a == 2, 0, a + 1)
    da, db = d[n, a], d[n, b]
    best = np.where(db > da, 0, 1 << a) | np.where(db >= da, 1 << b, 0)
    dc, m = d[:, 2], np.maximum(da, db)
    return np.where(out < 3, best, np.where(dc > m, 0, best) | np.where(dc >= m, 4, 0))


@pytest.mark.parametrize("seed", [1, 20240321])
def test_edge_left_out_is_shorter_and_ties_are_complete(seed):
    left_out = {0: 0, 1: 0, 2: 0, 3: 0}
    for name, p in _triangle_sets(np.random.default_rng(seed), 200_000).items():
        out = edge_left_out(p)
        d = longest_f64(p)
        d_out = d[np.arange(len(p)), np.minimum(out, 2)]
        wrong = (out < 3) & ~(d_out < d.max(axis=1))
        assert not wrong.any(), f"{name}: the edge left out is a longest one at {np.flatnonzero(wrong)[:5]}"
        full = ((d == d.max(axis=1, keepdims=True)) << np.arange(3)).sum(axis=1)
        got = ties_without(p, out)
        assert np.array_equal(got, full), f"{name}: ties differ at {np.flatnonzero(got != full)[:5]}"
        exact = ~shared_bound_filter(p)[0]           # the triangles that take this path
        for k in left_out:
            left_out[k] += int((out[exact] == k).sum())
    assert min(left_out.values()) > 1000, left_out   # every form of the path was met
