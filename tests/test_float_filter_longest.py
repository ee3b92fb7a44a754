"""The longest-edge kernels' filter with one bound for a triangle's three
edges, restated in numpy and searched for counterexamples on the adversarial
triangles of test_float_filters: it must answer only where the binary64 argmax
is unique and is its answer, and answer on ordinary triangles."""
import numpy as np
import pytest

from tests.test_float_filters import U, _triangle_sets, fma32, longest_f64, trunc_to_f32


@np.errstate(over="ignore", invalid="ignore")
def shared_bound_filter(p):
    """p [n, 3, 2] float64 -> (sure [n], k [n])."""
    t, bad = trunc_to_f32(p.reshape(-1))
    t = t.reshape(p.shape)
    e = np.roll(t, -1, axis=1) - t                                     # (dx, dy) of the three edges
    d = fma32(e[..., 0], e[..., 0], e[..., 1] * e[..., 1])
    s = np.sort(d, axis=1)
    k = d.argmax(axis=1)
    X, Y = np.abs(t).max(axis=1).T
    DX, DY = np.abs(e).max(axis=1).T
    c1, c2, c3 = np.float32(24.6) * U, np.float32(73.0) * U * U, np.float32(9.0) * U

    def full(c, like):
        return np.full_like(like, c)

    dm = s[:, 2]
    b2 = fma32(full(c1, X), fma32(X, DX, Y * DY),
               fma32(full(c2, X), fma32(X, X, Y * Y), fma32(full(c3, dm), dm, full(np.float32(6.0e-36), dm))))
    return ~bad.reshape(p.shape).any(axis=(1, 2)) & (dm - s[:, 1] > b2), k


@pytest.mark.parametrize("seed", [1, 20240321])
def test_shared_bound_never_contradicts_binary64(seed):
    decided = total = 0
    for name, p in _triangle_sets(np.random.default_rng(seed), 200_000).items():
        sure, k = shared_bound_filter(p)
        d = longest_f64(p)
        n = np.arange(len(p))
        rest = np.maximum(d[n, (k + 1) % 3], d[n, (k + 2) % 3])
        wrong = sure & ~(d[n, k] > rest)
        assert not wrong.any(), f"{name}: filter sure but binary64 disagrees at {np.flatnonzero(wrong)[:5]}"
        decided += int(sure.sum())
        total += len(p)
    assert decided > 0.5 * total


def test_shared_bound_decides_ordinary_triangles():
    rng = np.random.default_rng(7)
    sure, _ = shared_bound_filter(_triangle_sets(rng, 100_000)["grid_cell"])
    assert sure.mean() > 0.99
    sure, _ = shared_bound_filter(rng.random((100_000, 3, 2)))
    assert sure.mean() > 0.999
