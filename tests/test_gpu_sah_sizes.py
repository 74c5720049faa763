"""The SAH build at the edges of its phases: warps of 32 leaves, blocks of 256,
slices of 512, degenerate centroids and the depth budget.

The tree has to hold every leaf and node once, no deeper than the traversal
stack allows, with boxes that are exactly the unions of their leaves', the same
with and without slicing; and where cost decides, every split costs no more
than the best candidate in FP64 (up to the rounding of an FP32 cost: a few
products and sums of positive terms, below 1e-6 relative).
"""
import numpy as np
import pytest

from paper_1702_01530_gb300 import capi, scenegen as sg

pytestmark = pytest.mark.gpu

BINS = 16


def _scene(n, mode, seed):
    rng = np.random.default_rng(seed)
    ns = n // 3
    c = {"uniform": lambda: rng.uniform(-40, 40, (n, 3)),
         "grid": lambda: np.round(rng.uniform(-4, 4, (n, 3))),
         "point": lambda: np.zeros((n, 3)),
         "line": lambda: rng.uniform(-40, 40, (n, 1)) * [1.0, 0.0, -0.0],
         "powers": lambda: 2.0 ** -np.stack([np.arange(n) * (120.0 / n)] * 3, 1) * [1.0, 0.0, 0.0]}[mode]()
    sp, tr = np.zeros(ns, sg.SPHERE_DT), np.zeros(n - ns, sg.TRIANGLE_DT)
    sp["center"], sp["radius"] = c[:ns], 1e-20 if mode == "powers" else 0.3
    v = c[ns:, None, :] + rng.normal(0, 0.5 if mode == "uniform" else 0.0, (n - ns, 3, 3))
    tr["v0"], tr["v1"], tr["v2"] = v[:, 0], v[:, 1], v[:, 2]
    return sg.config_small(1, W=8, H=8).with_view(spheres=sp, triangles=tr)


def _tree(s, slicing=True):
    capi.rt_debug_set_sah_slicing(slicing)
    try:
        g = capi.GpuScene(s)
        try:
            return capi.rt_debug_get_sah_tree(g.handle)
        finally:
            g.close()
    finally:
        capi.rt_debug_set_sah_slicing(True)


def _boxes(t):
    """Child boxes (n - 1, 2, 6: lo, hi) and children (n - 1, 2)."""
    t = np.ascontiguousarray(t).view(np.float32)
    c0, c1 = t[:, [0, 2, 8, 1, 3, 9]], t[:, [4, 6, 10, 5, 7, 11]]
    return np.stack([c0, c1], 1), np.ascontiguousarray(t[:, 12:14]).view(np.int32)


def _check_tree(t):
    box, kids = _boxes(t)
    n = len(t) + 1
    assert np.array_equal(np.sort(~kids[kids < 0]), np.arange(n))
    assert np.array_equal(np.sort(kids[kids >= 0]), np.arange(1, n - 1))
    level, depth = np.array([0]), 0
    while len(level):
        k, b = kids[level], box[level]
        inner = k >= 0
        want = b[inner]                                     # the child's own two boxes, united
        got = box[k[inner]]
        assert np.array_equal(want[:, :3], got[:, :, :3].min(1))
        assert np.array_equal(want[:, 3:], got[:, :, 3:].max(1))
        level, depth = k[inner], depth + 1
    assert depth <= 60
    return box, kids


@pytest.mark.parametrize("n", [2, 3, 32, 33, 64, 255, 256, 257, 512, 513, 1024, 1025, 4097, 20000])
def test_sizes(n):
    t = _tree(_scene(n, "uniform", n))
    _check_tree(t)
    assert np.array_equal(t, _tree(_scene(n, "uniform", n), slicing=False))


@pytest.mark.parametrize("mode", ["grid", "point", "line", "powers"])
@pytest.mark.parametrize("n", [2, 33, 300, 5000])
def test_degenerate_centroids(mode, n):
    s = _scene(n, mode, n)
    t = _tree(s)
    _check_tree(t)
    assert np.array_equal(t, _tree(s, slicing=False))


def _area(b):
    d = np.maximum(b[..., 3:] - b[..., :3], 0.0)
    return d[..., 0] * d[..., 1] + d[..., 1] * d[..., 2] + d[..., 2] * d[..., 0]


def _union(b):
    return np.concatenate([b[:, :3].min(0), b[:, 3:].max(0)])


def test_splits_cost_least():
    box, kids = _check_tree(_tree(_scene(1500, "uniform", 5)))
    leaf = np.zeros((1500, 6), np.float32)
    leaf[~kids[kids < 0]] = box[kids < 0]

    def leaves(k):
        return [~k] if k < 0 else leaves(kids[k, 0]) + leaves(kids[k, 1])

    for node in range(len(kids)):
        l, r = leaves(kids[node, 0]), leaves(kids[node, 1])
        b = leaf[l + r]
        cost = _area(_union(b[:len(l)].astype(np.float64))) * len(l) + \
            _area(_union(b[len(l):].astype(np.float64))) * len(r)
        c = np.float32(0.5) * (b[:, :3] + b[:, 3:])
        best = np.inf
        for a in range(3):
            if len(b) <= 32 and node != 0:
                order = np.argsort(c[:, a], kind="stable")
                sides = [order[:i] for i in range(1, len(b))]
            else:
                ext = c[:, a].max() - c[:, a].min()
                q = np.minimum(BINS - 1, ((c[:, a] - c[:, a].min()) * (np.float32(BINS) / ext)).astype(np.int32))
                sides = [np.flatnonzero(q <= i) for i in range(BINS - 1)]
            for left in sides:
                right = np.setdiff1d(np.arange(len(b)), left)
                if len(left) and len(right):
                    x = b.astype(np.float64)
                    best = min(best, _area(_union(x[left])) * len(left) + _area(_union(x[right])) * len(right))
        assert cost <= best * (1 + 1e-6), (node, len(b), cost, best)
