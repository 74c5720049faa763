"""The LBVH build at the edges of its tiles and blocks, against the oracle.

The sort works on tiles of 2048 keys (256 per warp), the refit on blocks of 256
leaves whose nodes meet in shared memory, the keys by an FP32 estimate unless
a centroid lies next to a cell boundary. Everything is compared exactly: keys,
topology and boxes.
"""
import numpy as np
import pytest

import oracle
from paper_1702_01530_gb300 import capi, scenegen as sg

pytestmark = pytest.mark.gpu


def _scene(n_spheres, n_tris, seed, shift=0.0, step=None):
    rng = np.random.default_rng(seed)
    s = sg.config_small(1, W=8, H=8)
    sp, tr = np.zeros(n_spheres, sg.SPHERE_DT), np.zeros(n_tris, sg.TRIANGLE_DT)
    snap = (lambda a: a) if step is None else (lambda a: np.round(a / step) * step)
    sp["center"] = snap(rng.uniform(-40, 40, (n_spheres, 3))) + shift
    sp["radius"] = rng.uniform(0.01, 2.0, n_spheres)
    c = rng.uniform(-50, 50, (n_tris, 1, 3))
    v = snap(c + rng.normal(0, 0.5, (n_tris, 3, 3))) + shift
    tr["v0"], tr["v1"], tr["v2"] = v[:, 0], v[:, 1], v[:, 2]
    return s.with_view(spheres=sp, triangles=tr)


def _check(s):
    g = capi.GpuScene(s)
    try:
        got = capi.rt_scene_get_bvh(g.handle)
    finally:
        g.close()
    ref = oracle.OracleScene(s).lbvh()
    for k in ("keys", "left", "right", "leaf_box", "inner_box"):
        assert np.array_equal(got[k], ref[k]), k


@pytest.mark.parametrize("ns,nt", [(0, 1), (1, 0), (2, 0), (1, 1), (0, 255), (3, 253), (0, 257), (513, 0),
                                   (0, 2047), (1000, 1048), (1, 2048), (0, 4097), (777, 9000)])
def test_sizes(ns, nt):
    _check(_scene(ns, nt, 100 + ns + nt))


@pytest.mark.parametrize("shift,step", [(0.0, 0.5), (3000.0, None), (-1e6, 1.0), (0.0, 1e6)])
def test_cells_next_to_boundaries(shift, step):
    """Coordinates on a coarse grid (many centroids on cell boundaries and in
    one cell), far from the origin (the FP32 estimate decides nothing), and all
    coincident."""
    _check(_scene(300, 5000, 7, shift, step))


def test_device_records_of_any_alignment():
    """Triangle records need no more than the alignment of their floats."""
    import torch
    s = _scene(10, 3000, 3)
    n = s.n_prims
    raw = np.ascontiguousarray(s.triangles).view(np.uint8)
    sp = torch.from_numpy(np.ascontiguousarray(s.spheres).view(np.uint8).copy()).cuda()
    got = []
    for off in (0, 4):
        buf = torch.zeros(raw.size + 8, dtype=torch.uint8, device="cuda")
        buf[off:off + raw.size] = torch.from_numpy(raw.copy()).cuda()
        out = [torch.zeros((n - 1, 16), dtype=torch.int32, device="cuda"),
               torch.zeros((n, 12), dtype=torch.int32, device="cuda"),
               torch.zeros(n, dtype=torch.int64, device="cuda"),
               torch.zeros(2 * n - 1, dtype=torch.int32, device="cuda")]
        capi.rt_build_lbvh_noalloc(sp, 10, buf.data_ptr() + off, 3000, *out)
        got.append(out)
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n", [512, 4095, 4096, 4097, 65536, 65793])
def test_levels_of_runs(n):
    """Trees over runs of 256 leaves, over 16 of those, and over 256 of those."""
    _check(_scene(n // 2, n - n // 2, n))


def test_runs_that_leave_much_over():
    """Points at powers of two towards one corner: prefixes shorten by a bit from
    leaf to leaf, so that most subtrees hang off the path to one end of a run."""
    s = _scene(0, 6000, 1)
    tr = s.triangles.copy()
    p = np.float32(2.0) ** -np.random.default_rng(2).uniform(0, 12, (6000, 3)).astype(np.float32)
    for v in ("v0", "v1", "v2"):
        tr[v] = p
    _check(s.with_view(triangles=tr))


@pytest.mark.parametrize("scale", [1e-40, 1e37, 3e38])
def test_bounds_of_extreme_coordinates(scale):
    """Sums of vertices past the range of FP32, and denormal ones."""
    s = _scene(40, 3000, 9)
    tr, sp = s.triangles.copy(), s.spheres.copy()
    rng = np.random.default_rng(4)
    for v in ("v0", "v1", "v2"):
        tr[v] = (rng.uniform(-1, 1, (3000, 3)) * scale).astype(np.float32)
    sp["center"] = (rng.uniform(-1, 1, (40, 3)) * min(scale, 1e37)).astype(np.float32)
    _check(s.with_view(spheres=sp, triangles=tr))
