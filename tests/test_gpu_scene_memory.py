"""Device memory that a scene holds: 256 bytes a primitive, with the 4-wide tree's
112 and the LBVH's render nodes' 64 only once they are chosen, and none after it
is destroyed. The build's scratch is not kept."""
import numpy as np
import pytest

from paper_1702_01530_gb300 import capi, scenegen as sg

pytestmark = pytest.mark.gpu

SLACK = 8 << 20      # pages of the few allocations


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _scene(n):
    rng = np.random.default_rng(n)
    tr = np.zeros(n, sg.TRIANGLE_DT)
    c = rng.uniform(-40, 40, (n, 1, 3))
    v = (c + rng.normal(0, 0.2, (n, 3, 3))).astype(np.float32)
    tr["v0"], tr["v1"], tr["v2"] = v[:, 0], v[:, 1], v[:, 2]
    return sg.config_small(1, W=16, H=16).with_view(spheres=np.zeros(0, sg.SPHERE_DT), triangles=tr)


def test_a_scene_holds_what_it_renders_from():
    import torch
    w = capi.GpuScene(sg.config_blobs(1, n_blobs=8, n_spheres=10, W=16, H=16))     # the library's kernels are loaded
    for tree in (capi.RT_TREE_SAH, capi.RT_TREE_LBVH, capi.RT_TREE_WIDE):
        capi.rt_scene_set_traversal(w.handle, tree)
        w.render()
    w.close()
    n = 1_500_000
    s = _scene(n)
    before = _free()
    g = capi.GpuScene(s)
    try:
        held = before - _free()
        assert held <= 256 * n + SLACK
        for tree, more in ((capi.RT_TREE_LBVH, 64), (capi.RT_TREE_WIDE, 112), (capi.RT_TREE_LBVH, 0), (capi.RT_TREE_SAH, 0)):
            capi.rt_scene_set_traversal(g.handle, tree)
            now = before - _free()
            assert held <= now <= held + more * n + SLACK, tree
            held = now
        images = []
        for tree in (capi.RT_TREE_SAH, capi.RT_TREE_LBVH, capi.RT_TREE_WIDE):
            capi.rt_scene_set_traversal(g.handle, tree)
            images.append(g.render()["rgb"].clone())
            capi.rt_sync_status(g.handle)
        assert torch.equal(images[0], images[1]) and torch.equal(images[0], images[2])
    finally:
        g.close()
    del images
    torch.cuda.empty_cache()
    assert before - _free() <= SLACK


@pytest.mark.parametrize("n", [1, 2, 3, 255, 257, 511, 8191, 8193])
def test_scratch_of_small_scenes(n):
    """The scratch of a small scene is larger than its render nodes; it must not reach the error word behind them."""
    import torch
    g = capi.GpuScene(_scene(n))
    try:
        a = g.render()["rgb"].clone()
        for tree in (capi.RT_TREE_LBVH, capi.RT_TREE_WIDE):
            capi.rt_scene_set_traversal(g.handle, tree)
            assert torch.equal(a, g.render()["rgb"])
            capi.rt_sync_status(g.handle)
    finally:
        g.close()
