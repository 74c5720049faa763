"""The copies of the trees that renders walk (boxes as centre and extent).

Every tree holds the same leaf boxes in that form, so all walks of a scene give
the same image bit for bit, also where boxes are flat (axis-parallel triangles),
far from the origin, or tiny beside it; and editing the LBVH after it was chosen
reaches the copy.
"""
import numpy as np
import pytest

from paper_1702_01530_gb300 import capi, scenegen as sg

pytestmark = pytest.mark.gpu


def _moved(s, shift, scale):
    """The scene scaled about the origin, then shifted (camera and lights with it)."""
    f = lambda a: (np.asarray(a, np.float64) * scale + shift).astype(np.float32)   # noqa: E731
    sp, tr, li, cam = s.spheres.copy(), s.triangles.copy(), s.lights.copy(), s.camera.copy()
    sp["center"], sp["radius"] = f(sp["center"]), sp["radius"] * np.float32(scale)
    for k in ("v0", "v1", "v2"):
        tr[k] = f(tr[k])
    li["position"] = f(li["position"])
    cam["eye"] = f(cam["eye"])
    return s.with_view(spheres=sp, triangles=tr, lights=li, camera=cam, eye_sep=s.eye_sep * scale,
                       convergence=s.convergence * scale)


@pytest.mark.parametrize("shift,scale", [((0, 0, 0), 1.0), ((500, -300, 800), 1.0), ((0, 0, 0), 100.0),
                                         ((3, 2, 1), 0.05)])
@pytest.mark.parametrize("name", ["polyhedra", "blobs", "terrain"])
def test_all_walks_agree(name, shift, scale):
    import torch
    s = {"polyhedra": lambda: sg.config_polyhedra(6, 3, W=320, H=200, ground=True),
         "blobs": lambda: sg.config_blobs(9, n_blobs=6, n_spheres=20, box=15.0, W=320, H=200),
         "terrain": lambda: sg.config_terrain(9, n_grid=65, n_spheres=200, W=320, H=200)}[name]()
    g = capi.GpuScene(_moved(s, np.array(shift, np.float64), scale))
    try:
        sah = g.render()["rgb"].clone()
        capi.rt_sync_status(g.handle)
        assert sah.std() > 1e-3
        for tree in (capi.RT_TREE_LBVH, capi.RT_TREE_WIDE):
            capi.rt_scene_set_traversal(g.handle, tree)
            other = g.render()["rgb"]
            capi.rt_sync_status(g.handle)
            assert torch.equal(sah, other), tree
    finally:
        g.close()


def test_edit_after_choosing_the_lbvh():
    """A host-made cycle (node 0 its own left child, an empty right child)
    stops at the iteration bound whether the tree was chosen before or after."""
    s = sg.config_small(3, W=32, H=24)
    g = capi.GpuScene(s)
    try:
        bvh = capi.rt_scene_get_bvh(g.handle)
        capi.rt_scene_set_traversal(g.handle, capi.RT_TREE_LBVH)
        g.render()
        capi.rt_sync_status(g.handle)
        capi.rt_debug_set_node(g.handle, 0, 0, int(bvh["right"][0]), empty_right=True)
        g.render()
        with pytest.raises(capi.RtError) as e:
            capi.rt_sync_status(g.handle)
        assert e.value.code == capi.RT_ERR_TIMEOUT
        capi.rt_scene_set_traversal(g.handle, capi.RT_TREE_SAH)
        g.render()
        capi.rt_sync_status(g.handle)
    finally:
        g.close()
