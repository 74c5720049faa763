"""Short frames, whose warps begin with the tile of their own number, at the edges
of that rule: as many tiles as warps, one more and one less, and sixteen times
as many. The instrumented render asks for every tile; the images are the same.
"""
import pytest

from paper_1702_01530_gb300 import capi, scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [4, 64])
@pytest.mark.parametrize("more", [-1, 0, 1])
def test_images_at_the_rule_s_edges(rows, more):
    import torch
    # 8x4 tiles of one eye, both eyes; 9 blocks of 4 warps on an SM
    half = torch.cuda.get_device_properties(0).multi_processor_count * 36 // 2
    W, H = 8 * (half + more), rows
    s = sg.config_small(3)
    g = capi.GpuScene(s)
    try:
        a = g.render(W=W, H=H)["rgb"].clone()
        b = g.render(W=W, H=H, count_work=True)["rgb"]
        assert torch.equal(a, b)
    finally:
        g.close()


@pytest.mark.parametrize("W,H", [(1, 1), (7, 3), (33, 9)])
def test_fewer_tiles_than_warps(W, H):
    import torch
    s = sg.config_blobs(5, n_blobs=4, n_spheres=20)
    g = capi.GpuScene(s)
    try:
        a = g.render(W=W, H=H)["rgb"].clone()
        assert torch.equal(a, g.render(W=W, H=H, count_work=True)["rgb"])
    finally:
        g.close()
