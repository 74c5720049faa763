"""Short frames, whose warps begin with the tile of their own number, at the edges
of that rule: as many tiles as the launch has warps, one more and one less, and
sixteen times as many, one more and one less. The instrumented render asks the tile
counter for every tile; the images are the same. And in every frame some warp finds the
tiles handed out, which is what makes the others share their queues.
"""
import pytest

from paper_1702_01530_gb300 import capi, scenegen as sg

pytestmark = pytest.mark.gpu


def _same_as_counted(g, W, H):
    import torch
    a = g.render(W=W, H=H)["rgb"].clone()
    capi.rt_sync_status(g.handle)
    assert capi.rt_debug_render_state(g.handle)[1]
    b = g.render(W=W, H=H, count_work=True)["rgb"]
    assert torch.equal(a, b)


@pytest.fixture(scope="module")
def paired():
    """Enough primitives that a tile is 4x4 pixels of both eyes: any number of tiles."""
    s = sg.config_blobs(5, n_blobs=4, n_spheres=20)
    assert s.n_prims >= 1024
    g = capi.GpuScene(s)
    yield g
    g.close()


@pytest.mark.parametrize("times", [1, 2, 16])
@pytest.mark.parametrize("more", [-1, 0, 1])
def test_tiles_at_the_rule_s_edges(paired, times, more):
    warps = capi.rt_debug_render_state(paired.handle)[0]
    _same_as_counted(paired, 4 * (times * warps + more), 4)


@pytest.mark.parametrize("rows", [4, 64])
@pytest.mark.parametrize("more", [-1, 0, 1])
def test_tiles_of_one_eye(rows, more):
    """A small scene: 8x4 tiles of one eye, so two of them for every 8x4 pixels of the pair."""
    g = capi.GpuScene(sg.config_small(3))
    try:
        warps = capi.rt_debug_render_state(g.handle)[0]
        assert warps % 2 == 0
        _same_as_counted(g, 8 * (warps // 2 + more), rows)
    finally:
        g.close()


@pytest.mark.parametrize("W,H", [(1, 1), (7, 3), (33, 9)])
def test_fewer_tiles_than_warps(paired, W, H):
    _same_as_counted(paired, W, H)
