"""The batch's images where requests are read and written 16 bytes at a time and
where they are not: sizes that are no multiple of four values, sums that begin
off a 16-byte boundary behind such a request, images off one. All equal the
single renders bit for bit.
"""
import pytest

from paper_1702_01530_gb300 import capi, scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(64, 36, 0), (64, 36, 1)], [(5, 3, 0), (64, 36, 0), (7, 4, 0), (4, 1, 0)],
                                   [(1, 1, 0), (1, 1, 1), (2, 2, 0), (32, 8, 2)]])
def test_images_of_any_size_and_alignment(sizes):
    import torch
    s = sg.config_small(1)
    g = capi.GpuScene(s)
    try:
        outs, items = [], []
        for W, H, off in sizes:
            buf = torch.full((2 * H * W * 3 + off,), -1.0, device="cuda")
            o = buf[off:].view(2, H, W, 3)
            outs.append(o)
            items.append((g.handle, s.camera, s.eye_sep, s.convergence, W, H, 3, o[0], o[1]))
        batch = capi.rt_batch_create(capi.make_requests(items))
        capi.rt_batch_launch(batch)
        torch.cuda.synchronize()
        for (W, H, _), o in zip(sizes, outs):
            ref = torch.empty((2, H, W, 3), device="cuda")
            capi.rt_render_stereo(g.handle, s.camera, s.eye_sep, s.convergence, W, H, 3, ref[0], ref[1])
            assert torch.equal(o, ref), (W, H)
        capi.rt_batch_destroy(batch)
    finally:
        g.close()
