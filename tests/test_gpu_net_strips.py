"""The fused forward network at the edges of its strips and segments.

A strip is 122 output pixels wide, and its rows are cut into segments that
recompute 8 rows; a CTA walks several segments when there are more than SMs.
Widths on both sides of one, two and three strips, single rows and pixels, and
stacks of more images than SMs (several segments per CTA), against the oracle
that rounds where the kernel does. Tolerances as for the other network tests:
FP32 sums in another order can round an activation the other way, 2^-9 of it in
BF16 (5e-3 of a probability at most through two further layers), 2^-4 in E4M3
(3e-2), in few pixels (the means).
"""
import numpy as np
import pytest

from oracle import reproj as orp
from paper_1702_01530_gb300 import capi, scenegen as sg

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (122, 2, 1), (123, 3, 2), (121, 9, 1), (244, 1, 1), (245, 5, 3), (367, 20, 1),
         (7, 4, 200), (130, 33, 170)]


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("W,H,n", SIZES)
def test_forward_at_strip_and_segment_edges(W, H, n, fp8):
    import torch
    params = sg.net_params_he(81)
    rng = np.random.default_rng(82)
    params[orp.OFF_B[0]:orp.OFF_B[0] + 32] = rng.normal(0, 0.1, 32)
    params[orp.OFF_B[3]] = -0.5
    scales = (8.0, 16.0, 4.0)
    feat = sg.bf16_features_synthetic(83 + W, W, H * n).reshape(n, W * H, 16)
    net = capi.Net(params)
    try:
        if fp8:
            capi.rt_net_set_fp8(net.handle, scales)
        f16 = torch.from_numpy(feat).to(torch.bfloat16).cuda()
        prob = torch.full((n, H, W), float("nan"), dtype=torch.float32, device="cuda")
        capi.rt_net_forward_images(net.handle, f16, n, W, H, prob)
        one = torch.empty((H, W), dtype=torch.float32, device="cuda")
        for i in sorted({0, n // 2, n - 1}):
            capi.rt_net_forward(net.handle, f16[i].contiguous(), W, H, one)
            assert torch.equal(one, prob[i]), "a stacked image differs from the image alone"
        capi.rt_net_status(net.handle)
        got = prob.cpu().numpy()
    finally:
        net.close()
    assert np.isfinite(got).all()
    for i in sorted({0, n // 3, n - 1}):
        if fp8:
            err = np.abs(got[i] - orp.forward_fp8(params, feat[i], W, H, scales))
            assert err.max() <= 3e-2 and err.mean() <= 1e-3, (i, err.max(), err.mean())
        else:
            err = np.abs(got[i] - orp.forward(params, feat[i], W, H, bf16=True))
            assert err.max() <= 5e-3 and err.mean() <= 2e-4, (i, err.max(), err.mean())
