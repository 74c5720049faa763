"""Weight gradients on the tensor cores at the edges of their tiles.

The kernel takes tiles of 112 x 4 pixels, the SMs shared out among the layers,
sums 2 K steps of 16 pixels inside the tensor core where a CTA has at most 2
tiles, else 4, and writes partial sums every 16 tiles. Sizes on both sides of a
tile edge, a single pixel, enough tiles for the longer sums and for several
flushes, against the oracle's backward pass in float64 that rounds to BF16 where
the kernels do. What remains are FP32 sums (1e-6) and activations or data
gradients that round to BF16 the other way: a relative change of 2^-8 at most
in one factor, in about one value of a thousand, independently from pixel to
pixel, so 2^-8 / sqrt(P) of a sum over P pixels where one flips, and 1e-3 of
the whole with all layers and products between them.
"""
import numpy as np
import pytest

from oracle import reproj as orp
from paper_1702_01530_gb300 import capi, scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(1, 1), (111, 3), (112, 4), (113, 5), (225, 9), (3, 700), (900, 37),
                                 (1800, 340)])
def test_weight_gradients_at_tile_edges(W, H):
    import torch
    params = sg.net_params_he(71)
    params[orp.OFF_B[3]] = 0.2
    feat = sg.bf16_features_synthetic(72 + W, W, H)
    label = (np.random.default_rng(73).random(W * H) < 0.3).astype(np.float32)
    net = capi.Net(params)
    try:
        grads = torch.full((capi.RT_NET_PARAMS,), float("nan"), dtype=torch.float32, device="cuda")
        f16 = torch.from_numpy(feat).to(torch.bfloat16).cuda()
        capi.rt_net_train_step(net.handle, f16, torch.from_numpy(label).cuda(), W, H, 0.0, grads=grads)
        capi.rt_net_status(net.handle)
        g = grads.cpu().numpy().astype(np.float64)
    finally:
        net.close()
    emu = orp.grads_emulated(params, feat, label, W, H, bf16=True)
    bound = 1e-3 + 2.0 ** -8 / np.sqrt(W * H)
    k = 0
    for ci, co in orp.LAYERS:
        for n in (co * ci * 9, co):
            a, b = g[k:k + n], emu[k:k + n]
            assert np.linalg.norm(a - b) <= bound * np.linalg.norm(b) + 1e-12, (k, n)
            k += n


@pytest.mark.parametrize("W,H", [(2, 1), (123, 2), (124, 1), (125, 3), (128, 6), (248, 7), (249, 2), (372, 29)])
def test_data_gradients_at_strip_edges(W, H):
    """The data gradients stream through strips of 124 pixels and segments of
    rows; every layer's weight gradient but the last is a product of one."""
    test_weight_gradients_at_tile_edges(W, H)
