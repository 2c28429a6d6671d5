"""Convolutions of the CTA-pair kernel whose tiles are boxes of output pixels (tiled loads, filter taps outside
the image left out), against the direct convolution: boxes cut by the map's edges and by the last image,
an odd number of boxes, padding that leaves taps out, channel counts that are not whole chunks."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_1709_04060_b200 import synth
from qnn_testutil import decode_out
from test_gpu_conv import conv_desc, device_map, device_weights, qb  # noqa: F401

pytestmark = pytest.mark.gpu

BITPLANES, INT8 = 0, 1


@pytest.mark.parametrize("shape", [
    # B, H, W, C, OC, KH, KW, stride, pad, w_bits, a_bits
    (130, 5, 6, 96, 256, 5, 5, 1, 2, 1, 2),       # single pixels of 128 images, and of the last two
    (300, 4, 4, 144, 300, 3, 3, 1, 1, 2, 2),      # 128 + 16 channel bytes, a channel tile of 64
    (3, 13, 13, 256, 384, 3, 3, 1, 1, 1, 2),      # boxes of a few images: rows and columns
    (1, 33, 50, 32, 64, 5, 3, 1, 1, 4, 3),        # one image, rectangular filter
    (7, 9, 9, 64, 70, 3, 3, 1, 2, 2, 4),          # padding of two with three taps
    (5, 12, 7, 48, 130, 1, 1, 1, 0, 3, 1),        # a single tap
])
def test_box_tiles(qb, monkeypatch, shape):  # noqa: F811
    monkeypatch.setenv("QNN_TC_KERNEL", "pair")
    monkeypatch.setenv("QNN_CONV_BOX", "1")
    monkeypatch.setenv("QNN_CONV_LOWER", "0")
    monkeypatch.setenv("QNN_CONV_IMPLICIT", "1")
    case = synth.conv_case(1500 + shape[0], *shape)
    x, pitch = device_map(qb, case, INT8)
    Wp = device_weights(qb, case, INT8)
    npix = case.B * case.OH * case.OW
    want_raw = orc.qconv(case.In, case.Wt, None, case.stride, case.pad).reshape(npix, case.OC)
    want = (want_raw[:, :, None] >= case.thr[None]).sum(2)
    for out_fmt, raw in ((INT8, False), (BITPLANES, False), (INT8, True)):
        d = conv_desc(qb, case, INT8, out_fmt, pitch)
        nb = qb.qnn_conv_out_bytes(d, not raw)
        out = torch.full((nb + 64,), 0xEE, dtype=torch.uint8, device="cuda")
        ws = torch.zeros(qb.qnn_conv_workspace_bytes(d), dtype=torch.uint8, device="cuda")
        qb.check(qb.qnn_qconv(d, Wp, x, None if raw else torch.from_numpy(case.thr).cuda(), out, ws, ws.numel()))
        torch.cuda.synchronize()
        assert qb.qnn_device_status() == (0, 0)
        buf = out.cpu().numpy()
        assert (buf[nb:] == 0xEE).all() and not ws.any()
        assert np.array_equal(decode_out(buf[:nb], out_fmt, case.out_bits, npix, case.OC, raw), want_raw if raw else want)
