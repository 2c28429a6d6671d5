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


@pytest.mark.parametrize("shape,boxes", [
    # B, H, W, C, OC, KH, KW, stride, pad, w_bits, a_bits; number, width, height, images
    ((257, 5, 4, 96, 256, 5, 5, 1, 2, 1, 2), (60, 1, 1, 128)),       # single pixels of 128 images, and of the last one
    ((300, 2, 3, 144, 300, 3, 3, 1, 1, 2, 2), (20, 2, 1, 64)),       # 128 + 16 channel bytes, a channel tile of 44
    ((257, 17, 9, 48, 70, 5, 5, 1, 2, 4, 3), (405, 1, 4, 32)),       # an odd number; cut by the last row and image
    ((130, 10, 18, 144, 70, 3, 3, 1, 3, 2, 4), (385, 2, 3, 21)),     # boxes outside the image; cut at all edges
    ((3, 19, 3, 256, 300, 3, 5, 1, 1, 3, 1), (7, 1, 3, 3)),          # all images in a box, rectangular filter
    ((65, 11, 2, 96, 300, 3, 5, 1, 2, 1, 2), (17, 2, 13, 4)),        # whole images
])
def test_box_tiles(qb, monkeypatch, shape, boxes):  # noqa: F811
    monkeypatch.setenv("QNN_TC_KERNEL", "pair")
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
        assert qb.qnn_conv_boxes(d, not raw) == boxes
        nb = qb.qnn_conv_out_bytes(d, not raw)
        out = torch.full((nb + 64,), 0xEE, dtype=torch.uint8, device="cuda")
        ws = torch.zeros(qb.qnn_conv_workspace_bytes(d), dtype=torch.uint8, device="cuda")
        qb.check(qb.qnn_qconv(d, Wp, x, None if raw else torch.from_numpy(case.thr).cuda(), out, ws, ws.numel()))
        torch.cuda.synchronize()
        assert qb.qnn_device_status() == (0, 0)
        buf = out.cpu().numpy()
        assert (buf[nb:] == 0xEE).all() and not ws.any()
        assert np.array_equal(decode_out(buf[:nb], out_fmt, case.out_bits, npix, case.OC, raw), want_raw if raw else want)
