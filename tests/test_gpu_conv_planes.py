"""Convolutions whose route depends on sizes: rows too long to stage, bit-plane maps on the AND/POPC kernel
(which lowers on the fly), and bit-plane maps widened into the workspace for the 8-bit kernels."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

BITPLANES, INT8 = 0, 1


@pytest.fixture(scope="module")
def qb():
    from paper_1709_04060_b200 import binding
    return binding


def test_image_row_of_more_than_four_gigabytes(qb):
    """2^28 + 8 pixels of 16 bytes: the row's size does not fit 32 bits, so nothing may compute with it
    there.  1 x 1 convolution, one threshold; both ends, the wrap point and a random sample of pixels
    against dot products."""
    W, C, OC = (1 << 28) + 8, 16, 32
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randint(0, 4, (W, C), generator=g, device="cuda", dtype=torch.uint8)
    Wt = torch.randint(-2, 2, (OC, C), generator=g, device="cuda", dtype=torch.int8)
    thr = torch.randint(-12, 4, (OC, 1), generator=g, device="cuda", dtype=torch.int32)
    d = qb.qnn_conv_desc(1, 1, W, C, 0, OC, 1, 1, 1, 0, 2, 2, 1, 1, 0, INT8, BITPLANES, 0)
    out = qb.qconv(d, qb.pack(Wt, 2, 1, INT8), x, thr)
    torch.cuda.synchronize()
    assert qb.qnn_device_status() == (0, 0)
    at = torch.cat([torch.arange(0, 300), torch.arange(W - 300, W), torch.randint(0, W, (20000,))]).cuda()
    acc = x[at].double() @ Wt.double().T
    code = (acc >= thr[:, 0].double()).long()
    want = (code << torch.arange(32, device="cuda")).sum(1)
    got = out[: 4 * W].view(torch.int32)[at].long() & 0xFFFFFFFF
    assert torch.equal(got, want)
