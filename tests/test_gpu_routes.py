"""Routes that the library's own choice takes only at some sizes: image rows too long to stage, the
AND/POPC kernels (forced), bit-plane maps widened into the workspace, W4A4 planes on the tensor cores."""
import numpy as np
import pytest
import torch

import test_gpu_bitsparsity as sparsity
from oracle import oracle as orc
from paper_1709_04060_b200 import synth
from qnn_testutil import decode_out
from test_gpu_conv import CONV_CASES, conv_desc, device_map, device_weights
from test_gpu_conv import test_qconv_matches_direct_convolution as _direct_convolution

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


class Forced:
    """The binding with every descriptor's path set to the bit-serial one, so that a test written against
    the library's own choice also runs on the AND/POPC kernels."""

    def __init__(self, qb):
        self._qb = qb

    def __getattr__(self, name):
        f = getattr(self._qb, name)
        if name not in ("gemm_desc", "qnn_gemm_desc", "qnn_conv_desc"):
            return f

        def make(*args, **kw):
            d = f(*args, **kw)
            d.path = self._qb.QNN_PATH_BITSERIAL
            return d
        return make


@pytest.mark.parametrize("out_fmt", [BITPLANES, INT8])
@pytest.mark.parametrize("shape", CONV_CASES + [
    (2, 11, 14, 40, 70, 3, 3, 2, 1, 3, 4),       # stride 2 with padding, C not a multiple of 32
    (3, 9, 8, 33, 65, 5, 4, 3, 2, 4, 2),         # stride 3, rectangular filter, one channel past a word
])
def test_forced_bit_serial_convolution(qb, monkeypatch, out_fmt, shape):
    """AND/POPC with the lowering done by its staging code: padding, strides, several taps."""
    _direct_convolution(Forced(qb), monkeypatch, "auto", BITPLANES, out_fmt, shape)


@pytest.mark.parametrize("w_bits,a_bits,w_enc,a_enc", [
    (4, 4, 0, 0), (4, 4, 1, 0), (3, 4, 1, 1), (1, 4, 2, 0), (4, 1, 0, 2), (2, 3, 0, 1)])
def test_forced_bit_serial_product_with_empty_tiles(qb, w_bits, a_bits, w_enc, a_enc):
    """The tile skipping of the AND/POPC kernel, at the widths the library's own choice sends elsewhere."""
    sparsity.test_empty_planes_and_empty_blocks_change_nothing(Forced(qb), w_bits, a_bits, w_enc, a_enc)


def test_forced_bit_serial_product_of_zeros(qb):
    sparsity.test_all_zero_operands(Forced(qb))


S, U, B = synth.SIGNED, synth.UNSIGNED, synth.BIPOLAR


@pytest.mark.parametrize("lower", ["", "1"])
@pytest.mark.parametrize("shape,w_enc,a_enc", [
    # B, H, W, C, OC, KH, KW, stride, pad, w_bits, a_bits; all above 2^28 multiply-accumulates
    ((9, 33, 31, 40, 90, 3, 3, 1, 1, 3, 3), S, S),      # C = 40: rows of 48 bytes from pixels of two words
    ((12, 41, 40, 80, 100, 3, 3, 2, 1, 2, 4), S, U),    # stride 2, C = 80
    ((5, 30, 29, 96, 40, 5, 5, 1, 0, 1, 1), B, B),      # +-1 on both sides, no padding
    ((10, 30, 30, 40, 95, 3, 3, 1, 1, 1, 4), B, U),     # +-1 weights, pad elements of a word read as zero
    ((5, 24, 24, 128, 48, 5, 5, 1, 0, 2, 1), U, B),     # +-1 map
    ((40, 14, 14, 256, 300, 2, 2, 1, 1, 4, 3), S, S),   # many small images, two channel tiles
])
def test_maps_widened_into_the_workspace(qb, monkeypatch, lower, shape, w_enc, a_enc):
    """Bit-plane layers large enough to be widened to 8-bit containers first (two launches), with a
    workspace of exactly the size the library asks for and guard bytes behind it."""
    if lower:
        monkeypatch.setenv("QNN_CONV_LOWER", lower)
    case = synth.conv_case(1700 + shape[3] + shape[9], *shape, w_enc=w_enc, a_enc=a_enc, out_bits=1 + shape[4] % 4)
    npix = case.B * case.OH * case.OW
    assert npix * case.OC * 32 * case.KH * case.KW * ((case.C + 31) // 32) >= 1 << 28
    x, _ = device_map(qb, case, BITPLANES)
    Wp = device_weights(qb, case, BITPLANES)
    thr = torch.from_numpy(case.thr).cuda()
    want = orc.qconv(case.In, case.Wt, case.thr, case.stride, case.pad).reshape(npix, case.OC)
    for out_fmt, raw in ((INT8, False), (BITPLANES, False), (INT8, True)):
        d = conv_desc(qb, case, BITPLANES, out_fmt, 0)
        ws_bytes = qb.qnn_conv_workspace_bytes(d)
        ws = torch.full((ws_bytes + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
        nbytes = qb.qnn_conv_out_bytes(d, not raw)
        out = torch.full((nbytes,), 0xEE, dtype=torch.uint8, device="cuda")
        n0 = qb.qnn_launch_count()
        qb.check(qb.qnn_qconv(d, Wp, x, None if raw else thr, out, ws, ws_bytes))
        assert qb.qnn_launch_count() - n0 == 2
        torch.cuda.synchronize()
        assert qb.qnn_device_status() == (0, 0)
        assert bool((ws[ws_bytes:] == 0xA5).all())
        got = decode_out(out.cpu().numpy(), out_fmt, case.out_bits, npix, case.OC, raw)
        if raw:
            assert np.array_equal(got, orc.conv_direct(case.In, case.Wt, case.stride, case.pad).reshape(npix, case.OC))
        else:
            assert np.array_equal(got, want)


@pytest.mark.parametrize("w_enc,a_enc", [(S, U), (U, S)])
@pytest.mark.parametrize("out_fmt,raw,out_bits", [(INT8, False, 4), (BITPLANES, False, 1), (INT8, True, 2)])
@pytest.mark.parametrize("M,N,K", [(1100, 1001, 1000), (1030, 1027, 1040), (1024, 1025, 1024), (257, 4400, 993)])
def test_sixteen_plane_pairs_on_the_tensor_cores(qb, w_enc, a_enc, out_fmt, raw, out_bits, M, N, K):
    """W4A4 above 2^30 multiply-accumulates: the largest rings, copied in whole 16-byte units (K = 1024),
    in the units a row lies in, or word by word where those do not fit beside the thresholds."""
    case = synth.gemm_case(1800 + M + K, M, N, K, 4, 4, w_enc, a_enc, out_bits=out_bits)
    d = qb.gemm_desc(M, N, K, 4, 4, out_bits, w_enc, a_enc, BITPLANES, out_fmt)
    assert qb.qnn_qgemm_kernel_name(d, not raw) == "qgemm_tc_kernel"
    Wp = qb.pack(qb.to_device_logical(case.W, w_enc), 4, w_enc, BITPLANES)
    Ap = qb.pack(qb.to_device_logical(case.At, a_enc), 4, a_enc, BITPLANES)
    out = qb.qgemm(d, Wp, Ap, None if raw else torch.from_numpy(case.thr).cuda())
    torch.cuda.synchronize()
    assert qb.qnn_device_status() == (0, 0)
    got = decode_out(out.cpu().numpy().view(np.uint8).reshape(-1), out_fmt, out_bits, N, M, raw)
    assert np.array_equal(got, orc.qgemm(case.W, case.At, None if raw else case.thr).T)
