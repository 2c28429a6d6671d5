"""Three-channel layers whose image rows the tensor core reads in place, alone and with the 3 x 3,
stride 2 max-pool in the same kernel, against the oracle: tiles that end inside an image, rings that wrap,
several images per CTA and several CTAs per image, every stride the kernel takes, each output format."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_1709_04060_b200 import synth
from qnn_testutil import decode_out, round_up

pytestmark = pytest.mark.gpu

BITPLANES, INT8 = 0, 1


@pytest.fixture(scope="module")
def qb():
    from paper_1709_04060_b200 import binding
    return binding


def layer(qb, B, H, W, OC, KH, KW, stride, w_bits, a_bits, out_bits, w_enc, a_enc, seed):
    case = synth.conv_case(seed, B, H, W, 3, OC, KH, KW, stride, 0, w_bits, a_bits, w_enc=w_enc, a_enc=a_enc, out_bits=out_bits)
    rows = np.zeros((OC, KH, round_up(KW * 3, 16)), dtype=np.int32)
    rows[:, :, :KW * 3] = case.Wt.reshape(OC, KH, KW * 3)
    Wp = qb.pack(qb.to_device_logical(rows.reshape(OC, -1), w_enc), w_bits, w_enc, INT8)
    x = torch.from_numpy(case.In.astype(np.uint8)).cuda()
    return case, Wp, x, torch.from_numpy(case.thr).cuda()


# Layers that the library itself runs this way: five rounds of tiles on 148 SMs and full ones, or +-1 weights, which
# the kernel with lowering warps does not take.
SHAPES = [
    # B, H, W, OC, KH, KW, stride, w_bits, a_bits, out_bits, w_enc, a_enc
    (28, 227, 227, 96, 11, 11, 4, 8, 8, 2, 1, 0),     # the layer of the network; last tile half empty
    (760, 15, 15, 20, 11, 11, 4, 1, 8, 2, 2, 0),      # four pixels an image, several images a CTA
    (125, 61, 255, 128, 7, 5, 4, 1, 8, 1, 2, 0),      # 63 pixels a row, filter rows not a whole unit
    (40, 40, 131, 33, 3, 3, 2, 1, 8, 3, 2, 1),        # stride 2, signed activations, 65 pixels a row
    (44, 19, 100, 64, 3, 4, 1, 1, 8, 4, 2, 0),        # stride 1
    (250, 33, 37, 1, 1, 1, 4, 1, 8, 2, 2, 0),         # a single tap
    (373, 30, 29, 17, 9, 3, 2, 1, 4, 2, 2, 0),        # filter taller than wide
    (96, 26, 207, 100, 1, 5, 2, 8, 8, 3, 1, 1),       # signed operands, stride 2
    (223, 52, 210, 33, 2, 2, 2, 2, 8, 4, 0, 0),
]


@pytest.mark.parametrize("shape", SHAPES)
def test_rows_read_in_place(qb, shape):
    case, Wp, x, thr = layer(qb, *shape, seed=1700 + shape[1])
    npix = case.B * case.OH * case.OW
    want_raw = orc.qconv(case.In, case.Wt, None, case.stride, 0).reshape(npix, case.OC)
    want = (want_raw[:, :, None] >= case.thr[None]).sum(2)
    for out_fmt, raw in ((INT8, False), (BITPLANES, False), (INT8, True)):
        d = qb.qnn_conv_desc(case.B, case.H, case.Wd, 3, 3, case.OC, case.KH, case.KW, case.stride, 0, case.w_bits,
                             case.a_bits, case.out_bits, case.w_enc, case.a_enc, INT8, out_fmt, 0)
        assert qb.qnn_conv_in_place(d, not raw) == (not raw or case.w_enc == 2)       # sums: only +-1 weights
        nb = qb.qnn_conv_out_bytes(d, not raw)
        out = torch.full((nb + 64,), 0xEE, dtype=torch.uint8, device="cuda")
        ws = torch.zeros(qb.qnn_conv_workspace_bytes(d), dtype=torch.uint8, device="cuda")
        qb.check(qb.qnn_qconv(d, Wp, x, None if raw else thr, out, ws, ws.numel()))
        torch.cuda.synchronize()
        assert qb.qnn_device_status() == (0, 0)
        buf = out.cpu().numpy()
        assert (buf[nb:] == 0xEE).all()
        assert not ws.any()                               # nothing was lowered
        got = decode_out(buf[:nb], out_fmt, case.out_bits, npix, case.OC, raw)
        assert np.array_equal(got, want_raw if raw else want)


@pytest.mark.parametrize("shape,fuses", [(s, s[2] != 131) for s in SHAPES if s[2] in (227, 255, 131)] + [
    ((47, 143, 143, 96, 11, 11, 4, 1, 8, 2, 2, 0), True),      # 34 x 34 map, 16 pooled rows, CTAs that span images
    ((745, 19, 227, 32, 11, 11, 4, 1, 8, 2, 2, 0), True),      # three rows: one pooled row
    ((93, 20, 50, 40, 3, 3, 1, 1, 8, 1, 2, 0), True),          # stride 1, 48 pixels a row; one threshold
    ((107, 33, 101, 64, 5, 5, 2, 1, 8, 2, 2, 1), True),        # stride 2, 49 pixels a row
    ((257, 17, 94, 33, 2, 5, 2, 8, 8, 3, 1, 0), True),         # seven thresholds
    ((48, 142, 55, 70, 2, 3, 1, 8, 8, 4, 1, 0), True),         # stride 1, 8-bit weights, 15 thresholds
    ((59, 83, 115, 70, 3, 7, 2, 8, 8, 4, 1, 1), True),
    ((71, 65, 126, 70, 2, 7, 2, 8, 8, 1, 1, 0), True),
    ((93, 20, 40, 40, 3, 3, 1, 1, 8, 1, 2, 0), False),         # 40 units a row: three output rows a tile
])
def test_pool_in_the_same_kernel(qb, shape, fuses):
    case, Wp, x, thr = layer(qb, *shape, seed=1900 + shape[1])
    OH, OW, PH, PW = case.OH, case.OW, (case.OH - 3) // 2 + 1, (case.OW - 3) // 2 + 1
    codes = orc.qconv(case.In, case.Wt, case.thr, case.stride, 0).reshape(case.B, OH, OW, case.OC)
    want = np.max([codes[:, i:i + 2 * PH - 1:2, j:j + 2 * PW - 1:2] for i in range(3) for j in range(3)], axis=0)
    for out_fmt in (INT8, BITPLANES):
        d = qb.qnn_conv_desc(case.B, case.H, case.Wd, 3, 3, case.OC, case.KH, case.KW, case.stride, 0, case.w_bits,
                             case.a_bits, case.out_bits, case.w_enc, case.a_enc, INT8, out_fmt, 0)
        assert qb.qnn_conv_maxpool_fuses(d, 3, 2) == fuses
        if not fuses:
            assert qb.qnn_qconv_maxpool(d, 3, 2, Wp, x, thr, x) == qb.QNN_ERR_UNSUPPORTED
            continue
        npix = case.B * PH * PW
        nb = npix * round_up(case.OC, 16) if out_fmt == INT8 else case.out_bits * npix * round_up(case.OC, 32) // 8
        out = torch.full((nb + 64,), 0xEE, dtype=torch.uint8, device="cuda")
        qb.check(qb.qnn_qconv_maxpool(d, 3, 2, Wp, x, thr, out))
        torch.cuda.synchronize()
        assert qb.qnn_device_status() == (0, 0)
        buf = out.cpu().numpy()
        assert (buf[nb:] == 0xEE).all()
        assert np.array_equal(decode_out(buf[:nb], out_fmt, case.out_bits, npix, case.OC, False), want.reshape(npix, case.OC))


def test_only_that_pool_and_those_layers_fuse(qb):
    def d(**kw):
        v = dict(B=28, H=227, W=227, C=3, in_pitch=3, OC=96, KH=11, KW=11, stride=4, pad=0, w_bits=8, a_bits=8, out_bits=2,
                 w_enc=1, a_enc=0, fmt=INT8, out_fmt=INT8, path=0)
        v.update(kw)
        return qb.qnn_conv_desc(*v.values())
    assert qb.qnn_conv_maxpool_fuses(d(), 3, 2)
    assert not qb.qnn_conv_maxpool_fuses(d(), 2, 2)
    assert not qb.qnn_conv_maxpool_fuses(d(), 3, 1)
    assert not qb.qnn_conv_maxpool_fuses(d(in_pitch=0), 3, 2)
    assert not qb.qnn_conv_maxpool_fuses(d(C=4, in_pitch=4), 3, 2)
    assert not qb.qnn_conv_maxpool_fuses(d(OC=129), 3, 2)
    assert not qb.qnn_conv_maxpool_fuses(d(stride=3), 3, 2)
    assert not qb.qnn_conv_maxpool_fuses(d(pad=1), 3, 2)
    assert not qb.qnn_conv_maxpool_fuses(d(B=27), 3, 2)        # fewer than five rounds of pooled rows
    t = torch.zeros(64, dtype=torch.uint8, device="cuda")
    n0 = qb.qnn_launch_count()
    assert qb.qnn_qconv_maxpool(d(pad=1), 3, 2, t, t, t, t) == qb.QNN_ERR_UNSUPPORTED
    assert qb.qnn_qconv_maxpool(d(), 3, 2, t, t, None, t) == qb.QNN_ERR_INVALID_ARG
    assert qb.qnn_launch_count() == n0
