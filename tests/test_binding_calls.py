"""The binding's calls on the host: the extension in front of ctypes answers plain arguments as ctypes does
and leaves every other form to it.  No kernel is launched (the descriptors are refused)."""
import ctypes

import numpy as np
import pytest
import torch


@pytest.fixture(scope="module")
def qb():
    import __graft_entry__ as ge
    ge.build()
    from paper_1709_04060_b200 import binding
    return binding


def calls(qb):
    g = qb.qnn_gemm_desc(0, 256, 576, 1, 2, 2, 2, 0, 1, 1, 1, 0, 0)
    c = qb.qnn_conv_desc(1, 13, 13, 96, 0, 256, 3, 3, 1, 1, 1, 2, 2, 2, 0, 1, 1, 0)
    p = qb.qnn_pack_desc(4, 64, 2, 0, 1)
    pool = qb.qnn_pool_desc(1, 0, 6, 32, 3, 2, 2, 1)
    P = 0x10000
    return [
        (qb.qnn_qgemm, (g, P, P, P, P, None, 0, 0), qb.QNN_ERR_INVALID_ARG),
        (qb.qnn_qconv, (c, P, P, P, P, None, 0, 0), qb.QNN_ERR_WORKSPACE),
        (qb.qnn_qconv, (c, P, P, P + 1, P, P, 1 << 40, 0), qb.QNN_ERR_ALIGNMENT),
        (qb.qnn_qconv_static, (c, P, P, P, None, 0), qb.QNN_ERR_INVALID_ARG),
        (qb.qnn_pack, (p, P + 8, P, 0), qb.QNN_ERR_ALIGNMENT),
        (qb.qnn_planes_to_int8, (p, P, P, 0), qb.QNN_ERR_INVALID_ARG),
        (qb.qnn_im2col, (c, None, P, 0), qb.QNN_ERR_INVALID_ARG),
        (qb.qnn_maxpool, (pool, P, P, 0), qb.QNN_ERR_INVALID_ARG),
    ]


def test_plain_arguments(qb):
    for f, args, status in calls(qb):
        assert f(*args) == status, f.__name__


def test_extension_is_in_use(qb):
    assert qb._fastcall is not None and type(qb._qgemm).__name__ == "Entry"


def test_other_forms_go_the_ctypes_way(qb):
    g = calls(qb)[0][1][0]
    t = torch.zeros(64, 3, dtype=torch.int32)
    assert qb.qnn_qgemm(g, t, t, thr=t, out=t, workspace_bytes=np.int64(0), stream=np.int64(0)) == qb.QNN_ERR_INVALID_ARG
    assert qb.qnn_qgemm(g, torch.nn.Parameter(t, requires_grad=False), t, None, t, None, 0, True) == qb.QNN_ERR_INVALID_ARG
    with pytest.raises(AssertionError):
        qb.qnn_qgemm(g, t.t(), t, t, t, None, 0, 0)            # not contiguous
    with pytest.raises(TypeError):
        qb.qnn_qgemm(g, "x", t, t, t, None, 0, 0)
    with pytest.raises(TypeError):
        qb.qnn_qgemm(None, t, t, t, t, None, 0, 0)
    with pytest.raises(ctypes.ArgumentError):
        qb.qnn_qgemm(qb.qnn_pack_desc(), t, t, t, t, None, 0, 0)


def test_a_descriptor_changed_between_calls_is_read_again(qb):
    g = calls(qb)[0][1][0]
    P = 0x10000
    assert qb.qnn_qgemm(g, P, P, P, P, None, 0, 0) == qb.QNN_ERR_INVALID_ARG
    g.M, g.w_enc, g.w_bits = 64, 2, 2
    assert qb.qnn_qgemm(g, P, P, P, P, None, 0, 0) == qb.QNN_ERR_UNSUPPORTED
