"""The few-column tensor-core kernel (one to sixteen columns) at the edges of its plan, against the
oracle: groups of eight rows and pairs of them, depth slices that end inside a load, several passes over a
depth, warps that take other groups, each format and encoding."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_1709_04060_b200 import synth
from qnn_testutil import decode_out

pytestmark = pytest.mark.gpu

BITPLANES, INT8, FIELDS = 0, 1, 2


@pytest.fixture(scope="module")
def qb():
    from paper_1709_04060_b200 import binding
    return binding


@pytest.mark.parametrize("fmt,w,a,w_enc,a_enc", [
    (BITPLANES, 1, 2, 2, 0), (BITPLANES, 2, 4, 1, 1), (BITPLANES, 3, 1, 0, 2), (BITPLANES, 4, 3, 1, 0), (BITPLANES, 1, 1, 2, 2),
    (FIELDS, 1, 8, 2, 0), (FIELDS, 2, 2, 1, 1), (FIELDS, 4, 4, 1, 0), (INT8, 8, 8, 1, 0), (INT8, 3, 8, 0, 1),
])
@pytest.mark.parametrize("M,N,K", [
    (4100, 2, 4097), (1201, 8, 9216),          # rows past whole groups; one pass more than 16 warps hold
    (2500, 9, 1000), (321, 16, 9120),          # two blocks of columns; passes
    (4100, 5, 33), (1200, 3, 2080),            # shallow: several groups at a time
    (19000, 2, 512),                           # more groups a CTA than warps
    (4100, 4, 4097), (1200, 7, 2080),          # ... of few plane pairs too
    (4100, 8, 1025), (3000, 5, 9729),          # bytes as sums; three quarters of the steps of a warp
    (1000, 16, 11000), (500, 6, 20000),        # deeper than 16 warps hold
])
def test_plan_edges(qb, fmt, w, a, w_enc, a_enc, M, N, K):
    if fmt == INT8 and N > 8:
        N = 8
    case = synth.gemm_case(4400 + M + 3 * K + w, M, N, K, w, a, w_enc, a_enc, out_bits=3)
    a_fmt = INT8 if fmt == FIELDS else fmt
    Wp = qb.pack(qb.to_device_logical(case.W, w_enc), w, w_enc, fmt)
    Ap = qb.pack(qb.to_device_logical(case.At, a_enc), a, a_enc, a_fmt)
    thr = torch.from_numpy(case.thr).cuda()
    sums = orc.qgemm(case.W, case.At, None).T
    codes = (sums[:, :, None] >= case.thr[None]).sum(2)
    for out_fmt, raw in ((INT8, False), (BITPLANES, False), (INT8, True)):
        d = qb.qnn_gemm_desc(M, N, K, w, a, 3, w_enc, a_enc, fmt, a_fmt, out_fmt, 0, 0)
        name = qb.qnn_qgemm_kernel_name(d, not raw)
        if fmt == FIELDS or (fmt == BITPLANES and (a > 1 or (N > 3 and M > 1000))):
            assert name == "gemv_mma_kernel"
        elif fmt == INT8 and K <= 12288:                   # what the byte dot products stage
            assert (name == "gemv_mma_kernel") == ((not raw and (out_fmt == BITPLANES or M % 16 != 0)) or (N >= 4 and M * K >= 3 << 20))
        nb = qb.qnn_gemm_out_bytes(d, not raw)
        out = torch.full((nb + 64,), 0xEE, dtype=torch.uint8, device="cuda")
        qb.check(qb.qnn_qgemm(d, Wp, Ap, None if raw else thr, out))
        torch.cuda.synchronize()
        buf = out.cpu().numpy()
        assert (buf[nb:] == 0xEE).all()
        assert np.array_equal(decode_out(buf[:nb], out_fmt, 3, N, M, raw), sums if raw else codes)


@pytest.mark.parametrize("w,a,w_enc,a_enc", [(1, 2, 2, 0), (2, 2, 1, 0), (3, 1, 0, 2)])
@pytest.mark.parametrize("M,N,K", [(1, 1, 31), (17, 5, 128), (4097, 1, 4096), (9700, 3, 96), (10001, 16, 70)])
def test_counting_kernel_writes_whole_rows(qb, w, a, w_enc, a_enc, M, N, K):
    """The AND/POPC kernel writes pad bytes and pad bits itself: rows past whole groups of eight, several
    turns of a CTA."""
    case = synth.gemm_case(4700 + M + w, M, N, K, w, a, w_enc, a_enc, out_bits=3)
    Wp = qb.pack(qb.to_device_logical(case.W, w_enc), w, w_enc, BITPLANES)
    Ap = qb.pack(qb.to_device_logical(case.At, a_enc), a, a_enc, BITPLANES)
    thr = torch.from_numpy(case.thr).cuda()
    sums = orc.qgemm(case.W, case.At, None).T
    codes = (sums[:, :, None] >= case.thr[None]).sum(2)
    for out_fmt in (INT8, BITPLANES):
        d = qb.qnn_gemm_desc(M, N, K, w, a, 3, w_enc, a_enc, BITPLANES, BITPLANES, out_fmt, qb.QNN_PATH_BITSERIAL, 0)
        assert qb.qnn_qgemm_kernel_name(d, True) == "gemv_planes_kernel"
        nb = qb.qnn_gemm_out_bytes(d, True)
        out = torch.full((nb + 64,), 0xEE, dtype=torch.uint8, device="cuda")
        qb.check(qb.qnn_qgemm(d, Wp, Ap, thr, out))
        torch.cuda.synchronize()
        buf = out.cpu().numpy()
        assert (buf[nb:] == 0xEE).all()
        assert np.array_equal(decode_out(buf[:nb], out_fmt, 3, N, M, False), codes)
        if out_fmt == INT8:
            assert (buf[:nb].reshape(N, -1)[:, M:] == 0).all()
        elif M % 32:
            assert (buf[:nb].view(np.uint32).reshape(3 * N, -1)[:, -1] >> (M % 32) == 0).all()


@pytest.mark.parametrize("K,a,kernel", [
    (24576, 4, "gemv_planes_kernel"), (24577, 4, "qgemm_bitserial_kernel"),
    (98304, 1, "gemv_planes_kernel"), (98176, 1, "gemv_planes_kernel"), (98305, 1, "qgemm_bitserial_kernel"),
])
def test_deepest_columns_that_the_counting_kernel_stages(qb, K, a, kernel):
    """48 KB of columns, the kernel's own arrays beside them; deeper ones go to the tiled kernel."""
    case = synth.gemm_case(4900 + K, 9, 2, K, 1, a, 0, 0, out_bits=2)
    Wp = qb.pack(qb.to_device_logical(case.W, 0), 1, 0, BITPLANES)
    Ap = qb.pack(qb.to_device_logical(case.At, 0), a, 0, BITPLANES)
    d = qb.qnn_gemm_desc(9, 2, K, 1, a, 2, 0, 0, BITPLANES, BITPLANES, INT8, qb.QNN_PATH_BITSERIAL, 0)
    assert qb.qnn_qgemm_kernel_name(d, False) == kernel
    out = torch.zeros(qb.qnn_gemm_out_bytes(d, False), dtype=torch.uint8, device="cuda")
    qb.check(qb.qnn_qgemm(d, Wp, Ap, None, out))
    assert np.array_equal(out.cpu().numpy().view(np.int32).reshape(2, 9), orc.qgemm(case.W, case.At, None).T)
