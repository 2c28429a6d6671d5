"""CPU-side checks of the C ABI: the shared library loads, exports every symbol the
header declares, and its host-only logic (size queries, argument validation)
behaves as documented.  No kernel is launched here."""
import ctypes
import os
import re
import subprocess
import sys

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def qb():
    import __graft_entry__ as ge
    ge.build()
    from paper_1709_04060_b200 import binding
    return binding


def _declared_functions():
    text = open(os.path.join(ROOT, "include", "qnn.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(qnn_[a-z0-9_]+)\s*\(", text)))


def test_exports_match_header(qb):
    declared = _declared_functions()
    assert len(declared) >= 20
    lib = ctypes.CDLL(qb.LIB_PATH)
    for name in declared:
        assert hasattr(lib, name), f"{name} declared in qnn.h but not exported"
    assert sorted(qb.EXPORTS) == [d for d in declared if d in qb.EXPORTS]
    missing_in_binding = [d for d in declared if d not in qb.EXPORTS]
    assert missing_in_binding == [], missing_in_binding
    for name in declared:
        assert hasattr(qb, name), f"binding lacks {name}"


def test_no_oracle_or_cpu_fallback_in_product():
    """The product package must not reference the oracle."""
    pkg = os.path.join(ROOT, "paper_1709_04060_b200")
    for dirpath, _, files in os.walk(pkg):
        if "_build" in dirpath:
            continue
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                src = open(os.path.join(dirpath, f)).read()
                assert "import oracle" not in src and "from oracle" not in src, f
                assert "qnn_oracle" not in src, f


def test_version_and_status_strings(qb):
    assert qb.qnn_version() >= 100
    assert qb.qnn_status_string(0) == "ok"
    for s in range(-6, 0):
        assert qb.qnn_status_string(s) not in ("ok", "unknown status")


def test_packed_sizes(qb):
    assert qb.qnn_packed_ld(576, qb.QNN_FMT_BITPLANES) == 18
    assert qb.qnn_packed_ld(577, qb.QNN_FMT_BITPLANES) == 19
    assert qb.qnn_packed_ld(363, qb.QNN_FMT_INT8) == 368
    # config-1 operand sizes: W 1 x 64 x 18 words, A 2 x 256 x 18 words
    assert qb.qnn_packed_bytes(qb.qnn_pack_desc(64, 576, 1, 2, 0)) == 4608
    assert qb.qnn_packed_bytes(qb.qnn_pack_desc(256, 576, 2, 0, 0)) == 36864
    assert qb.qnn_packed_bytes(qb.qnn_pack_desc(256, 576, 2, 0, 1)) == 256 * 576
    assert qb.qnn_packed_bytes(qb.qnn_pack_desc(0, 576, 2, 0, 1)) == 0


def test_gemm_out_sizes(qb):
    d = qb.gemm_desc(64, 256, 576, 1, 2, 2, 2, 0, 0, qb.QNN_FMT_INT8)
    assert qb.qnn_gemm_out_bytes(d, True) == 256 * 64
    assert qb.qnn_gemm_out_bytes(d, False) == 256 * 64 * 4
    d = qb.gemm_desc(70, 10, 64, 1, 2, 2, 2, 0, 0, qb.QNN_FMT_BITPLANES)
    assert qb.qnn_gemm_out_bytes(d, True) == 2 * 10 * 3 * 4
    d = qb.gemm_desc(70, 10, 64, 1, 2, 2, 2, 0, 0, qb.QNN_FMT_INT8)
    assert qb.qnn_gemm_out_bytes(d, True) == 10 * 80


def test_conv_geometry(qb):
    # AlexNet conv2: 27x27x96, 5x5 pad 2 -> lowered (256, 2400, 729)
    d = qb.qnn_conv_desc(1, 27, 27, 96, 0, 256, 5, 5, 1, 2, 1, 2, 2, 2, 0, 0, 1, 0)
    assert qb.qnn_conv_out_h(d) == 27 and qb.qnn_conv_out_w(d) == 27
    assert qb.qnn_conv_lowered_k(d) == 2400
    assert qb.qnn_conv_lowered_bytes(d) == 2 * 729 * 75 * 4
    d.fmt = 1
    assert qb.qnn_conv_lowered_k(d) == 2400
    assert qb.qnn_conv_lowered_bytes(d) == 729 * 2400
    # conv1: 227x227x3, 11x11 stride 4 -> (96, 363, 3025); each filter row (33 bytes) is a
    # run padded to 48 bytes, so the lowered depth is 11 * 48
    d = qb.qnn_conv_desc(1, 227, 227, 3, 3, 96, 11, 11, 4, 0, 8, 8, 2, 1, 0, 1, 1, 0)
    assert qb.qnn_conv_out_h(d) == 55
    assert qb.qnn_conv_lowered_k(d) == 11 * 48
    assert qb.qnn_conv_lowered_bytes(d) == 3025 * 528
    # channel count not a multiple of 32: every pixel is padded to whole words
    d = qb.qnn_conv_desc(1, 8, 8, 40, 0, 16, 3, 3, 1, 1, 1, 2, 2, 2, 0, 0, 1, 0)
    assert qb.qnn_conv_lowered_k(d) == 32 * 9 * 2


def test_argument_validation_without_launch(qb):
    """Errors are detected on the host before any CUDA call (fake aligned addresses)."""
    P = 0x10000
    ok = dict(M=64, N=256, K=576, w_bits=1, a_bits=2, out_bits=2, w_enc=2, a_enc=0,
              fmt=0, out_fmt=1)

    def call(**kw):
        a = dict(ok); a.update(kw)
        ptrs = a.pop("ptrs", (P, P, P, P))
        path = a.pop("path", 0)
        d = qb.gemm_desc(a["M"], a["N"], a["K"], a["w_bits"], a["a_bits"], a["out_bits"],
                         a["w_enc"], a["a_enc"], a["fmt"], a["out_fmt"], path)
        if "a_fmt" in a:
            d.a_fmt = a["a_fmt"]
        return qb.qnn_qgemm(d, ptrs[0], ptrs[1], ptrs[2], ptrs[3], None, 0, stream=0)

    assert call(M=0) == qb.QNN_ERR_INVALID_ARG
    assert call(K=-1) == qb.QNN_ERR_INVALID_ARG
    assert call(w_bits=9) == qb.QNN_ERR_INVALID_ARG
    assert call(out_bits=5) == qb.QNN_ERR_INVALID_ARG
    assert call(w_enc=3) == qb.QNN_ERR_INVALID_ARG
    assert call(w_bits=2) == qb.QNN_ERR_UNSUPPORTED            # bipolar needs 1 bit
    assert call(a_fmt=1) == qb.QNN_ERR_UNSUPPORTED             # mixed operand formats
    assert call(path=qb.QNN_PATH_TCGEN05_I8) == qb.QNN_ERR_UNSUPPORTED   # planes on tensor path
    assert call(fmt=0, w_enc=1, w_bits=8, a_bits=8) == qb.QNN_ERR_UNSUPPORTED  # bit-serial > 4 bits
    assert call(ptrs=(None, P, P, P)) == qb.QNN_ERR_INVALID_ARG
    assert call(ptrs=(P, P, P, None)) == qb.QNN_ERR_INVALID_ARG
    assert call(ptrs=(P + 4, P, P, P)) == qb.QNN_ERR_ALIGNMENT
    assert call(ptrs=(P, P, P + 2, P)) == qb.QNN_ERR_ALIGNMENT

    pd = qb.qnn_pack_desc(4, 64, 2, qb.QNN_ENC_BIPOLAR, 0)
    assert qb.qnn_pack(pd, P, P, stream=0) == qb.QNN_ERR_UNSUPPORTED
    pd = qb.qnn_pack_desc(4, 64, 0, 0, 0)
    assert qb.qnn_pack(pd, P, P, stream=0) == qb.QNN_ERR_INVALID_ARG
    pd = qb.qnn_pack_desc(4, 64, 2, 0, 0)
    assert qb.qnn_pack(pd, P + 1, P, stream=0) == qb.QNN_ERR_ALIGNMENT

    cd = qb.qnn_conv_desc(1, 27, 27, 96, 0, 256, 5, 5, 1, 2, 1, 2, 2, 2, 0, 0, 1, 0)
    assert qb.qnn_qconv(cd, P, P, P, P, None, 0, stream=0) == qb.QNN_ERR_WORKSPACE
    assert qb.qnn_qconv(cd, P, P, P, P, P, 16, stream=0) == qb.QNN_ERR_WORKSPACE
    cd.a_enc, cd.a_bits = qb.QNN_ENC_BIPOLAR, 1
    assert qb.qnn_im2col(cd, P, P, stream=0) == qb.QNN_ERR_UNSUPPORTED    # zero pad not representable
    cd = qb.qnn_conv_desc(1, 3, 3, 96, 0, 256, 5, 5, 1, 0, 1, 2, 2, 2, 0, 0, 1, 0)
    assert qb.qnn_im2col(cd, P, P, stream=0) == qb.QNN_ERR_INVALID_ARG    # filter larger than image

    pl = qb.qnn_pool_desc(1, 2, 2, 16, 3, 2, 2, 1)
    assert qb.qnn_maxpool(pl, P, P, stream=0) == qb.QNN_ERR_INVALID_ARG


def test_gemm_workspace_size_rule(qb):
    """qnn_gemm_workspace_bytes (host only; 148 SMs assumed when there is no GPU): non-zero exactly
    where the CTA-pair kernel would leave a last round of tiles at most half full -- 8192 bytes of
    flags plus 256 KB per tile of that round."""
    if torch.cuda.is_available() and torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the expected sizes are those of 74 SM pairs")
    I8, PL = qb.QNN_FMT_INT8, qb.QNN_FMT_BITPLANES

    def ws(M, N, K, fmt=I8):
        return qb.qnn_gemm_workspace_bytes(qb.qnn_gemm_desc(M, N, K, 1, 2, 2, 2, 0, fmt, fmt, I8, 0, 0))

    assert ws(4096, 4096, 4096) == 8192 + 34 * 256 * 1024     # 256 tiles on 74 pairs: 3 rounds + 34
    assert ws(5120, 5120, 5120) == 8192 + 30 * 256 * 1024     # 400 tiles: 5 rounds + 30
    assert ws(8192, 8192, 8192) == 0                          # 1024 tiles: the last round holds 62 of 74
    assert ws(4096, 4096, 128) == 0                           # one k-block: nothing to split
    assert ws(4096, 1024, 4096) == 0                          # not the CTA-pair kernel
    assert ws(64, 256, 576) == 0
    assert ws(4096, 4096, 4096, PL) == 0                      # bit planes: another path


def test_kernel_choice_follows_the_documented_rule(qb):
    """qnn_qgemm_kernel (host only): the shape-driven choice documented in qnn.h -- the operand
    format is the caller's, the kernel follows from the shape (size sweep of Section 4.1.2)."""
    I8, PL, FL = qb.QNN_FMT_INT8, qb.QNN_FMT_BITPLANES, qb.QNN_FMT_FIELDS

    def k(M, N, K, w_fmt, a_fmt, path=0, w=2, a=2):
        d = qb.qnn_gemm_desc(M, N, K, w, a, 2, 1, 0, w_fmt, a_fmt, I8, path, 0)
        return qb.qnn_qgemm_kernel(d, True)

    assert k(4096, 4096, 4096, I8, I8) == qb.QNN_KERNEL_TENSOR_CTA_PAIR
    assert k(8192, 8192, 8192, I8, I8) == qb.QNN_KERNEL_TENSOR_CTA_PAIR
    assert k(4096, 1024, 4096, I8, I8) == qb.QNN_KERNEL_TENSOR            # fewer than 2048 columns
    assert k(128, 4096, 4096, I8, I8) == qb.QNN_KERNEL_TENSOR             # fewer than 256 channels
    assert k(64, 256, 576, I8, I8) == qb.QNN_KERNEL_TENSOR                # config 1
    assert k(8192, 1, 8192, I8, I8) == qb.QNN_KERNEL_BYTES_FEW_COLUMNS
    assert k(8192, 8, 8192, I8, I8) == qb.QNN_KERNEL_BYTES_FEW_COLUMNS
    assert k(8192, 16, 8192, I8, I8) == qb.QNN_KERNEL_TENSOR
    assert k(8192, 8, 8192, I8, I8, path=2) == qb.QNN_KERNEL_TENSOR       # path forced
    assert k(8192, 16, 8192, PL, PL) == qb.QNN_KERNEL_PLANES_FEW_COLUMNS
    assert k(8192, 17, 8192, PL, PL) == qb.QNN_KERNEL_PLANES_TILED
    assert k(64, 256, 576, PL, PL) == qb.QNN_KERNEL_PLANES_TILED
    assert k(8192, 16, 8192, FL, I8) == qb.QNN_KERNEL_FIELDS_FEW_COLUMNS
    assert k(8192, 17, 8192, FL, I8) == qb.QNN_ERR_UNSUPPORTED
    assert k(64, 64, 64, I8, PL) == qb.QNN_ERR_UNSUPPORTED                # mixed formats


def test_import_does_not_need_private_functions_of_torch(qb):
    """A torch build without the two functions behind the short way to the stream handle: the library
    still imports and answers host queries."""
    code = ("import torch\n"
            "for n in ('_cuda_getCurrentRawStream', '_cuda_getDevice'):\n"
            "    if hasattr(torch._C, n): delattr(torch._C, n)\n"
            "from paper_1709_04060_b200 import binding as qb\n"
            "assert qb.qnn_packed_ld(576, qb.QNN_FMT_BITPLANES) == 18\n"
            "assert qb.qnn_pack(qb.qnn_pack_desc(4, 64, 0, 0, 0), 16, 16, stream=0) == qb.QNN_ERR_INVALID_ARG\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-1500:]


def test_kernel_names_on_both_sides_of_every_rule(qb):
    """qnn_qgemm_kernel_name (host only) on both sides of each line the dispatch draws within a format;
    qnn_qgemm takes its decision from the same function."""
    I8, PL, FL = qb.QNN_FMT_INT8, qb.QNN_FMT_BITPLANES, qb.QNN_FMT_FIELDS
    S, B = qb.QNN_ENC_SIGNED, qb.QNN_ENC_BIPOLAR

    def k(M, N, K, fmt, w=2, a=2, out=I8, thr=True, path=0, skip=0, w_enc=S, a_enc=0):
        d = qb.qnn_gemm_desc(M, N, K, w, a, 2, w_enc, a_enc, fmt, PL if fmt == PL else I8, out, path, skip)
        return qb.qnn_qgemm_kernel_name(d, thr)

    mma, popc, tiled, tc = "gemv_mma_kernel", "gemv_planes_kernel", "qgemm_bitserial_kernel", "qgemm_tc_kernel"
    # packed weights: two columns on; one column where a clearing launch would be needed; depths that
    # an SM's shared memory does not hold
    assert k(8192, 1, 8192, FL) == "gemv_fields_dp4a_kernel"
    assert k(8192, 1, 8192, FL, out=PL) == mma
    assert k(8192, 1, 8192, FL, out=PL, thr=False) == "gemv_fields_dp4a_kernel"
    assert k(8192, 2, 8192, FL) == mma
    assert k(8192, 16, 9216, FL) == mma
    assert k(8192, 16, 13376, FL) == mma                      # 209 KB of column bytes
    assert k(8192, 16, 13377, FL) == "gemv_fields_kernel"
    assert k(8192, 8, 25000, FL, w=4, a=4) == mma
    assert k(8192, 8, 26000, PL) == mma
    assert k(8192, 16, 16384, FL) == "gemv_fields_kernel"
    # bytes: three columns on from 2^23 weights; fewer where pad bytes need clearing, below 2^26 weights
    assert k(2048, 3, 4096, I8) == mma
    assert k(2048, 3, 4080, I8) == "gemv_i8_kernel"
    assert k(4096, 2, 4096, I8) == "gemv_i8_kernel"
    assert k(4100, 1, 4096, I8) == mma
    assert k(4100, 1, 4096, I8, thr=False) == "gemv_i8_kernel"
    assert k(8200, 1, 8192, I8, out=PL) == "gemv_i8_kernel"
    assert k(4096, 9, 4096, I8) == tc
    assert k(4096, 4096, 4096, I8) == "qgemm_tc2_kernel"
    # planes, few columns: the estimate of both kernels, twelve plane pairs and more of 2^22 weights aside; neither
    # needs a clearing launch, so pad bytes and the output's format do not matter
    assert k(8192, 1, 8192, PL) == popc
    assert k(8192, 2, 8192, PL) == mma
    assert k(8192, 1, 8192, PL, w=3, a=4) == mma
    assert k(8192, 1, 8192, PL, w=4, a=4) == mma
    assert k(8192, 1, 8192, PL, w=3, a=3) == popc
    assert k(12000, 16, 64, PL, w=2, a=1) == mma
    assert k(960, 5, 64, PL, w=2, a=4) == mma
    assert k(5, 12, 647, PL, w=1, a=1, w_enc=B, thr=False) == popc
    for out, thr in ((I8, True), (PL, True), (I8, False)):
        assert k(4095, 1, 4096, PL, out=out, thr=thr) == popc
        assert k(4096, 1, 4096, PL, out=out, thr=thr) == popc
        assert k(101, 16, 64, PL, w=1, a=1, out=out, thr=thr) == popc
        assert k(961, 5, 64, PL, w=2, a=1, out=out, thr=thr) == mma
        assert k(1000, 1, 4096, PL, w=4, a=4, out=out, thr=thr) == mma
        assert k(352, 1, 512, PL, w=2, a=2, out=out, thr=thr) == popc
    assert k(8192, 2, 8192, PL, path=qb.QNN_PATH_BITSERIAL) == popc
    assert k(8192, 2, 8192, PL, skip=1) == popc
    # planes, tiled: sixteen plane pairs up to 2^30, a single pair between 2^24 and 2^27, the forced path
    # and skipped pairs stay with AND/POPC
    assert k(1024, 1024, 1024, PL) == tc
    assert k(1024, 1024, 1024, PL, w=4, a=4) == tiled
    assert k(1024, 1024, 1025, PL, w=4, a=4) == tc
    assert k(1024, 1024, 1024, PL, w=3, a=4) == tc
    assert k(512, 512, 512, PL, w=1, a=1, w_enc=B, a_enc=B) == tiled
    assert k(512, 512, 513, PL, w=1, a=1, w_enc=B, a_enc=B) == tc
    assert k(1024, 1024, 1024, PL, path=qb.QNN_PATH_BITSERIAL) == tiled
    assert k(1024, 1024, 1024, PL, skip=1) == tiled
    # ... and so do few plane pairs with little work, raw sums or many thresholds
    assert k(325, 313, 132, PL, w=1, a=1, thr=False) == tiled
    assert k(325, 313, 132, PL, w=2, a=3, thr=False) == tc
    assert k(133, 1948, 467, PL, w=2, a=1, thr=False) == tiled
    assert k(133, 1948, 467, PL, w=2, a=1) == tc
    assert k(325, 4000, 132, PL, w=2, a=2, thr=False) == tc
    assert k(64, 256, 576, PL, w=1, a=2, w_enc=B) == tc
    assert k(1000, 3025, 1363, PL, w=2, a=2, thr=False) == tc
    # depths whose tiles would outlast the bounded waits of the tensor-core kernel
    assert k(2, 17, 1 << 25, PL, w=1, a=2, w_enc=B) == tc
    assert k(2, 17, (1 << 25) + 1, PL, w=1, a=2, w_enc=B) == tiled
    assert k(64, 64, 64, I8, w=0) is None


@pytest.mark.parametrize("fmt", [0, 1])
def test_convolutions_refuse_misaligned_thresholds(qb, fmt):
    """As qnn_qgemm does, on the host, whichever kernel the layer would run on (fake addresses)."""
    P = 0x10000
    d = qb.qnn_conv_desc(1, 13, 13, 96, 0, 256, 3, 3, 1, 1, 1, 2, 2, 2, 0, fmt, 1, 0)
    for off in (1, 2, 3):
        assert qb.qnn_qconv(d, P, P, P + off, P, P, 1 << 30, stream=0) == qb.QNN_ERR_ALIGNMENT
        assert qb.qnn_qconv_static(d, P, P, P + off, P, stream=0) == qb.QNN_ERR_ALIGNMENT
