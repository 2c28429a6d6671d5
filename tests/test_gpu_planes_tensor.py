"""Bit planes multiplied on the tensor cores: the tiled product expands both operands to bytes inside the
kernel, the few-column product in registers.  Every output against the CPU oracle, at the sizes where a
tile, a ring slot, a step of the depth or a row of 32 ends; and against the AND/POPC kernels, which a
forced bit-serial path still runs."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_1709_04060_b200 import synth
from qnn_testutil import decode_out

pytestmark = pytest.mark.gpu

PLANES, INT8, FIELDS = 0, 1, 2
U, S, B = synth.UNSIGNED, synth.SIGNED, synth.BIPOLAR


@pytest.fixture(scope="module")
def qb():
    from paper_1709_04060_b200 import binding
    return binding


def check(qb, case, w_fmt, out_fmt, raw=False, path=0):
    a_fmt = INT8 if w_fmt == FIELDS else w_fmt
    Wp = qb.pack(qb.to_device_logical(case.W, case.w_enc), case.w_bits, case.w_enc, w_fmt)
    Ap = qb.pack(qb.to_device_logical(case.At, case.a_enc), case.a_bits, case.a_enc, a_fmt)
    d = qb.qnn_gemm_desc(case.M, case.N, case.K, case.w_bits, case.a_bits, case.out_bits, case.w_enc, case.a_enc,
                         w_fmt, a_fmt, out_fmt, path, 0)
    nbytes = qb.qnn_gemm_out_bytes(d, not raw)
    out = torch.full((max(nbytes, 16),), 0xEE, dtype=torch.uint8, device="cuda")
    qb.check(qb.qnn_qgemm(d, Wp, Ap, None if raw else torch.from_numpy(case.thr).cuda(), out))
    torch.cuda.synchronize()
    assert qb.qnn_device_status() == (0, 0)
    got = decode_out(out.cpu().numpy()[:nbytes], out_fmt, case.out_bits, case.N, case.M, raw)
    want = orc.qgemm(case.W, case.At, None if raw else case.thr).T
    bad = np.argwhere(got != want)
    assert bad.size == 0, f"{len(bad)} mismatches, first at (n,m)={bad[0]}"


ENCODINGS = [(1, B, 2, U), (1, B, 1, B), (1, U, 1, U), (1, S, 3, S), (2, S, 2, U), (2, U, 1, B), (3, S, 3, U),
             (3, U, 2, S), (4, S, 4, U), (4, U, 4, S), (2, S, 4, U), (4, S, 1, U)]


@pytest.mark.parametrize("w_bits,w_enc,a_bits,a_enc", ENCODINGS)
@pytest.mark.parametrize("M,N,K", [(64, 17, 31), (129, 127, 129), (257, 130, 513), (300, 260, 2100), (520, 129, 1024)])
def test_tiled_planes(qb, M, N, K, w_bits, w_enc, a_bits, a_enc):
    """Ragged tiles, depths that end inside a word, a k-block and a ring slot, rows that are and are not
    whole 16-byte units (K = 1024: they are), tiles whose depth two CTAs share."""
    case = synth.gemm_case(7000 + M + N + K, M, N, K, w_bits, a_bits, w_enc, a_enc, out_bits=1 + (M + w_bits) % 4)
    check(qb, case, PLANES, INT8)
    check(qb, case, PLANES, PLANES)
    check(qb, case, PLANES, INT8, raw=True)


@pytest.mark.parametrize("w_bits,w_enc,a_bits,a_enc", [(1, B, 1, U), (2, S, 2, U), (3, S, 3, U)])
def test_tiled_planes_with_a_shared_last_round(qb, w_bits, w_enc, a_bits, a_enc):
    """More tiles than SMs with at most half of them left for the last round, whose tiles are shared by
    two CTAs: their partial sums pass through the operand rings, 512 bytes per channel."""
    case = synth.gemm_case(7100 + w_bits, 256, 150 * 128 - 5, 256 if w_bits < 3 else 520, w_bits, a_bits, w_enc, a_enc, out_bits=2)
    check(qb, case, PLANES, INT8)


@pytest.mark.parametrize("fmt", [PLANES, FIELDS, INT8])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (31, 16, 100), (33, 8, 513), (700, 9, 2048), (96, 3, 4096), (4800, 2, 300),
                                   (65, 5, 8192), (64, 7, 9216), (40, 16, 9300), (50, 2, 70000)])
def test_few_columns(qb, M, N, K, fmt):
    """Tiles of 32 rows and steps of the depth that end early, one tile and several per CTA, loads of
    one, two and four words, depths past what the columns' shared memory holds (other kernels)."""
    if fmt == FIELDS and K == 70000:
        pytest.skip("packed fields refuse this depth")
    kinds = ENCODINGS if fmt == PLANES else [(w, we, a, ae) for (w, we, a, ae) in ENCODINGS if not (we == B and ae == B)]
    for i, (w_bits, w_enc, a_bits, a_enc) in enumerate(kinds if M * K < 300000 else kinds[i0(M, K)::5]):
        case = synth.gemm_case(7200 + M + N + K + i, M, N, K, w_bits, a_bits, w_enc, a_enc, out_bits=1 + (i + M) % 4)
        check(qb, case, fmt, INT8)
        check(qb, case, fmt, PLANES)
        check(qb, case, fmt, INT8, raw=True)


def i0(M, K):
    return (M + K) % 5


@pytest.mark.parametrize("N", [3, 40])
def test_forced_bit_serial_path(qb, N):
    """The AND/POPC kernels, which the library's own choice no longer reaches at these sizes."""
    for w_bits, w_enc, a_bits, a_enc in ENCODINGS:
        case = synth.gemm_case(7300 + N, 130, N, 700, w_bits, a_bits, w_enc, a_enc, out_bits=2)
        check(qb, case, PLANES, INT8, path=1)
        check(qb, case, PLANES, PLANES, path=1)
