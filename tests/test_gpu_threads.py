"""Several host threads and several streams.

First use of the kernels from several host threads at once: ctypes releases the interpreter lock, so
the library's one-time set-up of a kernel runs in all of them together, with problems of the same kernel
that need different amounts of shared memory."""
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# A process of its own: the kernels must not have been used before.
CHILD = """
import sys, threading
import torch
from paper_1709_04060_b200 import binding as qb
PL, I8, FL = qb.QNN_FMT_BITPLANES, qb.QNN_FMT_INT8, qb.QNN_FMT_FIELDS
buf = torch.zeros(96 << 20, dtype=torch.uint8, device="cuda")
out = [torch.empty(8 << 20, dtype=torch.uint8, device="cuda") for _ in range(8)]
torch.cuda.synchronize()
st = torch.cuda.current_stream().cuda_stream
bad = []

def call(i, d, barrier):
    barrier.wait()
    for _ in range(2):
        s = qb.qnn_qgemm(d, buf, buf, None, out[i], None, 0, st)
        if s != 0:
            bad.append((s, d.w_fmt, d.w_bits, d.a_bits, d.N, d.K))

def together(descs):
    barrier = threading.Barrier(len(descs))
    ts = [threading.Thread(target=call, args=(i, d, barrier)) for i, d in enumerate(descs)]
    [t.start() for t in ts]; [t.join() for t in ts]

for w in (1, 2, 3, 4):
    for a_enc in (0, 1):
        # few columns, one instantiation: 16 to 200 KB of activation columns
        for fmt, N, Ks in ((PL, 8, (10000, 2016, 6048, 10016)), (PL, 16, (7010, 480, 3040, 7010)),
                           (FL, 8, (9000, 512, 4096, 9000)), (FL, 16, (8000, 512, 4096, 8000))):
            if fmt == FL and w == 3:
                continue
            together([qb.qnn_gemm_desc(64, N, K, w, 2, 1, 1, a_enc, fmt, PL if fmt == PL else I8, I8, 0, 0) for K in Ks])
# bit planes expanded in the tensor-core kernel, one instantiation: rings of 32 to 100 KB
together([qb.qnn_gemm_desc(128, 200, K, w, a, 1, 1, 0, PL, PL, I8, 0, 0) for w, a, K in
          ((1, 1, 512), (4, 3, 500), (2, 2, 512), (3, 4, 500))])
torch.cuda.synchronize()
assert qb.qnn_device_status() == (0, 0)
print("failed calls:", bad)
sys.exit(1 if bad else 0)
"""


def test_threads_that_use_a_kernel_first_together():
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, (r.stdout + r.stderr)[-2000:]


def test_scratch_of_a_call_on_another_stream():
    """binding.qconv on a stream that is still busy: the workspace it drops on return must not be handed to
    the current stream's next tensor while the layer has yet to write it.  (Two layers: the widened bit
    planes and, for the explicit lowering, 8-bit containers.)"""
    from paper_1709_04060_b200 import binding as qb
    side = torch.cuda.Stream()
    for fmt in (qb.QNN_FMT_BITPLANES, qb.QNN_FMT_INT8):
        C, k = (96, 5) if fmt == qb.QNN_FMT_BITPLANES else (20, 3)
        d = qb.qnn_conv_desc(8, 27, 27, C, 0, 256, k, k, 1, k // 2, 1, 2, 2, 0, 0, fmt, qb.QNN_FMT_INT8, 0)
        x = torch.ones(1 << 20, dtype=torch.uint8, device="cuda")
        W = torch.ones(1 << 20, dtype=torch.uint8, device="cuda")
        thr = torch.arange(256 * 3, dtype=torch.int32, device="cuda")
        n = qb.qnn_conv_workspace_bytes(d)
        out = torch.empty(qb.qnn_conv_out_bytes(d, True), dtype=torch.uint8, device="cuda")
        for warm in range(2):                                  # the pools know the size
            qb.qconv(d, W, x, thr, out, stream=side.cuda_stream)
            torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(20_000_000)                      # about 10 ms
        qb.qconv(d, W, x, thr, out, stream=side.cuda_stream)
        mine = [torch.full((n,), 7, dtype=torch.uint8, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        assert all(bool((t == 7).all()) for t in mine)
