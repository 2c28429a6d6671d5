"""What the framework's users have it do, as cases that can be timed and compared.

Three kinds of work, all through the entry points of `paper_1709_04060_b200.binding` and
`paper_1709_04060_b200.alexnet`:

  gemm     one fused GEMM + threshold layer: a fully connected layer or a convolution that is a
           matrix product already.  Operands are few-bit values in 8-bit containers, bit planes or
           packed fields; the activations arrive from a previous layer, or (`feed`) are packed or
           widened in the same pass.
  conv     one convolution layer on a channels-last map, with its lowering and thresholds.
  alexnet  the whole AlexNet-shaped network: image to logits.

Every output is a whole number, so any two correct implementations agree on every bit.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1709_04060_b200 import alexnet, synth
from paper_1709_04060_b200 import binding as qb

UNSIGNED, SIGNED, BIPOLAR = qb.QNN_ENC_UNSIGNED, qb.QNN_ENC_SIGNED, qb.QNN_ENC_BIPOLAR
FMT = {"planes": qb.QNN_FMT_BITPLANES, "int8": qb.QNN_FMT_INT8, "fields": qb.QNN_FMT_FIELDS}


def _gemm(M, N, K, w, a, fmt, out="int8", feed="packed", xnor=False):
    return {"kind": "gemm", "M": M, "N": N, "K": K, "w": w, "a": a, "fmt": fmt, "out": out, "feed": feed, "xnor": xnor}


def _conv(B, H, C, OC, k, stride, pad, w, a, fmt):
    return {"kind": "conv", "B": B, "H": H, "C": C, "OC": OC, "k": k, "stride": stride, "pad": pad, "w": w, "a": a,
            "fmt": fmt}


def _net(B, mode, graph):
    return {"kind": "alexnet", "B": B, "mode": mode, "graph": graph}


def listed():
    return [
        # a small layer, one call of it: latency
        dict(_gemm(64, 256, 576, 1, 2, "int8"), name="gemm 64x256x576 w1a2"),
        # the microbenchmark sweep's square product, activations packed in the pass as a producer
        # that holds plain bytes does
        dict(_gemm(4096, 4096, 4096, 1, 2, "int8", feed="logical"), name="gemm 4096 w1a2, packed"),
        # the same product on data that is shipped and kept as bit planes, widened on the device
        dict(_gemm(4096, 4096, 4096, 4, 4, "int8", out="planes", feed="planes"), name="gemm 4096 w4a4, shipped"),
        # a layer kept in bit planes from end to end, sizes that are multiples of nothing
        dict(_gemm(1000, 3025, 1363, 3, 3, "planes", out="planes"), name="gemm ragged w3a3 planes"),
        # fully connected layers at batch 1, 4, 16 on packed weights (memory bound), in the two
        # packed formats, and the 8-bit classifier layer with raw logits at an odd small batch
        dict(_gemm(8192, 1, 8192, 2, 2, "fields"), name="fc 8192 N=1 w2a2 fields"),
        dict(_gemm(8192, 4, 8192, 2, 2, "planes"), name="fc 8192 N=4 w2a2 planes"),
        dict(_gemm(8192, 16, 8192, 4, 4, "fields"), name="fc 8192 N=16 w4a4 fields"),
        dict(_gemm(1000, 7, 4096, 8, 2, "int8", out="raw"), name="fc 1000 N=7 w8a2 logits"),
        # one convolution layer (27 x 27 x 96 -> 256, 5 x 5) at a middle batch in both formats
        dict(_conv(64, 27, 96, 256, 5, 1, 2, 1, 2, "int8"), name="conv 5x5 B=64 int8"),
        dict(_conv(8, 27, 96, 256, 5, 1, 2, 1, 2, "planes"), name="conv 5x5 B=8 planes"),
        # the network, one image at a time (a recorded graph is replayed) and in large batches
        dict(_net(1, "auto", True), name="alexnet B=1 graph"),
        dict(_net(256, "auto", False), name="alexnet B=256"),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "fc", "fc", "conv", "conv", "alexnet"])
    w, a = rng.randint(1, 4), rng.randint(1, 4)
    if kind == "gemm":
        fmt = rng.choice(["int8", "planes"])
        most = 1 << (34 if fmt == "int8" else 31)
        while True:
            M, N, K = _log(rng, 16, 8192), _log(rng, 17, 8192), _log(rng, 64, 8192)
            if M * N * K <= most:
                break
        feed = rng.choice(["packed", "logical", "planes"]) if fmt == "int8" else rng.choice(["packed", "logical"])
        return _gemm(M, N, K, w, a, fmt, rng.choice(["int8", "planes"]), feed, w == a == 1 and rng.random() < 0.5)
    if kind == "fc":
        M, N, K = _log(rng, 256, 12000), rng.randint(1, 16), _log(rng, 256, 9216)
        fmt = rng.choice(["fields", "planes", "int8"])
        if fmt == "int8" and rng.random() < 0.4:
            return _gemm(M, N, K, 8, a, fmt, "raw")
        return _gemm(M, N, K, w, a, fmt, rng.choice(["int8", "planes"]))
    if kind == "conv":
        fmt = rng.choice(["int8", "planes"])
        while True:
            k = rng.choice([1, 3, 3, 5])
            B, H, C, OC = _log(rng, 1, 64), rng.randint(7, 56), rng.choice([32, 64, 80, 96, 128, 192, 256, 384]), _log(rng, 32, 512)
            stride, pad = rng.choice([1, 1, 2]), rng.choice([0, k // 2])
            c = _conv(B, H, C, OC, k, stride, pad, w, a, fmt)
            if B * _oh(c) ** 2 * OC * k * k * C <= 1 << (34 if fmt == "int8" else 30):
                return c
    mode = rng.choice(["auto", "auto", "tensor", "bitserial"])
    B = _log(rng, 1, 16 if mode == "bitserial" else 224)
    return _net(B, mode, B <= 4)


def _oh(c):
    return (c["H"] + 2 * c["pad"] - c["k"]) // c["stride"] + 1


def _enc(c):
    """Weights: +-1 when they have one bit, two's complement otherwise; activations: codes from 0,
    or +-1 in a binary network."""
    return (BIPOLAR if c["w"] == 1 else SIGNED), (BIPOLAR if c.get("xnor") else UNSIGNED)


def _values(g, shape, bits, enc):
    """Uniform over the encoding's values, as the packer takes them: one byte per element."""
    lo, hi = synth.value_range(bits, enc)
    if enc == BIPOLAR:
        return torch.randint(0, 2, shape, generator=g, device="cuda", dtype=torch.int8).mul_(2).sub_(1)
    kind = torch.uint8 if enc == UNSIGNED else torch.int8
    return torch.randint(lo, hi + 1, shape, generator=g, device="cuda", dtype=kind)


def _thresholds(g, rows, n, K, w, w_enc, a, a_enc, spread):
    mu, sigma = synth.acc_stats(K, w, w_enc, a, a_enc)
    lo, hi = math.floor(mu - spread * sigma), math.ceil(mu + spread * sigma)
    t = torch.randint(lo, hi + 1, (rows, n), generator=g, device="cuda", dtype=torch.int32)
    return t.sort(dim=1).values.contiguous()


def _layer(case, seed):
    """Weights, activations and thresholds of a gemm or conv case."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)
    w_enc, a_enc = _enc(case)
    if case["kind"] == "gemm":
        W, A, K = (case["M"], case["K"]), (case["N"], case["K"]), case["K"]
    else:
        k, C, H = case["k"], case["C"], case["H"]
        W, A, K = (case["OC"], k, k, C), (case["B"], H, H, C), k * k * C
    W, A = _values(g, W, case["w"], w_enc), _values(g, A, case["a"], a_enc)
    if case.get("out") == "raw":
        return W, A, None
    return W, A, _thresholds(g, W.shape[0], (1 << case["a"]) - 1, K, case["w"], w_enc, case["a"], a_enc, 3.0)


def _network(case, seed):
    """An AlexNet-shaped network with random weights and thresholds, and a batch of images."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 29)
    net = synth.NetCase(B=case["B"], image=None)
    H, C = 227, 3
    for L in net.layers:
        shape = (L.OC, L.KH, L.KW, C) if L.kind == "conv" else (L.OC, H * H * C)
        net.weights[L.name] = _values(g, shape, L.w_bits, L.w_enc).cpu().numpy()
        if L.kind == "conv":
            H = (H + 2 * L.pad - L.KH) // L.stride + 1
            H = (H - 3) // 2 + 1 if L.pool else H
        else:
            H = 1
        C = L.OC
        if L.out_bits:
            K = int(np.prod(shape[1:]))
            net.thr[L.name] = _thresholds(g, L.OC, (1 << L.out_bits) - 1, K, L.w_bits, L.w_enc, L.a_bits, UNSIGNED,
                                          1.0).cpu().numpy()
    image = torch.randint(0, 256, (case["B"], 227, 227, 3), generator=g, device="cuda", dtype=torch.uint8)
    return net, image


def _buffer(n):
    return torch.zeros(max(int(n), 16), dtype=torch.uint8, device="cuda")


def _pad_channels(x, C):
    return F.pad(x, (0, C - x.shape[-1])).contiguous() if x.shape[-1] != C else x


def prepare(case, seed):
    kind = case["kind"]
    if kind == "alexnet":
        net, image = _network(case, seed)
        plan = alexnet.AlexNetPlan(net, case["B"], case["mode"])
        if not case["graph"]:
            return {"kind": kind, "plan": plan, "image": image}
        graph, logits = plan.capture(image)
        return {"kind": kind, "plan": plan, "image": image, "graph": graph, "logits": logits}
    W, A, thr = _layer(case, seed)
    w_enc, a_enc = _enc(case)
    fmt, w, a = FMT[case["fmt"]], case["w"], case["a"]
    if kind == "conv":
        C = case["C"]
        d = qb.qnn_conv_desc(case["B"], case["H"], case["H"], C, 0, case["OC"], case["k"], case["k"], case["stride"],
                             case["pad"], w, a, a, w_enc, a_enc, fmt, fmt, qb.QNN_PATH_AUTO)
        # planes pad every pixel to whole words, containers need no padding at these channel counts
        Cp = -(-C // 32) * 32 if fmt == qb.QNN_FMT_BITPLANES else C
        rows = _pad_channels(W, Cp).reshape(case["OC"], -1)
        s = {"kind": kind, "d": d, "W": qb.pack(rows, w, w_enc, fmt), "thr": thr,
             "A": qb.pack(A.reshape(-1, C), a, a_enc, fmt),
             "out": _buffer(qb.qnn_conv_out_bytes(d, True)), "ws": _buffer(qb.qnn_conv_workspace_bytes(d))}
        return s
    M, N, K = case["M"], case["N"], case["K"]
    a_fmt = qb.QNN_FMT_INT8 if case["fmt"] == "fields" else fmt
    out_fmt = qb.QNN_FMT_BITPLANES if case["out"] == "planes" else qb.QNN_FMT_INT8
    d = qb.qnn_gemm_desc(M, N, K, w, a, min(a, 4), w_enc, a_enc, fmt, a_fmt, out_fmt, qb.QNN_PATH_AUTO, 0)
    ws = qb.qnn_gemm_workspace_bytes(d)
    s = {"kind": kind, "feed": case["feed"], "d": d, "W": qb.pack(W, w, w_enc, fmt), "thr": thr,
         "out": _buffer(qb.qnn_gemm_out_bytes(d, thr is not None)), "ws": _buffer(ws) if ws else None, "ws_bytes": ws}
    packed = qb.pack(A, a, a_enc, a_fmt)
    if case["feed"] == "packed":
        s["A"] = packed
    else:
        src = qb.QNN_FMT_BITPLANES if case["feed"] == "planes" else a_fmt
        s["pd"] = qb.qnn_pack_desc(N, K, a, a_enc, src)
        s["src"] = A if case["feed"] == "logical" else qb.pack(A, a, a_enc, src)
        s["A"] = torch.zeros_like(packed)
    return s


def run(s):
    if s["kind"] == "alexnet":
        if "graph" in s:
            s["graph"].replay()
            return s["logits"]
        return s["plan"].forward(s["image"])
    if s["kind"] == "conv":
        qb.check(qb.qnn_qconv(s["d"], s["W"], s["A"], s["thr"], s["out"], s["ws"], s["ws"].numel()))
        return s["out"]
    if s["feed"] == "logical":
        qb.check(qb.qnn_pack(s["pd"], s["src"], s["A"]))
    elif s["feed"] == "planes":
        qb.check(qb.qnn_planes_to_int8(s["pd"], s["src"], s["A"]))
    qb.check(qb.qnn_qgemm(s["d"], s["W"], s["A"], s["thr"], s["out"], s["ws"], s["ws_bytes"]))
    return s["out"]


def _operand_bytes(rows, K, bits, fmt):
    if fmt == "int8":
        return rows * K
    return rows * K * (bits if fmt == "planes" else {1: 1, 2: 2, 3: 4, 4: 4}[bits]) / 8


def work(case):
    """Each operand read once in the form it is given, each result written once."""
    if case["kind"] == "alexnet":
        mode, B = case["mode"], case["B"]
        total, ops, H, C = B * 227 * 227 * 3 + B * 4000.0, 0, 227, 3
        for L in synth.ALEXNET_LAYERS:
            if L.kind == "conv":
                K, H = L.KH * L.KW * C, (H + 2 * L.pad - L.KH) // L.stride + 1
                ops += 2 * B * H * H * L.OC * K
                H = (H - 3) // 2 + 1 if L.pool else H
            else:
                K, H = H * H * C, 1
                ops += 2 * B * L.OC * K
            C = L.OC
            planes = L.w_bits < 8 and (mode == "bitserial" or (mode == "auto" and L.kind == "fc" and B <= 16))
            total += _operand_bytes(L.OC, K, L.w_bits, "planes" if planes else "int8") + 12 * L.OC * (L.out_bits > 0)
        return {"bytes": float(total), "flops": float(ops)}
    w, a, n_thr = case["w"], case["a"], (1 << case["a"]) - 1
    if case["kind"] == "conv":
        N, M, K, fmt = case["B"] * _oh(case) ** 2, case["OC"], case["k"] ** 2 * case["C"], case["fmt"]
        total = _operand_bytes(M, K, w, fmt) + _operand_bytes(case["B"] * case["H"] ** 2, case["C"], a, fmt)
        total += _operand_bytes(N, M, a, fmt) + 4 * M * n_thr
        return {"bytes": float(total), "flops": 2.0 * M * N * K}
    M, N, K = case["M"], case["N"], case["K"]
    fed = "planes" if case["feed"] == "planes" or (case["fmt"] == "planes" and case["feed"] == "packed") else "int8"
    total = _operand_bytes(M, K, w, case["fmt"]) + _operand_bytes(N, K, a, fed)
    total += 4 * M * N if case["out"] == "raw" else _operand_bytes(N, M, a, case["out"]) + 4 * M * n_thr
    return {"bytes": float(total), "flops": 2.0 * M * N * K}


def tolerance(case):
    return "exact"


def _count(acc, thr):
    """Number of thresholds that each accumulator [..., M] reaches."""
    code = torch.zeros(acc.shape, dtype=torch.uint8, device=acc.device)
    for i in range(thr.shape[1]):
        code += acc >= thr[:, i].double()
    return code


def _laid_out(code, fmt, bits):
    """Codes [N][M] as the framework's buffers hold them, as plain bytes."""
    N, M = code.shape
    if fmt == "int8":
        return F.pad(code, (0, -M % 16)).reshape(-1)
    code = F.pad(code, (0, -M % 32))
    weight = torch.tensor([1 << i for i in range(8)], dtype=torch.uint8, device=code.device)
    rows = [(((code >> b) & 1).view(N, -1, 8) * weight).sum(2, dtype=torch.uint8).reshape(-1) for b in range(bits)]
    return torch.cat(rows)


def _filled(x):
    """A buffer is never smaller than 16 bytes."""
    return F.pad(x, (0, max(0, 16 - x.numel())))


def _conv64(x, W, stride, pad):
    """Channels-last codes and filters to channels-last sums, 64-bit floats (exact: whole numbers
    far below 2^53)."""
    y = F.conv2d(x.permute(0, 3, 1, 2).double(), W.permute(0, 3, 1, 2).double(), stride=stride, padding=pad)
    return y.permute(0, 2, 3, 1)


def exact(case, seed):
    if case["kind"] == "alexnet":
        net, image = _network(case, seed)
        logits = []
        for part in image.split(16):
            x = part
            for L in net.layers:
                W = torch.from_numpy(net.weights[L.name]).cuda()
                if L.kind == "conv":
                    acc = _conv64(x, W, L.stride, L.pad)
                else:
                    acc = x.reshape(x.shape[0], -1).double() @ W.double().T
                if not L.out_bits:
                    logits.append(acc.to(torch.int32))
                    break
                x = _count(acc, torch.from_numpy(net.thr[L.name]).cuda())
                if L.pool:
                    x = F.max_pool2d(x.permute(0, 3, 1, 2).double(), 3, 2).permute(0, 2, 3, 1).to(torch.uint8)
        return torch.cat(logits)
    W, A, thr = _layer(case, seed)
    if case["kind"] == "conv":
        out = [_count(_conv64(x, W, case["stride"], case["pad"]), thr) for x in A.split(8)]
        return _filled(_laid_out(torch.cat(out).reshape(-1, case["OC"]), case["fmt"], case["a"]))
    acc = A.double() @ W.double().T
    if thr is None:
        return acc.to(torch.int32).reshape(-1).view(torch.uint8)
    return _filled(_laid_out(_count(acc, thr), case["out"], case["a"]))
