"""Which convolutions the library runs on which tiles, as its host queries answer (148 SMs, without a device)."""
import pytest


@pytest.fixture(scope="module")
def qb():
    import __graft_entry__ as ge
    ge.build()
    from paper_1709_04060_b200 import binding
    return binding


def conv(qb, B, H, W, C, OC, KH, KW, stride, pad, in_pitch=0):
    return qb.qnn_conv_desc(B, H, W, C, in_pitch, OC, KH, KW, stride, pad, 1, 2, 2, 2, 0, 1, 1, 0)


def test_the_environment_does_not_decide_what_fuses(qb, monkeypatch):
    """A plan asks once which layers run together with their pool; a later call must not answer otherwise."""
    big, small = (conv(qb, B, 227, 227, 3, 96, 11, 11, 4, 0, 3) for B in (28, 27))
    for value in (None, "0", "1"):
        if value is not None:
            monkeypatch.setenv("QNN_CONV_DIRECT", value)
        assert qb.qnn_conv_maxpool_fuses(big, 3, 2)
        assert not qb.qnn_conv_maxpool_fuses(small, 3, 2)


def first_layer(qb, B, H, W, OC, k, stride, out_bits, w_enc=1):
    return qb.qnn_conv_desc(B, H, W, 3, 3, OC, k, k, stride, 0, 1 if w_enc == 2 else 8, 8, out_bits, w_enc, 0, 1, 1, 0)


@pytest.mark.parametrize("layer,in_place", [
    # us, the kernel with lowering warps -> this one
    ((398, 91, 19, 32, 11, 2, 1), False),       # 16.5 -> 47.1
    ((78, 40, 40, 8, 7, 1, 1), False),          # 9.3 -> 20.9
    ((147, 197, 20, 96, 7, 1, 1), False),       # 32.9 -> 81.6
    ((425, 40, 40, 20, 11, 2, 3), False),       # 20.0 -> 32.5
    ((424, 256, 256, 48, 7, 4, 2), True),       # 264 -> 100
    ((479, 97, 23, 64, 1, 1, 2), True),         # 148 -> 68
    ((256, 227, 227, 96, 11, 4, 2), True),      # 128 -> 97
])
def test_first_layers_in_place_where_tiles_are_full(qb, layer, in_place):
    assert qb.qnn_conv_in_place(first_layer(qb, *layer)) == in_place
    assert not qb.qnn_conv_in_place(first_layer(qb, *layer), False)                  # sums
    assert qb.qnn_conv_in_place(first_layer(qb, *layer, w_enc=2), False)             # no other kernel lowers these inside


@pytest.mark.parametrize("layer,fuses", [
    ((162, 201, 137, 8, 11, 4, 3), False),      # 43.6 -> 84.0
    ((201, 82, 82, 20, 5, 2, 4), False),        # 55.8 -> 87.0
    ((500, 133, 133, 32, 5, 4, 1), False),      # 38.4 -> 66.8
    ((342, 159, 216, 64, 1, 4, 2), True),       # 109 -> 58
    ((32, 227, 227, 96, 11, 4, 2), True),       # 26.4 -> 22.4
    ((256, 227, 227, 96, 11, 4, 2), True),      # 151 -> 101
])
def test_first_layers_fuse_with_their_pool_where_tiles_are_full(qb, layer, fuses):
    assert qb.qnn_conv_maxpool_fuses(first_layer(qb, *layer), 3, 2) == fuses


def test_layers_of_plus_minus_one_fuse_where_few_thresholds_are_counted(qb):
    """36 x 47 -> 16, 3 x 3, batch 356, seven thresholds: 81 us apart, 106 in one kernel."""
    for layer in ((356, 43, 47, 16, 3, 1, 3), (131, 130, 130, 8, 5, 4, 3)):
        assert not qb.qnn_conv_maxpool_fuses(first_layer(qb, *layer, w_enc=2), 3, 2)
        assert qb.qnn_conv_maxpool_fuses(first_layer(qb, *layer[:6], 2, w_enc=2), 3, 2)
        assert qb.qnn_conv_in_place(first_layer(qb, *layer, w_enc=2))


def busiest_pair(cv, boxes):
    """k-blocks (one channel chunk) of the SM pair with the most, of 74: tiles of two boxes, or of 256
    consecutive pixels that meet every tap, dealt in turn."""
    B, H, W, OC, KH, KW, pad = cv.B, cv.H, cv.W, cv.OC, cv.KH, cv.KW, cv.pad
    OH, OW, tiles_c = H + 2 * pad - KH + 1, W + 2 * pad - KW + 1, -(-OC // 256)
    if boxes is None:
        tiles = [KH * KW] * -(-B * OH * OW // 256)
    else:
        count, w, h, n = boxes
        nn, nw = -(-B // n), -(-OW // w)
        assert count == nn * nw * -(-OH // h) and w * h * n <= 128

        def taps(q):
            oh, ow = q // nw * h, q % nw * w
            rows = {k for o in range(oh, oh + h) for k in range(KH) if 0 <= o + k - pad < H}
            cols = {k for o in range(ow, ow + w) for k in range(KW) if 0 <= o + k - pad < W}
            return rows or set(range(KH)), cols or set(range(KW))
        tiles = []
        for t in range(-(-count // 2)):
            (r0, c0), (r1, c1) = taps(2 * t // nn), taps(min(2 * t + 1, count - 1) // nn)
            r, c = r0 | r1, c0 | c1
            tiles.append((max(r) - min(r) + 1) * (max(c) - min(c) + 1))
    load = [0] * 74
    for u in range(len(tiles) * tiles_c):
        load[u % 74] += tiles[u % len(tiles)]
    return max(load)


@pytest.mark.parametrize("B,H,C,OC,k,boxes", [
    (64, 21, 512, 512, 3, False), (64, 17, 256, 512, 3, False), (14, 45, 96, 512, 3, False),      # a round more, or
    (21, 30, 128, 512, 3, False), (18, 56, 64, 256, 5, False), (64, 27, 96, 256, 5, False),       # nothing gained
    (256, 27, 96, 256, 5, True), (256, 13, 256, 384, 3, True), (256, 13, 384, 384, 3, True), (256, 13, 384, 256, 3, True),
])
def test_boxes_by_rounds(qb, B, H, C, OC, k, boxes):
    cv = conv(qb, B, H, H, C, OC, k, k, 1, k // 2)
    plan = qb.qnn_conv_boxes(cv)
    assert (plan is not None) == boxes
    if boxes:
        assert busiest_pair(cv, plan) < busiest_pair(cv, None)


def test_boxes_never_keep_a_pair_of_sms_busier(qb):
    import random
    rng, taken = random.Random(5), 0
    for _ in range(1500):
        k = rng.choice([3, 3, 5, 7])
        B, H, W, OC = rng.choice([8, 16, 33, 64, 128, 250]), rng.randint(4, 60), rng.randint(4, 60), rng.choice([256, 384, 512, 1000])
        if B * H * W > 300000:
            continue
        cv = conv(qb, B, H, W, rng.choice([96, 128, 256]), OC, k, k, 1, rng.choice([1, k // 2]))
        plan = qb.qnn_conv_boxes(cv)
        if plan is not None:
            taken += 1
            assert busiest_pair(cv, plan) <= 0.98 * busiest_pair(cv, None), (B, H, W, OC, k, plan)
    assert taken > 100


def test_boxes_save_more_where_the_epilogue_is_longer(qb):
    """Sums and codes of three or four bits: 34 x 34 x 32 -> 256, 5 x 5, 85 -> 100 us with single pixels."""
    cv = conv(qb, 118, 34, 34, 32, 256, 5, 5, 1, 2)
    assert qb.qnn_conv_boxes(cv) is not None and qb.qnn_conv_boxes(cv, False) is None
    cv.out_bits = 4
    assert qb.qnn_conv_boxes(cv) is None
    deep = conv(qb, 127, 10, 10, 32, 600, 7, 7, 1, 3)           # three taps of ten: 0.71 of the time
    assert qb.qnn_conv_boxes(deep, False) is not None


def test_only_padded_layers_of_stride_one_take_boxes(qb):
    assert qb.qnn_conv_boxes(conv(qb, 256, 27, 27, 96, 256, 5, 5, 1, 0)) is None
    assert qb.qnn_conv_boxes(conv(qb, 256, 27, 27, 96, 256, 5, 5, 2, 2)) is None
    assert qb.qnn_conv_boxes(conv(qb, 1, 27, 27, 96, 256, 5, 5, 1, 2)) is None          # too small for SM pairs
    assert qb.qnn_conv_boxes(conv(qb, 256, 27, 27, 90, 256, 5, 5, 1, 2)) is None        # not the tensor-map loader's


def test_the_choice_costs_a_call_next_to_nothing(qb):
    """Searched in every call it took 8 us for 56 x 56 maps and 300 for 1024 x 1024; a query is some 2."""
    import time
    for B, H, k in ((64, 56, 3), (64, 27, 5), (32, 224, 3), (2, 1024, 3)):
        cv = conv(qb, B, H, H, 64, 512, k, k, 1, k // 2)
        none = conv(qb, B, H, H, 64, 512, k, k, 1, 0)          # nothing to choose
        def us(c):
            best = 1.0
            for _ in range(20):
                t0 = time.perf_counter()
                for _ in range(50):
                    qb.qnn_conv_boxes(c)
                best = min(best, (time.perf_counter() - t0) / 50)
            return best * 1e6
        assert us(cv) < us(none) + 1.0, (B, H, k)


def test_shapes_that_share_a_place_in_the_table(qb):
    """More shapes than the table holds, twice and from two threads: the answers stay each shape's own."""
    from concurrent.futures import ThreadPoolExecutor
    shapes = [conv(qb, B, H, H, C, 512, 3, 3, 1, 1) for B in (64, 128, 250) for H in (7, 9, 13, 14, 21, 28) for C in (96, 256, 512)]
    first = [qb.qnn_conv_boxes(s) for s in shapes]
    assert any(first) and not all(first)
    with ThreadPoolExecutor(2) as pool:
        for got in pool.map(lambda order: [qb.qnn_conv_boxes(shapes[i]) for i in order], [range(len(shapes))] * 4):
            assert got == first
    for i in reversed(range(len(shapes))):
        assert qb.qnn_conv_boxes(shapes[i]) == first[i]
