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
