"""Which layers the convolution that walks along z takes: every shape that its emulation and its GPU
test run, on any number of SMs they name, with stages of one, two and four 16-channel chunks, the last
of them partly filled, and none of the others."""
import pytest

from test_conv_march import SHAPES, _plan

GPU_ONLY = [((40, 30, 128), 48, 16), ((33, 20, 64), 96, 32), ((30, 20, 96), 16, 48)]


@pytest.mark.parametrize("sms", [152, 148, 3])
def test_tested_shapes_are_taken(sms):
    plans = {}
    for shape, cin, cout in SHAPES + GPU_ONLY:
        p = _plan(shape, cin, cout, sms)
        assert p is not None, (shape, cin, cout)
        assert p["cps"] == (4 if cin > 32 else cin // 16), (shape, cin, cout)
        plans[p["cps"], cin // 16 % p["cps"] != 0] = True
    assert {(1, False), (2, False), (4, True)} <= set(plans)


@pytest.mark.parametrize("shape,cin,cout,taps", [
    ((4, 5, 16), 32, 16, 1),            # 1x1x1
    ((4, 5, 12), 16, 16, 27),           # rows that are not whole groups of eight slots
    ((4, 5, 240), 16, 16, 27),          # a row does not fit two tiles with their margins
    ((4, 5, 64), 256, 16, 27),          # the slice's weights leave no room for stages
])
def test_other_shapes_are_left(shape, cin, cout, taps):
    assert _plan(shape, cin, cout, 152, taps) is None
