"""Shapes at the edges of what each kernel serves, against the CPU oracle."""
import pytest

import smtm_inputs as si
import test_gpu_parity as parity

pytestmark = pytest.mark.gpu


# channels that are no multiple of 16 bytes: one element to a stage's worth, runs that begin inside a 16-byte piece,
# fewer channels than lanes, more frames than one listing holds
ANY_WIDTH = [
    (si.BF16, 5, 64, 15, 15), (si.F16, 3, 40, 9, 9), (si.F32, 4, 20, 15, 15), (si.F16, 3, 512, 2, 2), (si.BF16, 3, 2048, 3, 3),
    (si.BF16, 3, 16, 61, 61), (si.F32, 3, 4, 79, 79), (si.F16, 7, 24, 1, 1), (si.BF16, 3, 8, 113, 113), (si.F32, 3, 20, 1, 3),
    (si.BF16, 2100, 8, 5, 5), (si.F16, 300, 33, 4, 6),
]


@pytest.mark.parametrize("dt,B,C,H,W", ANY_WIDTH)
def test_pooling_of_channels_of_any_width(dt, B, C, H, W):
    parity.test_encode_matches_oracle(dt, si.NCHW, B, C, H, W)
