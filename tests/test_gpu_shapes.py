"""Shapes at the edges of what each kernel serves, against the CPU oracle."""
import pytest

import smtm_inputs as si
import test_gpu_parity as parity
from harness import run_workload

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


# lookups whose frames are small enough for a cluster of CTAs each: slices of one 16-byte piece and of a thousand
# channels, odd widths, clusters of 1, 2, 4 and 8, layers after most frames have left, more slots than warps
FRAME_LOOKUPS = [
    si.Workload("frame_2x2", si.F16, si.NCHW, B=200, stages=((64, 4, 4), (512, 2, 2), (512, 1, 1)), n=40, k_init=9, k_min=3,
                k_max=17, T=3, window_W=3, sigma=0.5, zipf_s=0.8, repeat_p=0.5, seed=51),
    si.Workload("frame_odd", si.BF16, si.NCHW, B=3, stages=((64, 15, 15), (136, 9, 9), (2048, 7, 7)), n=80, k_init=64,
                k_min=20, k_max=64, T=4, window_W=3, sigma=0.5, zipf_s=0.8, repeat_p=0.5, seed=52),
    si.Workload("frame_f32", si.F32, si.NCHW, B=1, stages=((20, 33, 31), (24, 17, 15), (4, 5, 3)), n=10, k_init=4, k_min=2,
                k_max=10, T=6, window_W=3, sigma=0.5, zipf_s=0.5, repeat_p=0.5, seed=53),
    si.Workload("frame_nhwc", si.BF16, si.NHWC, B=2, stages=((24, 30, 30), (264, 9, 7), (4096, 3, 1)), n=80, k_init=64,
                k_min=20, k_max=64, T=4, window_W=3, sigma=0.5, zipf_s=0.8, repeat_p=0.5, seed=54),
    si.Workload("frame_nhwc_f32", si.F32, si.NHWC, B=150, stages=((8, 5, 5), (20, 3, 3)), n=30, k_init=5, k_min=2, k_max=12,
                S=150, T=4, window_W=3, sigma=0.5, zipf_s=0.8, repeat_p=0.5, seed=55),
]


@pytest.mark.parametrize("w", FRAME_LOOKUPS, ids=lambda w: w.name)
def test_lookup_of_small_frames(w):
    rep = run_workload(w)
    assert rep.frames == w.B * w.T and sum(rep.exits) > 0 and rep.lookups > rep.frames


NHWC_POOLING = [(si.F16, 1, 24, 56, 56), (si.BF16, 3, 2056, 2, 3), (si.F32, 3, 8192, 1, 1), (si.F32, 5, 12, 64, 61), (si.F16, 700, 8, 2, 2)]


@pytest.mark.parametrize("dt,B,C,H,W", NHWC_POOLING)
def test_pooling_of_nhwc_maps_by_clusters(dt, B, C, H, W):
    parity.test_encode_matches_oracle(dt, si.NHWC, B, C, H, W)


# large fast memories on the tensor cores: class counts that are no multiple of four, vectors of one 16-byte piece and of
# less than a k-block per part, few tiles cut into many parts, a batch far below the largest
DENSE_LOOKUPS = [
    si.Workload("dense_101", si.F16, si.NCHW, B=130, stages=((1024, 4, 4), (2048, 2, 2)), n=101, k_init=101, k_min=70,
                k_max=101, T=3, sigma=0.6, zipf_s=0.9, repeat_p=0.3, seed=61),
    si.Workload("dense_short", si.BF16, si.NCHW, B=5, stages=((8, 9, 9), (24, 8, 8), (200, 5, 5)), n=67, k_init=66, k_min=65,
                k_max=67, T=4, tau=0.3, sigma=0.4, zipf_s=0.9, repeat_p=0.3, seed=62),
    si.Workload("dense_nhwc_601", si.BF16, si.NHWC, B=300, stages=((320, 3, 3), (640, 2, 2)), n=601, k_init=601, k_min=100,
                k_max=601, T=3, sigma=0.6, zipf_s=0.9, repeat_p=0.3, seed=63),
]


@pytest.mark.parametrize("w", DENSE_LOOKUPS, ids=lambda w: w.name)
def test_lookup_of_large_fast_memories(w):
    rep = run_workload(w)
    assert rep.frames == w.B * w.T and rep.routes == [0, w.L * w.T, 0, 0, 0]
