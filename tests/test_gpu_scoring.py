"""Scoring on the GPU: which frames a later layer's kernel takes up."""
import pytest

import smtm_inputs as si
from test_gpu_shapes import test_maps_ready_with_odd_widths as ready_steps

pytestmark = pytest.mark.gpu


def test_exits_of_a_later_layer_do_not_move_the_frames_of_clusters_that_begin_late():
    # more clusters than the chip holds beside the pooling kernel, and most frames exit at the layer they serve: a cluster
    # that begins after the first decisions takes up the frames it would have taken up before them
    ready_steps(si.Workload("late_clusters", si.BF16, si.NCHW, B=512, stages=((256, 14, 14), (2048, 7, 7)), n=60, k_init=12,
                            k_min=8, k_max=16, S=512, T=4, tau=0.81, sigma=1.0, zipf_s=0.5, repeat_p=0.8, seed=95))
