"""Scoring on the GPU: which frames a later layer's kernel takes up, and large fast memories that all frames share."""
import numpy as np
import pytest
import torch

import paper_2112_02644_b200 as smtm
import smtm_inputs as si
from harness import launches, run_workload
from test_gpu_shapes import kernels_of_lookup, test_maps_ready_with_odd_widths as ready_steps

pytestmark = pytest.mark.gpu


def test_exits_of_a_later_layer_do_not_move_the_frames_of_clusters_that_begin_late():
    # more clusters than the chip holds beside the pooling kernel, and most frames exit at the layer they serve: a cluster
    # that begins after the first decisions takes up the frames it would have taken up before them
    ready_steps(si.Workload("late_clusters", si.BF16, si.NCHW, B=512, stages=((256, 14, 14), (2048, 7, 7)), n=60, k_init=12,
                            k_min=8, k_max=16, S=512, T=4, tau=0.81, sigma=1.0, zipf_s=0.5, repeat_p=0.8, seed=95))


# clusters of the kernel of small frames after a first lookup, when half of the frames are taken to be still in
@pytest.mark.parametrize("B,begin,cluster", [(128, True, 1), (128, False, 2), (148, False, 2), (149, False, 1), (74, True, 2)])
def test_clusters_of_later_lookups_of_small_frames(B, begin, cluster):
    got = kernels_of_lookup(si.F16, si.NCHW, B, 256, 8, 8, 8, begin)
    assert [(g.kernel, g.cluster) for g in got] == [("k_lookup_frame", cluster)]


# later layers of large batches on the pipelined route: chunks in halves with a last one shorter than half a chunk, and of four
# channels; three whole chunks; channels that are no run of whole vectors (not pipelined); nine chunks (pooled and scored apart)
@pytest.mark.parametrize("dt,stages", [
    (si.BF16, ((64, 9, 9), (840, 8, 8))), (si.F16, ((32, 8, 8), (296, 9, 11), (1100, 5, 5))), (si.F32, ((16, 8, 8), (16, 40, 40))),
    (si.F32, ((64, 7, 7), (1028, 7, 7)))], ids=lambda v: str(v) if isinstance(v, tuple) else None)
def test_later_layers_of_large_batches(dt, stages):
    ready_steps(si.Workload("halves", dt, si.NCHW, B=450, stages=stages, n=40, k_init=8, k_min=4, k_max=12, S=450, T=3, tau=0.75,
                            sigma=1.0, zipf_s=0.5, repeat_p=0.8, seed=97))


# ... and the clusters that take chunks in halves, by the reducer: channels of odd widths from 128 bytes on and below (the halves
# meet on a 16-byte boundary), units of channels of 7x7 and 14x14 maps, whole vectors, a last chunk of one run of channels
@pytest.mark.parametrize("dt,stages,reducers", [
    (si.F16, ((64, 8, 8), (520, 9, 11), (2048, 5, 5)), ["TeamVectorsINS_3F16ELb1E", "LanePerChannelINS_3F16E"]),
    (si.BF16, ((64, 8, 8), (516, 9, 10), (2056, 5, 5)), ["TeamVectorsINS_4BF16ELb1E", "LanePerChannelINS_4BF16E"]),
    (si.F32, ((64, 7, 7), (1024, 7, 7), (640, 6, 6)), ["UnitPerLaneINS_3F32ELi49E", "TeamVectorsINS_3F32ELb0E"]),
    (si.BF16, ((64, 8, 8), (320, 14, 14), (1288, 7, 7)), ["UnitPerLaneINS_4BF16ELi196E", "UnitPerLaneINS_4BF16ELi49E"]),
], ids=lambda v: str(v) if isinstance(v, tuple) else None)
def test_chunks_in_halves(dt, stages, reducers):
    w = si.Workload("in_halves", dt, si.NCHW, B=450, stages=stages, n=40, k_init=8, k_min=4, k_max=12, S=450, T=3, tau=0.75,
                    sigma=1.0, zipf_s=0.5, repeat_p=0.8, seed=97)
    dtype = {si.F32: torch.float32, si.F16: torch.float16, si.BF16: torch.bfloat16}[dt]
    cache = smtm.smtm_cache_create(w.n, w.dims, [0.8] * w.L, [np.ones((w.n, d), np.float32) for d in w.dims], None, n_streams=w.S,
                                   k_init=8, k_min=4, k_max=12, max_batch=w.B, flags=smtm.FLAG_MAPS_READY)
    batch = smtm.Batch(cache, w.B, stream_id=si.stream_ids(w))
    for l, reducer in enumerate(reducers, 1):
        x = torch.zeros(si.shape4(w, l), dtype=dtype, device="cuda")
        got = launches(lambda: smtm.smtm_lookup_exit(cache, l, smtm.Fmap(x, dt, w.layout, *si.shape4(w, l)), batch))
        assert got[0].kernel == "k_lookup_sparse" and reducer in got[0].variant and "Lb1EEEvNS" in got[0].variant, got[0]
    smtm.smtm_cache_destroy(cache)
    ready_steps(w)


# fast memories of more than 64 slots that all frames share: eight, four, two or one frame to a cluster, slots in whole and
# ragged shares, warps that divide the vector length, a later layer with few frames left, one with vectors of odd widths
def shared(name, B, n, stages, **kw):
    kw = dict(dict(k_init=n, k_min=max(66, n // 2), k_max=n, T=3, window_W=3, sigma=0.5, zipf_s=0.8, repeat_p=0.3, seed=96), **kw)
    return si.Workload(name, si.F16, si.NHWC, B=B, stages=stages, n=n, **kw)


SHARED = [
    (shared("eight_frames", 150, 101, ((1024, 2, 2), (2048, 1, 1)), tau=0.3), [(8, 8), (4, 8)]),
    (shared("four_frames", 77, 201, ((128, 3, 3), (260, 2, 2))), [(4, 8), (2, 8)]),
    (shared("two_frames", 38, 75, ((2048, 2, 1),)), [(2, 8)]),
    (shared("one_frame", 5, 999, ((24, 3, 3), (1028, 1, 2)), k_min=60), [(1, 8), (1, 8)]),
    (shared("many_slots", 301, 1999, ((136, 1, 1), (36, 2, 2)), k_min=1500, T=2), [(8, 8), (8, 8)]),
    (shared("long_vector", 148, 66, ((9000, 1, 1),), T=2), [(4, 8)]),
    (shared("crowd", 601, 101, ((260, 2, 1), (64, 2, 2)), T=2), [(8, 2), (8, 4)]),
    (shared("queue", 400, 257, ((64, 3, 1),), T=2), [(8, 4)]),
]


@pytest.mark.parametrize("w,split", SHARED, ids=lambda v: getattr(v, "name", ""))
def test_scoring_of_large_fast_memories_that_all_frames_share(w, split):
    cache = smtm.smtm_cache_create(w.n, w.dims, [0.8] * w.L, [np.ones((w.n, d), np.float32) for d in w.dims], None,
                                   k_init=w.k_init, k_min=w.k_min, k_max=w.k_max, max_batch=w.B)
    batch = smtm.Batch(cache, w.B)
    for l in range(w.L):
        B, C, H, W = si.shape4(w, l)
        x = torch.zeros((B, H, W, C), dtype=torch.float16, device="cuda")
        call = smtm.smtm_lookup_exit if l else smtm.smtm_lookup_exit_begin
        got = launches(lambda: call(cache, l, smtm.Fmap(x, w.dtype, w.layout, B, C, H, W), batch))
        F, P = split[l]   # frames and CTAs of a cluster
        assert got[-1].kernel == "k_score_shared" and "ILi%dE" % F in got[-1].variant
        assert (got[-1].cluster, got[-1].grid) == (P, P * -(-B // F))
    smtm.smtm_cache_destroy(cache)
    rep = run_workload(w)
    assert rep.frames == w.B * w.T and rep.routes == [0, 0, w.L * w.T, 0, 0]


# maps of one pixel and equal channels, against centres with a single entry: a similarity is off by the rounding of the squared
# length, of its root, of one product and of the division.  Each is at most 2^-24 and 3.5e-8 in the mean square; a square root
# halves what the sum is off by, and a sum of D / 512 terms to a lane after sixteen in a tree is off by some 1.3e-7 (in fp32 on
# the CPU; a lane that adds D / 32 terms one by one is off by 4.7e-7 and 1.9e-6)
@pytest.mark.parametrize("D", [2048, 8192])
def test_lengths_of_long_vectors_in_nhwc_lookups(D):
    B, k = 300, 4
    cents = np.zeros((k, D), np.float32)
    cents[np.arange(k), np.arange(k) * 7] = 1.0
    cache = smtm.smtm_cache_create(k, [D], [0.8], [cents], None, k_init=k, k_min=k, k_max=k, max_batch=B)
    batch = smtm.Batch(cache, B)
    x = torch.linspace(0.3, 1.7, B, device="cuda").half()[:, None, None, None].expand(B, 1, 1, D).contiguous()
    fmap = smtm.Fmap(x, si.F16, si.NHWC, B, D, 1, 1)
    assert [g.kernel for g in launches(lambda: smtm.smtm_lookup_exit_begin(cache, 0, fmap, batch))] == ["k_lookup_nhwc"]
    smtm.smtm_lookup_exit_begin(cache, 0, fmap, batch)
    off = batch.sa.double().cpu() * D ** 0.5 - 1.0
    smtm.smtm_cache_destroy(cache)
    assert float(off.square().mean().sqrt()) <= 1.2e-7
