"""The update on the GPU at the sizes where its kernels change: one launch or two, the team that keeps the tables of an
only stream, the refresh of many classes.  Everything the update leaves behind is compared with the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2112_02644_b200 as smtm
import smtm_inputs as si
from harness import Report, compare_state, launches, run_workload

pytestmark = pytest.mark.gpu


def workload(name, B, n, stages=((64, 2, 2),), S=1, **kw):
    kw = dict(dict(k_init=4, k_min=3, k_max=12, T=4, window_W=2, sigma=0.4, zipf_s=0.6, repeat_p=0.3, seed=91), **kw)
    return si.Workload(name, si.F32, si.NCHW, B=B, stages=stages, n=n, S=S, **kw)


# one launch up to 512 frames, while its CTAs (one per frame and layer, and those of the tables) are at most nine to an SM, or
# sixteen where a thread has a frame; clusters of a CTA per 128 classes keep the tables of an only stream
@pytest.mark.parametrize("w,kernels,cluster", [
    (workload("frames_128", 128, 128), ["k_update_direct"], 1),
    (workload("frames_129", 129, 129), ["k_update_direct"], 2),
    (workload("frames_512", 512, 513, zipf_s=0.0), ["k_update_direct"], 8),
    (workload("frames_513", 513, 1024, zipf_s=0.0, k_max=900), ["k_update_plan_one", "k_update_apply"], 8),
    (workload("classes_1025", 40, 1025), ["k_update_direct", "k_resize"], 1),
    (workload("crowded", 300, 256, stages=((64, 2, 2),) * 5), ["k_update_plan_one", "k_update_apply"], 2),
    (workload("many_layers", 128, 30, stages=((64, 2, 2),) * 16), ["k_update_direct"], 1),
    (workload("wide_vector", 3, 5, stages=((16384, 1, 1),), k_max=5), ["k_update_direct"], 1),
    # (vectors of 210 and 274 16-byte pieces in sixteen blocks: with ceil(210 / 16) pieces to a block the last one had none)
    (workload("ragged_blocks", 300, 3, stages=((840, 1, 1), (1096, 1, 1)), k_init=3, k_max=3, tau=9.0), ["k_update_direct"], 1),
    (workload("ragged_blocks_600", 600, 3, stages=((840, 1, 1), (1096, 1, 1)), k_init=3, k_max=3, tau=9.0),
     ["k_update_plan_one", "k_update_apply"], 1),
    (workload("odd_vector", 130, 20, stages=((37, 3, 2), (66, 2, 2))), ["k_update_direct"], 1),
    (workload("one_frame", 1, 1, k_init=1, k_min=1, k_max=1), ["k_update_direct"], 1),
    (workload("forgets", 200, 300, forgetting=True, T=6), ["k_update_direct"], 4),
    (workload("streams_600", 300, 600, S=300), ["k_update_direct"], 1),
    (workload("seen_many", 512, 700, S=2, zipf_s=0.0, repeat_p=0.0), ["k_update_direct"], 1),
], ids=lambda v: getattr(v, "name", None))
def test_update_at_the_lines_between_its_kernels(w, kernels, cluster):
    cache = smtm.smtm_cache_create(w.n, w.dims, [0.8] * w.L, [np.ones((w.n, d), np.float32) for d in w.dims], None, n_streams=w.S,
                                   k_init=w.k_init, k_min=w.k_min, k_max=w.k_max, window_W=w.window_W, max_batch=w.B)
    sid = np.arange(w.B, dtype=np.int32) % w.S
    batch = smtm.Batch(cache, w.B, stream_id=sid if w.S > 1 else None)
    got = launches(lambda: smtm.smtm_cache_update_resize(cache, batch, None))
    smtm.smtm_cache_destroy(cache)
    assert [g.kernel for g in got] == kernels and got[len(kernels) - 1 if "k_resize" not in kernels else 0].cluster == cluster
    if w.S in (1, w.B):
        assert run_workload(w).frames == w.B * w.T
        return
    _run(w, sid)


def _run(w, sid):
    """The workload's steps with the frames' streams given; frames of streams the cache does not have are left out of the
    oracle's batch."""
    cents, counts = si.initial_centers(w)
    cache = smtm.smtm_cache_create(w.n, w.dims, [w.tau] * w.L, cents, counts, n_streams=w.S, k_init=w.k_init, k_min=w.k_min,
                                   k_max=w.k_max, window_W=w.window_W, max_batch=w.B)
    mem = oracle.OracleMemory(w.n, w.dims, [w.tau] * w.L, cents, counts, w.S, w.k_init, w.k_min, w.k_max, w.window_W)
    keep = (sid >= 0) & (sid < w.S)
    gb, labs = smtm.Batch(cache, w.B, stream_id=sid), si.labels(w)
    for t in range(w.T):
        fb = si.fallback_labels(w, labs[t])
        ob = mem.new_batch(int(keep.sum()), np.ascontiguousarray(sid[keep]))
        for l in range(w.L):
            x = si.frames(w, l, labs[t], t, device="cuda")
            (smtm.smtm_lookup_exit_begin if l == 0 else smtm.smtm_lookup_exit)(
                cache, l, smtm.Fmap(x, w.dtype, w.layout, *si.shape4(w, l)), gb)
            B, C, H, W = si.shape4(w, l)
            mem.lookup_exit(l, x.cpu()[torch.from_numpy(keep)].contiguous(), w.dtype, w.layout, (int(keep.sum()), C, H, W), ob)
        assert np.array_equal(gb.done.cpu().numpy()[keep], ob["done"])
        smtm.smtm_cache_update_resize(cache, gb, torch.from_numpy(fb).cuda())
        mem.update(ob, fb[keep])
        mem.resize()
    if keep.all():
        compare_state(w, cache, mem, Report())
    else:
        assert smtm.smtm_cache_status(cache) == 1
        smtm.smtm_cache_clear_status(cache)
        compare_state(w, cache, mem, Report())
    smtm.smtm_cache_destroy(cache)


def test_frames_of_no_stream_beside_an_only_stream():
    w = workload("strays", 300, 300, T=3)
    sid = np.zeros(w.B, np.int32)
    sid[[0, 7, 150, 299]] = 1, -2, 5, 9
    _run(w, sid)


# vectors of more than 4096 channels have several CTAs per frame in the one launch, fewer where the frames are many: one block, a
# block more than frames, as many blocks as there are, and (by the frames) one CTA each again; every frame of one class, and a
# layer of short vectors beside the long ones
@pytest.mark.parametrize("B,stages,parts,zipf", [
    (1, ((4100, 1, 1),), 4, 0.0), (3, ((4096, 1, 1),), 1, 0.0), (3, ((8192, 1, 1), (36, 2, 2)), 4, 9.0),
    (2, ((32772, 1, 1),), 16, 9.0), (40, ((8200, 1, 1),), 4, 0.5), (100, ((16388, 1, 1),), 2, 9.0), (150, ((4104, 1, 1),), 1, 9.0)])
def test_updates_of_long_vectors(B, stages, parts, zipf):
    w = workload("long", B, 6, stages=stages, k_init=3, k_max=6, zipf_s=zipf, tau=9.0)
    cache = smtm.smtm_cache_create(w.n, w.dims, [0.8] * w.L, [np.ones((w.n, d), np.float32) for d in w.dims], None, k_init=3,
                                   k_min=3, k_max=6, window_W=2, max_batch=B)
    batch = smtm.Batch(cache, B)
    got = launches(lambda: smtm.smtm_cache_update_resize(cache, batch, None))
    smtm.smtm_cache_destroy(cache)
    assert [(g.kernel, g.grid) for g in got] == [("k_update_direct", 1 + B * w.L * parts)]
    assert run_workload(w).frames == B * w.T
