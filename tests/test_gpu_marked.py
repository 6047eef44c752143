"""Frames that the caller takes out of a batch itself (padding, frames decided elsewhere): every route leaves them alone,
at whichever layer they were marked as gone."""
import numpy as np
import pytest
import torch

import oracle
import paper_2112_02644_b200 as smtm
import smtm_inputs as si
from harness import Report, compare_layer, compare_state, launches

pytestmark = pytest.mark.gpu


def _w(name, dt, layout, B, stages, n, k, S=1, **kw):
    kw = dict(dict(T=3, tau=0.6, window_W=3, sigma=0.8, zipf_s=0.5, repeat_p=0.5, seed=98), **kw)
    return si.Workload(name, dt, layout, B=B, stages=stages, n=n, k_init=k, k_min=k, k_max=k, S=S, **kw)


READY = smtm.FLAG_MAPS_READY
# the workload, the cache's flags and the kernel that decides
CASES = [
    (_w("frame_nchw", si.F16, si.NCHW, 100, ((64, 9, 9), (256, 4, 4)), 40, 12, 100), 0, "k_lookup_frame"),
    (_w("streamed_nchw", si.F32, si.NCHW, 300, ((1024, 7, 7), (1024, 7, 7)), 20, 4), 0, "k_lookup_nchw"),
    (_w("streamed_few", si.BF16, si.NCHW, 13, ((256, 56, 56), (256, 56, 56)), 20, 10), 0, "k_lookup_nchw"),
    (_w("frame_nhwc", si.F16, si.NHWC, 3, ((64, 50, 50), (104, 31, 31)), 20, 6), 0, "k_lookup_frame_nhwc"),
    (_w("nhwc", si.BF16, si.NHWC, 260, ((64, 8, 8), (128, 4, 4)), 20, 6, 260), 0, "k_lookup_nhwc"),
    (_w("apart", si.F16, si.NCHW, 70, ((64, 4, 4), (36, 5, 5)), 80, 70, 70), 0, "k_score_exit"),
    (_w("dense", si.BF16, si.NCHW, 130, ((256, 7, 7), (512, 4, 4)), 100, 70), 0, "k_finish_dense"),
    (_w("shared", si.F16, si.NHWC, 150, ((1024, 2, 2), (260, 1, 1)), 101, 101), 0, "k_score_shared"),
    (_w("shared_crowd", si.F16, si.NHWC, 1300, ((64, 2, 1), (96, 1, 1)), 301, 301), 0, "k_score_shared"),
    (_w("sparse", si.BF16, si.NCHW, 60, ((256, 14, 14), (512, 7, 7)), 60, 12, 60), READY, "k_lookup_sparse"),
    # more clusters than the chip holds: some begin when others have decided
    (_w("sparse_late", si.BF16, si.NCHW, 512, ((256, 14, 14), (2048, 7, 7)), 60, 12, 512, tau=0.81, sigma=1.0), READY, "k_lookup_sparse"),
    (_w("sparse_apart", si.F32, si.NCHW, 50, ((1028, 7, 7), (2052, 7, 7)), 30, 8, 50), READY, "k_score_exit"),
]


@pytest.mark.parametrize("w,flags,kernel", CASES, ids=lambda v: getattr(v, "name", ""))
def test_frames_marked_as_gone_are_left_alone(w, flags, kernel):
    cents, counts = si.initial_centers(w)
    mem = oracle.OracleMemory(w.n, w.dims, [w.tau] * w.L, cents, counts, w.S, w.k_init, w.k_min, w.k_max, w.window_W)
    cache = smtm.smtm_cache_create(w.n, w.dims, [w.tau] * w.L, cents, counts, n_streams=w.S, k_init=w.k_init, k_min=w.k_min,
                                   k_max=w.k_max, window_W=w.window_W, max_batch=w.B, flags=flags)
    sid = si.stream_ids(w) if w.S > 1 else None
    gbs, labs, rng, looked_up = [smtm.Batch(cache, w.B, stream_id=sid) for _ in range(2)], si.labels(w), np.random.default_rng(5), 0
    for t in range(w.T):
        gb, ob = gbs[t % 2], mem.new_batch(w.B, sid)
        smtm.smtm_batch_reset(cache, gb)
        for l in range(w.L):
            x = si.frames(w, l, labs[t], t, device="cuda")
            # a third of the frames still in, marked as exits at this layer, some of them at the last one
            marked = np.nonzero((ob["done"] == 0) & (rng.random(w.B) < 0.34))[0]
            stop = np.where(rng.random(len(marked)) < 0.7, l + 1, w.L).astype(np.int32)
            at = torch.from_numpy(marked).cuda()
            gb.done[at], gb.exit_layer[at], gb.pred[at] = 1, torch.from_numpy(stop).cuda(), -1
            gb.sv[l][at] = torch.rand((len(marked), w.dims[l]), device="cuda")   # (vectors of the caller's own)
            ob["done"][marked], ob["exit_layer"][marked] = 1, stop
            gone, todo = torch.from_numpy(np.nonzero(ob["done"])[0]).cuda(), ob["done"] == 0
            fields = (gb.done, gb.exit_layer, gb.pred, gb.sa, gb.ac, gb.sep, gb.top, gb.sv[l])
            before = [f[gone].cpu().numpy() for f in fields]
            torch.cuda.synchronize()
            got = launches(lambda: smtm.smtm_lookup_exit(cache, l, smtm.Fmap(x, w.dtype, w.layout, *si.shape4(w, l)), gb)) if t == 2 else []
            assert not got or kernel in [g.kernel for g in got]
            smtm.smtm_lookup_exit(cache, l, smtm.Fmap(x, w.dtype, w.layout, *si.shape4(w, l)), gb)
            torch.cuda.synchronize()
            for f, kept in zip(fields, before):
                assert np.array_equal(f[gone].cpu().numpy(), kept, equal_nan=kept.dtype == np.float32)
            mem.lookup_exit(l, x.cpu(), w.dtype, w.layout, si.shape4(w, l), ob)
            for f in ("done", "exit_layer", "pred"):
                assert np.array_equal(getattr(gb, f).cpu().numpy(), ob[f]), f
            compare_layer(w, l, x, gb, ob, todo, Report())
            looked_up += int(todo.sum())
        fb = si.fallback_labels(w, labs[t])
        smtm.smtm_cache_update_resize(cache, gb, torch.from_numpy(fb).cuda())
        mem.update(ob, fb)
        mem.resize()
        compare_state(w, cache, mem, Report())
    ctr = smtm.smtm_cache_get_counters(cache)
    assert int(ctr[smtm.CTR_LOOKUPS]) == looked_up and sum(mem.exits_per_layer) > 0
    assert [int(v) for v in ctr[: w.L]] == [int(v) for v in mem.exits_per_layer]
    smtm.smtm_cache_destroy(cache)
