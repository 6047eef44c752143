"""The work users have this library do, as cases that can be timed and compared.

Each case is a plain dict; `prepare` builds what a program holds before the call (maps on the device,
the cache, the carries, a CUDA graph where a program would use one), `run` is one pass through the
public entry points, `exact` the same pass in 64-bit torch.  `stay` is the share of
frames that go on to the later exit layers, as measured (for `work`).  Inputs are synthetic: a class centroid per
label broadcast over the map plus Gaussian noise, rectified where a backbone would rectify, labels
from a bounded Zipf law, a share of frames from classes the memory does not hold.

Kinds:
  step    lookups of all exit layers, then update and resize of the memory; `steps` > 0: that many
          consecutive steps captured in one CUDA graph, 0: one step by eager calls
  encode  smtm_encode alone
  warmup  smtm_cache_warmup with labelled frames, then a lookup of other frames
  host    smtm_step_host: one step on maps in pinned host memory, then the memory read back
"""
import numpy as np
import torch

import paper_2112_02644_b200 as smtm

TAU, CL_NUM, CL_DEN = 0.8, 19, 20
WARM_M = 32          # update count attached to the initial centres
REPEAT_P = 0.85      # per stream: the last label repeats with this probability
EXPONENT_MAX = 12    # floor(TS / W) is clamped here in Eq. 5
FT_MAX, FT_FRAC = 1 << 20, 10
DTYPES = {"f32": (smtm.F32, torch.float32, 4), "f16": (smtm.F16, torch.float16, 2), "bf16": (smtm.BF16, torch.bfloat16, 2)}

RESNET50 = "256x56x56 512x28x28 1024x14x14 2048x7x7"
MOBILENETV2 = "24x56x56 32x28x28 96x14x14 320x7x7"
VGG16_CIFAR = ("64x32x32 64x32x32 128x16x16 128x16x16 256x8x8 256x8x8 256x8x8 512x4x4 512x4x4 512x4x4 "
               "512x2x2 512x2x2 512x2x2")


def _case(name, **kw):
    c = dict(name=name, kind="step", dtype="bf16", layout="nchw", B=64, stages=RESNET50, n=100, k_init=10, k_min=10,
             k_max=10, streams=False, window=16, sigma=0.5, relu=True, zipf=1.1, novel=0.2, stay=0.3, forget=False,
             ready=False, steps=0)
    c.update(kw)
    return c


def listed():
    return [
        # One exit layer, a handful of frames, fp32: the smallest call, eager.
        _case("one_layer_fp32", dtype="f32", B=8, stages="64x56x56", n=10, sigma=0.3, relu=False, zipf=0.0, novel=0.0),
        # One video stream frame by frame, as on a phone: clips of 8 frames, four exits of a mobile network.
        _case("one_stream_clip", dtype="f16", layout="nhwc", B=1, stages=MOBILENETV2, n=200, k_init=16, k_min=16,
              k_max=16, zipf=1.2, stay=0.4, steps=8),
        # A batch of frames whose maps the backbone has just produced on the same stream (no promise about them).
        _case("four_exits_eager", B=64, stay=0.5),
        # Mobile network, channels last, batches resident; a fifth of the frames is of unknown classes.
        _case("mobile_nhwc", dtype="f16", layout="nhwc", B=256, stages=MOBILENETV2, n=200, k_init=16, k_min=16,
              k_max=16, zipf=1.2, stay=0.6, ready=True, steps=4),
        # Every one of 1000 classes cached: scoring is a dense contraction.
        _case("thousand_classes", B=1024, stages="2048x7x7", n=1000, k_init=1000, k_min=1000, k_max=1000, sigma=1.0,
              zipf=1.0, novel=0.0, stay=1.0, ready=True, steps=4),
        # 512 video streams, each with its own adaptive fast memory: the serving workload.
        _case("streams_512", B=512, stages="1024x14x14 2048x7x7", n=500, k_init=8, k_min=8, k_max=64, streams=True,
              novel=0.12, stay=0.1, ready=True, steps=8),
        # Thirteen shallow exits with tiny maps, rapidly changing scenes (the frequency table forgets).
        _case("thirteen_exits", dtype="f16", B=128, stages=VGG16_CIFAR, n=100, k_init=5, k_min=5, k_max=20,
              streams=True, window=4, zipf=1.0, forget=True, stay=0.2, steps=4),
        # Pooling alone, the largest maps.
        _case("encode_large", kind="encode", B=1024, stages="256x56x56", novel=0.0),
        # Another input resolution: maps whose rows are odd numbers of bytes.
        _case("odd_maps", B=96, stages="256x60x60 512x30x30 1024x15x15 2048x8x8", k_init=10, k_min=5, k_max=20, stay=0.5),
        # All classes of a 101-class data set cached, two exits.
        _case("all_101_classes", dtype="f16", B=256, stages="1024x14x14 2048x7x7", n=101, k_init=101, k_min=101,
              k_max=101, zipf=1.0, stay=0.2),
        # Building the centres of one layer from labelled frames, then looking other frames up.
        _case("enrol", kind="warmup", dtype="f16", layout="nhwc", B=512, stages="512x28x28", n=200, k_init=16, k_min=16,
              k_max=16, zipf=1.0, novel=0.0),
        # Maps in pinned host memory, the whole step through one call, centres and tables read back.
        _case("host_step", kind="host", B=16, stay=0.5),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choices(("step", "encode", "warmup", "host"), (8, 2, 1, 1))[0]
    dtype, layout = rng.choice(("f32", "f16", "bf16", "bf16")), rng.choice(("nchw", "nchw", "nhwc"))
    es = DTYPES[dtype][2]
    layers = 1 if kind in ("encode", "warmup") else rng.choice((1, 2, 3, 4))
    stages, side, ch = [], _log(rng, 4, 64), 0
    for _ in range(layers):  # deeper layers are smaller and have more channels, as in a backbone
        ch = max(ch, rng.choice((16, 24, 32, 40, 64, 96, 128, 160, 256, 320, 512, 768, 1024, 2048)))
        w = side if rng.random() < 0.7 else max(2, side + rng.choice((-1, 1)))
        stages.append((ch, side, w))
        side = max(2, (side + rng.choice((0, 1))) // rng.choice((1, 2, 2)))
    frame = sum(c * h * w * es for c, h, w in stages)
    most = (1.2e9 if kind == "encode" else 5e7 if kind == "host" else 2.5e8) / frame
    B = max(1, min(_log(rng, 1, 1024), int(most)))
    n = _log(rng, 10, 1000)
    k_max = max(2, min(n, rng.choice((_log(rng, 4, 64), _log(rng, 4, 64), n))))
    k_min = k_max if rng.random() < 0.5 else max(2, k_max // 4)
    streams = B > 1 and k_max <= 64 and rng.random() < 0.5
    ready = kind == "step" and rng.random() < 0.5
    steps = 0 if kind != "step" else rng.choice((0, 2, 4)) if frame * B < 1e8 else rng.choice((0, 2))
    return _case("", kind=kind, dtype=dtype, layout=layout, B=B, stages=" ".join("%dx%dx%d" % s for s in stages), n=n,
                 k_init=k_min, k_min=k_min, k_max=k_max, streams=streams, window=rng.choice((4, 16)),
                 sigma=rng.choice((0.3, 0.5, 1.0)), zipf=rng.choice((1.0, 1.1, 1.2)),
                 novel=0.0 if kind in ("encode", "warmup") else rng.choice((0.1, 0.2)), stay=0.4,
                 forget=streams and rng.random() < 0.3, ready=ready, steps=steps)


# ---- inputs -----------------------------------------------------------------------------------

def _stages(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["stages"].split()]


def _labels(case, rng, steps, B):
    n, outside = case["n"], max(1, case["n"] // 4)
    p = np.arange(1, n + 1, dtype=np.float64) ** -case["zipf"]
    lab = rng.choice(n, size=(steps, B), p=p / p.sum())
    unknown = rng.random((steps, B)) < case["novel"]
    lab = np.where(unknown, n + rng.integers(0, outside, (steps, B)), lab)
    if case["streams"]:
        for t in range(1, steps):
            lab[t] = np.where(rng.random(B) < REPEAT_P, lab[t - 1], lab[t])
    return lab


class _Inputs:
    """Maps, labels and initial centres of a case, from the seed alone."""

    def __init__(self, case, seed):
        self.stages, self.dims = _stages(case), [s[0] for s in _stages(case)]
        self.steps = max(1, case["steps"])
        if case["ready"] and not case["steps"]:
            self.steps = 2  # an eager program that promises resident maps alternates two sets
        rng = np.random.default_rng([seed, 1])
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed * 2 + 1)
        n_all = case["n"] + max(1, case["n"] // 4)
        mu = [torch.randn((n_all, d), generator=gen, device="cuda") for d in self.dims]
        if not case["relu"]:
            mu = [m / m.norm(dim=1, keepdim=True) for m in mu]
        lab = _labels(case, rng, self.steps, case["B"])
        self.labels = torch.from_numpy(lab).cuda()
        self.fallback = torch.where(self.labels < case["n"], self.labels, -1).int()
        self.maps = [[self._map(case, gen, mu[l], self.labels[t], l) for l in range(len(mu))] for t in range(self.steps)]
        self.probe, self.probe_B = None, min(64, case["B"])
        if case["kind"] == "warmup":
            other = torch.from_numpy(_labels(case, rng, 1, self.probe_B)[0]).cuda()
            self.probe = self._map(case, gen, mu[0], other, 0)
        # centres: the expected activation of a class plus the noise a mean over WARM_M frames carries
        self.centers = []
        for m, (c, h, w) in zip(mu, self.stages):
            m = m[: case["n"]].double()
            if case["relu"]:
                t = m / case["sigma"]
                m = m * torch.special.ndtr(t) + case["sigma"] * torch.exp(-0.5 * t * t) / (2 * np.pi) ** 0.5
                noise = torch.randn(m.shape, generator=gen, device="cuda", dtype=torch.float64)
                m = m + noise * (case["sigma"] / (WARM_M * h * w) ** 0.5)
            self.centers.append(m.float().cpu().numpy())
        self.count = 0 if case["kind"] == "warmup" else WARM_M
        self.streams = np.arange(case["B"], dtype=np.int32) if case["streams"] else None

    def _map(self, case, gen, mu, lab, l):
        c, h, w = self.stages[l]
        m = mu[lab]
        if case["layout"] == "nchw":
            x = torch.randn((len(lab), c, h, w), generator=gen, device="cuda").mul_(case["sigma"]).add_(m[:, :, None, None])
        else:
            x = torch.randn((len(lab), h, w, c), generator=gen, device="cuda").mul_(case["sigma"]).add_(m[:, None, None, :])
        return (x.clamp_(min=0) if case["relu"] else x).to(DTYPES[case["dtype"]][1])


class _State:
    pass


def _fmap(case, x, B, stage):
    return smtm.Fmap(x, DTYPES[case["dtype"]][0], smtm.NCHW if case["layout"] == "nchw" else smtm.NHWC, B, *stage)


def prepare(case, seed):
    x, s = _Inputs(case, seed), _State()
    s.case, s.L, s.keep = case, len(x.dims), x
    s.cache = smtm.smtm_cache_create(
        case["n"], x.dims, [TAU] * s.L, x.centers, [np.full(case["n"], x.count, np.uint32)] * s.L,
        n_streams=case["B"] if case["streams"] else 1, k_init=case["k_init"], k_min=case["k_min"], k_max=case["k_max"],
        window_W=case["window"], cl_num=CL_NUM, cl_den=CL_DEN, max_batch=case["B"],
        flags=(smtm.FLAG_FORGET_FT if case["forget"] else 0) | (smtm.FLAG_MAPS_READY if case["ready"] else 0))
    if case["kind"] == "host":
        s.host = [m.cpu().pin_memory() for m in x.maps[0]]
        s.fmaps = [_fmap(case, None, case["B"], st) for st in x.stages]
        s.fallback = x.fallback[0].cpu().numpy()
        s.out = [np.zeros(case["B"], np.uint8), np.zeros(case["B"], np.int32), np.zeros(case["B"], np.int32)]
        return s
    s.fmaps = [[_fmap(case, m, case["B"], st) for m, st in zip(maps, x.stages)] for maps in x.maps]
    if case["kind"] == "encode":
        s.sv = torch.zeros((case["B"], x.dims[0]), device="cuda")
        return s
    if case["kind"] == "warmup":
        s.labels = x.labels[0].int()
        s.probe = _fmap(case, x.probe, x.probe_B, x.stages[0])
        s.carries = [smtm.Batch(s.cache, x.probe_B)]
        return s
    s.carries = [smtm.Batch(s.cache, case["B"], stream_id=x.streams) for _ in range(2)]
    s.turn, s.graph = 0, None
    if case["steps"]:
        # a program warms its kernels up, then captures its steps; the memory starts as it was created
        before = smtm.smtm_cache_export(s.cache)
        spare = [smtm.Batch(s.cache, case["B"], stream_id=x.streams) for _ in range(2)]
        torch.cuda.synchronize()
        for t in range(2):
            _step(s, spare[t], t % x.steps)
        smtm.smtm_cache_import(s.cache, before)
        s.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s.graph):
            for t in range(x.steps):
                _step(s, s.carries[t % 2], t)
    torch.cuda.synchronize()
    return s


def _step(s, carry, t):
    smtm.smtm_lookup_exit_begin(s.cache, 0, s.fmaps[t][0], carry)
    for l in range(1, s.L):
        smtm.smtm_lookup_exit(s.cache, l, s.fmaps[t][l], carry)
    smtm.smtm_cache_update_resize(s.cache, carry, s.keep.fallback[t])


def _carry_out(b):
    return {"sa": b.sa, "done": b.done, "exit_layer": b.exit_layer, "pred": b.pred, "ac": b.ac, "sep": b.sep,
            "top": b.top, "sv": b.sv}


def run(s):
    kind = s.case["kind"]
    if kind == "encode":
        smtm.smtm_encode(s.cache, 0, s.fmaps[0][0], s.sv)
        return s.sv
    if kind == "warmup":
        smtm.smtm_cache_warmup(s.cache, 0, s.fmaps[0][0], s.labels)
        smtm.smtm_lookup_exit_begin(s.cache, 0, s.probe, s.carries[0])
        return _carry_out(s.carries[0])
    if kind == "host":
        # ... and the memory as the step left it, which such a program keeps with its results
        smtm.smtm_step_host(s.cache, s.fmaps, s.host, s.keep.streams, s.fallback, True, *s.out)
        centers = [smtm.smtm_cache_get_centers(s.cache, l)[0] for l in range(s.L)]
        return {"out": list(s.out), "centers": centers, "tables": smtm.smtm_cache_get_tables(s.cache)}
    if s.graph is not None:
        s.graph.replay()
        return [_carry_out(b) for b in s.carries]
    carry = s.carries[s.turn % 2]
    _step(s, carry, s.turn % s.keep.steps)
    s.turn += 1
    return _carry_out(carry)


def work(case):
    stages, B = _stages(case), case["B"]
    es = DTYPES[case["dtype"]][2]
    steps = max(1, case["steps"])
    read = B * stages[0][0] * (stages[0][1] * stages[0][2] * es + 4)
    flops = B * stages[0][0] * stages[0][1] * stages[0][2]
    if case["kind"] == "encode":
        return {"bytes": read, "flops": flops}
    if case["kind"] == "warmup":
        frames = B + min(64, B)
        return {"bytes": read * frames // B + 2 * 4 * case["n"] * stages[0][0], "flops": flops * frames // B}
    for c, h, w in stages[1:]:  # frames that have exited need nothing of the later layers
        read += int(case["stay"] * B * c * (h * w * es + 4))
        flops += int(case["stay"] * B * c * h * w)
    for i, (c, _, _) in enumerate(stages):  # the centres once, the dot products against the fast memory
        read += 4 * case["n"] * c
        flops += int((case["stay"] if i else 1) * 2 * B * case["k_max"] * c)
    return {"bytes": steps * (read + 8 * case["n"] * (B if case["streams"] else 1) + 4 * B * case["k_max"]),
            "flops": steps * flops}


def tolerance(case):
    # Pooling is a 32-bit sum; a similarity is a 32-bit dot product over up to 2048 channels (three bf16 products
    # with 32-bit sums against more than 64 classes).  The second best class of a frame may be tied.
    return {"rel": 1e-5, "max": 2e-4, "differ": 0.005}


# ---- the same in 64 bits -------------------------------------------------------------------------

class _Memory:
    def __init__(self, case, x):
        self.case, self.n, self.S = case, case["n"], case["B"] if case["streams"] else 1
        self.cen = [torch.from_numpy(c).cuda().double() for c in x.centers]
        self.m = [torch.full((self.n,), float(x.count), device="cuda", dtype=torch.float64) for _ in x.centers]
        self.ft = torch.zeros((self.S, self.n), dtype=torch.int64, device="cuda")
        self.ts = torch.zeros_like(self.ft)
        self.members = (torch.arange(case["k_max"], device="cuda") % self.n).repeat(self.S, 1)
        self.k = torch.full((self.S,), case["k_init"], dtype=torch.int64, device="cuda")
        self.sid = torch.arange(case["B"], device="cuda") if case["streams"] else torch.zeros(case["B"], dtype=torch.int64, device="cuda")

    def carry(self, B, L):
        dev, f = "cuda", torch.float64
        return {"sa": torch.zeros((B, self.case["k_max"]), dtype=f, device=dev), "done": None, "exit_layer": None,
                "pred": None, "ac": torch.full((B, L), float("nan"), dtype=f, device=dev),
                "sep": torch.full((B, L), float("nan"), dtype=f, device=dev), "top": None,
                "sv": [torch.zeros((B, c.shape[1]), dtype=f, device=dev) for c in self.cen]}

    def lookup(self, l, maps, layout, sid, carry, done, stop, pred):
        """One exit layer for the frames not done; done, stop and pred are changed in place."""
        at = (~done).nonzero().flatten()
        if not len(at):
            return
        sv = _pool(maps, layout, at)
        carry["sv"][l][at] = sv
        mem, k = self.members[sid[at]], self.k[sid[at]]
        used = torch.arange(mem.shape[1], device="cuda")[None] < k[:, None]
        dots = (sv @ self.cen[l].T).gather(1, mem)
        length = sv.norm(dim=1, keepdim=True) * self.cen[l].norm(dim=1)[mem]
        s = torch.where(used & (length > 0), dots / length, 0.0)
        sa = torch.where(used, carry["sa"][at] + s * 2.0 ** l, 0.0)
        carry["sa"][at] = sa
        low = torch.tensor(-float("inf"), dtype=torch.float64, device="cuda")

        def top(v):
            v, i = torch.where(used, v, low).topk(2, dim=1)
            gap = torch.where(v[:, 1] > 0, (v[:, 0] - v[:, 1]) / v[:, 1], float("inf"))
            return torch.where(v[:, 0] > 0, gap, 0.0), v, i

        ac, v, i = top(sa)
        carry["ac"][at, l], carry["sep"][at, l] = ac, top(s)[0]
        leave = (v[:, 0] > 0) & (v[:, 0] - v[:, 1] > TAU * v[:, 1].clamp(min=0))
        out = at[leave]
        done[out], stop[out] = True, l + 1
        pred[out] = mem[leave].gather(1, i[leave][:, :1]).flatten()

    def fold(self, l, sv, lab):
        q = torch.bincount(lab, minlength=self.n).double()
        total = torch.zeros_like(self.cen[l]).index_add_(0, lab, sv)
        hit = q > 0
        self.cen[l][hit] = ((self.cen[l] * self.m[l][:, None] + total) / (self.m[l] + q)[:, None])[hit]
        self.m[l] += q

    def update(self, carry, lab, stop):
        for l in range(len(self.cen)):
            at = (lab >= 0) & (stop >= l + 1)
            self.fold(l, carry["sv"][l][at], lab[at])
        W, forget = self.case["window"], self.case["forget"]
        # one frame of every stream at a time, in ascending order
        for lb in ([lab] if self.case["streams"] else lab[:, None]):
            seen = torch.arange(self.n, device="cuda")[None] == lb[:, None]
            self.ts = torch.where(seen, 0, self.ts + 1)
            if forget:
                aged = torch.where(~seen & (self.ts % W == 0), self.ft >> 2, self.ft)
                self.ft = torch.where(seen, (self.ft + (1 << FT_FRAC)).clamp(max=FT_MAX << FT_FRAC), aged)
            else:
                self.ft = (self.ft + seen).clamp(max=FT_MAX)
        score = self.ft if forget else self.ft << (2 * (EXPONENT_MAX - (self.ts // W).clamp(max=EXPONENT_MAX)))
        best, order = score.sort(dim=1, descending=True, stable=True)
        total = best.sum(dim=1)
        best, order = best[:, : self.case["k_max"]], order[:, : self.case["k_max"]]
        enough = CL_DEN * best.cumsum(dim=1) > CL_NUM * total[:, None]
        enough[:, : self.case["k_min"] - 1] = False
        size = torch.where(enough.any(dim=1), enough.int().argmax(dim=1) + 1, self.case["k_max"])
        moved = total > 0
        self.members = torch.where(moved[:, None], order, self.members)
        self.k = torch.where(moved, size, self.k)


def _pool(maps, layout, at):
    return torch.cat([maps[i].double().mean(dim=(2, 3) if layout == "nchw" else (1, 2)) for i in at.split(64)])


def exact(case, seed):
    x = _Inputs(case, seed)
    if case["kind"] == "encode":
        return _pool(x.maps[0][0], case["layout"], torch.arange(case["B"], device="cuda"))
    mem, L = _Memory(case, x), len(x.dims)
    if case["kind"] == "warmup":
        every = torch.arange(case["B"], device="cuda")
        mem.fold(0, _pool(x.maps[0][0], case["layout"], every), x.labels[0])
        steps, maps, B = 1, [[x.probe]], x.probe_B
    else:
        steps, maps, B = max(1, case["steps"]), x.maps, case["B"]
    carries = [mem.carry(B, L) for _ in range(2)]
    sid = mem.sid[:B]
    for t in range(steps):
        c = carries[t % 2]
        c["sa"].zero_()
        done = torch.zeros(B, dtype=torch.bool, device="cuda")
        stop, pred = torch.full((B,), L, device="cuda"), torch.full((B,), -1, device="cuda")
        for l in range(L):
            mem.lookup(l, maps[t][l], case["layout"], sid, c, done, stop, pred)
        if case["kind"] != "warmup":
            mem.update(c, torch.where(done, pred, x.fallback[t].long()), stop)
    if case["kind"] == "host":
        return {"out": None, "centers": mem.cen, "tables": None}
    return carries if case["steps"] else carries[0]
