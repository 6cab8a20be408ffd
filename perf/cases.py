"""Timed cases of the Spatial Pooler library: the work its users have it do,
through the public entry points of paper_1608_01966_gb300, from one frame of
one small pooler to a run of 256 poolers.

Every case draws its pools, permanences and frames from the seed with the
package's generators (the recipes of workloads.py): permanences U[0.1, 0.3)
around the threshold 0.2, blobbed video frames of 5-20 % density, Bernoulli
frames elsewhere.  A state keeps what a program keeps between calls: handles
(the learnt permanences live in them), frames on the device or in pinned
memory, and output buffers.

Kinds of cases (the "kind" of a case):
  call     one frame of one pooler per call, host frame in, active list out
  noalloc  one frame on permanences the caller owns on the device
  frames   a sequence of device frames of one pooler in one call
  batch    a run of frames of many equal poolers in one call
  uneven   the same for poolers of uneven shapes
  dense    inference over frames of poolers whose pools are the whole input
  encode   colour or gray camera frames to packed input bits
  serve    one frame of every stream of a server, submitted and collected
"""
import concurrent.futures as cf
import math
import os

import numpy as np
import torch

import paper_1608_01966_gb300 as spg
from paper_1608_01966_gb300 import synth, workloads as wl

VIDEO_POOL = 64  # distinct video frames behind a longer sequence
RESOLUTIONS = ((320, 180), (640, 360), (960, 540))


def listed():
    return [
        # the 32x32 workload: 256 columns, a hundred learning frames in one
        # call, every frame's overlaps recorded
        dict(name="small_frames", kind="frames", W=32, H=32, pool="uniform", C=256, S=16, m=4,
             k=10, inh=0, frames=100, learn=True, ovs=True),
        # a live camera: one 960x540 frame per call, the active columns back
        # on the host before the next one
        dict(name="live_call", kind="call", W=960, H=540, pool="window", C=1024, S=256, m=4,
             k=40, inh=0, learn=True),
        # a real-time stage that owns its memory: the paper's default pooler
        # (2048 x 128 on 240x134), one learning frame, nothing allocated
        dict(name="noalloc_default", kind="noalloc", W=240, H=134, pool="uniform", C=2048, S=128,
             m=8, k=40, inh=0, learn=True),
        # training one paper-scale pooler on a 500-frame video, with the record
        # of its overlaps that shows how the training goes
        dict(name="video_500", kind="frames", W=960, H=540, pool="window", C=1024, S=256, m=4,
             k=40, inh=0, frames=500, learn=True, ovs=True),
        # two points of the paper's parameter sweep, 200 learning frames each:
        # many columns of small pools competing in 9x9 neighbourhoods, and
        # the largest pooler of the sweep
        dict(name="sweep_local", kind="frames", W=960, H=540, pool="window", C=4096, S=64, m=2,
             k=32, inh=1, frames=200, learn=True, ovs=False),
        dict(name="sweep_large", kind="frames", W=960, H=540, pool="window", C=4096, S=256, m=8,
             k=128, inh=0, frames=200, learn=True, ovs=True),
        # a video server's poolers trained side by side: 256 of paper scale
        dict(name="batch_256", kind="batch", members=256, W=960, H=540, C=1024, S=256, m=4, k=40,
             frames=20, learn=True, ovs=False),
        # 64 poolers of odd and uneven shapes in one batch, overlaps recorded
        dict(name="uneven_64", kind="uneven", members=64, c_lo=128, c_hi=4096, s_lo=16, s_hi=256,
             n_lo=256, n_hi=16384, frames=16, learn=True, ovs=True),
        # classification with dense pools: 16 poolers x 256 frames
        dict(name="dense_16", kind="dense", members=16, C=1024, n_in=1024, k=20, frames=256,
             ovs=False),
        # camera frames to input bits: at the pooler's size, and full-HD
        # frames halved to it
        dict(name="encode_540p", kind="encode", W=960, H=540, ch=3, reduce=1, block=11,
             frames=128),
        dict(name="encode_1080p", kind="encode", W=1920, H=1080, ch=3, reduce=2, block=11,
             frames=64),
        # 32 live streams of mixed resolution on the server, a frame of each
        dict(name="serve_32", kind="serve", streams=32, C=1024, S=256, k=40, learn=True),
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, its logarithm spread evenly."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _pooler(rng, c_hi=4096, s_hi=256):
    """One pooler: a video frame with windowed pools on a square grid, or a
    flat or small input with uniform pools of any size."""
    S = _log(rng, 16, s_hi)
    m = rng.choice((2, 4, 8))
    if rng.random() < 0.5:
        W, H = rng.choice(RESOLUTIONS)
        g = _log(rng, 16, int(c_hi ** 0.5))
        C = g * g
        inh = 1 if rng.random() < 0.3 else 0
        pool = "window"
    else:
        W, H = _log(rng, 16, 256), _log(rng, 8, 256)
        C, inh, pool = _log(rng, 64, c_hi), 0, "uniform"
        S = min(S, W * H)
    return dict(W=W, H=H, pool=pool, C=C, S=S, m=m, k=_log(rng, 1, max(2, C // 16)), inh=inh)


def draw(rng):
    kind = rng.choice(("call", "noalloc", "frames", "frames", "batch", "uneven", "dense",
                       "encode", "encode", "serve"))
    learn = rng.random() < 0.7
    if kind in ("call", "noalloc"):
        return dict(kind=kind, learn=learn, **_pooler(rng))
    if kind == "frames":
        p = _pooler(rng)
        return dict(kind=kind, frames=_log(rng, 1, 200), learn=learn,
                    ovs=p["inh"] == 0 and rng.random() < 0.3, **p)
    if kind == "batch":
        W, H = rng.choice(RESOLUTIONS)
        g = _log(rng, 16, 32)
        return dict(kind=kind, members=_log(rng, 8, 200), W=W, H=H, C=g * g,
                    S=_log(rng, 32, 256), m=4, k=_log(rng, 4, 64), frames=_log(rng, 1, 20),
                    learn=learn, ovs=rng.random() < 0.3)
    if kind == "uneven":
        return dict(kind=kind, members=_log(rng, 4, 64), c_lo=_log(rng, 64, 256),
                    c_hi=_log(rng, 512, 4096), s_lo=16, s_hi=_log(rng, 32, 256), n_lo=256,
                    n_hi=_log(rng, 1024, 16384), frames=_log(rng, 1, 16), learn=learn,
                    ovs=rng.random() < 0.3)
    if kind == "dense":
        return dict(kind=kind, members=_log(rng, 1, 16), C=_log(rng, 64, 1024),
                    n_in=_log(rng, 64, 1024), k=_log(rng, 1, 32), frames=_log(rng, 16, 256),
                    ovs=rng.random() < 0.3)
    if kind == "encode":
        f = rng.choice((1, 1, 2, 3, 4, 5, 8))
        W, H, ch = _log(rng, 96, 1920), _log(rng, 64, 1080), rng.choice((1, 3))
        most = max(1, min(128, (128 * 960 * 540 * 3) // (W * H * ch)))
        return dict(kind=kind, W=W, H=H, ch=ch, reduce=f, block=rng.choice((3, 5, 7, 9, 11, 13)),
                    frames=_log(rng, 1, most))
    return dict(kind=kind, streams=_log(rng, 1, 48), C=rng.choice((256, 576, 1024)),
                S=_log(rng, 64, 256), k=_log(rng, 8, 40), learn=learn)


# ---- inputs -------------------------------------------------------------------

def _base(seed):
    return synth.derive_seed(wl.BASE_SEED + 7, synth.PURPOSE_INSTANCE, seed)


def _par(fn, items):
    """The generators are C code called without the interpreter's lock."""
    with cf.ThreadPoolExecutor(max_workers=min(16, os.cpu_count() or 4)) as ex:
        return list(ex.map(fn, items))


def _case(c, seed):
    """The package's description of one pooler (pools, permanences, sizes)."""
    if c["pool"] == "window":
        return wl.grid_case("perf", c["C"], c["S"], seed, W=c["W"], H=c["H"], min_overlap=c["m"],
                            k=c["k"], inhibition=c["inh"], radius=4)
    idx = synth.pool_uniform(synth.derive_seed(seed, synth.PURPOSE_POOL, 0), c["C"], c["S"],
                             c["W"] * c["H"])
    perm = synth.perm_uniform(synth.derive_seed(seed, synth.PURPOSE_PERM, 0), (c["C"], c["S"]),
                              0.1, 0.3)
    return wl.Case("perf", c["W"], c["H"], c["C"], c["S"], idx, perm, np.ones(c["C"], np.float32),
                   min_overlap=c["m"], k=c["k"], inhibition=c["inh"])


def _frames(c, seed, n):
    """n frames of a pooler's input, 0/1 bytes: blobbed video, or Bernoulli
    with a tenth of the bits set."""
    def one(t):
        s = synth.derive_seed(seed, synth.PURPOSE_FRAME, t)
        if c["pool"] == "window":
            return synth.frame_blobbed(s, c["W"], c["H"])
        return synth.frame_bernoulli(s, c["W"] * c["H"], 0.10)
    return np.stack(_par(one, range(n)))


def _device(words):
    return torch.from_numpy(np.ascontiguousarray(words).view(np.int32)).cuda()


def _create(case):
    return spg.sp_create_from_state(case.config(), case.idx, case.perm, case.boost)


def _zeros(shape, dtype=torch.int32):
    return torch.zeros(shape, dtype=dtype, device="cuda")


class State:
    """What a program keeps; gives the library's objects back when it goes."""

    def __init__(self, **kw):
        self.handles, self.batch, self.encoder, self.server = [], None, None, None
        self.__dict__.update(kw)

    def __del__(self):
        try:
            if self.server is not None:
                spg.sp_server_destroy(self.server)
            if self.encoder is not None:
                spg.sp_encoder_destroy(self.encoder)
            if self.batch is not None:
                spg.sp_batch_destroy(self.batch)
            for h in self.handles:
                spg.sp_destroy(h)
        except Exception:
            pass


def _batch_state(c, cases, per_member, n):
    """Handles, batch, device batch frames and output records.  per_member[i]:
    member i's packed frames [n][words]."""
    s = State(case=c, handles=[_create(x) for x in cases])
    s.batch = spg.sp_batch_create(s.handles)
    info = spg.sp_batch_get_info(s.batch)
    off, _ = spg.sp_batch_offsets(s.batch)
    s.stride = (info["frame_words"] + 3) // 4 * 4
    s.d = _device(wl.batch_frames(per_member, off, s.stride))
    s.mw = info["mask_words"]
    s.masks = _zeros((n, s.mw))
    _, s.ow = spg.sp_batch_overlap_offsets(s.batch)
    s.ov = _zeros((n, s.ow), torch.float32) if c["ovs"] else None
    return s


def _shapes(c):
    """Columns, synapses, input bits and frame density of an uneven batch's
    poolers: drawn evenly from the case's ranges, the same for every seed."""
    out = []
    for i in range(c["members"]):
        r, _ = synth.splitmix64(synth.derive_seed(wl.BASE_SEED + 4, synth.PURPOSE_SHAPE, i), 4)
        C = c["c_lo"] + r[0] % (c["c_hi"] - c["c_lo"] + 1)
        n_in = c["n_lo"] + r[2] % (c["n_hi"] - c["n_lo"] + 1)
        S = min(c["s_lo"] + r[1] % (c["s_hi"] - c["s_lo"] + 1), n_in)
        out.append((C, S, n_in, 0.02 + 0.18 * ((r[3] >> 11) / float(1 << 53))))
    return out


def _uneven(c, seed):
    """The poolers (k = 2 % of the columns) and their 0/1 frames."""
    base = _base(seed)

    def one(i):
        C, S, n_in, p = _shapes(c)[i]
        sd = synth.derive_seed(base, synth.PURPOSE_INSTANCE, i)
        sp = _case(dict(W=n_in, H=1, pool="uniform", C=C, S=S, m=4, k=max(1, (2 * C + 50) // 100),
                        inh=0), sd)
        return sp, np.stack([synth.frame_bernoulli(synth.derive_seed(sd, synth.PURPOSE_FRAME, t),
                                                   n_in, p) for t in range(c["frames"])])
    got = _par(one, range(c["members"]))
    return [g[0] for g in got], [g[1] for g in got]


def prepare(case, seed):
    c, kind, base = case, case["kind"], _base(seed)
    if kind == "call":
        sp = _case(c, base)
        f = torch.from_numpy(wl.pack(_frames(c, base, 16)).view(np.int32)).pin_memory()
        return State(case=c, handles=[_create(sp)], pinned=f, t=0, f=f.numpy().view(np.uint32),
                     out=np.empty(sp.C, np.int32))
    if kind == "noalloc":
        sp = _case(c, base)
        return State(case=c, cfg=sp.config(), idx=_device(sp.idx),
                     perm=torch.from_numpy(sp.perm).cuda(), boost=torch.from_numpy(sp.boost).cuda(),
                     d=_device(wl.pack(_frames(c, base, 16))), t=0, mask=_zeros((sp.C + 31) // 32),
                     list=_zeros(1 + sp.C))
    if kind == "frames":
        sp, n = _case(c, base), c["frames"]
        few = wl.pack(_frames(c, base, min(n, VIDEO_POOL)))
        s = State(case=c, handles=[_create(sp)], d=_device(few[np.arange(n) % len(few)]),
                  masks=_zeros((n, (sp.C + 31) // 32)))
        s.ov = _zeros((n, sp.C), torch.float32) if c["ovs"] else None
        return s
    if kind == "batch":
        one = dict(c, pool="window", inh=0)
        cases = _par(lambda i: _case(one, synth.derive_seed(base, synth.PURPOSE_INSTANCE, i)),
                     range(c["members"]))
        few = wl.pack(_frames(one, base, VIDEO_POOL))
        t = np.arange(c["frames"])
        # every pooler watches the videos from another place
        return _batch_state(c, cases, [few[(7 * i + t) % VIDEO_POOL] for i in range(len(cases))],
                            c["frames"])
    if kind == "uneven":
        cases, fr = _uneven(c, seed)
        return _batch_state(c, cases, [wl.pack(f) for f in fr], c["frames"])
    if kind == "dense":
        cases, fr = wl.dense_cases(c["members"], c["frames"], C=c["C"], n_in=c["n_in"], k=c["k"],
                                   seed=base)
        return _batch_state(c, cases, [wl.pack(f) for f in fr], c["frames"])
    if kind == "encode":
        few = np.stack(_par(lambda t: synth.frame_rgb(synth.derive_seed(base, synth.PURPOSE_FRAME, t),
                                                      c["W"], c["H"]), range(min(c["frames"], 8))))
        if c["ch"] == 1:
            few = np.ascontiguousarray(few[..., 1])
        d = torch.from_numpy(few.reshape(len(few), -1)).cuda()
        d = d[torch.arange(c["frames"], device="cuda") % len(few)].contiguous()
        e = spg.sp_encoder_create(spg.sp_encoder_config_init(
            src_w=c["W"], src_h=c["H"], channels=c["ch"], reduce=c["reduce"], block=c["block"]))
        info = spg.sp_encoder_get_info(e)
        return State(case=c, encoder=e, d=d, src=info["src_bytes"],
                     bits=_zeros((c["frames"], info["out_words"])))
    # serve: stream i at resolution i mod 3, eight frames of it in host memory
    cases, frames = [], []
    for i in range(c["streams"]):
        W, H = RESOLUTIONS[i % 3]
        one = dict(W=W, H=H, pool="window", C=c["C"], S=c["S"], m=4, k=c["k"], inh=0)
        cases.append((one, synth.derive_seed(base, synth.PURPOSE_INSTANCE, i)))
    sps = _par(lambda x: _case(*x), cases)
    for i, (one, sd) in enumerate(cases):
        frames.append(wl.pack(np.stack([synth.frame_blobbed(
            synth.derive_seed(sd, synth.PURPOSE_FRAME, t), one["W"], one["H"]) for t in range(8)])))
    s = State(case=c, frames=frames, t=0)
    s.server = spg.sp_server_create(c["streams"], 4, max(f.shape[1] for f in frames), 8 << 30,
                                    c["k"])
    s.ids = np.array([spg.sp_server_open_stream(s.server, x.config(duty_period=1000.0),
                                                (x.idx, x.perm, x.boost)) for x in sps], np.uint32)
    s.at = {int(v): i for i, v in enumerate(s.ids)}
    s.ptrs = [np.array([f[t].ctypes.data for f in frames], np.uint64) for t in range(8)]
    s.learn = np.full(len(sps), 1 if c["learn"] else 0, np.int32)
    return s


def run(state):
    s, c = state, state.case
    kind = c["kind"]
    if kind == "call":
        f = s.f[s.t % len(s.f)]
        s.t += 1
        spg.sp_compute(s.handles[0], f, c["learn"])
        active = spg.sp_active_columns(s.handles[0])
        s.out[:len(active)] = active
        s.out[len(active):] = -1
        return [s.out]
    stream = torch.cuda.current_stream()
    if kind == "noalloc":
        x = s.d[s.t % len(s.d)]
        s.t += 1
        spg.sp_step_noalloc(s.cfg, s.idx, s.perm, s.boost, x, c["learn"], s.mask, s.list, stream)
        return [s.perm, s.mask]
    if kind == "frames":
        if s.ov is None:
            spg.sp_compute_frames_device(s.handles[0], s.d, c["frames"], s.d.shape[1], c["learn"],
                                         s.masks, stream)
            return [s.masks]
        spg.sp_compute_frames_overlaps_device(s.handles[0], s.d, c["frames"], s.d.shape[1],
                                              c["learn"], s.masks, s.ov, stream)
        return [s.masks, s.ov]
    if kind in ("batch", "uneven"):
        if s.ov is None:
            spg.sp_batch_compute_device(s.batch, s.d, c["frames"], s.stride, c["learn"], s.masks,
                                        s.mw, stream)
            return [s.masks]
        spg.sp_batch_compute_overlaps_device(s.batch, s.d, c["frames"], s.stride, c["learn"],
                                             s.masks, s.mw, s.ov, s.ow, stream)
        return [s.masks, s.ov]
    if kind == "dense":
        if s.ov is None:
            spg.sp_batch_infer_device(s.batch, s.d, c["frames"], s.stride, s.masks, s.mw, stream)
            return [s.masks]
        spg.sp_batch_infer_overlaps_device(s.batch, s.d, c["frames"], s.stride, s.masks, s.mw,
                                           s.ov, s.ow, stream)
        return [s.masks, s.ov]
    if kind == "encode":
        spg.sp_encode_device(s.encoder, s.d, c["frames"], s.src, s.bits, s.bits.shape[1], stream)
        return [s.bits]
    spg.sp_server_submit_many_ptrs(s.server, s.ids, s.ptrs[s.t % len(s.ptrs)], s.learn)
    s.t += 1
    out = np.full((len(s.ids), c["k"]), -1, np.int32)
    got = 0
    while got < len(s.ids):
        for r, active in spg.sp_server_poll(s.server, max_results=64, active_cap=64 * c["k"],
                                            wait_ms=1000):
            out[s.at[r["stream_id"]], :len(active)] = active
            got += 1
    return [out]


# ---- what a pass cannot do without ----------------------------------------------

def work(case):
    c, kind = case, case["kind"]
    if kind == "encode":
        px = (c["W"] // c["reduce"]) * (c["H"] // c["reduce"])
        # block sums and luma per source pixel, two symmetric window passes,
        # rounding and comparison per output pixel
        ops = px * (c["reduce"] ** 2 * c["ch"] + 3 + 2 * c["block"] + 3)
        return {"bytes": c["frames"] * (c["W"] * c["H"] * c["ch"] + px / 8),
                "flops": c["frames"] * ops}
    if kind == "uneven":
        b = ops = 0.0
        for C, S, bits, _ in _shapes(c):
            one = work(dict(kind="frames", C=C, S=S, W=bits, H=1, k=max(1, (2 * C + 50) // 100),
                            frames=c["frames"], learn=c["learn"], ovs=c["ovs"]))
            b, ops = b + one["bytes"], ops + one["flops"]
        return {"bytes": b, "flops": ops}
    if kind == "dense":
        n, C, S, bits, k = c["members"], c["C"], c["n_in"], c["n_in"], c["k"]
        frames = c["frames"]
    elif kind == "serve":
        n, C, S, k, frames = c["streams"], c["C"], c["S"], c["k"], 1
        bits = sum(w * h for w, h in RESOLUTIONS) / 3
    else:
        n, C, S, bits, k = c.get("members", 1), c["C"], c["S"], c["W"] * c["H"], c["k"]
        frames = c.get("frames", 1)
    # pools and permanences once, every frame in, every mask (and overlap
    # record) out, the permanences of a frame's winners back where it learns
    b = n * (C * S * 8 + frames * (bits / 8 + C / 8))
    if c.get("ovs"):
        b += n * frames * C * 4
    if c.get("learn"):
        b += n * min(C, frames * k) * S * 4
    return {"bytes": b, "flops": 2.0 * n * C * S * frames}


# ---- the same in 64 bits, without the library -------------------------------------

def _winners(ov, k):
    order = np.lexsort((np.arange(len(ov)), -ov))[:k]
    return order[ov[order] > 0]


def _exact_one(sp, frames, learn):
    """Overlaps of every frame and the permanences after the last, global
    inhibition and unit boosts, in numpy's 64 bits."""
    perm = sp.perm.astype(np.float64)
    thr, inc, dec = (float(np.float32(v)) for v in (sp.thr, sp.inc, sp.dec))
    out = np.empty((len(frames), sp.C))
    for t, x in enumerate(frames):
        on = x[sp.idx] != 0
        n = ((perm >= thr) & on).sum(axis=1)
        out[t] = np.where(n < sp.min_overlap, 0, n)
        if learn:
            w = _winners(out[t], sp.k)
            perm[w] = np.where(on[w], np.minimum(1.0, perm[w] + inc),
                               np.maximum(0.0, perm[w] - dec))
    return out, perm


def exact(case, seed):
    c, kind, base = case, case["kind"], _base(seed)
    if kind == "noalloc":
        sp = _case(c, base)
        if c["inh"]:
            return None
        _, perm = _exact_one(sp, _frames(c, base, 1), c["learn"])
        return [perm, None]
    if not c.get("ovs"):
        return None
    if kind == "frames":
        if c["C"] * c["S"] * c["frames"] > 1 << 30:
            return None
        few = _frames(c, base, min(c["frames"], VIDEO_POOL))
        fr = [few[t % len(few)] for t in range(c["frames"])]
        return [None, _exact_one(_case(c, base), fr, c["learn"])[0]]
    if kind == "uneven":
        if sum(C * S for C, S, _, _ in _shapes(c)) * c["frames"] > 1 << 30:
            return None
        cases, fr = _uneven(c, seed)
        got = _par(lambda i: _exact_one(cases[i], fr[i], c["learn"])[0], range(len(cases)))
        return [None, np.concatenate(got, axis=1)]
    if kind == "dense":
        cases, fr = wl.dense_cases(c["members"], c["frames"], C=c["C"], n_in=c["n_in"], k=c["k"],
                                   seed=base)
        out = []
        for sp, f in zip(cases, fr):
            n = f.astype(np.float64) @ (sp.perm.astype(np.float64)
                                        >= float(np.float32(sp.thr))).astype(np.float64).T
            out.append(np.where(n < sp.min_overlap, 0.0, n))
        return [None, np.concatenate(out, axis=1)]
    return None
