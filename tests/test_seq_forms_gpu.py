"""Frame sequences of one SP (Alg. 1, Alg. 2 and Section 1.1, one persistent
launch per call): the forms its state takes -- pools, bitmaps of 64 x 64 boxes
with or without the permanences in shared memory, one CTA or a cluster -- at
the edges of their tilings, against the oracle.  Masks, every frame's overlaps
and the permanences are compared exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1608_01966_gb300 as spg  # noqa: E402
from paper_1608_01966_gb300 import synth, workloads as wl  # noqa: E402
from helpers import oracle_run  # noqa: E402

pytestmark = pytest.mark.gpu


def _box_pools(rng, C, S, W, H, box):
    """Ascending pools of S distinct pixels, each inside a box x box window
    that may touch any edge of the frame."""
    idx = np.empty((C, S), np.uint32)
    for c in range(C):
        x0 = rng.integers(0, max(1, W - box + 1))
        y0 = rng.integers(0, max(1, H - box + 1))
        w, h = min(box, W), min(box, H)
        px = np.sort(rng.choice(w * h, S, replace=False))
        idx[c] = (y0 + px // w) * W + x0 + px % w
    return idx


def _check(W, H, C, idx, k, m, boost=None, inh=0, gw=0, gh=0, radius=0, frames=11, stride_pad=0,
           density=0.3, offset=0):
    S = idx.shape[1]
    perm = synth.perm_uniform(77, (C, S), 0.1, 0.3)
    boost = np.ones(C, np.float32) if boost is None else boost
    case = wl.Case("seq", W, H, C, S, idx, perm, boost, min_overlap=m, k=k, inhibition=inh, gw=gw,
                   gh=gh, radius=radius)
    fr = (np.random.default_rng(5).random((frames, W * H)) < density).astype(np.uint8)
    act, want_perm, ov = oracle_run(case, fr, True, want_ov=True)
    packed = wl.pack(fr)
    nw = packed.shape[1]
    buf = np.zeros(offset + frames * (nw + stride_pad), np.uint32)
    for t in range(frames):
        o = offset + t * (nw + stride_pad)
        buf[o:o + nw] = packed[t]
    d = torch.from_numpy(buf.view(np.int32)).cuda()
    h = spg.sp_create_from_state(case.config(), idx, perm, boost)
    masks = torch.zeros((frames, (C + 31) // 32), dtype=torch.int32, device="cuda")
    got_ov = torch.zeros((frames, C), dtype=torch.float32, device="cuda")
    # two calls, so that the second one starts from what the first wrote back
    n1 = frames - 9 if frames > 17 else frames
    st = torch.cuda.current_stream()
    spg.sp_compute_frames_overlaps_device(h, d[offset:], n1, nw + stride_pad, True, masks, got_ov, st)
    if n1 < frames:
        spg.sp_compute_frames_overlaps_device(h, d[offset + n1 * (nw + stride_pad):], frames - n1,
                                              nw + stride_pad, True, masks[n1:], got_ov[n1:], st)
    spg.sp_sync(h)
    np.testing.assert_array_equal(got_ov.cpu().numpy(), ov)
    np.testing.assert_array_equal(spg.masks_to_dense(masks.cpu().numpy().view(np.uint32), C), act)
    np.testing.assert_array_equal(spg.sp_get_permanences(h), want_perm)
    np.testing.assert_array_equal(spg.sp_active_columns(h), np.flatnonzero(act[-1]))
    spg.sp_destroy(h)


@pytest.mark.parametrize("W,H,C,S,box,k", [
    (64, 64, 1024, 100, 64, 20),     # every box is the frame
    (96, 70, 1000, 97, 64, 40),      # three words a row, columns not a multiple of 32
    (32, 300, 600, 130, 32, 9),      # one word a row, tall band
    (960, 80, 2047, 96, 64, 130),    # Table-like wide frame, odd column count
    (224, 64, 4096, 256, 64, 128),   # permanences do not fit: learnt from global memory
    (128, 64, 512, 96, 20, 3),       # small boxes inside the 64 x 64 ones
])
def test_window_forms(W, H, C, S, box, k):
    idx = _box_pools(np.random.default_rng(W + C), C, S, W, H, box)
    _check(W, H, C, idx, k, 4, frames=20)


@pytest.mark.parametrize("pad,offset", [(0, 1), (3, 0), (5, 3)])
def test_window_form_unaligned_frames(pad, offset):
    idx = _box_pools(np.random.default_rng(3), 512, 128, 160, 90, 64)
    _check(160, 90, 512, idx, 25, 4, stride_pad=pad, offset=offset)


@pytest.mark.parametrize("order", ["descending", "repeated", "wide", "tall"])
def test_pools_that_no_bitmap_can_hold(order):
    """Orders, repeats (a synapse listed twice counts twice) and extents that
    the bitmap form must leave to the pools form."""
    rng = np.random.default_rng(9)
    idx = _box_pools(rng, 300, 120, 128, 100, 64)
    if order == "descending":
        idx = np.ascontiguousarray(idx[:, ::-1])
    elif order == "repeated":
        idx[7, 5] = idx[7, 4]
        idx[::3, 60] = idx[::3, 59]
    elif order == "wide":
        idx[11, 0] = idx[11, 1] // 128 * 128  # another pixel of the first row
        row = np.unique(np.concatenate([idx[11], [idx[11, 1] // 128 * 128 + 127]]))[:120]
        idx[11, :len(row)] = row
    else:
        idx[200, -1] = 128 * 100 - 1
        idx[200, 0] = 0
    _check(128, 100, 300, idx.astype(np.uint32), 12, 3)


@pytest.mark.parametrize("C,S,n_in", [(1, 1, 33), (64, 4, 40), (256, 16, 1024), (500, 7, 900),
                                      (512, 32, 2000), (33, 33, 512), (129, 128, 4096)])
def test_small_poolers_in_one_cta(C, S, n_in):
    rng = np.random.default_rng(C)
    idx = np.sort(np.stack([rng.choice(n_in, S, replace=False) for _ in range(C)]), axis=1)
    _check(n_in, 1, C, idx.astype(np.uint32), max(1, C // 20), 1, frames=19)


@pytest.mark.parametrize("gw,gh,r,k", [(33, 31, 4, 5), (64, 16, 0, 1), (16, 64, 7, 20),
                                       (7, 200, 3, 2), (40, 30, 40, 3)])
@pytest.mark.parametrize("S", [24, 112])
def test_local_inhibition_rows(gw, gh, r, k, S):
    """Odd and even grid widths (a row's first column at either half of a
    word), radii from 0 to past the grid, both forms."""
    C = gw * gh
    idx = _box_pools(np.random.default_rng(gw), C, S, 192, 96, 64)
    _check(192, 96, C, idx, k, 2, inh=1, gw=gw, gh=gh, radius=r)


@pytest.mark.parametrize("inh", [0, 1])
def test_boosts_on_the_window_form(inh):
    C = 32 * 20
    boost = (0.5 + np.random.default_rng(2).integers(0, 4, C) / 4).astype(np.float32)
    idx = _box_pools(np.random.default_rng(4), C, 100, 160, 80, 64)
    _check(160, 80, C, idx, 17, 4, boost=boost, inh=inh, gw=32, gh=20, radius=3)


def test_all_columns_tie():
    """Every column sees the same pool: all counts tie in every frame."""
    one = _box_pools(np.random.default_rng(8), 1, 128, 96, 64, 64)
    idx = np.repeat(one, 777, axis=0)
    perm = np.full((777, 128), 0.25, np.float32)
    case = wl.Case("ties", 96, 64, 777, 128, idx, perm, np.ones(777, np.float32), min_overlap=1,
                   k=333, dec=0.0, inc=0.0)
    fr = (np.random.default_rng(1).random((9, 96 * 64)) < 0.4).astype(np.uint8)
    act, _, _ = oracle_run(case, fr, True, want_ov=True)
    h = spg.sp_create_from_state(case.config(), idx, perm, case.boost)
    masks = torch.zeros((9, 25), dtype=torch.int32, device="cuda")
    d = torch.from_numpy(wl.pack(fr).view(np.int32)).cuda()
    spg.sp_compute_frames_device(h, d, 9, d.shape[1], True, masks, torch.cuda.current_stream())
    spg.sp_sync(h)
    np.testing.assert_array_equal(spg.masks_to_dense(masks.cpu().numpy().view(np.uint32), 777), act)
    assert (act.sum(axis=1) == 333).all()
    spg.sp_destroy(h)


@pytest.mark.parametrize("n", [1, 2, 3, 5, 7])
@pytest.mark.parametrize("inh", [0, 1])
def test_short_sequences_and_single_frames(n, inh):
    """Runs of every short length from the two frame APIs in turn, learning on
    and off, so that each launch form takes over pending learning from the
    others."""
    C, W, H, S = 32 * 17, 96, 80, 100
    idx = _box_pools(np.random.default_rng(12), C, S, W, H, 64)
    perm = synth.perm_uniform(78, (C, S), 0.1, 0.3)
    case = wl.Case("short", W, H, C, S, idx, perm, np.ones(C, np.float32), min_overlap=3, k=9,
                   inhibition=inh, gw=32, gh=17, radius=3)
    fr = (np.random.default_rng(6).random((4 * (n + 2), W * H)) < 0.3).astype(np.uint8)
    packed = wl.pack(fr)
    d = torch.from_numpy(packed.view(np.int32)).cuda()
    h = spg.sp_create_from_state(case.config(), idx, perm, case.boost)
    p, t, st = perm, 0, torch.cuda.current_stream()
    for turn in range(4):
        learn = turn != 2
        spg.sp_compute_frames_device(h, d[t], n, packed.shape[1], learn, None, st)
        spg.sp_compute_device(h, d[t + n], learn, st)
        spg.sp_compute(h, packed[t + n + 1], learn)
        act, p, _ = oracle_run(case, fr[t:t + n + 2], learn, perm=p)
        np.testing.assert_array_equal(spg.sp_active_columns(h), np.flatnonzero(act[-1]))
        t += n + 2
    np.testing.assert_array_equal(spg.sp_get_permanences(h), p)
    spg.sp_destroy(h)
