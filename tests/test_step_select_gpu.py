"""Alg. 2 in the last CTA of the per-frame kernels: column counts around its
16-byte copies, mask words and warps, winner sets from none to all, ties, and
overlaps that are counts, whole numbers, or neither.  Every entry point that
runs a frame by itself, against the oracle, exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1608_01966_gb300 as spg  # noqa: E402
from paper_1608_01966_gb300 import synth, workloads as wl  # noqa: E402
from helpers import dense, oracle_run  # noqa: E402

pytestmark = pytest.mark.gpu


def _case(C, S, k, boost=None, n_in=700, seed=5):
    idx = synth.pool_uniform(seed, C, S, n_in)
    perm = synth.perm_uniform(seed + 1, (C, S), 0.1, 0.3)
    boost = np.ones(C, np.float32) if boost is None else np.asarray(boost, np.float32)
    return wl.Case("select", n_in, 1, C, S, idx, perm, boost, min_overlap=1, k=k)


def _frames(c, n, seed=8):
    return (np.random.default_rng(seed).random((n, c.n_in)) < 0.3).astype(np.uint8)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def _single(c, fr):
    """sp_compute, sp_compute_device and sp_step_noalloc, a learning frame each."""
    act, perm, ov = oracle_run(c, fr, True, want_ov=True)
    x = wl.pack(fr)
    h = spg.sp_create_from_state(c.config(), c.idx, c.perm, c.boost)
    st = torch.cuda.current_stream()
    for t in range(len(fr)):
        if t % 2:
            spg.sp_compute_device(h, _dev(x[t]), True, st)
        else:
            spg.sp_compute(h, x[t], True)
        np.testing.assert_array_equal(spg.sp_active_columns(h), np.flatnonzero(act[t]))
        np.testing.assert_array_equal(spg.sp_get_overlaps(h), ov[t])
    np.testing.assert_array_equal(spg.sp_get_permanences(h), perm)
    spg.sp_destroy(h)
    idx, p, b = _dev(c.idx), torch.from_numpy(c.perm.copy()).cuda(), torch.from_numpy(c.boost).cuda()
    mask = torch.zeros((c.C + 31) // 32, dtype=torch.int32, device="cuda")
    lst = torch.full((1 + c.C,), -1, dtype=torch.int32, device="cuda")
    for t in range(len(fr)):
        spg.sp_step_noalloc(c.config(), idx, p, b, _dev(x[t]), True, mask, lst, st)
        got = lst.cpu().numpy()
        np.testing.assert_array_equal(got[1:1 + got[0]], np.flatnonzero(act[t]))
        np.testing.assert_array_equal(dense(mask.cpu().numpy().view(np.uint32), c.C), act[t])
    np.testing.assert_array_equal(p.cpu().numpy(), perm)


def _batch(cases, frames, calls):
    """One batch of the cases, its frames in calls of the given lengths."""
    hs = [spg.sp_create_from_state(c.config(), c.idx, c.perm, c.boost) for c in cases]
    b = spg.sp_batch_create(hs)
    fo, mo = spg.sp_batch_offsets(b)
    fw, mw = spg.sp_batch_get_info(b)["frame_words"], spg.sp_batch_get_info(b)["mask_words"]
    d = _dev(wl.batch_frames([wl.pack(f) for f in frames], fo, fw))
    masks = torch.zeros((sum(calls), mw), dtype=torch.int32, device="cuda")
    t = 0
    for n in calls:
        spg.sp_batch_compute_device(b, d[t], n, fw, True, masks[t], mw, torch.cuda.current_stream())
        t += n
    spg.sp_batch_sync(b)
    m = masks.cpu().numpy().view(np.uint32)
    spg.sp_batch_destroy(b)
    for i, c in enumerate(cases):
        act, perm, _ = oracle_run(c, frames[i], True)
        at = int(mo[i])
        np.testing.assert_array_equal(dense(m[:, at:at + (c.C + 31) // 32], c.C), act,
                                      err_msg=f"member {i}")
        np.testing.assert_array_equal(spg.sp_active_columns(hs[i]), np.flatnonzero(act[-1]))
        np.testing.assert_array_equal(spg.sp_get_permanences(hs[i]), perm, err_msg=f"member {i}")
        spg.sp_destroy(hs[i])


@pytest.mark.parametrize("C", [1, 2, 3, 4, 5, 29, 31, 32, 33, 127, 128, 129, 509, 512, 513, 1025,
                               2047, 2116, 16383, 16384])
def test_column_counts(C):
    for k in sorted({0, 1, max(1, C // 10), C, C + 3}):
        c = _case(C, 9, k)
        _single(c, _frames(c, 2))


def test_column_counts_in_one_batch():
    """Members of every size in one launch, whose shared memory is the largest's."""
    cases = [_case(C, S, max(1, C // 7), seed=20 + i)
             for i, (C, S) in enumerate([(1, 16), (5, 40), (31, 16), (33, 256), (127, 9), (513, 100),
                                         (2116, 20), (1030, 64)])]
    frames = [_frames(c, 6, 30 + i) for i, c in enumerate(cases)]
    _batch(cases, frames, [1, 1, 2, 1, 1])


def test_counts_on_both_sides_of_the_bins():
    """1022 synapses are counted in shared memory, 1023 in global memory, in
    one batch and alone."""
    cases = [_case(70, S, 9, n_in=4000, seed=S) for S in (1022, 1023, 1021)]
    frames = [_frames(c, 5, 40 + i) for i, c in enumerate(cases)]
    _batch(cases, frames, [1, 4])
    for c, f in zip(cases, frames):
        _single(c, f[:2])


@pytest.mark.parametrize("boosts", ["twos", "halves", "whole_mix", "zeros", "thirds"])
@pytest.mark.parametrize("S", [8, 64])
def test_boosted_overlaps(boosts, S):
    """Whole overlaps up to S go through the bins, larger ones (a count above
    S / 2 doubled) or fractions through the radix select; boosts of 0 make
    overlaps of 0."""
    C = 700
    r = np.random.default_rng(S)
    b = {"twos": np.full(C, 2.0), "halves": np.full(C, 0.5),
         "whole_mix": r.integers(1, 4, C).astype(float), "zeros": r.integers(0, 2, C).astype(float),
         "thirds": r.integers(1, 7, C) / 3.0}[boosts]
    for k in (1, 60, C):
        c = _case(C, S, k, boost=b)
        # a frame with every input set makes counts of up to S: doubled, they leave the bins
        fr = _frames(c, 4)
        fr[2] = 1
        _single(c, fr)
    _batch([c, _case(C, S, 60, boost=b[::-1].copy())], [fr, fr], [1, 3])


def test_every_column_ties():
    C = 300
    idx = np.repeat(synth.pool_uniform(3, 1, 32, 700), C, axis=0)
    perm = np.full((C, 32), 0.25, np.float32)
    for k in (0, 1, 31, 33, 299, 300):
        c = wl.Case("ties", 700, 1, C, 32, idx, perm, np.ones(C, np.float32), min_overlap=1, k=k,
                    inc=0.0, dec=0.0)
        _single(c, _frames(c, 2))
