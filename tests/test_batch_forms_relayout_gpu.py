"""Batch members whose frame bands fit the window form for fine splits only:
whatever splits were tried or set before, the form in use follows the
permanences.  Winners, overlaps and permanences against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1608_01966_gb300 as spg  # noqa: E402
from paper_1608_01966_gb300 import synth, workloads as wl  # noqa: E402
from helpers import dense, oracle_run  # noqa: E402

pytestmark = pytest.mark.gpu

W, C, S, DY = 960, 1024, 256, 6  # the columns' boxes, DY rows apart
H = C * DY + 64
N = 3  # members


def _case(i):
    """Ascending pools inside 64 x 64 boxes going down a tall frame: the 64
    columns of a CTA at 16 columns per warp need 448 rows of 120 bytes, more
    than the 48 KB a CTA may stage; at 8 they need 256."""
    rng = np.random.default_rng(40 + i)
    px = np.sort(rng.permuted(np.tile(np.arange(4096), (C, 1)), axis=1)[:, :S], axis=1)
    x0 = rng.integers(0, W - 64, C)
    idx = (np.arange(C)[:, None] * DY + px // 64) * W + x0[:, None] + px % 64
    perm = synth.perm_uniform(90 + i, (C, S), 0.1, 0.3)
    return wl.Case("tall", W, H, C, S, idx.astype(np.uint32), perm, np.ones(C, np.float32),
                   min_overlap=4, k=40)


@pytest.fixture(scope="module")
def work():
    cases = [_case(i) for i in range(N)]
    frames = [(np.random.default_rng(60 + i).random((6, W * H)) < 0.2).astype(np.uint8)
              for i in range(N)]
    return cases, frames, [oracle_run(c, f, True, want_ov=True) for c, f in zip(cases, frames)]


def _batch(cases, frames):
    hs = [spg.sp_create_from_state(c.config(), c.idx, c.perm, c.boost) for c in cases]
    b = spg.sp_batch_create(hs)
    fo, _ = spg.sp_batch_offsets(b)
    fw = spg.sp_batch_get_info(b)["frame_words"]
    d = torch.from_numpy(wl.batch_frames([wl.pack(f) for f in frames], fo, fw).view(np.int32)).cuda()
    return hs, b, d, fw


def _check(hs, b, d, fw, cases, want, t0=0):
    """Frames t0.. of the batch, learning, against the oracle's."""
    _, mo = spg.sp_batch_offsets(b)
    oo, ow = spg.sp_batch_overlap_offsets(b)
    n, mw = d.shape[0] - t0, spg.sp_batch_get_info(b)["mask_words"]
    masks = torch.zeros((n, mw), dtype=torch.int32, device="cuda")
    ov = torch.zeros((n, ow), dtype=torch.float32, device="cuda")
    spg.sp_batch_compute_overlaps_device(b, d[t0], n, fw, True, masks, mw, ov, ow,
                                         torch.cuda.current_stream())
    spg.sp_batch_sync(b)
    m, o = masks.cpu().numpy().view(np.uint32), ov.cpu().numpy()
    spg.sp_batch_destroy(b)
    for i, c in enumerate(cases):
        act, perm, wov = want[i]
        np.testing.assert_array_equal(o[:, int(oo[i]):int(oo[i]) + C], wov[t0:], err_msg=f"member {i}")
        np.testing.assert_array_equal(dense(m[:, int(mo[i]):int(mo[i]) + C // 32], C), act[t0:],
                                      err_msg=f"member {i}")
        np.testing.assert_array_equal(spg.sp_get_permanences(hs[i]), perm, err_msg=f"member {i}")
        spg.sp_destroy(hs[i])


def test_autotune_trials_leave_no_stale_form(work):
    """The tuner tries splits whose bands do not fit, on frames that learn,
    and puts the permanences back."""
    cases, frames, want = work
    hs, b, d, fw = _batch(cases, frames)
    assert (spg.sp_batch_forms(b) == spg.SP_FORM_WINDOW).all()
    spg.sp_batch_autotune(b, d, 4, fw)
    _check(hs, b, d, fw, cases, want)


def test_window_form_comes_back_with_a_finer_split(work):
    """Two frames on a split that fits, two on one that does not, the rest on
    the first again."""
    cases, frames, want = work
    hs, b, d, fw = _batch(cases, frames)
    st = torch.cuda.current_stream()
    for cpw, form, t in ((4, spg.SP_FORM_WINDOW, 0), (16, spg.SP_FORM_COMPACT, 2)):
        spg.sp_batch_set_schedule(b, 8, 4, [cpw] * N)
        assert (spg.sp_batch_forms(b) == form).all()
        spg.sp_batch_compute_device(b, d[t], 2, fw, True, None, 0, st)
        spg.sp_batch_sync(b)
        spg.sp_batch_destroy(b)  # applies what is pending; the split is the batch's
        b = spg.sp_batch_create(hs)
    spg.sp_batch_set_schedule(b, 8, 4, [16] * N)
    spg.sp_batch_set_schedule(b, 8, 4, [4] * N)
    assert (spg.sp_batch_forms(b) == spg.SP_FORM_WINDOW).all()
    _check(hs, b, d, fw, cases, want, t0=4)
