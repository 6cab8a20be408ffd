"""The bounded waits inside a sequence launch, made to expire by a limit of
1 ns: the launch ends early and reports SP_ETIMEOUT, in every form of the
state; the handle works on, and a fresh one computes what the oracle does."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1608_01966_gb300 as spg  # noqa: E402
from paper_1608_01966_gb300 import synth, workloads as wl  # noqa: E402
from helpers import dense, oracle_run  # noqa: E402

pytestmark = pytest.mark.gpu


def _uniform(C, S, n, inh=0, gw=0, gh=0):
    return wl.Case("wait", n, 1, C, S, synth.pool_uniform(61, C, S, n),
                   synth.perm_uniform(62, (C, S), 0.1, 0.3), np.ones(C, np.float32), min_overlap=2,
                   k=12, inhibition=inh, gw=gw, gh=gh, radius=2)


def _case(form):
    if form == "pools":
        return _uniform(2000, 36, 5000)
    if form == "two_ctas":
        return _uniform(64, 150, 3000)
    if form == "local":
        return _uniform(960, 40, 4000, 1, 40, 24)
    return wl.grid_case("wait", 1024 if form == "window" else 4096, 256, 63, W=960, H=540,
                        min_overlap=4, k=40, inhibition=0, radius=4)


@pytest.mark.parametrize("form", ["pools", "two_ctas", "local", "window", "window_l2"])
def test_expired_wait_ends_the_launch(form):
    c = _case(form)
    fr = (np.random.default_rng(7).random((24, c.n_in)) < 0.15).astype(np.uint8)
    x = torch.from_numpy(wl.pack(fr).view(np.int32)).cuda()
    st = torch.cuda.current_stream()
    masks = torch.zeros((24, (c.C + 31) // 32), dtype=torch.int32, device="cuda")
    h = spg.sp_create_from_state(c.config(), c.idx, c.perm, c.boost)
    for n in (24, 8, 9):  # the wait that expires may be the last frame's
        spg.sp_set_device_wait_ns(h, 1)
        spg.sp_compute_frames_device(h, x, n, x.shape[1], True, masks, st)
        with pytest.raises(spg.SpError) as e:
            spg.sp_sync(h)
        assert e.value.status == 4  # SP_ETIMEOUT
        spg.sp_sync(h)  # reported once
        spg.sp_set_device_wait_ns(h, 0)
        spg.sp_compute_frames_device(h, x, n, x.shape[1], True, masks, st)
        spg.sp_sync(h)
    spg.sp_destroy(h)
    act, perm, _ = oracle_run(c, fr, True)
    h = spg.sp_create_from_state(c.config(), c.idx, c.perm, c.boost)
    spg.sp_compute_frames_device(h, x, 24, x.shape[1], True, masks, st)
    spg.sp_sync(h)
    np.testing.assert_array_equal(dense(masks.cpu().numpy().view(np.uint32), c.C), act)
    np.testing.assert_array_equal(spg.sp_get_permanences(h), perm)
    spg.sp_destroy(h)
