"""Calls recorded into the caller's CUDA graph and replayed between live ones."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1608_01966_gb300 as spg  # noqa: E402
from paper_1608_01966_gb300 import synth, workloads as wl  # noqa: E402
from helpers import oracle_run  # noqa: E402

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def _local_case():
    C, S, n = 640, 24, 3000
    idx = synth.pool_uniform(31, C, S, n)
    perm = synth.perm_uniform(32, (C, S), 0.1, 0.3)
    return wl.Case("local", n, 1, C, S, idx, perm, np.ones(C, np.float32), min_overlap=1, k=4,
                   inhibition=1, gw=32, gh=20, radius=3)


@pytest.mark.parametrize("which", ["global", "local"])
@pytest.mark.parametrize("frames", [1, 4])
def test_active_columns_after_a_replay(which, frames):
    """Inference recorded from device frames; live sp_compute calls, whose list
    the kernel writes to the host, come between the replays."""
    c = wl.frame_case(seed=wl.BASE_SEED + 51) if which == "global" else _local_case()
    fr = (np.random.default_rng(3).random((6 * frames, c.n_in)) < 0.2).astype(np.uint8)
    act = oracle_run(c, fr, False)[0]
    x, d = wl.pack(fr), _dev(wl.pack(fr))
    h = spg.sp_create_from_state(c.config(), c.idx, c.perm, c.boost)
    buf = torch.zeros_like(d[:frames])
    st = torch.cuda.Stream()

    def call():
        if frames == 1:
            spg.sp_compute_device(h, buf, False, st)
        else:
            spg.sp_compute_frames_device(h, buf, frames, buf.shape[1], False, None, st)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        call()  # the handle's stream is st from here on
        st.synchronize()
        g.capture_begin()
        call()
        g.capture_end()
    for t in range(6):
        live = (t * frames + 7) % len(x)
        spg.sp_compute(h, x[live], False)
        np.testing.assert_array_equal(spg.sp_active_columns(h), np.flatnonzero(act[live]))
        with torch.cuda.stream(st):
            buf.copy_(d[t * frames:(t + 1) * frames])
            g.replay()
        st.synchronize()
        np.testing.assert_array_equal(spg.sp_active_columns(h),
                                      np.flatnonzero(act[(t + 1) * frames - 1]), err_msg=f"replay {t}")
    torch.cuda.synchronize()
    spg.sp_destroy(h)
