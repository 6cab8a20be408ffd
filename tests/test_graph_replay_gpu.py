"""Calls recorded into the caller's CUDA graph and replayed between live ones."""
import ctypes as ct

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1608_01966_gb300 as spg  # noqa: E402
from paper_1608_01966_gb300 import synth, workloads as wl  # noqa: E402
from helpers import dense, oracle_run  # noqa: E402

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


def _node_types(graph):
    """CUgraphNodeType of every node (0 kernel, 2 memset)."""
    cu = ct.CDLL("libcuda.so.1")
    n = ct.c_size_t(0)
    assert cu.cuGraphGetNodes(ct.c_void_p(graph), None, ct.byref(n)) == 0
    nodes = (ct.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(ct.c_void_p(graph), nodes, ct.byref(n)) == 0
    kinds = []
    for x in nodes:
        k = ct.c_int(-1)
        assert cu.cuGraphNodeGetType(ct.c_void_p(x), ct.byref(k)) == 0
        kinds.append(k.value)
    return sorted(kinds)


@pytest.mark.parametrize("learn", [False, True])
def test_noalloc_replays_between_live_calls(learn):
    """Two recorded calls, replayed between live ones on permanences that all
    of them share.  A recorded call clears the shared counter itself: its
    replays cannot start above what an earlier call left there."""
    c = wl.frame_case(seed=wl.BASE_SEED + 52)
    n = 12
    fr = (np.random.default_rng(4).random((n, c.n_in)) < 0.2).astype(np.uint8)
    act, want, _ = oracle_run(c, fr, learn)
    d = _dev(wl.pack(fr))
    buf = torch.zeros_like(d[:2])
    idx, perm, boost = _dev(c.idx), torch.from_numpy(c.perm.copy()).cuda(), torch.from_numpy(c.boost).cuda()
    masks = torch.zeros((2, 32), dtype=torch.int32, device="cuda")
    lst = torch.zeros(1 + c.C, dtype=torch.int32, device="cuda")
    st = torch.cuda.Stream()

    def call(x, mask):
        spg.sp_step_noalloc(c.config(), idx, perm, boost, x, learn, mask, lst, st)

    g = torch.cuda.CUDAGraph(keep_graph=True)
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        spg.sp_step_noalloc(c.config(), idx, perm, boost, d[0], False, masks[0], lst, st)  # loads the code
        st.synchronize()
        g.capture_begin()
        call(buf[0], masks[0])
        call(buf[1], masks[1])
        g.capture_end()
        kinds = _node_types(g.raw_cuda_graph())
        assert kinds == sorted([0, 2] * 2 + [0] * (2 if learn else 0))
        g.instantiate()
        for t in range(0, n, 4):
            call(d[t], masks[0])
            np.testing.assert_array_equal(dense(masks.cpu().numpy().view(np.uint32)[:1], c.C)[0], act[t])
            for s in (t + 1, t + 3):
                k = 2 if s == t + 1 else 1
                if k == 2:
                    buf.copy_(d[s:s + 2])
                    g.replay()
                else:
                    call(d[s], masks[0])
                got = dense(masks.cpu().numpy().view(np.uint32), c.C)
                np.testing.assert_array_equal(got[:k], act[s:s + k], err_msg=f"frame {s}")
    torch.cuda.synchronize()
    np.testing.assert_array_equal(perm.cpu().numpy(), want)
