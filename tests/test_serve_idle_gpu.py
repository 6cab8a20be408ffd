"""What an idle server costs its host, and frames whose words the gather cannot
read 16 bytes at a time."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1608_01966_gb300 as spg  # noqa: E402
from paper_1608_01966_gb300 import synth, workloads as wl  # noqa: E402
from helpers import oracle_run  # noqa: E402

pytestmark = pytest.mark.gpu


def _case(n_in, i):
    C, S = 200 + 31 * i, 20
    return wl.Case("serve", n_in, 1, C, S, synth.pool_uniform(80 + i, C, S, n_in),
                   synth.perm_uniform(81 + i, (C, S), 0.1, 0.3), np.ones(C, np.float32),
                   min_overlap=1, k=12)


def test_idle_server_takes_no_processor_time():
    """With nothing outstanding a poll goes to sleep at once (it used to yield
    for 100 us first), and so does the worker (which did so every 5 ms)."""
    c = _case(640, 0)
    s = spg.sp_server_create(2, 4, 64, 1 << 28, 16)
    sid = spg.sp_server_open_stream(s, c.config(duty_period=0.0), (c.idx, c.perm, c.boost))
    spg.sp_server_submit(s, sid, np.zeros(20, np.uint32), False)
    assert spg.sp_server_drain(s, wait_ms=1000)[0] == 1
    time.sleep(0.05)
    polls = []
    for _ in range(20):
        t = time.thread_time()
        assert not list(spg.sp_server_poll(s, wait_ms=3))
        polls.append(time.thread_time() - t)
    assert min(polls) < 60e-6
    t, w = time.process_time(), time.perf_counter()
    time.sleep(1.0)
    assert (time.process_time() - t) / (time.perf_counter() - w) < 0.01
    spg.sp_server_destroy(s)


@pytest.mark.parametrize("words", [1, 2, 3, 5, 31, 257, 2049])
def test_frames_of_any_number_of_words(words):
    """Ring slots of odd sizes: every second or fourth frame of a stream lies on
    a 16-byte boundary, the others do not."""
    cases = [_case(32 * words - 5 * i, i) for i in range(3)]
    s = spg.sp_server_create(3, 5, words, 1 << 28, 16)
    ids = [spg.sp_server_open_stream(s, c.config(), (c.idx, c.perm, c.boost)) for c in cases]
    frames = [(np.random.default_rng(i).random((7, c.n_in)) < 0.3).astype(np.uint8)
              for i, c in enumerate(cases)]
    want = [oracle_run(c, f, True) for c, f in zip(cases, frames)]
    packed = [wl.pack(f) for f in frames]
    for t in range(7):
        for i, sid in enumerate(ids):
            spg.sp_server_submit(s, sid, packed[i][t], True)
        got = {}
        while len(got) < 3:
            for r, active in spg.sp_server_poll(s, wait_ms=1000):
                got[r["stream_id"]] = np.array(active)
        for i, sid in enumerate(ids):
            np.testing.assert_array_equal(got[sid], np.flatnonzero(want[i][0][t]), err_msg=f"frame {t}")
    for i, (sid, c) in enumerate(zip(ids, cases)):
        np.testing.assert_array_equal(
            spg.sp_server_get_permanences(s, sid, (c.C, 20)), want[i][1])
    spg.sp_server_destroy(s)
