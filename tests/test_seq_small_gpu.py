"""Sequences of small poolers around the sizes where the launch changes: one
CTA or a cluster, 1 to 8 columns of a warp side by side, a last group of
columns that is not full, pools of whole 16-byte loads or not.  Masks, overlaps
and permanences against the oracle, exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1608_01966_gb300 as spg  # noqa: E402
from paper_1608_01966_gb300 import synth, workloads as wl  # noqa: E402
from helpers import dense, oracle_run  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [31, 32, 33, 64, 65, 96, 128, 129, 160, 161, 256, 257, 320, 512, 513,
                               1025])
@pytest.mark.parametrize("inh", [0, 1])
def test_small_sequences(C, inh):
    n = 611
    gw = next(w for w in (8, 5, 3, 1) if C % w == 0)
    for S in (1, 3, 4, 16, 18, 26, 32, 48, 90):
        idx = synth.pool_uniform(C + S, C, S, n)
        perm = synth.perm_uniform(C + S + 1, (C, S), 0.1, 0.3)
        c = wl.Case("small", n, 1, C, S, idx, perm, np.ones(C, np.float32), min_overlap=1,
                    k=max(1, C // 9) if not inh else 2, inhibition=inh, gw=gw if inh else 0,
                    gh=C // gw if inh else 0, radius=2 if inh else 0)
        fr = (np.random.default_rng(S).random((7, n)) < 0.3).astype(np.uint8)
        act, want, wov = oracle_run(c, fr, True, want_ov=True)
        h = spg.sp_create_from_state(c.config(), idx, perm, c.boost)
        x = torch.from_numpy(wl.pack(fr).view(np.int32)).cuda()
        masks = torch.zeros((7, (C + 31) // 32), dtype=torch.int32, device="cuda")
        ov = torch.zeros((7, C), dtype=torch.float32, device="cuda")
        spg.sp_compute_frames_overlaps_device(h, x, 7, x.shape[1], True, masks, ov,
                                              torch.cuda.current_stream())
        spg.sp_sync(h)
        np.testing.assert_array_equal(ov.cpu().numpy(), wov, err_msg=f"S {S}")
        np.testing.assert_array_equal(dense(masks.cpu().numpy().view(np.uint32), C), act)
        np.testing.assert_array_equal(spg.sp_get_permanences(h), want)
        spg.sp_destroy(h)
