"""The default schedule of a batch's persistent pass: 8 x 4 (CTAs per SM x
columns in flight) up to 18 CTAs of a frame per SM, 10 x 4 above."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1608_01966_gb300 as spg  # noqa: E402
from paper_1608_01966_gb300 import workloads as wl  # noqa: E402
from helpers import dense, oracle_run  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extra,schedule", [(0, (8, 4)), (1, (10, 4))])
def test_default_schedule_by_ctas_per_sm(extra, schedule):
    """One-CTA members, exactly 18 per SM and one more: the schedule reported,
    and every member's winners on learning frames against the oracle."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 18 * sms + extra
    c = wl.uneven_cases(1, c_range=(8, 8), n_in_range=(256, 256))[0][0]
    frames = wl.bernoulli_frames(3, c.n_in, 0.3, 4)
    hs = [spg.sp_create_from_state(c.config(), c.idx, c.perm, c.boost) for _ in range(n)]
    b = spg.sp_batch_create(hs)
    assert spg.sp_batch_schedule(b, n) == (*schedule, [0] * n)
    info = spg.sp_batch_get_info(b)
    fo, mo = spg.sp_batch_offsets(b)
    fw, mw = info["frame_words"], info["mask_words"]
    words = wl.pack(frames)
    d = torch.from_numpy(wl.batch_frames([words] * n, fo, fw).view(np.int32)).cuda()
    dm = torch.zeros((4, mw), dtype=torch.int32, device="cuda")
    spg.sp_batch_compute_device(b, d, 4, fw, True, dm, mw, torch.cuda.current_stream())
    spg.sp_batch_sync(b)
    masks = dm.cpu().numpy().view(np.uint32)
    spg.sp_batch_destroy(b)
    for h in hs:
        spg.sp_destroy(h)
    want = oracle_run(c, frames, True)[0]
    for i in range(n):
        got = dense(masks[:, int(mo[i]):int(mo[i]) + 1], c.C)
        np.testing.assert_array_equal(got, want, err_msg=f"member {i}")
