"""Dense members of very different shapes inferred in one call: one with the
most columns there are, one with a histogram that does not fit beside them.
Every overlap and winner against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1608_01966_gb300 as spg  # noqa: E402
from paper_1608_01966_gb300 import synth, workloads as wl  # noqa: E402
from helpers import dense, oracle_run  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in", [40447, 40448, 40700, 40959, 41000])
def test_many_columns_beside_many_inputs(n_in):
    cases, frames = [], []
    for i, (C, n, k) in enumerate([(16384, 64, 300), (32, n_in, 5), (200, 500, 9)]):
        cases.append(wl.Case("mixed", n, 1, C, n, synth.pool_dense(C, n),
                             synth.perm_uniform(70 + i, (C, n), 0.1, 0.3), np.ones(C, np.float32),
                             min_overlap=2, k=k))
        frames.append((np.random.default_rng(i).random((20, n)) < 0.2).astype(np.uint8))
    hs = [spg.sp_create_from_state(c.config(), c.idx, c.perm, c.boost) for c in cases]
    b = spg.sp_batch_create(hs)
    fo, mo = spg.sp_batch_offsets(b)
    oo, ow = spg.sp_batch_overlap_offsets(b)
    fw, mw = spg.sp_batch_get_info(b)["frame_words"], spg.sp_batch_get_info(b)["mask_words"]
    d = torch.from_numpy(wl.batch_frames([wl.pack(f) for f in frames], fo, fw).view(np.int32)).cuda()
    masks = torch.zeros((20, mw), dtype=torch.int32, device="cuda")
    ov = torch.zeros((20, ow), dtype=torch.float32, device="cuda")
    spg.sp_batch_infer_overlaps_device(b, d, 20, fw, masks, mw, ov, ow, torch.cuda.current_stream())
    spg.sp_batch_sync(b)
    m, o = masks.cpu().numpy().view(np.uint32), ov.cpu().numpy()
    spg.sp_batch_destroy(b)
    for i, c in enumerate(cases):
        act, _, want = oracle_run(c, frames[i], False, want_ov=True)
        np.testing.assert_array_equal(o[:, int(oo[i]):int(oo[i]) + c.C], want, err_msg=f"member {i}")
        at = int(mo[i])
        np.testing.assert_array_equal(dense(m[:, at:at + (c.C + 31) // 32], c.C), act,
                                      err_msg=f"member {i}")
        spg.sp_destroy(hs[i])
