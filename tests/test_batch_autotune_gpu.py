"""The splits that the batch autotuner tries."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1608_01966_gb300 as spg  # noqa: E402
from paper_1608_01966_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


def test_every_split_is_tried():
    """Members of 8 columns are one CTA in every split, so a layout launches
    nothing, and a single frame is timed in three launches: the default and
    2, 4, 8, 16 and 32 columns per warp.  (32 used to be what members of 128 and
    more synapses got by default.)"""
    c = wl.uneven_cases(1, c_range=(8, 8), n_in_range=(256, 256))[0][0]
    hs = [spg.sp_create_from_state(c.config(), c.idx, c.perm, c.boost) for _ in range(3)]
    b = spg.sp_batch_create(hs)
    fw = spg.sp_batch_get_info(b)["frame_words"]
    x = torch.from_numpy(np.zeros((1, fw), np.int32)).cuda()
    spg.sp_batch_autotune(b, x, 1, fw)  # what forms allocate is there afterwards
    before = spg.sp_kernel_launch_count()
    spg.sp_batch_autotune(b, x, 1, fw)
    derived = sum(f == spg.SP_FORM_COMPACT for f in spg.sp_batch_forms(b))  # at the end, once each
    assert spg.sp_kernel_launch_count() - before - derived == 3 * 6
    spg.sp_batch_destroy(b)
    for h in hs:
        spg.sp_destroy(h)
