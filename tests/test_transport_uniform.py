"""The transport loop's control values are the same in all lanes of a warp.  The
counter of histories handed out is moved by the other warps of a CTA at any
time, so a lane may use it only through the value its own atomic returned, and
the end of a work item is a vote on those values: two lanes that read the
counter itself could choose different sections, or leave the loop apart.
The hazard needs an unlucky schedule, so the rule is checked on the source; the
accumulators at the ends of work items are compared on the GPU."""
import os
import re

import numpy as np
import pytest

import workloads as W

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_05047_gb300", "csrc", "transport.cu")


def test_history_counter_is_read_by_atomics_only():
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(SOURCE).read(), flags=re.S)
    rest = text.replace("atomicAdd(&s_next, 1u)", "").replace("s_next = 0;", "")
    rest = re.sub(r"__shared__ unsigned [^;]*;", "", rest)
    assert "atomicAdd(&s_next, 1u)" in text and "s_next" not in rest
    # what masks the section counts changes only by a vote of the whole warp
    writes = [w.strip() for w in re.findall(r"[^\n;{}]*\bwaiting\s*=[^;]*;", text)]
    assert [w for w in writes if not w.startswith("unsigned waiting")] and all(
        "__any_sync(0xffffffffu" in w for w in writes if not w.startswith("unsigned waiting")), writes


@pytest.mark.gpu
@pytest.mark.parametrize("block", [32, 64, 512])
@pytest.mark.parametrize("n", [1, 31, 95, 97, 129, 1535, 1537, 40_001])   # around a warp's, a CTA's slots and an item's histories
def test_ends_of_work_items(block, n):
    from gpu_helpers import Session, sinogram_from
    sc = W.scanner_tiny()
    s = Session(sc, W.standard_materials(), W.phantom_water_cylinder(), W.lut_tiny(sc))
    try:
        lm = s.run(7, 3, n, bin_mask=3)
        assert np.all(lm["cls"] >= 0)    # every history of every item was followed
        exp = sinogram_from(lm["key"], lm["q"], lm["cls"], sc.n_bins, (6, 7))
        for grid in (0, 1, 3):
            s.zero()
            s.run(7, 3, n, listmode=False, stats=False, bin_mask=3, block=block, grid=grid)
            np.testing.assert_array_equal(s.acc().cpu().numpy(), exp)
    finally:
        s.close()
