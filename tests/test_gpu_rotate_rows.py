"""The rotation sum with rows that are shorter and longer than a CTA, and just at
its sizes: the exact sums of the definition."""
import numpy as np
import pytest

import paper_2509_05047_gb300 as psc
import workloads as W
from oracle import sinogram as S

from test_gpu_postproc import _acc, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rad,n_tof", [(1, 1), (3, 10), (31, 1), (33, 1), (9, 7), (51, 5), (51, 7)])   # rows of 1, 30, 31, 33, 63, 255, 357
@pytest.mark.parametrize("step", [1, 4, 13, 26])      # 52, 13 (odd), 4 and 2 members an orbit
def test_rotation_sum_of_row_sizes(env, n_rad, n_tof, step):  # noqa: F811
    ctx, torch = env
    sc = W.scanner_small(n_crystals=52, n_rings=3, n_tof=n_tof, n_rad=n_rad)
    x = np.random.default_rng(step).integers(0, 1 << 40, size=sc.shape, dtype=np.int64)
    s_id, a_id = _acc(ctx, torch, sc, x)
    o_id, stream = psc.psc_acc_create(ctx, s_id), torch.cuda.current_stream().cuda_stream
    psc.psc_acc_rotate_sum(ctx, a_id, step, o_id, stream)
    out = torch.empty(sc.shape, dtype=torch.int64, device="cuda")
    psc.psc_acc_read(ctx, o_id, out, stream)
    np.testing.assert_array_equal(out.cpu().numpy(), S.rotational_average(x, 52, sc.n_rings, step, average=False))
    for i in (a_id, o_id, s_id):
        psc.psc_unload(ctx, i)
