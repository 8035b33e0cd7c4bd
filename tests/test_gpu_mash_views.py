"""View mashing at every factor with a kernel of its own and one beyond, view
counts that leave rows over, and rows that are not whole blocks."""
import numpy as np
import pytest

from oracle import sinogram as S
import paper_2509_05047_gb300 as psc
import workloads as W

from test_gpu_postproc import _acc, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vf", range(1, 10))
@pytest.mark.parametrize("groups,n_tof", [(1, 1), (5, 7), (9, 3)])
def test_view_mashing_matches_oracle(env, vf, groups, n_tof):  # noqa: F811
    ctx, torch = env
    n = 2 * vf * groups
    if n < 4:
        n = 4
    sc = W.scanner_small(n_crystals=n, n_rings=2, n_tof=n_tof, n_rad=n - 1)
    x = np.random.default_rng(vf).integers(0, 1 << 40, size=sc.shape, dtype=np.int64)
    s_id, a_id = _acc(ctx, torch, sc, x)
    out = torch.full((sc.n_planes, sc.n_views // vf, sc.n_rad, sc.n_tof), -1, dtype=torch.int64, device="cuda")
    psc.psc_acc_mash(ctx, a_id, vf, 1, out, torch.cuda.current_stream().cuda_stream)
    np.testing.assert_array_equal(out.cpu().numpy(), S.mash(x, vf, 1))
    psc.psc_unload(ctx, a_id)
    psc.psc_unload(ctx, s_id)
