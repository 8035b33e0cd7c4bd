"""Mashing by many views and by TOF bins: the exact int64 sums, at remainders of
the loads that go out together (8 views, 4 TOF bins)."""
import numpy as np
import pytest

import paper_2509_05047_gb300 as psc
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_crystals,n_rad,n_tof,views,bins", [
    (18, 17, 1, 9, 1), (20, 19, 5, 10, 1), (34, 33, 3, 17, 1), (48, 47, 2, 24, 1),          # 9, 10, 17, 24 views
    (20, 19, 3, 1, 3), (20, 19, 9, 2, 3), (24, 23, 10, 3, 5), (24, 9, 27, 12, 9), (12, 11, 8, 6, 4), (20, 19, 13, 10, 13), (10, 9, 27, 5, 27)])
def test_mash_sums(n_crystals, n_rad, n_tof, views, bins):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc = W.scanner_small(n_crystals=n_crystals, n_rings=3, n_tof=n_tof, n_rad=n_rad)
    ctx = psc.psc_create(0)
    try:
        acc = np.random.default_rng(views).integers(0, 1 << 55, size=sc.shape)
        sums = torch.from_numpy(acc).cuda().flatten()
        a = psc.psc_acc_wrap(ctx, psc.psc_load_scanner(ctx, psc.scanner_desc(sc)), sums)
        V = n_crystals // 2
        out = torch.full((9, V // views, n_rad, n_tof // bins), -1, dtype=torch.int64, device="cuda")
        psc.psc_acc_mash(ctx, a, views, bins, out, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        want = acc.reshape(9, V // views, views, n_rad, n_tof // bins, bins).sum(axis=(2, 5))
        np.testing.assert_array_equal(out.cpu().numpy(), want)
    finally:
        psc.psc_destroy(ctx)
