"""The axial pass gives a thread two neighbouring columns of a shared-memory
tile, in blocks of 8 outputs: the same bits as the pass that loads its rows
directly (PSC_AXIAL_TMA=0), at the edges of blocks, tiles and windows."""
import numpy as np
import pytest

import paper_2509_05047_gb300 as psc
import workloads as W

from test_gpu_finalize import Fin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rings", [1, 8, 9, 17, 37])        # segments of 1 .. 37 planes: whole and partial blocks, both tile widths
@pytest.mark.parametrize("radius", [1, 7, 8, 10, 20, 24, 25, 31, 32])     # also windows longer than the segment
@pytest.mark.parametrize("offset", [0, 1])                    # an estimate on a 16-byte boundary, and 8 bytes past one
def test_pairs_equal_direct_pass(n_rings, radius, offset, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc = W.scanner_small(n_crystals=8, n_rings=n_rings, n_tof=9, n_rad=7)   # 252 bins a plane: a partial tile, LORs across pairs
    f = Fin(sc)
    try:
        rng = np.random.default_rng(radius)
        acc = rng.integers(0, 1 << 40, size=sc.shape, dtype=np.int64)
        acc[rng.uniform(size=sc.shape) < 0.5] = 0
        f.write_acc(acc)
        kw = dict(sens=f.sino(rng.uniform(0.5, 1.5, size=sc.lor_shape), True), sigma=(1.0, 1.0, radius / 4.0), scale=0.37)
        norm = f.sino(rng.uniform(0.2, 2.0, size=sc.shape), False)
        stream = torch.cuda.current_stream().cuda_stream
        for extra in ({}, {"norm": norm}, {"sens_first": True}):
            got = []
            for tma in ("1", "0"):
                monkeypatch.setenv("PSC_AXIAL_TMA", tma)
                out = torch.full((sc.n_bins + offset,), np.nan, dtype=torch.float64, device="cuda")[offset:].view(sc.shape)
                psc.psc_finalize(f.ctx, psc.finalize_args(f.a_id, **kw, **extra), out, stream)
                torch.cuda.synchronize()
                got.append(out.cpu().numpy().view(np.int64))
            np.testing.assert_array_equal(got[0], got[1])
    finally:
        f.close()


@pytest.mark.parametrize("n_crystals,n_rad,n_tof", [(10, 9, 5), (10, 9, 1), (12, 7, 3), (38, 33, 27)])  # planes of 225, 45, 126, 16929 bins
@pytest.mark.parametrize("radius", [3, 31])
@pytest.mark.parametrize("value", [1.0, np.inf])              # an infinite factor spreads over the window and no further
def test_padded_planes_equal_direct_pass(n_crystals, n_rad, n_tof, radius, value, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc = W.scanner_small(n_crystals=n_crystals, n_rings=37, n_tof=n_tof, n_rad=n_rad)
    f = Fin(sc)
    try:
        rng = np.random.default_rng(radius)
        acc = rng.integers(1, 1 << 40, size=sc.shape, dtype=np.int64)
        f.write_acc(acc)
        sens = rng.uniform(0.5, 1.5, size=sc.shape)
        sens[18 * 37 + 18, 1, 2, 0] = value
        sid = f.sino(sens, False)
        for first in (True, False):
            got = []
            for tma in ("1", "0"):
                monkeypatch.setenv("PSC_AXIAL_TMA", tma)
                got.append(f.run(sens=sid, sens_first=first, sigma=(0.5, 0.5, radius / 4.0), scale=0.37).cpu().numpy())
            np.testing.assert_array_equal(got[0], got[1])
    finally:
        f.close()
