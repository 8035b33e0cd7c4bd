"""The axial tiles in every form of the epilogue (sensitivity, a normalisation per
LOR or per bin, the normalisation sinogram's division), on planes of odd and even
size and in the radius-32 window: the same bits as the pass that loads its rows
directly, and each of the two passes is the one that ran."""
import numpy as np
import pytest

import paper_2509_05047_gb300 as psc
import workloads as W

from gpu_kernels import kernels_of
from test_gpu_finalize import Fin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_crystals,n_rad,n_tof,n_rings", [(38, 33, 27, 37),   # 16929 bins: an odd plane, columns across LORs, half-width tiles
                                                             (40, 33, 25, 20),   # 16500 bins: whole quads
                                                             (76, 65, 25, 9)])   # 61750 bins: even, no whole quads
@pytest.mark.parametrize("radius", [9, 16, 31, 32])
@pytest.mark.parametrize("form", ["sens", "norm_lor", "norm_bin", "sens_bin_norm", "divide"])
def test_tiles_equal_direct_pass(n_crystals, n_rad, n_tof, n_rings, radius, form, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc = W.scanner_small(n_crystals=n_crystals, n_rings=n_rings, n_tof=n_tof, n_rad=n_rad)
    f = Fin(sc)
    try:
        rng = np.random.default_rng(radius)
        acc = rng.integers(0, 1 << 40, size=sc.shape, dtype=np.int64)
        acc[rng.random(size=sc.shape, dtype=np.float32) < 0.5] = 0
        f.write_acc(acc)
        sigma = (0.25, 0.25, radius / 4.0)
        kw = dict(sigma=sigma, scale=0.37)
        if form in ("sens", "norm_lor"):
            kw["sens"] = f.sino(rng.uniform(0.5, 1.5, size=sc.lor_shape), True)
        if form == "norm_lor":
            norm = rng.uniform(0.2, 2.0, size=sc.lor_shape)
            norm[:, 0, :3] = 0.0
            kw["norm"] = f.sino(norm, True)
        if form in ("norm_bin", "sens_bin_norm"):
            kw["norm"] = f.sino(rng.uniform(0.2, 2.0, size=sc.shape), False)
        if form == "sens_bin_norm":
            kw["sens"] = f.sino(rng.uniform(0.5, 1.5, size=sc.shape), False)
        got = []
        for tma, kernel in (("1", "smooth_axial_tma_kernel"), ("0", "smooth_axial_kernel")):
            monkeypatch.setenv("PSC_AXIAL_TMA", tma)
            out = torch.full(sc.shape, np.nan, dtype=torch.float64, device="cuda")

            def call(stream):
                if form == "divide":
                    psc.psc_norm_sinogram(f.ctx, f.a_id, sigma, out, stream)
                else:
                    psc.psc_finalize(f.ctx, psc.finalize_args(f.a_id, **kw), out, stream)
            assert kernel in kernels_of(call)
            torch.cuda.synchronize()
            got.append(out.view(torch.int64))
        assert torch.equal(got[0], got[1])
    finally:
        f.close()


def test_planes_that_cannot_be_described_take_the_direct_pass(monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for n_rad in (33, 32 + 5):    # odd planes that would be padded; the radius-31 window has no other instantiation
        sc = W.scanner_small(n_crystals=38, n_rings=12, n_tof=5, n_rad=n_rad)
        f = Fin(sc)
        try:
            acc = np.random.default_rng(n_rad).integers(0, 1 << 40, size=sc.shape, dtype=np.int64)
            f.write_acc(acc)
            got = []
            for refused, kernel in (("0", "smooth_axial_tma_kernel"), ("1", "smooth_axial_kernel")):
                monkeypatch.setenv("PSC_FAULT_TMA_MAP", refused)
                out = torch.full(sc.shape, np.nan, dtype=torch.float64, device="cuda")
                args = psc.finalize_args(f.a_id, sigma=(0.25, 0.25, 31 / 4.0), scale=0.37)
                assert kernel in kernels_of(lambda stream: psc.psc_finalize(f.ctx, args, out, stream))
                torch.cuda.synchronize()
                got.append(out.view(torch.int64))
            assert torch.equal(got[0], got[1])
        finally:
            f.close()
