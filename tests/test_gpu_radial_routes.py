"""The radial pass at the wide radii, on whole lines and on columns: the lines
against the FP64 oracle, and the columns of a large sinogram against the lines
that a few of its segments take (the same bits), with the factors of the pass,
finite and not."""
import numpy as np
import pytest

import oracle
import paper_2509_05047_gb300 as psc
import workloads as W

from gpu_kernels import kernels_of
from test_gpu_finalize import Fin, SMOOTH_RTOL

pytestmark = pytest.mark.gpu

LINES, COLUMNS = "smooth_radial_lines_kernel", "smooth_radial_kernel"


def _factors(f, sc, rng, factors, special=False):
    sens, norm = rng.uniform(0.5, 1.5, size=sc.lor_shape), rng.uniform(0.2, 2.0, size=sc.shape)
    if special:
        sens[3, 1, 5], sens[7, 2, 0], norm[9, 0, 2, 1], norm[-1, -1, -1, -1] = np.inf, np.nan, np.inf, 0.0
    kw, host = {}, {}
    if "sens" in factors:
        kw.update(sens=f.sino(sens, True), sens_first=True)
        host.update(sens=sens, smooth_before_sensitivity=False)
    if "norm" in factors:
        kw["norm"], host["norm"] = f.sino(norm, False), norm
    return kw, host


@pytest.mark.parametrize("n_crystals,n_rad,n_tof", [(46, 45, 4), (60, 49, 1), (34, 33, 12)])
@pytest.mark.parametrize("radius", [9, 10, 12, 16, 17, 20, 24])
@pytest.mark.parametrize("factors", ["", "sens", "norm", "sens norm"])
def test_lines_match_oracle(n_crystals, n_rad, n_tof, radius, factors):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc = W.scanner_small(n_crystals=n_crystals, n_rings=4, n_tof=n_tof, n_rad=n_rad)
    f = Fin(sc)
    try:
        rng = np.random.default_rng(radius)
        acc = rng.integers(0, 1 << 62, size=sc.shape) >> rng.integers(0, 62, size=sc.shape)
        acc[rng.uniform(size=sc.shape) < 0.3] = 0
        f.write_acc(acc)
        kw, host = _factors(f, sc, rng, factors)
        sigma = (radius / 4.0, 0.0, 0.0)
        out = torch.empty(sc.shape, dtype=torch.float64, device="cuda")
        args = psc.finalize_args(f.a_id, sigma=sigma, scale=0.37, **kw)
        assert LINES in kernels_of(lambda stream: psc.psc_finalize(f.ctx, args, out, stream))
        got = f.run(sigma=sigma, scale=0.37, **kw).cpu().numpy()
        np.testing.assert_allclose(got, oracle.finalize(acc, sc.n_rings, sigma=sigma, scale=0.37, **host), rtol=SMOOTH_RTOL,
                                   atol=1e-300)
    finally:
        f.close()


@pytest.mark.parametrize("radius", [0, 3, 8, 9, 10, 12, 16, 17, 20, 24])
@pytest.mark.parametrize("factors", ["", "sens", "norm", "sens norm"])
def test_columns_equal_lines(radius, factors):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc = W.scanner_small(n_crystals=198, n_rings=24, n_tof=5, n_rad=49)   # 285,000 columns; 34,650 in three segments; 99 views
    f = Fin(sc)
    try:
        rng = np.random.default_rng(radius)
        acc = rng.integers(0, 1 << 45, size=sc.shape)
        acc[rng.random(size=sc.shape, dtype=np.float32) < 0.5] = 0
        f.write_acc(acc)
        kw, _ = _factors(f, sc, rng, factors, special=True)
        got = []
        for segments, kernel in ((None, COLUMNS), ((22, 25), LINES)):
            args = psc.finalize_args(f.a_id, sigma=(radius / 4.0, 0.0, 0.0), scale=0.37, segments=segments, **kw)
            out = torch.zeros(sc.shape, dtype=torch.float64, device="cuda")
            names = kernels_of(lambda stream: psc.psc_finalize(f.ctx, args, out, stream))
            assert kernel in names and (LINES in names) == (kernel == LINES)
            torch.cuda.synchronize()
            got.append(out.view(torch.int64))
        planes = [ra * 24 + ra + d for d in (-1, 0, 1) for ra in range(max(0, -d), min(24, 24 - d))]
        assert torch.equal(got[0][planes], got[1][planes]) and bool((got[1][planes] != 0).any())
    finally:
        f.close()
